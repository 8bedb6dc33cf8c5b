"""The binding refuses a schedule with a stream missing before it reaches the
library, in every run mode."""
import pytest

from paper_2203_02530_gb300 import build as B


@pytest.mark.parametrize("flags", [0, 1, 2])
@pytest.mark.parametrize("streams", [[None], [7, None]])
def test_missing_stream_is_refused(monkeypatch, streams, flags):
    B.build()
    from paper_2203_02530_gb300 import spmv

    class Lib:
        def spmv_schedule_run(self, *args):
            raise AssertionError("reached the library")

    monkeypatch.setattr(spmv, "lib", Lib())
    with pytest.raises((TypeError, AttributeError)):
        spmv.spmv_schedule_run(None, [0], [0], streams, 16, 32, flags)
