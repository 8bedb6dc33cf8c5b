"""The hashes of served requests start at zero whatever the caller has queued on
the default stream, which the serving streams do not wait for."""
import numpy as np
import pytest

from paper_2203_02530_gb300 import workloads as W
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layout", ["buckets", "sliced"])
def test_hashes_beside_work_on_the_default_stream(layout):
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    mats = [W.stencil_7pt(11, seed=1), W.zipf_random(5000, seed=2)]
    rng = np.random.default_rng(3)
    args = (rng.integers(0, 2, size=40).astype(np.int32), rng.integers(1, 9, size=40).astype(np.int32),
            rng.integers(0, 2**63, size=40, dtype=np.uint64), np.zeros(40))
    a = torch.rand((4096, 4096), device="cuda") / 2048
    with spmv.Batch(mats) as b:
        if layout == "sliced":
            spmv.spmv_batch_set_lanes(b.h, -1, spmv.BATCH_SLICED)
        with spmv.Server(b, n_streams=4, budget_bytes=1 << 30) as sv:
            want = sv.run(*args)[1]
            assert np.count_nonzero(want) == 40
            for _ in range(3):
                for _ in range(40):   # tens of milliseconds
                    a = a @ a
                got = sv.run(*args)[1]
                torch.cuda.synchronize()
                assert np.array_equal(got, want)
