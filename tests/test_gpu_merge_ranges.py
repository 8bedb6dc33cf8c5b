"""Merge-path product at the edges of its lanes (8 entries), chunks (256
entries) and ranges: row lengths on both sides of them, runs of empty rows,
one row over every range; integer data, so the result is exact."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import dev, synced, torch_cuda

pytestmark = pytest.mark.gpu


def _csr(lens, seed):
    rng = np.random.default_rng(seed)
    n = len(lens)
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rp[1:])
    return (n, rp, rng.integers(0, n, size=rp[-1]).astype(np.int32),
            rng.integers(-4, 5, size=rp[-1]).astype(np.float64))


CASES = {
    "one_row": [5],
    "one_row_of_a_lane": [8],
    "only_empty_rows": [0] * 3000,
    "edges": [7, 8, 9, 0, 0, 255, 256, 257, 1, 0, 503, 504, 505, 247, 248, 249] * 9,
    "empty_runs": ([0] * 700 + [3, 1]) * 20,
    "ones": [1] * 5003,
    "eights": [8] * 4000,
    "row_over_every_range": [2] * 100 + [1_400_000] + [0, 3] * 100,
    "many_long": [2500] * 700,
    "mixed_large": list(np.random.default_rng(7).integers(0, 30, size=150_001)),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_merge_ranges_exact(name):
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    n, rp, ci, va = _csr(CASES[name], 11)
    x = np.random.default_rng(12).integers(-4, 5, size=n).astype(np.float64)
    want = oracle.csr_spmv(n, rp, ci, va, x)
    s = torch.cuda.Stream()
    args = [dev(rp.astype(np.int32)), dev(ci), dev(va), dev(x)]
    for call in (spmv.spmv_csr_merge, spmv.spmv_csr_merge_noalloc):
        y = synced(torch.full((n + 64,), float("nan"), dtype=torch.float64, device="cuda"))
        call(n, int(rp[-1]), *args, y, s)
        s.synchronize()
        got = y.cpu().numpy()
        assert np.array_equal(got[:n], want), call.__name__
        assert np.isnan(got[n:]).all()
    assert spmv.spmv_csr_error() == 0
    if rp[-1] < 1_000_000:   # the plan's ranges, whole and per rank, local and remote
        with spmv.Part(n, rp, ci, va, 3, spmv.PER_PARTITION) as part:
            part.set_variant(spmv.VARIANT_MERGE, 0)
            y = synced(torch.full((n,), float("nan"), dtype=torch.float64, device="cuda"))
            order = [4 * p + k for k in range(4) for p in range(3)]
            part.run(order, [0] * 12, [s], args[3], y)
            s.synchronize()
            assert np.array_equal(y.cpu().numpy(), want)


@pytest.mark.parametrize("n", [115_000, 135_000])
def test_plan_range_lengths(n):
    """A plan's ranges are one chunk up to 2 x 4864 x 256 items, else two: a
    local product on each side of the line, a small remote one."""
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    rng = np.random.default_rng(n)
    lens = rng.integers(0, 41, size=n)
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rp[1:])
    assert (n + rp[-1] > 2 * 4864 * 256) == (n == 135_000)
    rows = np.repeat(np.arange(n), lens)
    ci = np.clip(rows + rng.integers(-300, 301, size=rp[-1]), 0, n - 1).astype(np.int32)
    va = rng.integers(-4, 5, size=rp[-1]).astype(np.float64)
    x = rng.integers(-4, 5, size=n).astype(np.float64)
    want = oracle.csr_spmv(n, rp, ci, va, x)
    s, x_d = torch.cuda.Stream(), dev(x)
    for gran in (spmv.COARSE, spmv.PER_PARTITION):
        ops = 3 if gran else 1
        order = [4 * p + k for k in range(4) for p in range(ops)]
        with spmv.Part(n, rp, ci, va, 3, gran) as part:
            part.set_variant(spmv.VARIANT_MERGE, 0)
            y = synced(torch.full((n,), float("nan"), dtype=torch.float64, device="cuda"))
            part.run(order, [0] * len(order), [s], x_d, y)
            s.synchronize()
            assert np.array_equal(y.cpu().numpy(), want), gran
