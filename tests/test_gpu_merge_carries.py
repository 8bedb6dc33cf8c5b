"""Rows carried over many ranges of the merge path (248 items each here): runs of
carries on both sides of the 8 that a thread adds and of the 256 that a warp adds
per round, plan-free and in plans; integer data, so the result is exact."""
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


@pytest.mark.parametrize("ranges", [[7, 8, 9, 10, 11], [263, 264, 265, 266], [519, 520, 521, 522], [3, 1200, 2, 40]])
@pytest.mark.parametrize("extra", [-1, 0, 1])
def test_runs_of_carries_exact(ranges, extra):
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    n, rp, ci, va = _csr(sum([[3, 248 * r + extra, 0, 5] for r in ranges], []), 11)
    x = np.random.default_rng(12).integers(-4, 5, size=n).astype(np.float64)
    want = oracle.csr_spmv(n, rp, ci, va, x)
    s = torch.cuda.Stream()
    args = [dev(rp.astype(np.int32)), dev(ci), dev(va), dev(x)]
    for call in (spmv.spmv_csr_merge, spmv.spmv_csr_merge_noalloc):
        y = synced(torch.full((n + 64,), float("nan"), dtype=torch.float64, device="cuda"))
        call(n, int(rp[-1]), *args, y, s)
        s.synchronize()
        got = y.cpu().numpy()
        assert np.array_equal(got[:n], want) and np.isnan(got[n:]).all(), call.__name__
    for P in (1, 2):
        order = [4 * p + k for k in range(4) for p in range(P)]
        with spmv.Part(n, rp, ci, va, P, spmv.PER_PARTITION) as part:
            part.set_variant(spmv.VARIANT_MERGE, 0)
            y = synced(torch.full((n,), float("nan"), dtype=torch.float64, device="cuda"))
            part.run(order, [0] * len(order), [s], args[3], y)
            s.synchronize()
            assert np.array_equal(y.cpu().numpy(), want), P


def test_one_row_over_every_range_keeps_up():
    """Half the entries in one row take little more than the same entries in
    short rows (one thread adding the run of carries: 15 times as long)."""
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    s = torch.cuda.Stream()
    best = []
    for long_row in (5, 1_000_000):
        n = 100_000 if long_row > 5 else 300_000
        lens = np.full(n, 5)
        lens[n // 3] = long_row
        m = _csr(lens, 1)
        x_d, y = dev(np.ones(n)), synced(torch.zeros(n, dtype=torch.float64, device="cuda"))
        with spmv.Part(*m, 1, spmv.COARSE) as part:
            part.set_variant(spmv.VARIANT_MERGE, 0)
            times = []
            for _ in range(8):
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                a.record(s)
                spmv.spmv_local(part.h, -1, x_d, y, s)
                b.record(s)
                b.synchronize()
                times.append(a.elapsed_time(b))
            best.append(min(times))
    assert best[1] < 5 * best[0], best
