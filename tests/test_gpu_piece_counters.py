"""The counters of rows summed in pieces after launches that overlapped on two
streams (whose own results are not defined): the next product is right, for
batches with and without a ticket and for the sliced products of a plan."""
import numpy as np
import pytest

from paper_2203_02530_gb300 import workloads as W
from tests.gpu_util import assert_fp64_close, dev, reference, synced, torch_cuda

pytestmark = pytest.mark.gpu


def _long_rows(n, rows, seed):
    rng = np.random.default_rng(seed)
    lens = rng.integers(0, 6, size=n)
    lens[rng.choice(n, size=rows, replace=False)] = 4096
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rp[1:])
    return n, rp, rng.integers(0, n, size=rp[-1]).astype(np.int32), rng.uniform(-1, 1, size=rp[-1])


@pytest.mark.parametrize("rows,lanes", [(3000, 2), (3000, 64), (300_000, 2), (300_000, 64)])
def test_batch_after_overlapped_launches(rows, lanes):
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    mats = [_long_rows(rows, 40, 1), W.stencil_7pt(9, seed=2), _long_rows(700, 9, 3)]
    with spmv.Batch(mats) as b:
        offs = b.offsets()
        x = W.uniform_x(offs[-1], seed=5)
        refs = [reference(*m, x[offs[i]:offs[i + 1]]) for i, m in enumerate(mats)]
        want, scale = (np.concatenate([r[k] for r in refs]) for k in range(2))
        spmv.spmv_batch_set_lanes(b.h, -1, lanes)
        x_d, s, s2 = dev(x), torch.cuda.Stream(), torch.cuda.Stream()
        y, y2 = (synced(torch.full((offs[-1],), float("nan"), dtype=torch.float64, device="cuda")) for _ in range(2))
        for _ in range(50):
            spmv.spmv_batch_run(b.h, x_d, y, s)
            spmv.spmv_batch_run(b.h, x_d, y2, s2)
        torch.cuda.synchronize()
        for _ in range(2):
            synced(y.fill_(float("nan")))
            spmv.spmv_batch_run(b.h, x_d, y, s)
            s.synchronize()
            assert_fp64_close(y.cpu().numpy(), want, scale)


def test_plan_after_overlapped_launches():
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    n, rp, ci, va = _long_rows(20_000, 60, 4)
    x = W.uniform_x(n, seed=6)
    want, scale = reference(n, rp, ci, va, x)
    x_d, s, s2 = dev(x), torch.cuda.Stream(), torch.cuda.Stream()
    y, y2 = (synced(torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")) for _ in range(2))
    with spmv.Part(n, rp, ci, va, 1, spmv.COARSE) as part:
        part.set_variant(spmv.VARIANT_SELL, 8)
        for _ in range(50):
            spmv.spmv_local(part.h, -1, x_d, y, s)
            spmv.spmv_local(part.h, -1, x_d, y2, s2)
        torch.cuda.synchronize()
        for _ in range(2):
            synced(y.fill_(float("nan")))
            spmv.spmv_local(part.h, -1, x_d, y, s)
            s.synchronize()
            assert_fp64_close(y.cpu().numpy(), want, scale)
