"""Cut rows in the per-matrix launches: a CTA per row, its warps sharing the
pieces; y is the whole-batch launch's bit for bit, in every layout and with the
CSR copy released, for rows of one piece more than a warp round, of one round of
pieces and of many."""
import numpy as np
import pytest

from paper_2203_02530_gb300 import workloads as W
from tests.gpu_util import dev, reference, synced, torch_cuda

pytestmark = pytest.mark.gpu

LONG = [513, 1024, 32 * 512 - 1, 32 * 512, 32 * 512 + 1, 200_001]


def _matrix(n, seed):
    rng = np.random.default_rng(seed)
    lens = rng.integers(0, 6, size=n)
    lens[rng.choice(n, size=len(LONG), replace=False)] = LONG
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rp[1:])
    return n, rp, rng.integers(0, n, size=rp[-1]).astype(np.int32), rng.uniform(-1, 1, size=rp[-1])


@pytest.mark.parametrize("lanes", [0, 1, 32, 64])
def test_cut_rows_of_separate_launches(lanes):
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    mats = [W.stencil_7pt(5, seed=2), _matrix(3001, 1), W.stencil_7pt(6, seed=3), _matrix(700, 2)]
    with spmv.Batch(mats) as b:
        offs = b.offsets()
        x = W.uniform_x(offs[-1], seed=5)
        refs = [reference(*m, x[offs[i]:offs[i + 1]]) for i, m in enumerate(mats)]
        want, scale = (np.concatenate([r[k] for r in refs]) for k in range(2))
        spmv.spmv_batch_set_lanes(b.h, -1, lanes)
        if lanes == 64:
            spmv.spmv_batch_release_csr(b.h)
        x_d, s, s2 = dev(x), torch.cuda.Stream(), torch.cuda.Stream()
        y, y2 = (synced(torch.full((offs[-1],), float("nan"), dtype=torch.float64, device="cuda")) for _ in range(2))
        spmv.spmv_batch_run(b.h, x_d, y, s)
        for m in range(4):   # per-matrix launches keep no state: two streams at once
            spmv.spmv_batch_run_separate(b.h, m, x_d, y2, (s, s2)[m // 2])
        torch.cuda.synchronize()
        got = y.cpu().numpy()
        # two sums of the same k products differ by at most 2 k u sum |a x|
        k = max(LONG)
        assert (np.abs(got - want) <= 2 * k * 2.0**-53 * scale + 1e-300).all()
        assert np.array_equal(got.view(np.uint64), y2.cpu().numpy().view(np.uint64))
