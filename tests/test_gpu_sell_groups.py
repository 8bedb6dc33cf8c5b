"""Groups of short slices in the sorted sliced layout: every group kind (0 to 4
entries a row), left-over slices and rows cut by a rank's end, against the
launches that take slices (4 entries per lane and step) and the oracle."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import dev, synced, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,P", [(2000, 1), (40_000, 3), (400_003, 3)])
def test_groups_exact(n, P):
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    rng = np.random.default_rng(n)
    lens = rng.choice([0, 1, 2, 3, 4, 5, 6, 9, 40, 70], size=n, p=[.2, .2, .2, .1, .1, .05, .05, .05, .04, .01])
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rp[1:])
    ci = rng.integers(0, n, size=rp[-1]).astype(np.int32)
    va = rng.integers(-4, 5, size=rp[-1]).astype(np.float64)
    x = rng.integers(-4, 5, size=n).astype(np.float64)
    want = oracle.csr_spmv(n, rp, ci, va, x)
    s, x_d = torch.cuda.Stream(), dev(x)
    for gran in (spmv.COARSE, spmv.PER_PARTITION):
        ops = P if gran else 1
        order = [4 * p + k for k in range(4) for p in range(ops)]
        with spmv.Part(n, rp, ci, va, P, gran) as part:
            for param in (4, 8, 9, 105, 106, 107, 2008, 2105, 2107):
                part.set_variant(spmv.VARIANT_SELL, param)
                y = synced(torch.full((n,), float("nan"), dtype=torch.float64, device="cuda"))
                part.run(order, [0] * len(order), [s], x_d, y)
                s.synchronize()
                assert np.array_equal(y.cpu().numpy(), want), (gran, param)
            assert spmv.spmv_part_check(part.h) == 0
