"""Work units of the batched products: rows at the piece lengths' edges, and
batches on both sides of the line between the small and the persistent
launches, in every layout."""
import numpy as np
import pytest

from paper_2203_02530_gb300 import workloads as W
from tests.gpu_util import assert_fp64_close, dev, reference, torch_cuda

pytestmark = pytest.mark.gpu


def _edge_rows(n, seed, filler):
    """Row lengths around 64, 512, 1024 and 2048 entries among rows of up to
    `filler` entries; columns repeat and are in no order."""
    rng = np.random.default_rng(seed)
    lens = rng.integers(0, filler + 1, size=n)
    edges = [63, 64, 65, 511, 512, 513, 1023, 1024, 1025, 2047, 2048, 2049, 4096]
    lens[rng.choice(n, size=len(edges), replace=False)] = edges
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rp[1:])
    return n, rp, rng.integers(0, n, size=rp[-1]).astype(np.int32), rng.uniform(-1, 1, size=rp[-1])


# rows of the large matrix: the batch takes the small launches (1000), the
# persistent ones with parts of items (200 000), longer pieces (2 000 000)
@pytest.mark.parametrize("rows", [1000, 200_000, 2_000_000])
@pytest.mark.parametrize("lanes", [0, 2, 32, 64])
def test_pieces_and_parts_match_oracle_and_separate_launches(rows, lanes):
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    mats = [_edge_rows(777, 1, 5), W.stencil_7pt(9, seed=2), _edge_rows(rows, 3, 3),
            (0, np.zeros(1, np.int64), np.zeros(0, np.int32), np.zeros(0)), W.random_csr(33, density=0.3, seed=4)]
    with spmv.Batch(mats) as b:
        offs = b.offsets()
        x = W.uniform_x(offs[-1], seed=5)
        refs = [reference(*m, x[offs[i]:offs[i + 1]]) for i, m in enumerate(mats)]
        want, scale = (np.concatenate([r[k] for r in refs]) for k in range(2))
        spmv.spmv_batch_set_lanes(b.h, -1, lanes)
        spmv.spmv_batch_set_lanes(b.h, 1, 2 if lanes == 64 else 64)   # both layouts in one batch
        x_d = dev(x)
        y, y2 = (torch.full((offs[-1],), float("nan"), dtype=torch.float64, device="cuda") for _ in range(2))
        torch.cuda.synchronize()
        s = torch.cuda.Stream()
        spmv.spmv_batch_run(b.h, x_d, y, s)
        spmv.spmv_batch_run_separate(b.h, -1, x_d, y2, s)
        s.synchronize()
        first = y.cpu().numpy()
        assert_fp64_close(first, want, scale, "rows %d lanes %d" % (rows, lanes))
        assert np.array_equal(first.view(np.uint64), y2.cpu().numpy().view(np.uint64))
        spmv.spmv_batch_run(b.h, x_d, y, s)   # the pieces' counters are ready again
        s.synchronize()
        assert np.array_equal(first.view(np.uint64), y.cpu().numpy().view(np.uint64))
        xh, yh = torch.from_numpy(x).pin_memory(), torch.zeros(offs[-1], dtype=torch.float64).pin_memory()
        spmv.spmv_batch_run_host(b.h, xh, yh, 3, s, torch.cuda.Stream(), torch.cuda.Stream())
        assert np.array_equal(first.view(np.uint64), yh.numpy().view(np.uint64))
