"""TILE and WARP products of rows that a lane does not sum: rows on both sides of
32, 64 and 1024 entries, of a CTA's round and of a tile's 1792 entries, among
short rows and alone, whole and per rank; integer data, so the result is exact."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import dev, synced, torch_cuda

pytestmark = pytest.mark.gpu

_rng = np.random.default_rng(3)
CASES = {
    "edges": list(_rng.permutation([1, 0, 31, 32, 33, 63, 64, 65, 96, 97, 1023, 1024, 1025, 1791, 1792, 1793, 2047, 2048,
                                    2049, 4097] + [3] * 400)),
    "one_row": [5000],
    "one_row_of_a_tile_most": [1024],
    "first_and_last": [3000] + [2] * 100 + [1500],
    "only_cta_rows": [2000] * 300,
    "one_huge": [4] * 1000 + [300_001] + [4] * 1000,
    "as_long_as_each_other": [70] * 700,
    "over_64_by_a_little": list(_rng.integers(33, 67, size=5000)),
    "tile_full_of_entries": [56] * 320 + [57] * 320 + [1024, 768, 1, 1024, 769, 1] * 9,
}


def _csr(lens, seed):
    rng = np.random.default_rng(seed)
    n = len(lens)
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rp[1:])
    return (n, rp, rng.integers(0, n, size=rp[-1]).astype(np.int32),
            rng.integers(-4, 5, size=rp[-1]).astype(np.float64))


@pytest.mark.parametrize("name", sorted(CASES))
def test_long_rows_exact(name):
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    n, rp, ci, va = _csr(CASES[name], 11)
    x = np.random.default_rng(12).integers(-4, 5, size=n).astype(np.float64)
    want = oracle.csr_spmv(n, rp, ci, va, x)
    s, x_d = torch.cuda.Stream(), dev(x)
    for P in sorted({1, min(3, n)}):
        order = [4 * p + k for k in range(4) for p in range(P)]
        with spmv.Part(n, rp, ci, va, P, spmv.PER_PARTITION) as part:
            for variant in (spmv.VARIANT_TILE, spmv.VARIANT_WARP):
                for param in range(5):
                    part.set_variant(variant, param)
                    y = synced(torch.full((n,), float("nan"), dtype=torch.float64, device="cuda"))
                    part.run(order, [0] * len(order), [s], x_d, y)
                    s.synchronize()
                    assert np.array_equal(y.cpu().numpy(), want), (P, variant, param)
            y = synced(torch.full((n,), float("nan"), dtype=torch.float64, device="cuda"))
            part.set_variant(spmv.VARIANT_TILE, 0)
            spmv.spmv_pack(part.h, -1, x_d, s)   # every rank in one launch
            spmv.spmv_local(part.h, -1, x_d, y, s)
            spmv.spmv_halo_copy(part.h, -1, s)
            spmv.spmv_remote(part.h, -1, y, s)
            s.synchronize()
            assert np.array_equal(y.cpu().numpy(), want), P
            assert part.query(spmv.Q_ERROR) == 0


@pytest.mark.parametrize("lens", [[20_000] * 400, [3000] * 4000], ids=["20000", "3000"])
def test_long_rows_are_spread_over_the_chip(lens):
    """A few hundred long rows keep up with a warp per row over all of them (the
    VECTOR variant): one warp after another for 32 rows took 38 to 150 times the
    time before rows went to CTAs."""
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    n, rp, ci, va = _csr(lens, 5)
    s, x_d = torch.cuda.Stream(), dev(np.ones(n))
    y = synced(torch.zeros(n, dtype=torch.float64, device="cuda"))

    def best(variant, param):
        part.set_variant(variant, param)
        times = []
        for _ in range(8):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record(s)
            spmv.spmv_local(part.h, -1, x_d, y, s)
            b.record(s)
            b.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)

    with spmv.Part(n, rp, ci, va, 1, spmv.COARSE) as part:
        base = best(spmv.VARIANT_VECTOR, 32)
        for variant, param in ((spmv.VARIANT_TILE, 0), (spmv.VARIANT_TILE, 4), (spmv.VARIANT_WARP, 3)):
            assert best(variant, param) < 5 * base, (variant, param)
