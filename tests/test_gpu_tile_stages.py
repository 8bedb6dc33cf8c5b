"""Staged kernel (variants TILE and WARP) at the edges of its tiles: row
lengths on both sides of the whole-warp lines (32 and 64 entries), tiles wider
than the stage, empty and partial tiles; integer data, so the result is exact."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import dev, synced, torch_cuda

pytestmark = pytest.mark.gpu


def _lens(name):
    rng = np.random.default_rng(3)
    if name == "thresholds":      # a long row decides how its tile's rows of 33 to 64 are summed
        return [31, 32, 33, 63, 64, 65] * 16 + [31, 32, 33, 63, 64] * 13 + [1] * 5
    if name == "wide_tiles":      # 2 % of the tiles need more than the others' stage
        return list(np.where(np.arange(32 * 120) // 32 % 60 == 7, 64, rng.integers(0, 9, size=32 * 120)))
    if name == "largest_stage":   # tiles of 1792 entries and more
        return [56] * 96 + [57] * 96 + [64] * 40
    if name == "very_long":
        return [3] * 40 + [5000] + [0] * 70 + [129, 128, 127, 4096]
    if name == "mostly_empty":
        return [0] * 1000 + [1] + [0] * 30
    return [7] * 33               # one full tile and one row


@pytest.mark.parametrize("name", ["thresholds", "wide_tiles", "largest_stage", "very_long", "mostly_empty", "one_over"])
@pytest.mark.parametrize("P", [1, 3])
def test_staged_tiles_exact(name, P):
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    lens = np.array(_lens(name))
    n = max(lens.size, 5000 if name == "very_long" else 0)
    lens = np.concatenate([lens, np.zeros(n - lens.size, dtype=lens.dtype)])
    rng = np.random.default_rng(4)
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rp[1:])
    ci = rng.integers(0, n, size=rp[-1]).astype(np.int32)
    va = rng.integers(-4, 5, size=rp[-1]).astype(np.float64)
    x = rng.integers(-4, 5, size=n).astype(np.float64)
    want = oracle.csr_spmv(n, rp, ci, va, x)
    s, x_d = torch.cuda.Stream(), dev(x)
    with spmv.Part(n, rp, ci, va, P) as part:
        for variant in (spmv.VARIANT_TILE, spmv.VARIANT_WARP):
            for param in range(5):
                part.set_variant(variant, param)
                y = synced(torch.full((n,), float("nan"), dtype=torch.float64, device="cuda"))
                part.run([0, 1, 2, 3], [0] * 4, [s], x_d, y)
                s.synchronize()
                assert np.array_equal(y.cpu().numpy(), want), (variant, param)
        assert part.query(spmv.Q_ERROR) == 0
