"""Sides of dispatch rules that no other test is large or odd enough to reach:
streams of products that go rank by rank with x in one copy, the plan-free merge
product on arrays at 16 but not 32 bytes, and the coarsest pieces of a batch."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import dev, synced, torch_cuda

pytestmark = pytest.mark.gpu


def _csr(lens, seed, near=None):
    rng = np.random.default_rng(seed)
    n = len(lens)
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rp[1:])
    ci = rng.integers(0, n, size=rp[-1])
    if near:
        ci = np.clip(np.repeat(np.arange(n), lens) + rng.integers(-near, near + 1, size=rp[-1]), 0, n - 1)
    return n, rp, ci.astype(np.int32), rng.integers(-4, 5, size=rp[-1]).astype(np.float64)


# one product above 65 536 rows a rank and two above 131 072 go rank by rank
@pytest.mark.parametrize("rows_per_rank,count", [(65_536, 1), (65_537, 1), (131_072, 2), (131_073, 2)])
def test_host_streams_on_both_sides_of_the_line(rows_per_rank, count):
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    P = 2
    n, rp, ci, va = _csr(np.random.default_rng(1).integers(0, 6, size=P * rows_per_rank), 2, near=rows_per_rank // 2)
    xs = torch.from_numpy(np.random.default_rng(3).integers(-9, 10, size=(count, n)).astype(np.float64)).pin_memory()
    want = [oracle.csr_spmv(n, rp, ci, va, xs[k].numpy()) for k in range(count)]
    s, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    with spmv.Part(n, rp, ci, va, P, spmv.COARSE) as part:
        for variant in ((spmv.VARIANT_TILE, 0), (spmv.VARIANT_SELL, 8)):
            part.set_variant(*variant)
            for flags in range(4):
                ys = torch.full((count, n), float("nan"), dtype=torch.float64).pin_memory()
                for _ in range(2):   # the second call finds the events and vectors of the first
                    spmv.spmv_apply_host_many(part.h, count, xs, n, ys, n, flags, s2, s)
                for k in range(count):
                    assert np.array_equal(ys[k].numpy(), want[k]), (variant, flags, k)


@pytest.mark.parametrize("name,lens", [("edges", [7, 8, 9, 0, 255, 256, 257, 1, 247, 248, 249, 503, 504] * 7),
                                       ("one_row", [5]), ("long", [2] * 40 + [70_000] + [0, 3] * 40),
                                       ("mixed", list(np.random.default_rng(7).integers(0, 30, size=150_001)))])
@pytest.mark.parametrize("shift_col,shift_val", [(4, 0), (0, 2), (4, 2)])
def test_merge_on_arrays_at_16_bytes(name, lens, shift_col, shift_val):
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    n, rp, ci, va = _csr(lens, 11)
    x = np.random.default_rng(12).integers(-4, 5, size=n).astype(np.float64)
    want = oracle.csr_spmv(n, rp, ci, va, x)

    def shifted(a, k):   # at 16 bytes past a multiple of 32, nothing of the array's own after its end
        t = torch.empty(a.size + k, dtype=torch.int32 if a.dtype == np.int32 else torch.float64, device="cuda")
        t[k:] = dev(a)
        assert t.data_ptr() % 32 == 0
        return t[k:]

    s = torch.cuda.Stream()
    col, val = shifted(ci, shift_col), shifted(va, shift_val)
    assert (col.data_ptr() | val.data_ptr()) % 32 == 16
    for call in (spmv.spmv_csr_merge, spmv.spmv_csr_merge_noalloc):
        y = synced(torch.full((n + 64,), float("nan"), dtype=torch.float64, device="cuda"))
        call(n, int(rp[-1]), dev(rp.astype(np.int32)), col, val, dev(x), y, s)
        s.synchronize()
        got = y.cpu().numpy()
        assert np.array_equal(got[:n], want) and np.isnan(got[n:]).all(), call.__name__


@pytest.mark.parametrize("lanes", [2, 64])
def test_batch_with_the_longest_pieces(lanes):
    """More rows than 4 x 128 for each of 48 warps per SM: pieces of 2048 entries
    and 16 long rows a unit."""
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = 4 * sms * 48 * 128 + 1
    lens = np.random.default_rng(5).integers(0, 3, size=rows)
    lens[::1009] = 65
    edges = [2047, 2048, 2049, 4095, 4096, 4097, 70_000]
    lens[np.random.default_rng(6).choice(rows, size=len(edges), replace=False)] = edges
    mats = [_csr(lens, 7), _csr(np.array([3000] * 9 + [2] * 500), 8)]
    with spmv.Batch(mats) as b:
        offs = b.offsets()
        assert offs[-1] > rows
        x = np.random.default_rng(9).integers(-4, 5, size=offs[-1]).astype(np.float64)
        want = np.concatenate([oracle.csr_spmv(*m, x[offs[i]:offs[i + 1]]) for i, m in enumerate(mats)])
        spmv.spmv_batch_set_lanes(b.h, -1, lanes)
        x_d, s = dev(x), torch.cuda.Stream()
        for run in (lambda y: spmv.spmv_batch_run(b.h, x_d, y, s),
                    lambda y: spmv.spmv_batch_run_separate(b.h, -1, x_d, y, s)):
            y = synced(torch.full((offs[-1],), float("nan"), dtype=torch.float64, device="cuda"))
            run(y)
            s.synchronize()
            assert np.array_equal(y.cpu().numpy(), want)
