"""PACK and COPY in one launch (streams of products through host buffers): the
send and receive buffers and y are those of the operations one by one."""
import numpy as np
import pytest

from tests.gpu_util import dev, synced, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,P", [(64, 1), (37, 2), (1025, 3), (40_003, 4)])
def test_pack_and_copy_in_one(n, P):
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    rng = np.random.default_rng(n)
    lens = rng.integers(0, 9, size=n)
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rp[1:])
    ci = rng.integers(0, n, size=rp[-1]).astype(np.int32)
    va = rng.integers(-4, 5, size=rp[-1]).astype(np.float64)
    xs = torch.from_numpy(rng.integers(-9, 10, size=(4, n)).astype(np.float64)).pin_memory()
    ys = torch.full((4, n), float("nan"), dtype=torch.float64).pin_memory()
    s, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    bufs = (spmv.X_SENDBUF, spmv.X_RECVBUF)
    with spmv.Part(n, rp, ci, va, P, spmv.COARSE) as part:
        part.set_variant(spmv.VARIANT_SELL, 8)
        spmv.spmv_apply_host_many(part.h, 4, xs, n, ys, n, 0, s2, s)
        torch.cuda.synchronize()
        got = [part.export(w, 0).copy() for w in bufs]
        for k in range(4):
            x_d = dev(xs[k].numpy())
            y = synced(torch.full((n,), float("nan"), dtype=torch.float64, device="cuda"))
            spmv.spmv_pack(part.h, -1, x_d, s)
            spmv.spmv_local(part.h, -1, x_d, y, s)
            spmv.spmv_halo_copy(part.h, -1, s)
            spmv.spmv_remote(part.h, -1, y, s)
            s.synchronize()
            assert np.array_equal(y.cpu().numpy(), ys[k].numpy()), k
        for a, w in zip(got, bufs):   # both hold the last product's
            assert np.array_equal(a, part.export(w, 0))
