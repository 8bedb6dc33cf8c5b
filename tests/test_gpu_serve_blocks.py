"""Served blocks at the edges of the row classes (64, 65, 2048, 2049 entries)
and of the widths: every width alone, with X at 32- and only 16-byte aligned
addresses, and in merged blocks whose columns belong to several requests, gives
the same bits and the oracle's product."""
import numpy as np
import pytest

import oracle
from paper_2203_02530_gb300 import workloads as W
from tests.gpu_util import assert_fp64_close, torch_cuda
from tests.test_gpu_serve import host_hash

pytestmark = pytest.mark.gpu


def _edges(n, seed):
    rng = np.random.default_rng(seed)
    lens = rng.integers(0, 12, size=n)
    lens[rng.choice(n, size=9, replace=False)] = [63, 64, 65, 96, 128, 129, 2047, 2048, 2049]
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(lens, out=rp[1:])
    return n, rp, rng.integers(0, n, size=rp[-1]).astype(np.int32), rng.uniform(-1, 1, size=rp[-1])


def test_widths_alignments_and_merged_blocks():
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    mats = [_edges(5003, 1), W.stencil_7pt(9, seed=2), _edges(3000, 3)]
    mat = np.repeat(np.arange(3), 24).astype(np.int32)
    wid = np.tile(np.arange(1, 9), 9).astype(np.int32)
    seed = np.arange(100, 172).astype(np.uint64)
    s = torch.cuda.Stream()
    with spmv.Batch(mats) as b:
        spmv.spmv_batch_set_lanes(b.h, -1, spmv.BATCH_SLICED)
        with spmv.Server(b, n_streams=3, budget_bytes=1 << 30) as sv:
            _, hashes, stats = sv.run(mat, wid, seed, np.zeros(72))
            assert stats["blocks"] < 72   # requests were merged
            _, plain, _ = sv.run(mat, wid, seed, np.zeros(72), spmv.SERVE_PLAIN)
            assert np.array_equal(hashes, plain)
            for r in range(72):
                n, rp, ci, va = mats[mat[r]]
                w, bits = int(wid[r]), []
                for shift in (0, 2):   # doubles: X at a multiple of 32 bytes, and 16 bytes off one
                    x = torch.zeros(n * w + 4, dtype=torch.float64, device="cuda")[shift:]
                    y = torch.zeros(n * w, dtype=torch.float64, device="cuda")
                    torch.cuda.synchronize()
                    spmv.spmv_serve_single(sv.h, int(mat[r]), w, int(seed[r]), y, x, s)
                    s.synchronize()
                    bits.append(y.cpu().numpy().reshape(n, w))
                assert np.array_equal(bits[0].view(np.uint64), bits[1].view(np.uint64)), (r, w)
                assert host_hash(bits[0], w) == hashes[r], (r, w)
                if r % 7 == 0:
                    X = W.request_x(int(seed[r]), n, w)
                    for j in range(w):
                        assert_fp64_close(bits[0][:, j], oracle.csr_spmv(n, rp, ci, va, X[:, j]),
                                          oracle.csr_absdot(n, rp, ci, va, X[:, j]), "request %d column %d" % (r, j))
