"""Device memory that a plan or a batch makes is zero-filled when the call that
makes it returns, also with the caller's work queued on the default stream: the
products' streams do not wait for that stream."""
import numpy as np
import pytest

from paper_2203_02530_gb300 import workloads as W
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


class _Device:   # n doubles at a device address, for torch.as_tensor
    def __init__(self, address, n):
        self.__cuda_array_interface__ = {"data": (address, False), "shape": (n,), "typestr": "<f8", "version": 3}


def _busy(torch):
    a = torch.rand((4096, 4096), device="cuda") / 2048
    for _ in range(40):   # tens of milliseconds
        a = a @ a


def test_io_buffers_are_not_filled_late():
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    n, rp, ci, va = W.stencil_7pt(12, seed=1)[:4]
    xh = torch.from_numpy(W.uniform_x(n, seed=2)).pin_memory()
    yh = torch.zeros(n, dtype=torch.float64).pin_memory()
    s = torch.cuda.Stream()
    with spmv.Part(n, rp, ci, va, 2, spmv.COARSE) as part:
        _busy(torch)
        xi, yi = spmv.spmv_part_io_buffers(part.h)
        g = part.run([0, 1, 2, 3], [0, 0, 0, 0], [s], xi, yi, spmv.RUN_CAPTURE)
        spmv.spmv_apply_host(part.h, g, xh, yh, s)
        torch.cuda.synchronize()
        x, y = (torch.as_tensor(_Device(int(getattr(p, "value", p)), n), device="cuda").cpu() for p in (xi, yi))
        assert np.array_equal(x.numpy(), xh.numpy())
        assert np.count_nonzero(yh.numpy()) and np.array_equal(y.numpy(), yh.numpy())


def test_plan_and_batch_made_beside_other_work():
    from paper_2203_02530_gb300 import spmv
    torch = torch_cuda()
    m = W.zipf_random(4000, seed=3)[:4]
    x = torch.from_numpy(W.uniform_x(m[0], seed=4)).cuda()
    s = torch.cuda.Stream()
    got = []
    for busy in (False, True):
        y, z = (torch.zeros(m[0], dtype=torch.float64, device="cuda") for _ in range(2))
        torch.cuda.synchronize()
        if busy:
            _busy(torch)
        with spmv.Part(*m, 2, spmv.COARSE) as part:
            if busy:
                _busy(torch)
            part.set_variant(spmv.VARIANT_SELL, 2008)
            part.run([0, 1, 2, 3], [0, 0, 0, 0], [s], x, y)
            s.synchronize()
        if busy:
            _busy(torch)
        with spmv.Batch([m]) as b:
            spmv.spmv_batch_set_lanes(b.h, -1, 64)
            spmv.spmv_batch_run(b.h, x, z, s)
            s.synchronize()
        torch.cuda.synchronize()
        got.append((y.cpu().numpy(), z.cpu().numpy()))
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
