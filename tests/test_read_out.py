"""Where the reading calls' outputs may lie: which buffers a kernel of the
context stores to (without a GPU), and that every other kind gets a copy."""
import ctypes as C

import numpy as np
import pytest

from paper_1807_04733_gb300 import build as B
from paper_1807_04733_gb300 import pic
from paper_1807_04733_gb300 import workloads as W

torch = pytest.importorskip("torch")

UNREGISTERED, HOST, DEVICE, MANAGED = 0, 1, 2, 3     # cudaMemoryType


def test_kernel_stores_to_its_own_device_only():
    B.build()
    f = pic.lib().pic_kernel_stores
    f.argtypes = [C.c_int, C.c_int, C.c_int, C.c_uint64]
    assert f(DEVICE, 0, 0, 4096) and f(DEVICE, 3, 3, 4100)
    assert not f(DEVICE, 1, 0, 4096) and not f(DEVICE, 0, 1, 4096)
    for kind in (UNREGISTERED, HOST, MANAGED):
        assert not f(kind, 0, 0, 4096)
    for p in (4097, 4098, 4099):
        assert not f(DEVICE, 0, 0, p)


@pytest.mark.gpu
def test_window_into_any_buffer():
    wl = W.config(0, scale=0.02, flags=W.FLAG_DETERMINISTIC).replace(n_steps=60)
    ctx = pic.Context(wl)
    ctx.step(60)
    n, J, _ = ctx.moments(0)
    n, J = n[50].cpu().numpy().view(np.uint8).ravel(), J[50].cpu().numpy().view(np.uint8).ravel()
    assert n.any()
    buf = [lambda k: torch.zeros(k + 8, dtype=torch.uint8, device="cuda"),
           lambda k: torch.zeros(k + 8, dtype=torch.uint8),
           lambda k: torch.zeros(k + 8, dtype=torch.uint8).pin_memory()]
    for make in buf:
        for off in (0, 4, 1, 2):
            a, b = make(n.size), make(J.size)
            pic.pic_moment_window(ctx.ctx, 0, 50, a.data_ptr() + off, b.data_ptr() + off)
            for got, want in ((a, n), (b, J)):
                got = got.cpu().numpy()
                assert np.array_equal(got[off: off + want.size], want)
                assert not got[:off].any() and not got[off + want.size:].any()
    ctx.close()
