"""What a context does after a failure status.  A full buffer in strict mode
(PIC_F_STRICT_CAPACITY) sets the status and drops the carrier; the steps go on
as they do otherwise, in every form, and what can be read is that of single
steps bit for bit (deterministic build)."""
import ctypes as C

import numpy as np
import pytest

from paper_1807_04733_gb300 import pic
from paper_1807_04733_gb300 import workloads as W

from .test_gpu_group import records

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

STRICT = W.FLAG_DETERMINISTIC | W.FLAG_STRICT_CAPACITY


def overflowing(me, ce=25):
    """A stack whose buffer is loaded full and one with room, both with a source."""
    wl = W.batched(n_stacks=2, scale=2e-3, n_steps=300, moment_every=me, compact_every=ce, flags=STRICT)
    wl.stacks[0].capacity = 9_001
    return wl


def begin(wl, **kw):
    ctx = pic.Context(wl, **kw)
    ctx.set_records(records(wl, 9_001), 9_001)
    return ctx


def moments(ctx, wl):
    """The moments and ledgers of a context whatever its status, and that."""
    out = []
    for s in range(len(wl.stacks)):
        nc, no, _ = ctx.shape(s)
        n = torch.zeros((no, 2, wl.n_e, nc), dtype=torch.int32, device="cuda")
        J = torch.zeros((no, 2, nc + 1), dtype=torch.int32, device="cuda")
        led = pic.pic_ledger()
        st = pic.lib().pic_moments(ctx.ctx, s, C.c_void_p(n.data_ptr()), C.c_void_p(J.data_ptr()), C.byref(led))
        out += [st, led.as_dict(), n.cpu().numpy(), J.cpu().numpy()]
    return out


def same(a, b):
    for i, (x, y) in enumerate(zip(a, b)):
        assert np.array_equal(x, y) if isinstance(x, np.ndarray) else x == y, i


@pytest.mark.parametrize("graph", [0, 1, 2])
@pytest.mark.parametrize("me", [1, 5])
def test_steps_go_on_after_an_overflow(me, graph):
    """Several calls of whole groups and shorter ones, the overflow in the first."""
    wl = overflowing(me)
    a, b = begin(wl, use_graph=graph), begin(wl, event_pass=1)
    for n in (25, 60, 3, 1, 61):
        a.step(n)
        b.step(n)
        x = moments(a, wl)
        same(x, moments(b, wl))
        assert x[0] == 3 and x[1]["spawn_dropped"] > 0
    a.close()
    b.close()


def test_windows_after_an_overflow_inside_one():
    """Windows of 50 steps that calls of different lengths end, a whole group's
    launch and a short one's, after an overflow within the first window."""
    wl = overflowing(50, ce=40)
    a, b = begin(wl), begin(wl, event_pass=1)
    for n in (45, 5, 47, 3, 100, 50):
        a.step(n)
        b.step(n)
    same(moments(a, wl), moments(b, wl))
    for s in range(2):
        assert torch.equal(a.gen_moments(s), b.gen_moments(s))
    a.close()
    b.close()


@pytest.mark.parametrize("graph", [0, 1, 2])
def test_checkpoint_loaded_after_a_failure(graph):
    """The context steps on from the checkpoint as a fresh one does."""
    wl = overflowing(5)
    a = pic.Context(wl, use_graph=graph)
    a.step(30)
    blob = a.save()
    a.set_records(records(wl, 9_001), 9_001)
    a.step(70)
    assert moments(a, wl)[0] == 3
    a.load(blob)
    b = pic.Context(wl, use_graph=graph)
    b.load(blob)
    for n in (20, 70):
        a.step(n)
        b.step(n)
        same(moments(a, wl), moments(b, wl))
    a.close()
    b.close()
