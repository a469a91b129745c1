"""pic_step captured by the caller in a graph of its own: every replay runs the
captured steps, in grouped steps as in single ones (bit for bit, deterministic
build)."""
import numpy as np
import pytest

from paper_1807_04733_gb300 import pic
from paper_1807_04733_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("me,steps", [(1, 5), (1, 30), (50, 30), (5, 55)])
@pytest.mark.parametrize("capacity", [5_001, 9_000_000])
def test_replays_of_a_captured_call(capacity, me, steps):
    wl = W.config(0, scale=0.02, flags=W.FLAG_DETERMINISTIC).replace(n_steps=190, moment_every=me)
    wl.stacks[0].capacity = capacity
    out = []
    for event_pass in (0, 1):
        stream = torch.cuda.Stream()
        ctx = pic.Context(wl, event_pass=event_pass, stream=stream)
        ctx.step(97)
        ctx.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            ctx.step(steps)
        for _ in range(3):
            with torch.cuda.stream(stream):
                g.replay()
        ctx.step(9)
        n, J, led = ctx.moments(0)
        out.append((n.cpu().numpy(), J.cpu().numpy(), led, ctx.records(0).view(np.uint32)))
        ctx.close()
        del g
    for a, b in zip(*out):
        assert np.array_equal(a, b) if isinstance(a, np.ndarray) else a == b
