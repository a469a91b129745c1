"""pic_load into a context that has stepped further than the checkpoint."""
import pytest

from paper_1807_04733_gb300 import pic
from paper_1807_04733_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, W.FLAG_WEIGHTS])
def test_windows_ahead_of_the_checkpoint_are_empty(flags):
    wl = W.config(0, scale=0.02, flags=W.FLAG_DETERMINISTIC | flags).replace(n_steps=200, moment_every=5)
    a = pic.Context(wl)
    a.step(60)
    blob = a.save()
    a.step(100)
    assert a.moments(0)[1][12:].any()
    if flags:
        a.weighted_moments(0)
    a.load(blob)
    n, J, _ = a.moments(0)
    assert J[:12].any() and not n[12:].any() and not J[12:].any()
    if flags:
        nw, Jw, _ = a.weighted_moments(0)
        assert not nw[12:].any() and not Jw[12:].any()
    a.close()
