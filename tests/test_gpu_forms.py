"""The forms of the step that the context's sizes and tables choose, against
single steps with a separate event pass (event_pass 1): bit-identical records,
moments and ledgers (deterministic build)."""
import numpy as np
import pytest

from paper_1807_04733_gb300 import pic
from paper_1807_04733_gb300 import workloads as W

from .test_gpu_group import check, hot, outcome, records

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DET = W.FLAG_DETERMINISTIC


@pytest.mark.parametrize("cells", [260, 315])
@pytest.mark.parametrize("me", [1, 3])
def test_large_density_grid(cells, me):
    """Grids whose density histograms leave room for eight warps (260 cells of
    60 bins) and for fewer, with the slots of many sub-tiles."""
    wl = W.bilayer(fe_nm=15, au_nm=cells - 15, n0=300_000, capacity=1_200_000, n_e=60,
                   n_steps=130, moment_every=me, flags=DET)
    assert check(wl, [101, 1, 28])[3]["eventful"] > 0


@pytest.mark.parametrize("flags", [0, W.FLAG_WEIGHTS, W.FLAG_VELOCITY])
@pytest.mark.parametrize("me", [1, 4])
def test_calls_of_one_step_between_others(me, flags):
    """More slots than LONE_SLOTS: a step by itself takes the single-step kernels,
    and the groups before and after it go on from its state."""
    wl = W.bilayer(n0=300_000, capacity=2_500_000, n_steps=160, moment_every=me, flags=DET | flags)
    led = check(wl, [95, 1, 1, 3, 1, 20, 1, 1, 1, 36])[3]
    assert led["injected"] > 0 and led["spawned"] > 0
    check(wl, [101, 1, 58], graph=1)


def test_many_stacks_and_a_large_one():
    """One block for a stack of more slots than 32-bit sums are safe for."""
    wl = W.batched(n_stacks=151, scale=2e-4, n_steps=120, flags=DET)
    wl.stacks[3].capacity = 9_000_000
    led = check(wl, [100, 20])[3]
    assert led["injected"] > 0


@pytest.mark.parametrize("stacks", [1, 3])
def test_autotune_tries_grouped_steps_once(stacks):
    """One trial of grouped steps, also beside the little that 16 layers of 100 bins
    leave of the fused form, and for several stacks."""
    if stacks == 1:
        st = W.make_stack([5] * 16, [i % 3 for i in range(16)], 100, 0.02, 30_000, 10_000)
        wl = W.Workload("layers", 100, 0.02, 1.0, 1.0, 900, 50, 50, 3, DET, [st])
    else:
        wl = W.batched(n_stacks=3, scale=1e-3, n_steps=900, moment_every=50, flags=DET)
    ctx = pic.Context(wl)
    ctx.step(100)
    trials = ctx.autotune(3)
    assert sum(t["event_pass"] == 0 for t in trials) == 1
    assert sum(t["chosen"] for t in trials) == 1
    ctx.close()


def single(wl):
    """The workload with one certain scattering (the lowest bin of one table):
    thresholds that close to 1 keep its steps from being grouped."""
    wl.stacks[0].tau_in = wl.stacks[0].tau_in.copy()
    wl.stacks[0].tau_in[1, 1, 0] = 1e-9
    return wl


@pytest.mark.parametrize("graph", [0, 1, 2])
@pytest.mark.parametrize("me,flags", [(1, 0), (50, 0), (5, W.FLAG_VELOCITY), (5, W.FLAG_WEIGHTS)])
def test_single_steps(me, flags, graph):
    """Steps that are not grouped: the general step inside the streaming pass
    (fused), graphs of single steps and the persistent kernel of their passes."""
    wl = single(W.bilayer(n0=20_000, capacity=50_000, n_steps=250, moment_every=me, flags=DET | flags))
    ctx = pic.Context(wl)
    ctx.step(10)
    assert ctx.launches >= 20                      # a launch per pass and step
    ctx.close()
    assert check(wl, [50, 130, 70], graph=graph)[3]["spawn_dropped"] > 0


@pytest.mark.parametrize("graph", [0, 2])
@pytest.mark.parametrize("me,chunks", [(1, [60, 40, 100]), (5, [200]), (50, [75, 125])])
def test_persistent_groups(me, chunks, graph):
    wl = W.spin_valve(True, fe_nm=5, au_nm=30, n0=20_000, capacity=60_000, n_steps=200, moment_every=me,
                      flags=DET | W.FLAG_VELOCITY)
    check(wl, chunks, graph=graph)


@pytest.mark.parametrize("graph", [0, 1, 2])
@pytest.mark.parametrize("capacity,n", [(3_000_000, 3_000_000), (9_000_000, 8_990_000)])
def test_closed_groups_of_large_sub_tiles(capacity, n, graph):
    """1024-slot sub-tiles and groups of up to 50 steps: a full buffer, and one
    that fills up in the first steps, above the size of the plain persistent form
    (several launches per range, of which a closed group's successors leave)."""
    wl = W.bilayer(n0=0, capacity=capacity, n_steps=170, moment_every=50, flags=DET)
    led = check(wl, [20, 100, 50], records(wl, n), graph=graph)[3]
    assert led["spawn_dropped"] > 0 and led["absorbed"] > 0
