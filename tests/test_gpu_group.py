"""Grouped time steps (event_pass 0) against single steps with a separate
event pass (event_pass 1): bit-identical records, moments and ledgers
(deterministic build), at the sizes and options where a group can go wrong:
ragged sub-tiles with old records behind the last slot, long closed groups,
events for more than one round per sub-tile, record lists that fill up,
secondaries of secondaries within one group, many layers, edges that half
precision cannot hold, weights, velocities, several stacks with empty ones."""
import numpy as np
import pytest

from paper_1807_04733_gb300 import pic
from paper_1807_04733_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DET = W.FLAG_DETERMINISTIC


def outcome(wl, event_pass, chunks, recs=None, graph=0):
    ctx = pic.Context(wl, event_pass=event_pass, use_graph=graph)
    if recs is not None:
        ctx.set_records(recs, len(recs))
    status = 0
    for n in chunks:
        ctx.step(n)
    try:
        ctx.sync()
    except pic.PicError as e:
        status = e.status
    out = [status]
    if status == 0:
        for s in range(len(wl.stacks)):
            n, J, led = ctx.moments(s)
            out += [n.cpu().numpy(), J.cpu().numpy(), led, ctx.gen_moments(s).cpu().numpy(),
                    ctx.records(s).view(np.uint32)]
            if wl.flags & W.FLAG_VELOCITY:
                out.append(ctx.vel_moments(s).cpu().numpy())
            if wl.flags & W.FLAG_WEIGHTS:
                nw, Jw, wi = ctx.weighted_moments(s)
                out += [nw.cpu().numpy(), Jw.cpu().numpy(), wi, ctx.weights(s)]
    ctx.close()
    return out


def check(wl, chunks, recs=None, graph=0):
    a, b = outcome(wl, 0, chunks, recs, graph), outcome(wl, 1, chunks, recs)
    assert len(a) == len(b)
    for i, (x, y) in enumerate(zip(a, b)):
        if isinstance(x, np.ndarray):
            assert x.shape == y.shape and np.array_equal(x, y), i
        else:
            assert x == y, (i, x, y)
    return a


def hot(wl, rate=0.2):
    """Every carrier scatters, mostly inelastically, in most steps."""
    for st in wl.stacks:
        st.tau_in[:] = rate * wl.dt
    return wl


def records(wl, n, seed=1):
    st = wl.stacks[0]
    rng = np.random.default_rng(seed)
    edges = np.cumsum([0] + list(st.layer_cells)).astype(np.float64)
    r = np.zeros(n, pic.REC_DTYPE)
    lay = rng.integers(0, len(st.layer_cells), n)
    r["z"] = (edges[lay] + rng.random(n) * np.array(st.layer_cells)[lay] * 0.999).astype(np.float32)
    mu = rng.uniform(-1, 1, n).astype(np.float32)
    r["mu"] = np.where(mu == 0, np.float32(0.5), mu)
    k = rng.integers(0, wl.n_e + 1, n)                 # some slots removed already
    r["packed"] = (k | (rng.integers(0, 2, n) << 8) | (lay << 9) | (1 << 13)).astype(np.uint32)
    r["id"] = np.arange(n)
    return r


@pytest.mark.parametrize("me,ce", [(1, 50), (3, 7), (50, 50)])
def test_ragged_sub_tiles_over_many_steps(me, ce):
    """A few slots per sub-tile, compacted often: the memory behind the last
    slot holds old records; closed groups once the buffer is full."""
    wl = W.config(0, scale=0.003, flags=DET).replace(n_steps=3000, moment_every=me, compact_every=ce)
    led = check(wl, [200, 1, 2, 2797])[3]
    assert led["absorbed"] > 0 and led["spawn_dropped"] > 0


@pytest.mark.parametrize("me", [1, 2, 50])
def test_secondaries_of_secondaries_in_one_group(me):
    """Most carriers scatter in every step and the buffer has room for all:
    long lists, several event rounds per sub-tile, new carriers that create
    carriers before the group ends, and the capacity reached inside a group."""
    wl = hot(W.bilayer(n0=0, capacity=60_000, n_steps=40, moment_every=me, flags=DET))
    led = check(wl, [3, 9, 28], records(wl, 9_001))[3]
    assert led["spawned"] > 20_000 and led["spawn_dropped"] > 0


@pytest.mark.parametrize("flags", [W.FLAG_NO_SECONDARIES, W.FLAG_TRANSPARENT, W.FLAG_LOWEST_BIN_ANY,
                                   W.FLAG_VELOCITY, W.FLAG_WEIGHTS])
@pytest.mark.parametrize("me", [1, 50])
def test_options(flags, me):
    wl = W.spin_valve(True, fe_nm=3, au_nm=7, n0=3_000, capacity=9_001, n_steps=420, flags=DET | flags,
                      moment_every=me, compact_every=64)
    check(wl, [150, 270])


def test_strict_capacity_reported():
    wl = hot(W.bilayer(n0=0, capacity=9_100, n_steps=8, moment_every=8,
                       flags=DET | W.FLAG_STRICT_CAPACITY))
    assert check(wl, [8], records(wl, 9_001))[0] == 3


def test_many_layers_and_coarse_edges():
    n_e, cells = 4, [3, 1, 2, 2100, 5, 4, 1, 1, 2, 6, 3, 2, 1, 700, 2, 1]
    st = W.make_stack(cells, [i % 3 for i in range(16)], n_e, 0.2, 50_000, 0)
    wl = W.Workload("layers", n_e, 0.2, 2.0, 1.0, 60, 10, 25, 3, DET | W.FLAG_VELOCITY, [st])
    check(wl, [60], records(wl, 30_011))


@pytest.mark.parametrize("graph", [0, 1])
def test_stacks_with_empty_ones(graph):
    wl = W.batched(n_stacks=7, scale=2e-3, n_steps=250, flags=DET)
    wl.stacks[0].n0 = 0
    wl.stacks[4].n0 = 0
    wl.stacks[4].capacity = 0
    wl.stacks[6].n0 = 1
    check(wl, [3, 247] if graph == 0 else [250], graph=graph)
