"""Performance cases of the hot-electron PIC library: what its users run.

A case is a dict of plain values.  ``kind`` says which public entry points a
pass goes through:

* ``kept``: a context that is past its pump pulse; a pass advances it by
  ``steps`` time steps and reads the moment window just finished
  (``pic_step``, ``pic_moment_window``), as a program does that follows a
  simulation.  The state moves on from pass to pass.
* ``run``: a simulation from nothing: context, pulse, ``steps`` time steps,
  all moments, destruction.
* ``grad``: the gradient of a linear functional of a finished run's moments
  (``pic_grad``).
* ``fit``: one training step of a table fit: forward run and backward pass
  through ``PicTransport``.
* ``compact``: ``pic_compact_static`` on particle arrays of the caller's own.

Every output is an exact integer (counts, fixed-point sums, ledgers) except
the gradients, which are float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1807_04733_gb300 import pic
from paper_1807_04733_gb300 import workloads as W

FLAGS = {"deterministic": W.FLAG_DETERMINISTIC, "no_secondaries": W.FLAG_NO_SECONDARIES,
         "transparent": W.FLAG_TRANSPARENT, "velocity": W.FLAG_VELOCITY,
         "weights": W.FLAG_WEIGHTS}

BASE = dict(kind="kept", stack="bilayer", fe=15, au=100, n0=100_000, capacity=400_000, n_e=30,
            dt=1.0, pre=0, steps=50, n_max=0, moment_every=1, compact_every=50, graph=0, flags="")


def _case(name=None, **kw):
    c = dict(BASE, **kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one time step of the 1e5-carrier bilayer and its
        # window, as an interactive program does it; launches and latency
        _case("bilayer_step", pre=200, steps=1, n_max=200_000),
        # the smallest standard workload as a whole: 1e5 carriers, 500 steps
        # of 1 fs, densities every step
        _case("bilayer_run", kind="run", steps=500),
        # a medium simulation from nothing: antiparallel spin valve, ragged
        # sizes, the velocity moment behind the spin current
        _case("valve_ap_run", kind="run", stack="valve_ap", fe=10, au=50, n0=1_200_007,
              capacity=6_000_035, dt=0.5, steps=600, flags="velocity"),
        # the standard spin valve (1e7 carriers, capacity 5e7), densities and
        # fluxes every step, 50 steps of a run that is past its pulse
        _case("valve", stack="valve", fe=10, au=50, n0=10_000_000, capacity=50_000_000, dt=0.5,
              pre=300, steps=50, n_max=50_300, graph=1),
        # the largest standard workload (2e8 carriers, capacity 4e8): one
        # moment and compaction period of 50 steps, the buffer full
        _case("large", au=300, n0=200_000_000, capacity=400_000_000, n_e=60, dt=0.5, pre=300,
              steps=50, n_max=100_300, moment_every=50, graph=1),
        # the same bilayer with room for every secondary, from nothing: the
        # pulse, then the growing cascade
        _case("growing_run", kind="run", au=300, n0=20_000_000, capacity=160_000_000, n_e=60,
              dt=0.5, steps=500, moment_every=50, graph=1),
        # 64 stacks of differing thickness, tables and size in one context,
        # replayed from graphs: a parameter scan
        _case("batched", stack="batched64", n0=0, capacity=0, pre=150, steps=50, n_max=3150,
              graph=1),
        # a small scan from nothing, each period one persistent launch
        _case("scan_run", kind="run", stack="batched13", n0=300_000, capacity=0, steps=200,
              graph=2),
        # importance-sampled source: weighted moments every 10 steps
        _case("weighted_run", kind="run", n0=1_000_003, capacity=4_000_012, steps=300,
              moment_every=10, flags="weights"),
        # the gradient of the standard 1e7-carrier run of 800 steps
        _case("adjoint", kind="grad", n0=10_000_000, capacity=50_000_000, steps=800),
        # one step of fitting the tables to measured moments
        _case("fit", kind="fit", n0=200_000, capacity=800_000, steps=250, moment_every=5),
        # compaction of a caller's arrays, an odd number of slots
        _case("compact", kind="compact", n0=100_000_007, capacity=0, steps=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _steps_kept(stack, fe, au, n_e, me, pre, steps):
    """Room for 10000 passes, or for 4 GB of moment windows (about 10 bytes
    per bin)."""
    cells = (fe + au) * 2 if not stack.startswith("batched") else 125 * int(stack[7:])
    windows = 4e9 / (10.0 * 2 * n_e * cells)
    return int(max(pre + 4 * steps, min(pre + 10000 * steps, me * windows)))


def draw(rng):
    """One more case: sizes over their logarithms, every option in turn."""
    kind = rng.choice(["kept", "kept", "run", "run", "run", "grad", "fit", "compact"])
    if kind == "compact":
        return _case(kind=kind, n0=_log(rng, 1000, 1.0e8), capacity=0, steps=1)
    n_e = rng.choice([12, 25, 30, 30, 41, 60])
    dt = rng.choice([0.5, 1.0])
    stack = rng.choice(["bilayer", "bilayer", "valve", "valve_ap", "batched%d" % rng.randint(2, 24)])
    if kind == "fit":
        stack = rng.choice(["bilayer", "valve"])
    fe, au = rng.randint(5, 20), rng.randint(20, 5000 // n_e)
    ratio = rng.choice([2.0, 3.0, 4.0, 5.0, 8.0])
    hi = {"kept": 8e6, "run": 2e6, "grad": 2e6, "fit": 5e5}[kind]
    n0 = _log(rng, 1e4, hi)
    flags = [f for f, p in (("deterministic", 0.2), ("no_secondaries", 0.15),
                            ("transparent", 0.1), ("velocity", 0.25)) if rng.random() < p]
    if kind == "run" and not stack.startswith("batched") and rng.random() < 0.25:
        flags.append("weights")
    pre = int(math.ceil(150.0 / dt))
    steps = {"kept": rng.randint(2, 60), "run": rng.randint(pre, pre + 250),
             "grad": rng.randint(pre, pre + 150), "fit": rng.randint(pre, pre + 100)}[kind]
    me = rng.choice([1, 1, 1, 2, 5, 10, 50])
    if kind == "fit":
        me = rng.choice([5, 10, 25])
    return _case(kind=kind, stack=stack, fe=fe, au=au, n0=n0, capacity=int(n0 * ratio), n_e=n_e,
                 dt=dt, pre=pre if kind == "kept" else 0, steps=steps,
                 n_max=_steps_kept(stack, fe, au, n_e, me, pre, steps) if kind == "kept" else 0,
                 moment_every=me, compact_every=rng.choice([20, 50, 50, 64]),
                 graph=rng.choice([0, 0, 1, 2]) if kind in ("kept", "run") else 0,
                 flags=",".join(flags))


# ---------------------------------------------------------------------------
def _workload(case, seed):
    c = case
    flags = 0
    for f in c["flags"].split(","):
        flags |= FLAGS[f] if f else 0
    n_e, de = c["n_e"], 1.5 / c["n_e"]
    n_max = c["n_max"] or c["steps"]
    rng = np.random.default_rng(seed)
    common = dict(n_e=n_e, de=de, dt=c["dt"], n_steps=n_max, moment_every=c["moment_every"],
                  compact_every=c["compact_every"], seed=seed & 0x7FFFFFFF, flags=flags)
    if c["stack"].startswith("batched"):
        n = int(c["stack"][7:])
        # the standard scan's stacks (n0 = 0), or its shapes with carriers
        # spread over two decades up to n0
        wl = W.batched(n_stacks=n, scale=c["n0"] / 1e7 if c["n0"] else 1.0, **common)
        wl.stacks = [W.perturb(st, rng, rel=0.05) for st in wl.stacks]
    else:
        mats = {"bilayer": [W.MAT_FE, W.MAT_AU], "valve": [W.MAT_FE, W.MAT_AU, W.MAT_FE],
                "valve_ap": [W.MAT_FE, W.MAT_AU, W.MAT_FE_AP]}[c["stack"]]
        st = W.make_stack([c["fe"], c["au"], c["fe"]][: len(mats)], mats, n_e, de, c["capacity"], c["n0"])
        # the fitted and scanned tables differ from run to run
        st = W.perturb(st, rng, rel=0.05)
        if flags & W.FLAG_WEIGHTS:
            depth = np.arange(st.n_cells)
            st.cell_bias = 1.0 + 3.0 * np.exp(-((depth - c["fe"]) / 4.0) ** 2)
            st.e_bias = np.linspace(0.5, 1.5, n_e)
        wl = W.Workload("case", n_e, de, c["dt"], 1.0, n_max, c["moment_every"], c["compact_every"],
                        common["seed"], flags, [st])
    return wl


def _weights(ctx, case, seed):
    """Weights of a functional of the moments: the spin density of ten cells
    and the spin flux at the first interface."""
    S, ncm = len(ctx.wl.stacks), ctx.n_cells_max
    _, n_out, _ = ctx.shape(0)
    rng = np.random.default_rng(seed)
    gn = torch.zeros((S, n_out, 2, ctx.wl.n_e, ncm), dtype=torch.float32, device="cuda")
    gJ = torch.zeros((S, n_out, 2, ncm + 1), dtype=torch.float32, device="cuda")
    c0 = int(rng.integers(0, max(1, ncm - 10)))
    for s, st in enumerate(ctx.wl.stacks):
        gn[s, :, 0, :, c0: min(c0 + 10, st.n_cells)] = 1.0
        gn[s, :, 1, :, c0: min(c0 + 10, st.n_cells)] = -1.0
        gJ[s, :, 0, st.layer_cells[0]] = 1.0
        gJ[s, :, 1, st.layer_cells[0]] = -1.0
    return gn, gJ


def _begin(state):
    """A context that has run through its pulse (kept) or to its end (grad)."""
    case = state["case"]
    state["done"] = case["pre"] if case["kind"] == "kept" else case["steps"]
    ctx = state["ctx"] = pic.Context(state["wl"], use_graph=case["graph"])
    ctx.step(state["done"])
    ctx.sync()
    return ctx


def prepare(case, seed):
    if case["kind"] == "compact":
        n = case["n0"]
        g = torch.Generator(device="cuda").manual_seed(seed)
        z = torch.rand(n, device="cuda", generator=g) * 115.0
        mu = torch.rand(n, device="cuda", generator=g) * 2.0 - 1.0
        ids = torch.randperm(n, device="cuda", generator=g, dtype=torch.int32) if n < 1 << 22 else \
            torch.arange(n, device="cuda", dtype=torch.int32)
        pk = torch.randint(1, 31, (n,), device="cuda", generator=g, dtype=torch.int32) | (1 << 13)
        # a tenth of the slots removed, as after some periods without compaction
        pk[torch.randperm(n, device="cuda", generator=g)[: n // 10]] &= ~0xFF
        out = [torch.empty_like(x) for x in (z, mu, ids, pk)]
        return {"case": case, "in": [z, mu, ids, pk], "out": out}
    wl = _workload(case, seed)
    state = {"case": case, "wl": wl}
    if case["kind"] in ("kept", "grad"):
        ctx = _begin(state)
        if case["kind"] == "kept":
            cells = [st.n_cells for st in wl.stacks]
            state["n"] = torch.zeros(sum(2 * wl.n_e * c for c in cells), dtype=torch.int32, device="cuda")
            state["J"] = torch.zeros(sum(2 * (c + 1) for c in cells), dtype=torch.int32, device="cuda")
        else:
            state["gn"], state["gJ"] = _weights(ctx, case, seed)
    elif case["kind"] == "fit":
        st = wl.stacks[0]
        g = torch.Generator(device="cuda").manual_seed(seed)
        n_out = (case["steps"] + case["moment_every"] - 1) // case["moment_every"]
        state["tau"] = torch.tensor(st.tau_in[None], device="cuda", requires_grad=True)
        state["T"] = torch.tensor(st.T[None], device="cuda", requires_grad=True)
        # the measured moments that the fit aims at
        state["target"] = torch.rand((1, n_out, 2, wl.n_e, st.n_cells), device="cuda", generator=g) * \
            (4.0 * st.n0 / (2 * wl.n_e * st.n_cells))
    return state


def _ledgers(leds):
    return torch.tensor([[led[k] for k in pic.LEDGER_FIELDS] for led in leds], dtype=torch.int64)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "compact":
        (z, mu, i, p), (zo, muo, io, po) = state["in"], state["out"]
        n = z.numel()
        alive = pic.pic_compact_static(z.data_ptr(), mu.data_ptr(), i.data_ptr(), p.data_ptr(), n,
                                       zo.data_ptr(), muo.data_ptr(), io.data_ptr(), po.data_ptr(),
                                       torch.cuda.current_stream().cuda_stream)
        return [alive, zo[:alive], muo[:alive], io[:alive], po[:alive]]
    wl = state["wl"]
    if kind == "kept":
        if state["done"] + case["steps"] > wl.n_steps:
            state["ctx"].close()        # the simulation has ended: the next one
            _begin(state)
        ctx, n, J = state["ctx"], state["n"], state["J"]
        ctx.step(case["steps"])
        state["done"] += case["steps"]
        # the last window that has ended (the running one if none has)
        win = max(0, state["done"] // case["moment_every"] - 1)
        leds, on, oj = [], 0, 0
        for s, st in enumerate(wl.stacks):
            leds.append(pic.pic_moment_window(ctx.ctx, s, win, n.data_ptr() + 4 * on, J.data_ptr() + 4 * oj))
            on += 2 * wl.n_e * st.n_cells
            oj += 2 * (st.n_cells + 1)
        return [n, J, _ledgers(leds)]
    if kind == "run":
        ctx = pic.Context(wl, use_graph=case["graph"])
        ctx.step(case["steps"])
        ns, Js, gs, vs, leds = [], [], [], [], []
        for s in range(len(wl.stacks)):
            n, J, led = ctx.moments(s)
            ns.append(n.reshape(-1))
            Js.append(J.reshape(-1))
            leds.append(led)
            gs.append(ctx.gen_moments(s).reshape(-1))
            if wl.flags & W.FLAG_VELOCITY:
                vs.append(ctx.vel_moments(s).reshape(-1))
        out = {"led": _ledgers(leds)}
        for k, v in (("n", ns), ("J", Js), ("gen", gs), ("vel", vs)):
            if v:
                out[k] = v[0] if len(v) == 1 else torch.cat(v)
        if wl.flags & W.FLAG_WEIGHTS:
            out["nw"], out["Jw"], out["w_injected"] = ctx.weighted_moments(0)
        ctx.close()
        return out
    if kind == "grad":
        g_tau, g_T = state["ctx"].grad(state["gn"], state["gJ"])
        return [g_tau, g_T]
    tau, T = state["tau"], state["T"]
    tau.grad = T.grad = None
    n, J = pic.PicTransport.apply(tau, T, wl, case["steps"])
    loss = ((n - state["target"]) ** 2).sum() / n.numel()
    loss.backward()
    return [n.detach(), J.detach(), tau.grad, T.grad]


def _carriers(case):
    """(live carriers, slots, histogram bins per window) of a context, about."""
    if case["stack"].startswith("batched"):
        k = int(case["stack"][7:])
        mean = (case["n0"] or 1e7) * 0.215          # mean of a log-uniform over two decades
        return 3.5 * k * mean, 4 * k * mean, k * 2 * case["n_e"] * 125
    cells = case["fe"] * (1 if case["stack"] == "bilayer" else 2) + case["au"]
    return min(0.95 * case["capacity"], 4.0 * case["n0"]), case["capacity"], 2 * case["n_e"] * cells


def work(case):
    """A carrier-step is about 32 operations (a quarter of a Philox4x32-10
    call, two half flights, three comparisons, its deposit).  Bytes: the
    particle state that a kept context holds read and written once per pass
    (16 B each way), or created and read once; the moments written."""
    if case["kind"] == "compact":
        n = case["n0"]
        return {"bytes": 16.0 * n + 16.0 * 0.9 * n, "flops": 0.0}
    live, _, bins = _carriers(case)
    steps = case["steps"]
    windows = max(1.0, steps / case["moment_every"])
    passes = {"kept": 1.0, "run": 0.8, "grad": 2.0, "fit": 2.4}[case["kind"]]
    out = 4.0 * bins * (1.0 if case["kind"] == "kept" else windows)
    return {"bytes": 32.0 * live + out, "flops": 32.0 * live * steps * passes}


def exact(case, seed):
    """The compaction's outputs; the other cases are random walks whose
    outputs are whole numbers, or gradients that no closed form gives."""
    if case["kind"] != "compact":
        return None
    z, mu, i, p = prepare(case, seed)["in"]
    live = (p & 0xFF) != 0
    return [int(live.sum()), z[live].double(), mu[live].double(), i[live].long(), p[live].long()]
