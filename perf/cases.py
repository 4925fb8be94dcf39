"""The workloads whose time is followed: what a user of this package runs,
through its public entry points, from the smallest call to the largest.

Simulation cases are cattle-shaped populations (log-normal herds, a few
infected ones, geometric event sizes), the package's example models, and the
option sets of the engine: both solvers, models from transition strings,
dense and sparse output, one replicate and many.  The learned one-day
emulator is there with its two network entry points.  ``prepare`` builds what
a program keeps (the model handle, device buffers, a stream), ``run`` makes
one call.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1605_01421_gb300 import binding, emulator
from paper_1605_01421_gb300 import workloads as W

# --------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------


def listed():
    return [
        # The first example of the paper (Sec. 4.1) as a beginner runs it: a
        # small SIR model, the default stream; latency and launches count.
        dict(name="sir_100x99", family="sir", nodes=100, days=99, reps=1),
        # The call of the README, everything in it: model, event planning,
        # upload, run, trajectory back in numpy (the paper's 1,600 herds).
        dict(name="simulate_sise_1600x365", family="simulate", nodes=1600, days=365, reps=1),
        # The same benchmark with the model kept: what a parameter study or
        # a fit does thousands of times.
        dict(name="sise_1600x365", family="sise", nodes=1600, days=365, reps=1),
        # The paper's spatially coupled example (Sec. 4.2).
        dict(name="sise_sp_1600x365", family="sise_sp", nodes=1600, days=365, reps=1),
        # The all events method on the same herds.
        dict(name="aem_sise_1600x365", family="aem", nodes=1600, days=365, reps=1),
        # A model given as transition strings (Sec. 3.5, predator and prey).
        dict(name="predator_prey_1000x30", family="predator_prey", nodes=1000, days=30, reps=1),
        # One national population: few large herds carry most transitions.
        dict(name="sise3_37000x365", family="sise3", nodes=37000, days=365, reps=1),
        # Many replicates, each with its own events: the benchmark's shape.
        dict(name="sise3_256x5000x60", family="sise3", nodes=5000, days=60, reps=256),
        # A scenario study: shared events, a ragged node count, no dense
        # trajectory, prevalence counters and the sparse output of 100 herds.
        dict(name="sise3_prevalence_48x5003x120", family="prevalence", nodes=5003, days=120,
             reps=48),
        # Every herd large and infected: the throughput of the SSA itself.
        dict(name="endemic_100000x20", family="endemic", nodes=100000, days=20, reps=1),
        # One training step's gradients of the emulator network (BF16).
        dict(name="emulator_gradients_8192", family="emu_gradients", rows=8192),
        # The emulator network on a population, E4M3 inference.
        dict(name="emulator_forward_e4m3_100000", family="emu_forward", rows=100000, fp8=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["sir", "simulate", "sise", "sise_sp", "aem", "predator_prey", "sise3",
                         "sise3_batch", "prevalence", "endemic", "emu_gradients",
                         "emu_forward"])
    if family == "sir":
        return dict(family=family, nodes=_log_int(rng, 10, 20000), days=rng.randint(5, 200),
                    reps=rng.choice([1, 1, 3]))
    if family in ("simulate", "sise", "aem"):
        return dict(family=family, nodes=_log_int(rng, 50, 6000), days=rng.randint(20, 365),
                    reps=rng.choice([1, 1, 2, 7]))
    if family == "sise_sp":
        return dict(family=family, nodes=_log_int(rng, 50, 4000), days=rng.randint(20, 365),
                    reps=rng.choice([1, 1, 2]))
    if family == "predator_prey":
        return dict(family=family, nodes=_log_int(rng, 10, 1000), days=rng.randint(5, 30),
                    reps=1)
    if family == "sise3":
        return dict(family=family, nodes=_log_int(rng, 1000, 37000), days=rng.randint(30, 365),
                    reps=1)
    if family == "sise3_batch":
        return dict(family="sise3", nodes=_log_int(rng, 200, 5000), days=rng.randint(10, 60),
                    reps=_log_int(rng, 8, 256))
    if family == "prevalence":
        return dict(family=family, nodes=_log_int(rng, 200, 6000), days=rng.randint(20, 120),
                    reps=_log_int(rng, 2, 48))
    if family == "endemic":
        return dict(family=family, nodes=_log_int(rng, 1000, 100000), days=rng.randint(3, 20),
                    reps=1)
    if family == "emu_gradients":
        return dict(family=family, rows=_log_int(rng, 512, 8192) // 8 * 8)
    return dict(family=family, rows=_log_int(rng, 100, 100000), fp8=rng.random() < 0.5)


# --------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------

# exit, enter, ageing, external transfer
MIX_SISE = (1 / 3, 1 / 3, 0.0, 1 / 3)
MIX_SISE3 = (0.3, 0.3, 0.2, 0.2)


def _herds(rng, n, median, sigma, hi):
    return np.clip(np.rint(np.exp(np.log(median) + sigma * rng.standard_normal(n))), 1,
                   hi).astype(np.int64)


def _seeded(rng, ages, share):
    """1% of the herds (at least one) with `share` of each age infected."""
    infected = np.zeros_like(ages)
    n = ages.shape[0]
    j = rng.choice(n, size=max(1, n // 100), replace=False)
    infected[j] = np.maximum((ages[j] > 0).astype(np.int64),
                             np.rint(share * ages[j]).astype(np.int64))
    u0 = np.stack([ages - infected, infected], axis=2)
    return u0.reshape(n, -1).astype(np.int32)


def _take(pool, key, want):
    """Grants `want` animals from the groups `key` of `pool`, each group's
    grants in order and together at most what it holds; takes them out."""
    o = np.argsort(key, kind="stable")
    k, w = key[o], want[o]
    first = np.r_[True, k[1:] != k[:-1]]
    cs = np.cumsum(w)
    base = np.r_[0, cs][np.flatnonzero(first)][np.cumsum(first) - 1]
    upto = np.minimum(cs - base, pool[k])
    got = upto - np.r_[0, upto[:-1]]
    got[first] = upto[first]
    np.subtract.at(pool, k, got)
    out = np.empty_like(got)
    out[o] = got
    return out


def _events(rng, ages, days, reps, rate, mix, enter_sel, exit_sel, ageing):
    """Daily exit, enter, ageing and external-transfer events of `reps`
    replicates (their own events when reps > 1), geometric sizes with mean 3,
    sources of transfers by a heavy-tailed out-degree.  The animals of every
    group are tracked in the order the solver runs a day, so every event is
    valid on every path."""
    n, a_n = ages.shape
    pool = np.tile(ages.reshape(-1), reps)
    k = np.arange(1, 1001, dtype=np.float64)
    p = k ** -2.2
    deg = rng.choice(k, size=n, p=p / p.sum())
    cdf = np.cumsum(deg / deg.sum())
    cols = []

    def emit(kind, T, rep, node, dest, cnt, sel, shift):
        ok = cnt > 0
        m = int(ok.sum())
        full = lambda x: np.broadcast_to(np.asarray(x), ok.shape)[ok].astype(np.int32)  # noqa: E731
        if m:
            cols.append((np.full(m, kind, np.int32), np.full(m, T, np.int32), full(node),
                         full(dest), full(cnt), full(sel), full(shift), full(rep)))

    for d in range(days):
        T = d + 1
        per = rng.multinomial(rng.poisson(rate * n, size=reps), mix)
        rep = [np.repeat(np.arange(reps), per[:, i]) for i in range(4)]
        node = [rng.integers(0, n, r.size) for r in rep[:3]]
        node.append(np.minimum(np.searchsorted(cdf, rng.random(rep[3].size)), n - 1))
        size = [rng.geometric(1 / 3, r.size) for r in rep]
        if rep[0].size:
            a = rng.integers(0, a_n, rep[0].size)
            got = _take(pool, (rep[0] * n + node[0]) * a_n + a, size[0])
            emit(W.EXIT, T, rep[0], node[0], 0, got, exit_sel + a, -1)
        if rep[1].size:
            np.add.at(pool, (rep[1] * n + node[1]) * a_n, size[1])
            emit(W.ENTER, T, rep[1], node[1], 0, size[1], enter_sel, -1)
        if ageing and rep[2].size:
            a = rng.integers(0, a_n - 1, rep[2].size)
            key = (rep[2] * n + node[2]) * a_n + a
            got = _take(pool, key, size[2])
            np.add.at(pool, key + 1, got)
            emit(W.INTERNAL, T, rep[2], node[2], 0, got, exit_sel + a, a)
        if rep[3].size and n > 1:
            a = rng.integers(0, a_n, rep[3].size)
            dest = (node[3] + rng.integers(1, n, rep[3].size)) % n
            got = _take(pool, (rep[3] * n + node[3]) * a_n + a, size[3])
            np.add.at(pool, (rep[3] * n + dest) * a_n + a, got)
            emit(W.EXTERNAL, T, rep[3], node[3], dest, got, exit_sel + a, -1)
    ev = W.empty_events()
    if cols:
        for i, name in enumerate(("event", "time", "node", "dest", "n", "select", "shift")):
            ev[name] = np.concatenate([c[i] for c in cols])
        ev["proportion"] = np.zeros(ev["event"].size)
        if reps > 1:
            ev["rep"] = np.concatenate([c[7] for c in cols])
    return ev


def _sise(rng, case, seed, solver=W.SSM):
    """SISe on herds of median 50 with enter, exit and transfer events
    (0.41 a node-day), as the paper's 1,600-herd benchmark."""
    ages = _herds(rng, case["nodes"], 50, 1.0, 5000)[:, None]
    ev = _events(rng, ages, case["days"], 1, 0.41, MIX_SISE, 0, 2, False)
    w = W.plain_model(W.SISE, _seeded(rng, ages, 0.1), np.arange(case["days"] + 1),
                      W.sise_gdata(), seed=seed, n_rep=case["reps"], events=ev)
    w.solver = solver
    return w


def _sise_sp(rng, case, seed):
    """SISe with coupling between farms within 2,500 m; the farms' density is
    that of 1,600 in a square of 50 km."""
    n = case["nodes"]
    herd = _herds(rng, n, 50, 1.0, 5000)
    ev = _events(rng, herd[:, None], case["days"], 1, 0.41, MIX_SISE, 0, 2, False)
    infected = np.zeros(n, np.int64)
    j = rng.choice(n, size=max(1, n // 10), replace=False)
    infected[j] = (herd[j] * 0.05).astype(np.int64)
    side = 50000.0 * math.sqrt(n / 1600)
    w = W.plain_model(W.SISE_SP, np.stack([herd - infected, infected], 1),
                      np.arange(case["days"] + 1), W.sise_sp_gdata(), seed=seed,
                      n_rep=case["reps"], events=ev)
    w.neighbors = W.distance_neighbors(rng.uniform(0, side, n), rng.uniform(0, side, n), 2500.0)
    return w


def _sise3(rng, case, seed, own_events):
    """SISe3 herds with the cattle events (0.111 a node-day): the national
    population (median 60, up to 10,000 animals) or the batched one."""
    national = case["reps"] == 1
    herd = (_herds(rng, case["nodes"], 60, 1.2, 10000) if national
            else _herds(rng, case["nodes"], 50, 1.0, 5000))
    ages = W.split_ages(herd)
    ev = _events(rng, ages, case["days"], case["reps"] if own_events else 1, 0.111, MIX_SISE3,
                 0, 3, True)
    return W.plain_model(W.SISE3, _seeded(rng, ages, 0.1), np.arange(case["days"] + 1),
                         W.sise3_gdata(), seed=seed, n_rep=case["reps"], events=ev)


def _workload(case, seed):
    rng = np.random.default_rng(seed)
    f = case["family"]
    if f == "sir":
        # 100 animals a node, one of them (or a few) infected
        i = rng.integers(1, 4, case["nodes"])
        u0 = np.stack([100 - i, i, 0 * i], 1)
        return W.plain_model(W.SIR, u0, np.arange(1, case["days"] + 2), [0.16, 0.077],
                             seed=seed, n_rep=case["reps"])
    if f in ("simulate", "sise"):
        return _sise(rng, case, seed)
    if f == "aem":
        return _sise(rng, case, seed, W.AEM)
    if f == "sise_sp":
        return _sise_sp(rng, case, seed)
    if f == "predator_prey":
        w = W.config_predator_prey(case["nodes"], case["days"], seed=seed)
        w.u0 = (w.u0 + rng.integers(-20, 21, w.u0.shape)).astype(np.int32)
        return w
    if f == "sise3":
        return _sise3(rng, case, seed, case["reps"] > 1)
    if f == "prevalence":
        return _sise3(rng, case, seed, False)
    assert f == "endemic"
    return W.config_endemic(case["nodes"], case["days"], gen_seed=seed, seed=seed)


# -- emulator network -------------------------------------------------------

DIMS = [(256, 16), (256, 256), (256, 256), (392, 256)]
USED, BINS = 387, 129


def _network(seed):
    """FP32 weights of the emulator's 16-256-256-256-392 network."""
    g = torch.Generator().manual_seed(seed)
    ws, bs = [], []
    for layer, (o, i) in enumerate(DIMS):
        w = torch.randn(o, i, generator=g) * math.sqrt(2.0 / i) * (0.25 if layer == 3 else 1.0)
        b = 0.05 * torch.randn(o, generator=g)
        if layer == 3:
            w[USED:] = 0.0
            b[USED:] = 0.0
        ws.append(w)
        bs.append(b)
    return ws, bs


def _features(rows, seed):
    """BF16 input rows of nodes the emulator meets (counts, phi, rates), and
    the one-day increments it is trained on."""
    rng = np.random.default_rng(seed)
    u, phi = emulator.random_states(rng, rows)
    f = np.zeros((rows, 16), np.float32)
    f[:, :6] = np.log1p(u)
    f[:, 6] = phi
    f[:, 7:10] = 50 * 0.0173 * rng.uniform(0.5, 1.5, 3)
    f[:, 10:13] = 10 * 0.1 * rng.uniform(0.5, 1.5, 3)
    t = np.clip(np.rint(64 + 3 * rng.standard_normal((rows, 3))), 0, 128).astype(np.int32)
    return torch.from_numpy(f).to(torch.bfloat16), torch.from_numpy(t)


# --------------------------------------------------------------------------
# prepare, run
# --------------------------------------------------------------------------


def _prepare_emulator(case, seed):
    emu = emulator.Emulator("cuda", seed=0)
    for layer, (w, b) in enumerate(zip(*_network(seed))):
        emu.W32[layer].copy_(w)
        emu.W16[layer].copy_(w.to(torch.bfloat16))
        emu.b32[layer].copy_(b)
    f, t = _features(case["rows"], seed)
    state = dict(case=case, emu=emu, f=f.cuda(), t=t.cuda())
    if case.get("fp8"):
        emu.quantize_fp8(_features(4096, seed + 1)[0].cuda())
    return state


def prepare(case, seed):
    f = case["family"]
    if f.startswith("emu_"):
        return _prepare_emulator(case, seed)
    w = _workload(case, seed)
    if f == "simulate":
        return dict(case=case, w=w)  # the call takes numpy and gives numpy
    m = binding.Model(w)
    R, M, n = case["reps"], len(w.tspan), m.n_nodes
    state = dict(case=case, w=w, m=m,
                 u0=torch.as_tensor(np.ascontiguousarray(w.u0), device="cuda"),
                 v0=torch.as_tensor(np.ascontiguousarray(w.v0), device="cuda"),
                 U=None, V=None, stream=None)
    if f == "prevalence":
        # all counts of 100 herds (or all), and phi of them, at every day
        nodes = np.unique(np.linspace(0, n - 1, min(n, 100)).astype(np.int64))
        urow = (nodes[:, None] * m.n_comp + np.arange(m.n_comp)).reshape(-1)
        up = (np.arange(M + 1) * urow.size, np.tile(urow, M).astype(np.int32))
        vp = (np.arange(M + 1) * nodes.size, np.tile(nodes, M).astype(np.int32))
        state["uval"] = torch.empty((R, up[1].size), dtype=torch.int32, device="cuda")
        state["vval"] = torch.empty((R, vp[1].size), dtype=torch.float64, device="cuda")
        state["prev"] = torch.empty((R, M, 4), dtype=torch.int64, device="cuda")
        m.set_output(dense=False, n_tspan=M, u_pattern=up, u_values=state["uval"], v_pattern=vp,
                     v_values=state["vval"], prevalence=([1, 3, 5], range(6)),
                     prev_out=state["prev"])
    else:
        state["U"] = torch.empty((R, M, n, m.n_comp), dtype=torch.int32, device="cuda")
        state["V"] = torch.empty((R, M, n, m.n_v), dtype=torch.float64, device="cuda")
    if f not in ("sir", "predator_prey"):
        # the examples stay on the default stream; longer jobs use their own
        state["stream"] = torch.cuda.Stream()
    torch.cuda.synchronize()
    return state


def run(state):
    case = state["case"]
    f = case["family"]
    if f == "simulate":
        w = state["w"]
        U, V, st = binding.simulate(w)
        return dict(U=U, V=V, reactions=int(st["reactions"]))
    if f == "emu_gradients":
        loss, dW, db = state["emu"].gradients(state["f"], state["t"])
        return dict(loss=loss, dW=dW, db=db)
    if f == "emu_forward":
        emu = state["emu"]
        return emu.forward_fp8(state["f"]) if case["fp8"] else emu.forward(state["f"])[0]
    w = state["w"]
    rc, st, er = state["m"].run(w.tspan, w.seed, case["reps"], state["u0"], state["v0"],
                                state["U"], state["V"], stream=state["stream"])
    out = dict(reactions=int(st["reactions"]), events=int(st["events_applied"]))
    if f == "prevalence":
        out |= dict(uval=state["uval"], vval=state["vval"], prev=state["prev"])
    else:
        out |= dict(U=state["U"])
        if state["V"].numel():
            out |= dict(V=state["V"])
    return out


# --------------------------------------------------------------------------
# work, exact
# --------------------------------------------------------------------------


def work(case):
    f = case["family"]
    if f.startswith("emu_"):
        rows = case["rows"]
        weights = sum(o * i for o, i in DIMS)
        flops = 2.0 * rows * weights
        if f == "emu_forward":
            return dict(bytes=rows * (2 * 16 + 4 * 392) + weights * (1 if case["fp8"] else 2),
                        flops=flops)
        # forward, both products of the backward pass (none into the inputs)
        return dict(bytes=rows * (2 * 16 + 12) + 6 * weights,
                    flops=3 * flops - 2.0 * rows * DIMS[0][0] * DIMS[0][1])
    C, T, NV, rate = {"sir": (3, 2, 0, 0.0), "predator_prey": (2, 5, 0, 0.0),
                      "sise3": (6, 6, 1, 0.111), "prevalence": (6, 6, 1, 0.111),
                      "endemic": (6, 6, 1, 0.0)}.get(f, (2, 2, 1, 0.41))
    units = case["nodes"] * case["reps"]
    points = case["days"] + 1
    events = rate * case["nodes"] * case["days"]
    if f == "sise3":
        events *= case["reps"]
    if f == "prevalence":
        herds = min(case["nodes"], 100)
        written = case["reps"] * points * (herds * (4 * C + 8 * NV) + 32)
    else:
        written = units * points * (4 * C + 8 * NV)
    # each event once: type, node, destination, size, select, shift, time
    moved = units * (4 * C + 8 * NV) + written + 23 * events
    # expected draws a node-day (each one logarithm, one division, its rates)
    draws = {"sir": 4.0, "endemic": 100.0, "predator_prey": 4000.0}.get(f, 0.1)
    return dict(bytes=moved, flops=units * case["days"] * (8.0 + draws * (4 * T + 30)))


def _gelu(x):
    return torch.nn.functional.gelu(x, approximate="tanh")


def exact(case, seed):
    """The emulator network in 64 bits; a simulated path has no such value
    (its counts are compared as whole numbers)."""
    f = case["family"]
    if not f.startswith("emu_"):
        return None
    ws, bs = _network(seed)
    x, t = _features(case["rows"], seed)
    x, t = x.double().cuda(), t.long().cuda()
    used = []
    for layer, w in enumerate(ws):
        if case.get("fp8") and layer > 0:
            top = w.abs().amax(1, keepdim=True)
            scale = torch.where(top > 0, top / 448.0, torch.ones_like(top))
            w = (w / scale).to(torch.float8_e4m3fn).double() * scale.double()
        else:
            w = w.to(torch.bfloat16).double()
        used.append(w.cuda().requires_grad_(f == "emu_gradients"))
    bs = [b.double().cuda().requires_grad_(f == "emu_gradients") for b in bs]
    h = x
    for layer in range(3):
        h = _gelu(h @ used[layer].T + bs[layer])
    logits = h @ used[3].T + bs[3]
    if f == "emu_forward":
        return logits
    heads = logits[:, :USED].reshape(-1, 3, BINS)
    loss = -torch.log_softmax(heads, 2).gather(2, t[:, :, None]).sum() / case["rows"]
    loss.backward()
    return dict(loss=float(loss.item()), dW=[w.grad for w in used], db=[b.grad for b in bs])
