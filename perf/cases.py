"""Performance cases: the work a user of this framework has it do.

A case is a dict of plain values; its "kind" names the calls of one pass:

  window  one window of the minimum delay on a running network: step(n), the
          voltage of every compartment into a pinned host frame, and the
          spikes of the window (the recording loop of a simulation);
  state   the same with the gates and the synaptic conductances read too
          (a recording of the whole state);
  closed  one step of a loop with an outside world: new stimuli in, one time
          step, soma voltages and spikes out;
  hines   Algorithm 1 on a batch of trees in device memory (mm.hines_solve);
  cost    the learned cost model: its loss and gradient on the timed sample
          and its prediction for every neuron of the network.

Networks are drawn by the repository's generator with the repository's
parameters (tree shapes, cylinders, weights, stimuli) and have run for three
windows (120 steps) before the first pass, so that spikes and synaptic
events are under way.  FP64 networks return what the calls return; FP32c networks
keep their frames and spike times in single precision, the precision of
their increments.  Spikes are kept in a raster of
fixed size, ordered by neuron, compartment and time.
"""
import math

import numpy as np
import torch

from paper_2005_06332_gb300 import mm, netgen

WARM = 120  # steps before the first pass: three minimum delays of 1 ms


def _net(name, kind, neurons, dist, precision, syn, steps=40, p_lo=0.1, p_hi=0.1, mono=False, delay_lo=1.0,
         delay_hi=1.0, giants=0, giant_size=0, points=False, ordered=False):
    return dict(name=name, kind=kind, neurons=neurons, dist=dist, precision=precision, syn=syn, steps=steps, p_lo=p_lo,
                p_hi=p_hi, mono=mono, delay_lo=delay_lo, delay_hi=delay_hi, giants=giants, giant_size=giant_size,
                points=points, ordered=ordered)


def listed():
    return [
        # the smallest call: 64 identical neurons in a closed loop, where the latency of a step counts
        _net("closed_mono64", "closed", 64, "mono:255", "fp32c", 10, steps=1, mono=True),
        # the single-morphology network in plain FP64
        _net("mono64_fp64", "window", 64, "mono:255", "fp64", 10, mono=True),
        # a closed loop over a mid-size network
        _net("closed_multi2k", "closed", 2000, "loguniform:50:5000", "fp32c", 100, steps=1, p_lo=0.02, p_hi=0.2),
        # a small network of F-distributed sizes, an odd number of neurons, its whole state recorded
        _net("fisher333", "state", 333, "fisher:10:5000", "fp32c", 100),
        # the mix of 20 sizes (mean 300) of the load-balance test
        _net("multi20_10k", "window", 10000, "group:20:700:300", "fp32c", 100),
        # the multi-morphology network in plain FP64
        _net("multi2k_fp64", "window", 2000, "loguniform:50:5000", "fp64", 100, p_lo=0.02, p_hi=0.2),
        # the multi-morphology network in compensated FP32: the main workload
        _net("multi10k_fp32c", "window", 10000, "loguniform:50:5000", "fp32c", 100, p_lo=0.02, p_hi=0.2),
        # lognormal sizes with 1000 synapses per neuron
        _net("lognormal3k", "window", 3000, "lognormal:800:20000", "fp32c", 1000),
        # a mixed network with giant neurons and a spread of delays
        _net("mixed_giants", "window", 1500, "lognormal:1000:20000", "fp32c", 300, delay_lo=1.0, delay_hi=5.0, giants=2,
             giant_size=100000),
        # spikes detected at the synapse points, events added in a fixed order (reproducible runs), FP64
        _net("points_ordered_fp64", "state", 701, "loguniform:50:3000", "fp64", 100, p_lo=0.02, p_hi=0.2, points=True,
             ordered=True),
        # the standalone batched tree solve on trees of the main workload's sizes
        dict(name="hines_multi3k", kind="hines", trees=3000, lo=50, hi=5000, p_branch=0.1),
        # the cost model of the learned schedule: 5000 timed neurons, a network of 100,000
        dict(name="cost_model", kind="cost", timed=5000, neurons=100000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.random()
    if what < 0.12:
        return dict(kind="hines", trees=_log_int(rng, 16, 3000), lo=_log_int(rng, 8, 200), hi=_log_int(rng, 300, 5000),
                    p_branch=round(rng.uniform(0.02, 0.3), 3))
    if what < 0.2:
        return dict(kind="cost", timed=_log_int(rng, 300, 5000), neurons=_log_int(rng, 1000, 100000))
    precision = "fp64" if rng.random() < 0.3 else "fp32c"
    dist, most = rng.choice([("loguniform:50:5000", 10000), ("group:20:700:300", 10000), ("fisher:10:5000", 10000),
                             ("lognormal:800:20000", 3000), ("mono:%d" % _log_int(rng, 30, 1500), 5000)])
    if precision == "fp64":
        if dist.startswith("lognormal"):
            dist = "lognormal:800:8192"  # the largest neuron the FP64 path holds
        most = min(most, 1500)
    giants = rng.choice([1, 2]) if precision == "fp32c" and rng.random() < 0.15 else 0
    if giants:
        most = 1500
    neurons = _log_int(rng, 40, most)
    closed = giants == 0 and rng.random() < 0.25
    options = not closed and giants == 0 and neurons <= 1500
    points = options and rng.random() < 0.2
    p = sorted(round(rng.uniform(0.02, 0.2), 3) for _ in range(2))
    wide = rng.random() < 0.25
    c = _net("", "closed" if closed else ("state" if options and rng.random() < 0.3 else "window"), neurons, dist, precision,
             min(neurons - 1, _log_int(rng, 10, 400)), steps=1 if closed else rng.choice([40, 40, 20, 33]), p_lo=p[0],
             p_hi=p[1], delay_lo=1.0, delay_hi=5.0 if wide else 1.0, giants=giants,
             giant_size=_log_int(rng, 20000, 100000) if giants else 0, points=points,
             ordered=options and rng.random() < 0.3)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs

def _dist(text):
    kind, *v = text.split(":")
    v = [int(x) for x in v]
    return {"mono": lambda: ("mono", v[0]), "loguniform": lambda: ("loguniform", v[0], v[1]),
            "group": lambda: ("group", v[0], v[1], v[2]), "fisher": lambda: ("fisher", 10, 40, 300, v[0], v[1]),
            "lognormal": lambda: ("lognormal", v[0], 1.0, 20, v[1])}[kind]()


def _draw_trees(r, n, p):
    """Local parents of trees of n[k] compartments and branch probability p[k], by netgen.random_tree's rule."""
    i = np.arange(n.sum()) - np.repeat(np.cumsum(n) - n, n)
    jump = r.random(len(i)) < np.repeat(p, n)
    return np.where(jump, np.minimum((r.random(len(i)) * i).astype(np.int64), i - 1), i - 1).astype(np.int32)


def _network(case, seed):
    """netgen.make_network's recipe; the case fixes the neurons' sizes, the seed draws everything else."""
    n = netgen.draw_sizes(np.random.default_rng(netgen.SEED_BASE), case["neurons"], _dist(case["dist"]))
    n = np.concatenate([n, np.full(case["giants"], case["giant_size"], np.int64)])
    N, r = len(n), np.random.default_rng(seed)
    p = np.concatenate([r.uniform(case["p_lo"], case["p_hi"], case["neurons"]), np.full(case["giants"], 0.05)])
    own = 1 if case["mono"] else N  # identical neurons: one tree and its cylinders for all
    parent = _draw_trees(r, n[:own], p[:own])
    length, diam = r.uniform(5.0, 20.0, len(parent)), r.uniform(0.5, 2.0, len(parent))
    if case["mono"]:
        parent, length, diam = (np.tile(v, N) for v in (parent, length, diam))
    dst = np.repeat(np.arange(N, dtype=np.int32), case["syn"])
    src = r.integers(0, N - 1, len(dst))
    src = (src + (src >= dst)).astype(np.int32)
    return netgen.Network(
        comp_offset=np.concatenate([[0], np.cumsum(n)]), parent=parent, length_um=length, diam_um=diam,
        stim_nA=r.uniform(0.1, 0.5, N), syn_src=src, syn_dst=dst,
        syn_comp=r.integers(0, n[dst]).astype(np.int32), syn_w=r.uniform(0.0, 0.05, len(dst)),
        syn_delay_ms=r.uniform(case["delay_lo"], case["delay_hi"], len(dst)), params=dict(netgen.DEFAULT_PARAMS),
        syn_src_comp=r.integers(0, n[src]).astype(np.int32) if case["points"] else None)


def _new_stimulus(net, seed):
    return net.stim_nA * (0.8 + 0.4 * np.random.default_rng([seed, 1]).random(net.n_neurons))


def _trees(case, seed):
    """Offsets, local parents and the four coefficient arrays of a batch of random trees (diagonally dominant)."""
    n = netgen.draw_sizes(np.random.default_rng(netgen.SEED_BASE), case["trees"], ("loguniform", case["lo"], case["hi"]))
    r = np.random.default_rng(seed)
    off = np.concatenate([[0], np.cumsum(n)])
    parent = _draw_trees(r, n, np.full(len(n), case["p_branch"]))
    t = {"offset": torch.from_numpy(off).cuda(), "parent": torch.from_numpy(parent).cuda()}
    a, c, b, rhs = (torch.from_numpy(r.random(off[-1])).cuda() for _ in range(4))
    root = t["parent"] < 0
    t["a"] = -(0.1 + 0.9 * a).masked_fill_(root, 0.0)
    t["c"] = -(0.1 + 0.9 * c).masked_fill_(root, 0.0)
    t["b"] = 0.5 + 1.5 * b + 2.0 * (t["a"].abs() + t["c"].abs())
    t["rhs"] = 2.0 * rhs - 1.0
    return t


def _features(case, seed):
    """Features and log times of `neurons` neurons, their normalisation, and the parameters of a model in training."""
    r = np.random.default_rng(seed)
    mean, spread = r.uniform(0.0, 6.0, 16), r.uniform(0.2, 1.5, 16)
    X = (mean + spread * r.standard_normal((case["neurons"], 16))).astype(np.float32)
    y = (X[:, 0] - 0.3 * X[:, 6] + 0.1 * X[:, 1] * X[:, 2] + 0.2 * r.standard_normal(case["neurons"])).astype(np.float32)
    s = min(case["timed"], case["neurons"])
    mu, sd = X[:s].mean(0).astype(np.float32), X[:s].std(0).astype(np.float32)
    y_mu, y_sd = float(np.float32(y[:s].mean())), float(np.float32(y[:s].std()))
    theta = np.zeros(mm.MLP_PARAMS, np.float32)
    theta[:1024] = r.uniform(-0.6, 0.6, 1024)
    theta[1024:1088] = r.uniform(-0.1, 0.1, 64)
    theta[1088:5184] = r.uniform(-0.3, 0.3, 4096)
    theta[5184:5248] = r.uniform(-0.1, 0.1, 64)
    theta[5248:5312] = r.uniform(-0.3, 0.3, 64)
    theta[5312] = 0.05
    return X, y, s, mu, sd, y_mu, y_sd, theta


def prepare(case, seed):
    if case["kind"] == "hines":
        return {"kind": "hines", **_trees(case, seed)}
    if case["kind"] == "cost":
        X, y, s, mu, sd, y_mu, y_sd, theta = _features(case, seed)
        mlp = mm.MLP(seed=1)
        mlp.set_params(theta)
        mlp.set_normalisation(mu, sd, y_mu, y_sd)
        return {"kind": "cost", "mlp": mlp, "X": X, "Xt": X[:s].copy(), "yt": y[:s].copy()}
    net = _network(case, seed)
    sim = mm.Network(net, precision=case["precision"], detect="points" if case["points"] else "soma",
                     deterministic=case["ordered"])
    sim.step(WARM)
    sim.read_spike_points()
    single = case["precision"] == "fp32c"
    st = {"kind": case["kind"], "sim": sim, "steps": case["steps"], "single": single, "held": _held(case)}
    if case["kind"] == "closed":
        st["stim"] = _new_stimulus(net, seed)
        st["soma"] = torch.empty(net.n_neurons, dtype=torch.float64, pin_memory=True)
        return st
    which = ("V", "m", "h", "n", "gsyn") if case["kind"] == "state" else ("V",)
    st["frame"] = {w: torch.empty(net.n_comp, dtype=torch.float64, pin_memory=True) for w in which}
    st["out"] = {w: torch.empty(net.n_comp, dtype=torch.float32) for w in which} if single \
        else st["frame"]
    return st


def _held(case):
    """Spikes the raster of a pass has room for: two per neuron, or one per synapse point."""
    return max(2 * (case["neurons"] + case["giants"]), case["neurons"] * case["syn"] if case["points"] else 0)


def _raster(spikes, held, single):
    nrn, comp, t = spikes
    k = np.lexsort((t, comp, nrn))[:held]
    out = {"neuron": np.full(held, -1, np.int32), "comp": np.full(held, -1, np.int32),
           "t": np.full(held, -1.0, np.float32 if single else np.float64)}
    out["neuron"][:len(k)], out["comp"][:len(k)], out["t"][:len(k)] = nrn[k], comp[k], t[k]
    return out


# -------------------------------------------------------------------- pass

def run(st):
    if st["kind"] == "hines":
        return mm.hines_solve(st["offset"], st["parent"], st["a"], st["b"], st["c"], st["rhs"])
    if st["kind"] == "cost":
        loss, grad = st["mlp"].loss_grad(st["Xt"], st["yt"])
        return {"loss": loss, "grad": grad, "y": st["mlp"].predict(st["X"])}
    sim, single = st["sim"], st["single"]
    if st["kind"] == "closed":
        sim.set_stimulus(st["stim"])
        sim.step(1)
        soma, spikes = sim.read_outputs(st["soma"].numpy())
        return {"soma": st["soma"].float() if single else st["soma"], **_raster(spikes, st["held"], single)}
    sim.step(st["steps"])
    for w, f in st["frame"].items():
        sim.read_state(w, f.numpy())
        if single:
            st["out"][w].copy_(f)
    return {**st["out"], **_raster(sim.read_spike_points(), st["held"], single)}


# -------------------------------------------------------------------- work

def _mean_size(text):
    d = _dist(text)
    if d[0] == "mono":
        return d[1]
    if d[0] == "loguniform":
        return (d[2] - d[1]) / math.log(d[2] / d[1])
    if d[0] == "lognormal":
        return d[1] * math.exp(0.5) * 0.98
    return d[3]


def work(case):
    if case["kind"] == "hines":
        comps = case["trees"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        return {"bytes": comps * (4 + 4 * 8 + 8), "flops": comps * 8}
    if case["kind"] == "cost":
        macs = 16 * 64 + 64 * 64 + 64
        return {"bytes": (case["timed"] * 17 + case["neurons"] * 17 + 2 * mm.MLP_PARAMS) * 4,
                "flops": case["timed"] * macs * 6 + case["neurons"] * macs * 2}
    comps = case["neurons"] * _mean_size(case["dist"]) + case["giants"] * case["giant_size"]
    syn = (case["neurons"] + case["giants"]) * case["syn"]
    word = 8 if case["precision"] == "fp64" else 4
    # the state (V, m, h, n) in and out, area, coupling and diagonal in, per synapse its conductance in and out;
    # the outputs.  Operations: about 90 per compartment and step (45 for the gates, counting an exponential as
    # one, 25 for the currents, 20 for assembly and solve)
    outs = {"closed": case["neurons"] * 8, "window": comps * word, "state": comps * 5 * word}[case["kind"]]
    return {"bytes": comps * 11 * word + syn * 2 * word + outs, "flops": comps * case["steps"] * 90}


# ------------------------------------------------- the same in 64 bits, plainly

def _levels(parent):
    """Compartments sorted by depth: (order, parent position in that order, level offsets); parent: global, -1 at roots."""
    depth = (parent >= 0).long()
    anc = parent.clone()
    while bool((anc >= 0).any()):
        up = anc.clamp_min(0)
        depth = depth + torch.where(anc >= 0, depth[up], 0)
        anc = torch.where(anc >= 0, anc[up], -1)
    order = torch.argsort(depth, stable=True)
    pos = torch.empty_like(order)
    pos[order] = torch.arange(order.numel(), device=order.device)
    par = parent[order]
    par = torch.where(par >= 0, pos[par.clamp_min(0)], 0)
    off = [0] + torch.cumsum(torch.bincount(depth), 0).tolist()
    return order, pos, par, off


def _tree_solve(par, off, a, c, d, r):
    """Algorithm 1 level by level, in place; the solution replaces r."""
    for l in range(len(off) - 2, 0, -1):
        s, e = off[l], off[l + 1]
        f = a[s:e] / d[s:e]
        d.index_add_(0, par[s:e], f * c[s:e], alpha=-1.0)
        r.index_add_(0, par[s:e], f * r[s:e], alpha=-1.0)
    r[:off[1]] /= d[:off[1]]
    for l in range(1, len(off) - 1):
        s, e = off[l], off[l + 1]
        r[s:e] = (r[s:e] - c[s:e] * r[par[s:e]]) / d[s:e]


def _exact_hines(case, seed):
    t = _trees(case, seed)
    off, p = t["offset"], t["parent"].long()
    base = torch.repeat_interleave(off[:-1], off[1:] - off[:-1])
    order, pos, par, lev = _levels(torch.where(p >= 0, p + base, -1))
    a, b, c, r = (t[k][order] for k in ("a", "b", "c", "rhs"))
    _tree_solve(par, lev, a, c, b, r)
    return r[pos]


def _exact_cost(case, seed):
    X, y, s, mu, sd, y_mu, y_sd, theta = _features(case, seed)
    th = torch.from_numpy(theta).bfloat16().double().requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = (v.reshape(sh) for v, sh in zip(
        torch.split(th, [1024, 64, 4096, 64, 64, 1]), [(64, 16), (64,), (64, 64), (64,), (64,), ()]))
    Z = (torch.from_numpy(X).double() - torch.from_numpy(mu).double()) / torch.from_numpy(sd).double()

    def model(z):
        return torch.relu(torch.relu(z @ W1.T + b1) @ W2.T + b2) @ W3 + b3
    loss = ((model(Z[:s]) - (torch.from_numpy(y[:s]).double() - y_mu) / y_sd) ** 2).mean()
    loss.backward()
    return {"loss": float(loss), "grad": th.grad.numpy(), "y": (model(Z) * y_sd + y_mu).detach().numpy()}


def _ratio(x):  # x / (e^x - 1)
    return torch.where(x.abs() < 1e-6, 1.0 - 0.5 * x, x / torch.expm1(torch.where(x.abs() < 1e-6, 1.0, x)))


def _rates(v):
    return ((_ratio(-(v + 40.0) * 0.1), 4.0 * torch.exp(-(v + 65.0) / 18.0)),
            (0.07 * torch.exp(-(v + 65.0) * 0.05), 1.0 / (1.0 + torch.exp(-(v + 35.0) * 0.1))),
            (0.1 * _ratio(-(v + 55.0) * 0.1), 0.125 * torch.exp(-(v + 65.0) * 0.0125)))


def _exact_network(case, seed):
    net = _network(case, seed)
    p, dt = net.params, net.dt
    dev = lambda v: torch.from_numpy(np.ascontiguousarray(v)).cuda()  # noqa: E731
    size = np.diff(net.comp_offset)
    base = np.repeat(net.comp_offset[:-1], size)
    order, pos, par, lev = _levels(dev(np.where(net.parent >= 0, net.parent + base, -1)))
    L, D = dev(net.length_um)[order], dev(net.diam_um)[order]
    area = math.pi * D * L * 1e-8
    half = p["Ra"] * (0.5e-4 * L) / (math.pi * (0.5e-4 * D) ** 2) * 1e-6
    g = 1.0 / (half + half[par])
    g[:lev[1]] = 0.0
    passive = area * (p["Cm"] * 1e3 / dt) + g
    passive.index_add_(0, par, g)
    soma = pos[dev(net.comp_offset[:-1])]
    # synapses: target, source point (a soma, or the compartment it leaves from), delay in steps, weight
    target = pos[dev(net.comp_offset[net.syn_dst] + net.syn_comp)]
    at = net.comp_offset[net.syn_src] + (net.syn_src_comp if case["points"] else 0)
    point, source = (np.unique(at, return_inverse=True) if case["points"] else (net.comp_offset[:-1], net.syn_src))
    nrn = np.searchsorted(net.comp_offset, point, side="right") - 1
    comp, source, where = dev(point - net.comp_offset[nrn]), dev(source.astype(np.int64)), pos[dev(point)]
    nrn = dev(nrn)
    delay = dev(np.floor(net.syn_delay_ms / dt + 0.5).astype(np.int64))
    weight = dev(net.syn_w)
    V = torch.full_like(area, p["v_init"])
    gates = [a / (a + b) for a, b in _rates(V)]
    gs = torch.zeros_like(V)
    stim = dev(net.stim_nA)
    fired = torch.zeros((int(delay.max()) + 1 if len(delay) else 1, len(where)), dtype=torch.bool, device="cuda")
    decay = math.exp(-dt / p["tau_syn"])
    d, r = torch.empty_like(V), torch.empty_like(V)

    def currents():
        m, h, n = gates
        s = area * 1e3
        ga, gk, gl = p["gNa"] * s * m ** 3 * h, p["gK"] * s * n ** 4, p["gL"] * s
        d.copy_(passive + ga + gk + gl + gs)
        r.copy_(-(ga * (V - p["ENa"]) + gk * (V - p["EK"]) + gl * (V - p["EL"]) + gs * (V - p["e_syn"])))
        axial = g * (V[par] - V)
        r.add_(axial)
        r.index_add_(0, par, axial, alpha=-1.0)
        r.index_add_(0, soma, stim)

    solve = torch.cuda.CUDAGraph()
    with torch.cuda.graph(solve):
        _tree_solve(par, lev, -g, -g, d, r)
    spikes = []
    for n in range(WARM + case["steps"]):
        if case["kind"] == "closed" and n == WARM:
            stim = dev(_new_stimulus(net, seed))
        if len(delay):
            hit = fired[(n - 1 - delay) % fired.shape[0], source]
            gs.index_add_(0, target, weight * hit)
        currents()
        solve.replay()
        old = V[where]
        V = V + r
        gs *= decay
        gates = [a / (a + b) + (x - a / (a + b)) * torch.exp(-dt * (a + b)) for x, (a, b) in zip(gates, _rates(V))]
        new = V[where]
        up = (old < p["threshold"]) & (new >= p["threshold"])
        fired[n % fired.shape[0]] = up
        if n >= WARM:
            k = up.nonzero()[:, 0]
            spikes.append((nrn[k], comp[k], n * dt + dt * (p["threshold"] - old[k]) / (new[k] - old[k])))
    raster = _raster(tuple(torch.cat([s[j] for s in spikes]).cpu().numpy() for j in range(3)), _held(case), False)
    if case["kind"] == "closed":
        return {"soma": V[soma], **raster}
    state = {"V": V, "m": gates[0], "h": gates[1], "n": gates[2], "gsyn": gs}
    return {**{w: state[w][pos] for w in (state if case["kind"] == "state" else ("V",))}, **raster}


def exact(case, seed):
    if case["kind"] == "hines":
        return _exact_hines(case, seed)
    if case["kind"] == "cost":
        return _exact_cost(case, seed)
    return _exact_network(case, seed)
