"""The measured calls of this framework: what a user's program runs, through the public entry points.

A case names a batch of graphs (family, size, count), a depth, a number of parameter points and the call:

* ``energy``   ``Plan.energy(theta)``, a landscape scan or a line search;
* ``terms``    ``Plan.energy(theta, terms=True)``, every edge's <ZZ>, as RQAOA reads it each round;
* ``grad``     ``Plan.energy_grad(theta)``, a caller with an optimiser of its own;
* ``train``    ``qaoa_energy(theta, plan)`` and ``loss.backward()``, the step of a torch training loop;
* ``graph``    ``Plan.graph(theta).run(theta)``, a captured evaluation replayed with new points;
* ``noalloc``  ``Plan.energy_noalloc(theta, out)``, callers that may not allocate.

``plan`` is ``orbits`` (the default plan) or ``plain`` (every edge its own representative, for graphs whose
symmetry is not worth searching, and wherever one term per edge is wanted).  The random graphs and the points
follow the seed; the families and depths are those of the benchmark configurations and tests.
"""
import math

import numpy as np
import torch

from paper_2101_10296_gb300 import inputs, qaoa


def _case(name, family, n, count, p, points, call, plan="orbits", signs=False):
    c = {"family": family, "n": n, "count": count, "p": p, "points": points, "call": call, "plan": plan,
         "signs": signs}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one point of one tiny graph: what a call costs when nearly nothing is computed
        _case("circulant20_p1_one_point", "circulant_1_4", 20, 1, 1, 1, "energy"),
        # the benchmark-shaped batch: 48 graphs of 100 to 10,000 vertices, replayed as a captured evaluation
        _case("mix48_p1_replay", "mix48", 0, 48, 1, 256, "graph"),
        # a large irregular graph without a symmetry search, every edge its own cone
        _case("random10000_p1_plain_grad", "er4", 10000, 1, 1, 101, "grad", "plain"),
        # RQAOA's reading of every edge's correlation at a few optimised points
        _case("cubic1000_p2_terms", "rr3", 1000, 1, 2, 3, "terms", "plain"),
        # a landscape of four cubic graphs, forward only
        _case("cubic2000x4_p2_energy", "rr3", 2000, 4, 2, 64, "energy"),
        # the same graphs in a training loop
        _case("cubic2000x4_p2_train", "rr3", 2000, 4, 2, 64, "train"),
        # a signed (Ising) objective
        _case("signed2000_p2_grad", "rr3", 2000, 1, 2, 33, "grad", "orbits", True),
        # a very symmetric graph of 10,000 vertices: a few cones, many points
        _case("torus100_p2_grad", "torus", 100, 1, 2, 32, "grad"),
        # the allocation-free entry point on a small torus
        _case("torus8_p2_noalloc", "torus", 8, 1, 2, 128, "noalloc"),
        # cones of up to 24 qubits with their gradients: states beyond one thread's registers
        _case("cubic24x4_p3_grad", "rr3", 24, 4, 3, 25, "grad"),
        # a 28-qubit cone: blocks of 2^18 amplitudes streamed through memory
        _case("torus6_p3_energy", "torus", 6, 1, 3, 32, "energy"),
        # a deeper circuit on a band graph, whose later layers mix more than a tile holds
        _case("circulant30_p4_grad", "circulant_1_2", 30, 1, 4, 64, "grad"),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["p1", "p1", "p2", "p2", "p2", "p3", "p3", "p4"])
    if kind == "p1":
        family = rng.choice(["er4", "rr3", "rr4", "circulant_1_7", "torus", "cube"])
        n = {"torus": _log_int(rng, 5, 100), "cube": rng.randint(5, 12)}.get(family) or 2 * _log_int(rng, 12, 5000)
        call = rng.choice(["energy", "terms", "grad", "train", "graph", "noalloc"])
        plan = "plain" if call == "terms" else rng.choice(["orbits", "plain"])
        return _case(None, family, n, rng.randint(1, 3), 1, _log_int(rng, 1, 100), call, plan)
    if kind == "p2":
        family = rng.choice(["rr3", "rr3", "rr3", "torus", "circulant_1_7"])
        call = rng.choice(["energy", "terms", "grad", "grad", "train", "graph", "noalloc"])
        if family == "rr3":
            n, count = 2 * _log_int(rng, 30, 1000), rng.randint(1, 4)
            plan = "plain" if call == "terms" else rng.choice(["orbits", "plain"])
            signs = rng.random() < 0.3
            points = _log_int(rng, 1, 16 if signs else 48)
            return _case(None, family, n, 1 if signs else count, 2, points, call, plan, signs)
        n = _log_int(rng, 7, 100) if family == "torus" else _log_int(rng, 40, 5000)
        call = "energy" if call == "terms" else call
        return _case(None, family, n, 1, 2, _log_int(rng, 1, 128), call)
    if kind == "p3":
        call = rng.choice(["energy", "grad", "train"])
        if rng.random() < 0.7:
            return _case(None, "rr3", 2 * rng.randint(8, 12), rng.randint(1, 4), 3, _log_int(rng, 1, 24), call,
                         rng.choice(["orbits", "plain"]))
        return _case(None, "torus", rng.choice([5, 6]), 1, 3, _log_int(rng, 1, 24 if call == "energy" else 8), call)
    return _case(None, "circulant_1_2", rng.randint(21, 60), 1, 4, _log_int(rng, 1, 64),
                 rng.choice(["energy", "grad", "train", "graph"]))


# ---------------------------------------------------------------- inputs

def _graphs(case, seed):
    f, n = case["family"], case["n"]
    if f == "mix48":
        return [b() for _, b in inputs.mixed_benchmark_graphs()]
    out = []
    for k in range(case["count"]):
        s = 97 * seed + k + 1
        if f == "er4":
            out.append(inputs.erdos_renyi(n, 4.0 / (n - 1), s))
        elif f in ("rr3", "rr4"):
            out.append(inputs.random_regular(n, int(f[2]), s))
        elif f == "torus":
            out.append(inputs.torus(n, n + k))
        elif f == "cube":
            out.append(inputs.hypercube(n + k if n + k <= 12 else n))
        else:
            out.append(inputs.circulant(n + k, [int(j) for j in f.split("_")[1:]]))
    return out


def _weights(case, graphs, seed):
    if not case["signs"]:
        return None
    return [np.random.default_rng(31 * seed + k + 7).choice([1, -1], len(e)) for k, (_, e) in enumerate(graphs)]


def _theta(case, seed):
    return np.stack([inputs.draw_params(case["p"], case["points"], 1009 * seed + k + 1)
                     for k in range(case["count"])])


def prepare(case, seed):
    graphs = _graphs(case, seed)
    plan = qaoa.Plan(graphs, case["p"], orbits=case["plan"] == "orbits", weights=_weights(case, graphs, seed))
    plan.upload()
    theta = torch.tensor(_theta(case, seed), device="cuda")
    state = {"call": case["call"], "plan": plan, "theta": theta}
    if case["call"] == "graph":
        state["graph"] = plan.graph(theta)
    elif case["call"] == "train":
        theta.requires_grad_(True)
    elif case["call"] == "noalloc":
        state["out"] = torch.empty(case["count"], case["points"], dtype=torch.float64, device="cuda")
    return state


def run(state):
    plan, theta, call = state["plan"], state["theta"], state["call"]
    if call == "energy":
        return plan.energy(theta)
    if call == "terms":
        return plan.energy(theta, terms=True)
    if call == "grad":
        return plan.energy_grad(theta)
    if call == "graph":
        return state["graph"].run(theta)
    if call == "noalloc":
        return plan.energy_noalloc(theta, out=state["out"])
    theta.grad = None
    e = qaoa.qaoa_energy(theta, plan)
    (-e.sum()).backward()
    return e.detach(), theta.grad


def work(case):
    """Parameters in and results out once; every cone that differs from the others evolved once per point.

    Operations per amplitude of an inner block: 4 for each qubit a layer mixes, 6 for each phase after the first
    (the first is a table entry), 4 for the observable; a gradient by reverse differentiation takes three times
    the forward sweep.
    """
    p, P = case["p"], case["points"]
    graphs = _graphs(case, 0)
    plan = qaoa.Plan(graphs, p, cone_classes=True, weights=_weights(case, graphs, 0))
    reps, blocks = plan.reps(), plan.shell_blocks()
    mix = reps["mix_qubits"].sum(axis=1).astype(np.float64)
    fwd = float((blocks * np.ldexp(1.0, reps["n_inner"]) * (4 * mix + 6 * (p - 1) + 4)).sum()) * P
    grad = case["call"] in ("grad", "train", "graph")
    m = sum(len(e) for _, e in graphs) if case["call"] == "terms" else 0
    rows = len(graphs) * P
    return {"bytes": 8.0 * (rows * 2 * p + rows + (rows * 2 * p if grad else 0) + m * P),
            "flops": fwd * (3 if grad else 1)}


# ---------------------------------------------------------------- values in 64 bits
# Plain torch on whole states, from the definition: |+>, then per layer exp(-i gamma C) and exp(-i beta X).

def _bit(n, q, device):
    return (torch.arange(1 << n, device=device, dtype=torch.int32) >> q) & 1


def _cut(n, edges, weights, device):
    c = torch.zeros(1 << n, device=device, dtype=torch.int32)
    for (a, b), w in zip(edges, weights):
        c += int(w) * (_bit(n, int(a), device) ^ _bit(n, int(b), device))
    return c


def _phase(psi, cut, gamma, lo, hi):
    tab = torch.polar(torch.ones(1, dtype=torch.float64, device=psi.device),
                      -gamma[:, None] * torch.arange(lo, hi + 1, device=psi.device, dtype=torch.float64)[None])
    psi *= tab[:, cut - lo]


def _halves(psi, q):
    v = psi.view(psi.shape[0], -1, 2, 1 << q)
    return v[:, :, 0], v[:, :, 1]


def _mix(psi, q, cos, isin):
    a, b = _halves(psi, q)
    t = a * cos
    t -= b * isin
    b *= cos
    b -= a * isin
    a.copy_(t)


def _imdot(lam, psi):
    """Im <lam|psi> per point."""
    return (lam.real * psi.imag - lam.imag * psi.real).flatten(1).sum(1)


def _state_values(n, edges, weights, obs, mixed, theta, grad):
    """<obs> (diagonal) and its derivatives for the circuit whose layer l mixes the qubits mixed[l]."""
    device = theta.device
    p = theta.shape[1] // 2
    cut = _cut(n, edges, weights, device)
    lo, hi = int(cut.min()), int(cut.max())
    val = torch.empty(theta.shape[0], dtype=torch.float64, device=device)
    der = torch.zeros_like(theta) if grad else None
    step = max(1, (1 << 26) >> n)
    for j in range(0, theta.shape[0], step):
        th = theta[j:j + step]
        B = th.shape[0]
        psi = torch.full((B, 1 << n), 2.0 ** (-n / 2), dtype=torch.complex128, device=device)
        cos = torch.cos(th[:, p:])
        isin = 1j * torch.sin(th[:, p:])
        for l in range(p):
            _phase(psi, cut, th[:, l], lo, hi)
            for q in mixed[l]:
                _mix(psi, q, cos[:, l, None, None], isin[:, l, None, None])
        val[j:j + B] = (torch.view_as_real(psi).square().sum(-1) * obs).sum(1)
        if not grad:
            continue
        lam = psi * obs
        for l in reversed(range(p)):
            for q in mixed[l]:
                (a, b), (la, lb) = _halves(psi, q), _halves(lam, q)
                der[j:j + B, p + l] += 2 * (_imdot(la, b) + _imdot(lb, a))
            for q in mixed[l]:
                for s in (psi, lam):
                    _mix(s, q, cos[:, l, None, None], -isin[:, l, None, None])
            der[j:j + B, l] = 2 * _imdot(lam, psi * cut)
            for s in (psi, lam):
                _phase(s, cut, -th[:, l], lo, hi)
    return val, der


def _ball(adj, u, v, p):
    """The edge's cone, with its vertices ordered by how they hang on those before them, so that equal cones get
    equal descriptions: (vertices, distances, local edges, their weights)."""
    pos, dist = {u: 0, v: 1}, [0, 0]
    frontier = [u, v]
    for d in range(1, p + 1):
        seen = {}
        for a in frontier:
            for b, w in adj[a]:
                if b not in pos:
                    seen.setdefault(b, []).append((pos[a], w))
        frontier = sorted(seen, key=lambda b: (sorted(seen[b]), b))
        for b in frontier:
            pos[b] = len(dist)
            dist.append(d)
    loc = sorted((pos[a], pos[b], w) for a in pos for b, w in adj[a]
                 if b in pos and pos[a] < pos[b] and min(dist[pos[a]], dist[pos[b]]) < p)
    return len(dist), tuple(dist), tuple(loc)


def _reps(case, graph, k):
    """(edge index, multiplicity): one edge per translation class of the regular families, else every edge."""
    n, e = graph
    f = case["family"]
    if case["call"] != "terms" and (f == "torus" or f.startswith("circulant")):
        if f == "torus":
            cols = case["n"] + k
            steps = [1, cols]
        else:
            steps = [int(j) for j in f.split("_")[1:]]
        index = {(int(a), int(b)): i for i, (a, b) in enumerate(e)}
        return [(index[(0, s)], n) for s in steps]
    return [(i, 1) for i in range(len(e))]


def _cone_values(case, graph, weights, theta, k, grad):
    """Energy, gradient and per-edge <ZZ> of one graph from its cones, equal cones evaluated once."""
    n, e = graph
    w = np.ones(len(e), dtype=np.int64) if weights is None else weights
    p = case["p"]
    adj = [[] for _ in range(n)]
    for (a, b), we in zip(e.tolist(), w.tolist()):
        adj[a].append((b, we))
        adj[b].append((a, we))
    groups = {}
    for i, mult in _reps(case, graph, k):
        groups.setdefault(_ball(adj, int(e[i][0]), int(e[i][1]), p), []).append((i, mult))
    energy = torch.full((theta.shape[0],), 0.5 * float(w.sum()), dtype=torch.float64, device=theta.device)
    der = torch.zeros_like(theta)
    terms = torch.zeros(len(e), theta.shape[0], dtype=torch.float64, device=theta.device)
    for (nq, dist, loc), members in groups.items():
        mixed = [[q for q in range(nq) if dist[q] <= p - 1 - l] for l in range(p)]
        obs = 1.0 - 2.0 * (_bit(nq, 0, theta.device) ^ _bit(nq, 1, theta.device)).to(torch.float64)
        t, dt = _state_values(nq, [x[:2] for x in loc], [x[2] for x in loc], obs, mixed, theta, grad)
        tot = float(sum(mult * int(w[i]) for i, mult in members))
        energy -= 0.5 * tot * t
        if grad:
            der -= 0.5 * tot * dt
        for i, _ in members:
            terms[i] = t
    return energy, der, terms


def _p1_values(graph, theta):
    """Depth 1 in closed form: per edge from its ends' other neighbours and the triangles on it."""
    n, e = graph
    nb = [set() for _ in range(n)]
    for a, b in e.tolist():
        nb[a].add(b)
        nb[b].add(a)
    sig = [(min(len(nb[a]), len(nb[b])) - 1, max(len(nb[a]), len(nb[b])) - 1, len(nb[a] & nb[b]))
           for a, b in e.tolist()]
    kinds = sorted(set(sig))
    row = {s: i for i, s in enumerate(kinds)}
    th = theta.detach().clone().requires_grad_(True)
    g, b = th[:, 0], th[:, 1]
    s2, c2 = torch.sin(2 * b), torch.cos(2 * b)
    zz = []
    for du, dv, f in kinds:
        pair = 0.5 * (torch.cos(g) ** (du + dv - 2 * f) * (1 - torch.cos(2 * g) ** f))
        zz.append(s2 * s2 * pair - s2 * c2 * torch.sin(g) * (torch.cos(g) ** du + torch.cos(g) ** dv))
    zz = torch.stack(zz)
    rows = torch.tensor([row[s] for s in sig], device=theta.device)
    count = torch.bincount(rows, minlength=len(kinds)).to(torch.float64)
    energy = 0.5 * (count[:, None] * (1 - zz)).sum(0)
    (der,) = torch.autograd.grad(energy.sum(), th)
    return energy.detach(), der, zz.detach()[rows]


def exact(case, seed):
    graphs = _graphs(case, seed)
    weights = _weights(case, graphs, seed)
    device = "cuda" if torch.cuda.is_available() else "cpu"
    theta = torch.tensor(_theta(case, seed), device=device)
    p, call = case["p"], case["call"]
    grad = call in ("grad", "train", "graph")
    es, gs, ts = [], [], []
    for k, graph in enumerate(graphs):
        n, e = graph
        if p == 1 and weights is None:
            en, der, t = _p1_values(graph, theta[k])
        elif p >= 3 and n <= 24:
            w = np.ones(len(e), dtype=np.int64)
            obs = _cut(n, e, w, device).to(torch.float64)
            en, der = _state_values(n, e, w, obs, [range(n)] * p, theta[k], grad)
            t = None
        else:
            en, der, t = _cone_values(case, graph, None if weights is None else weights[k], theta[k], k, grad)
        es.append(en)
        gs.append(der)
        ts.append(t)
    energy = torch.stack(es)
    if call in ("energy", "noalloc"):
        return energy
    if call == "terms":
        return energy, torch.cat(ts)
    der = torch.stack(gs)
    return energy, -der if call == "train" else der
