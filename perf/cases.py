"""What the framework is measured on: belief propagation runs through its public entry points.

A case is one call as a user's program makes it, on a graph compiled beforehand: the
smallest grid that fits one thread block, grids that fit a few or all SMs, graphs with
more states per variable, batches of uneven graphs, many evidence sets of one graph,
high-degree variables, logical factors, listed configurations, a gradient, a call from
host buffers and a burst of serving requests. Message and belief arrays come back whole.
Runs in the chaotic regime (max-product over hundreds of iterations) are kept to
iteration counts at which two rounding orders still agree.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2202_04110_gb300 import binding
from paper_2202_04110_gb300 import workloads as W

DAMPING = 0.5


def listed():
    return [
        # a program that queries a small model in a loop: launches and latency count
        {"name": "grid 10x10", "kind": "grid", "rows": 10, "cols": 10, "T": 1.0, "iters": 50},
        # an image-sized MAP query, sides that no tile divides
        {"name": "grid 317x241 max", "kind": "grid", "rows": 317, "cols": 241, "T": 0.0, "iters": 50},
        # the large single model: marginals of a million variables
        {"name": "grid 1000x1000", "kind": "grid", "rows": 1000, "cols": 1000, "T": 1.0, "iters": 200},
        # a training step: beliefs and their gradient with respect to couplings and fields
        {"name": "gradient 64x64", "kind": "grad", "rows": 64, "cols": 64, "iters": 100, "ckpt": 10},
        # one multi-label image model with a shared table
        {"name": "potts 181 K16", "kind": "potts", "side": 181, "K": 16, "T": 1.0, "iters": 100},
        # many uneven models and a restricted Boltzmann machine at once
        {"name": "batch 128+rbm", "kind": "batch", "grids": 128, "hi": 256, "n_vis": 784, "n_hid": 500, "iters": 60},
        # a restricted Boltzmann machine alone: every variable has hundreds of factors
        {"name": "rbm 784x500", "kind": "rbm", "n_vis": 784, "n_hid": 500, "T": 1.0, "iters": 100},
        # deconvolution of a set of images with OR / AND factors, max-product
        {"name": "deconvolution 100", "kind": "deconv", "images": 100, "iters": 10},
        # lateral layer of pools: large listed-configuration factors, max-product
        {"name": "pool 128 K49", "kind": "pool", "side": 128, "radius": 3, "slack": 1, "T": 0.0, "iters": 20},
        # one model, many observations at once
        {"name": "evidence 32 x 256x256", "kind": "multi", "rows": 256, "cols": 256, "K": 2, "samples": 32, "iters": 100},
        # a program whose data are in host memory: copies in and out count
        {"name": "host 500x500", "kind": "host", "rows": 500, "cols": 500, "T": 1.0, "iters": 100},
        # a burst of requests of every size at the serving loop
        {"name": "serve 16", "kind": "serve", "requests": 16, "hi": 512},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid", "grid", "grid", "grad", "potts", "potts", "batch", "rbm", "deconv", "pool", "multi", "multi", "host", "serve"])
    T = rng.choice([0.0, 1.0])
    if kind == "grid":
        return {"kind": kind, "rows": _log(rng, 3, 1200), "cols": _log(rng, 3, 1200), "T": T,
                "iters": rng.randint(20, 200) if T else rng.randint(20, 60)}
    if kind == "grad":
        return {"kind": kind, "rows": _log(rng, 8, 200), "cols": _log(rng, 8, 200), "iters": rng.randint(20, 120), "ckpt": rng.choice([5, 10, 16])}
    if kind == "potts":
        return {"kind": kind, "side": _log(rng, 16, 256), "K": rng.choice([4, 8, 16]), "T": T,
                "iters": rng.randint(20, 120) if T else rng.randint(10, 30)}
    if kind == "batch":
        return {"kind": kind, "grids": _log(rng, 8, 100), "hi": rng.randint(64, 256), "n_vis": _log(rng, 50, 784), "n_hid": _log(rng, 50, 500),
                "iters": rng.randint(20, 60)}
    if kind == "rbm":
        return {"kind": kind, "n_vis": _log(rng, 20, 1000), "n_hid": _log(rng, 20, 800), "T": T, "iters": rng.randint(20, 120) if T else rng.randint(10, 30)}
    if kind == "deconv":
        return {"kind": kind, "images": _log(rng, 2, 100), "iters": rng.randint(5, 10)}
    if kind == "pool":
        return {"kind": kind, "side": _log(rng, 12, 140), "radius": rng.choice([2, 3, 4]), "slack": rng.choice([1, 2]), "T": T, "iters": rng.randint(8, 20)}
    if kind == "multi":
        K = rng.choice([2, 2, 8])
        side = _log(rng, 10, 256) if K == 2 else _log(rng, 10, 96)
        return {"kind": kind, "rows": side, "cols": side + rng.randint(0, 9) if K == 2 else side, "K": K, "samples": rng.randint(3, 32), "iters": rng.randint(20, 100)}
    if kind == "host":
        return {"kind": kind, "rows": _log(rng, 10, 900), "cols": _log(rng, 10, 900), "T": 1.0, "iters": rng.randint(50, 200)}
    return {"kind": kind, "requests": rng.randint(4, 10), "hi": rng.randint(100, 450)}


# ---- inputs ---------------------------------------------------------------------------


@functools.lru_cache(maxsize=16)
def _grid_graph(rows, cols, K):
    cfg = W.PAIR2_CFG.copy() if K == 2 else W.dense_pair_cfg(K, K)
    return W.FactorGraph(np.full(rows * cols, K, np.int32), [W.EnumGroup(cfg, W.grid_pairs(rows, cols), K > 2)], [])


@functools.lru_cache(maxsize=4)
def _rbm_graph(n_vis, n_hid):
    return W.rbm(n_vis, n_hid, 0).graph


def _ising(rows, cols, seed, T, iters):
    """W.ising_grid with the graph's structure shared between seeds."""
    graph = _grid_graph(rows, cols, 2)
    rng = np.random.default_rng(seed)
    J = rng.uniform(-1.0, 1.0, size=graph.enum_groups[0].n_fac)
    h = rng.standard_normal(rows * cols)
    return W.Problem("ising", graph, np.stack([J, -J, -J, J], 1).astype(np.float32).ravel(), np.stack([-h, h], 1).astype(np.float32).ravel(), T, DAMPING, iters)


def _potts(side, K, seed, T, iters):
    """W.potts_grid with the graph's structure shared between seeds."""
    graph = _grid_graph(side, side, K)
    rng = np.random.default_rng(seed)
    w, cfg = rng.uniform(0.5, 2.0), graph.enum_groups[0].cfg
    return W.Problem("potts", graph, (-w * np.minimum(np.abs(cfg[:, 0] - cfg[:, 1]), 2)).astype(np.float32),
                     rng.standard_normal(side * side * K).astype(np.float32), T, DAMPING, iters)


def _problems(case, seed):
    """The case's workloads.Problem members (one for all but batches and serving)."""
    k, seed = case["kind"], int(seed)
    if k in ("grid", "host", "grad"):
        return [_ising(case["rows"], case["cols"], seed, case.get("T", 1.0), case["iters"])]
    if k == "potts":
        return [_potts(case["side"], case["K"], seed, case["T"], case["iters"])]
    if k == "multi":
        return [_ising(case["rows"], case["cols"], seed, 1.0, case["iters"]) if case["K"] == 2 else _potts(case["rows"], case["K"], seed, 1.0, case["iters"])]
    if k == "rbm":
        p = W.rbm(2, 2, 0, T=case["T"], n_iters=case["iters"])
        rng = np.random.default_rng(seed)
        p.graph = _rbm_graph(case["n_vis"], case["n_hid"])
        pot = np.zeros((case["n_vis"] * case["n_hid"], 4), np.float32)
        pot[:, 3] = rng.normal(0.0, 0.1, size=pot.shape[0])
        ev = np.zeros((p.graph.n_vars, 2), np.float32)
        ev[:, 1] = rng.standard_normal(p.graph.n_vars)
        p.log_pot, p.evidence = pot.ravel(), ev.ravel()
        return [p]
    if k == "deconv":
        return [W.deconvolution(seed, n_img=case["images"], n_iters=case["iters"])]
    if k == "pool":
        return [W.pool_grid(case["side"], case["radius"], case["slack"], seed, T=case["T"], n_iters=case["iters"])]
    if k == "batch":
        shapes = np.random.default_rng(case["grids"])  # the sizes belong to the case, the values to the seed
        sides = shapes.integers(16, case["hi"] + 1, size=case["grids"])
        Ks = shapes.choice([2, 4, 8, 16], size=case["grids"])
        members = [_potts_any(int(s), int(K), seed * 1000 + i, case["iters"]) for i, (s, K) in enumerate(zip(sides, Ks))]
        return members + _problems({"kind": "rbm", "n_vis": case["n_vis"], "n_hid": case["n_hid"], "T": 1.0, "iters": case["iters"]}, seed + 1)
    shapes = np.random.default_rng(1000 * case["requests"] + case["hi"])  # k == "serve"
    out = []
    for i in range(case["requests"]):
        side, K, iters = int(shapes.integers(16, case["hi"] + 1)), int(shapes.choice([2, 4, 16])), int(shapes.integers(50, 201))
        T = 1.0 if iters > 80 else float(shapes.choice([0.0, 1.0]))  # long max-product runs amplify rounding
        out.append(_ising(side, side, seed * 1000 + i, T, iters) if K == 2 else _potts(side, K, seed * 1000 + i, T, iters))
    return out


def _potts_any(side, K, seed, iters):
    if K > 2:
        return _potts(side, K, seed, 1.0, iters)
    return W.potts_grid(side, 2, seed, T=1.0, n_iters=iters)


def _gpu(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda()


def _extra(case, seed, p):
    """Per-sample evidence of a many-evidence run, or the cotangent of a gradient."""
    rng = np.random.default_rng(int(seed) + 77)
    if case["kind"] == "multi":
        return rng.standard_normal((case["samples"], p.evidence.size)).astype(np.float32)
    return rng.standard_normal(p.evidence.size).astype(np.float32)


def prepare(case, seed):
    k, ps = case["kind"], _problems(case, seed)
    p = ps[0]
    if k == "serve":
        server = binding.Server(8 << 30, 8)
        return {"kind": k, "server": server, "problems": ps, "descs": [binding.marshal_desc(q.graph) for q in ps]}
    if k == "batch":
        p = W.Problem("batch", None, np.concatenate([q.log_pot for q in ps]), np.concatenate([q.evidence for q in ps]), 1.0, DAMPING, case["iters"])
    g = binding.Graph([q.graph for q in ps] if k == "batch" else p.graph)
    s = {"kind": k, "g": g, "T": p.T, "iters": p.n_iters}
    if k == "host":
        s["lp"], s["ev"] = (torch.from_numpy(a).pin_memory().numpy() for a in (p.log_pot, p.evidence))
        s["bel"] = torch.empty(p.evidence.size, dtype=torch.float32).pin_memory().numpy()
        s["dec"] = torch.empty(g.info["n_vars"], dtype=torch.int32).pin_memory().numpy()
        return s
    s["lp"] = _gpu(p.log_pot)
    s["ev"] = _gpu(_extra(case, seed, p) if k == "multi" else p.evidence)
    if k == "grad":
        s["cot"], s["ckpt"] = _gpu(_extra(case, seed, p)), case["ckpt"]
        s["lp"].requires_grad_(True)
        s["ev"].requires_grad_(True)
    else:
        n = g.info["n_edge_states"]
        s["msgs"] = torch.zeros((case["samples"], n) if k == "multi" else (n,), device="cuda")
    return s


# ---- the call -------------------------------------------------------------------------


def run(s):
    k = s["kind"]
    if k == "serve":
        server = s["server"]
        ids = [server.submit(p.graph, p.log_pot, p.evidence, p.T, p.damping, p.n_iters, desc=d, borrow=True) for p, d in zip(s["problems"], s["descs"])]
        return [server.wait(i, 60.0)[0] for i in ids]
    g = s["g"]
    if k == "host":
        bel, _ = g.infer_host(s["lp"], s["ev"], s["T"], DAMPING, s["iters"], s["bel"], s["dec"])
        return bel
    if k == "grad":
        nb = binding.lbp_beliefs(s["lp"], s["ev"], g, 1.0, DAMPING, s["iters"], s["ckpt"])
        return (nb.detach(), *torch.autograd.grad(nb, (s["lp"], s["ev"]), s["cot"]))
    m = s["msgs"].zero_()
    if k == "multi":
        return g.run_bp_multi(s["lp"], s["ev"], 1.0, DAMPING, s["iters"], m)
    g.run_bp(s["lp"], s["ev"], s["T"], DAMPING, s["iters"], m)
    if k == "grid":
        return m, g.beliefs(s["ev"], m, True), g.decode(s["ev"], m)
    return m, g.beliefs(s["ev"], m, True)


# ---- what one pass cannot do without ----------------------------------------------------


def _sizes(case):
    """[(variable states, edge-states, edges, potentials, operations of one iteration, iterations)] per member."""
    def grid(rows, cols, K, iters, pots):
        F = rows * (cols - 1) + cols * (rows - 1)
        return rows * cols * K, 2 * F * K, 2 * F, pots, F * (4 * K * K + 14 * K), iters

    k = case["kind"]
    if k in ("grid", "grad", "host"):
        F = case["rows"] * (case["cols"] - 1) + case["cols"] * (case["rows"] - 1)
        return [grid(case["rows"], case["cols"], 2, case["iters"], 4 * F)]
    if k == "multi":
        one = grid(case["rows"], case["cols"], case["K"], case["iters"], 0)
        return [one] * case["samples"]
    if k == "potts":
        return [grid(case["side"], case["side"], case["K"], case["iters"], case["K"] ** 2)]
    if k in ("batch", "serve"):
        if k == "serve":
            return [grid(int(math.isqrt(p.graph.n_vars)), int(math.isqrt(p.graph.n_vars)), int(p.graph.num_states[0]), p.n_iters, p.log_pot.size) for p in _problems(case, 0)]
        shapes = np.random.default_rng(case["grids"])
        sides = shapes.integers(16, case["hi"] + 1, size=case["grids"])
        Ks = shapes.choice([2, 4, 8, 16], size=case["grids"])
        return [grid(int(s), int(s), int(K), case["iters"], int(K) ** 2) for s, K in zip(sides, Ks)] + _sizes({**case, "kind": "rbm"})
    if k == "rbm":
        F = case["n_vis"] * case["n_hid"]
        return [(2 * (case["n_vis"] + case["n_hid"]), 4 * F, 2 * F, 4 * F, 44 * F, case["iters"])]
    if k == "deconv":
        n = case["images"]
        V, E = 180 + n * (500 + 18000 + 225), n * (18000 * 3 + 18000 + 225)
        return [(2 * V, 2 * E, E, 0, 20 * E, case["iters"])]
    F = 2 * case["side"] * (case["side"] - 1)
    K, C = (2 * case["radius"] + 1) ** 2, W.pool_grid(2, case["radius"], case["slack"], 0).graph.enum_groups[0].n_cfg
    return [(case["side"] ** 2 * K, 2 * F * K, 2 * F, C, F * (4 * C + 14 * K), case["iters"])]


def work(case):
    """Every input read once (evidence, log-potentials, an index per edge, the messages that
    the run starts from) and every output written once; the arithmetic of all iterations,
    an exponential or a logarithm counted as one operation."""
    B = F = 0
    for vs, es, e, pot, ops, iters in _sizes(case):
        B += 4 * (2 * vs + 2 * es + e + pot)
        F += ops * iters
    if case["kind"] == "grad":
        B, F = B + 4 * (_sizes(case)[0][3] + 2 * _sizes(case)[0][0]), 3 * F
    return {"bytes": B, "flops": F}


# ---- the same in 64 bits, written with torch alone ----------------------------------------


def _d(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", torch.float64)


def _exact_pairs(p, evs=None):
    """Messages and normalised log-beliefs of a graph whose variables have K states each and
    whose factors are one group of pairwise tables (dense or listed)."""
    fg, e = p.graph, p.graph.enum_groups[0]
    K, F, V = int(fg.num_states[0]), e.n_fac, fg.n_vars
    vars_ = torch.from_numpy(e.vars.astype(np.int64)).cuda()
    cfg = torch.from_numpy(e.cfg.astype(np.int64)).cuda()
    ev = _d(p.evidence).reshape(V, K)
    pot = _d(p.log_pot)
    dense = e.n_cfg == K * K
    tab = pot.reshape(-1, K, K) if dense else pot
    m = torch.zeros(F, 2, K, dtype=torch.float64, device="cuda")

    def beliefs():
        return ev.clone().index_add_(0, vars_.reshape(-1), m.reshape(-1, K))

    def lse(v, side):  # towards neighbour `side` of every factor
        if dense:
            t = tab if side == 0 else tab.transpose(1, 2)
            if p.T == 0:
                return torch.cat([(t if t.shape[0] == 1 else t[i:i + 65536]).add(v[i:i + 65536, None, :]).amax(2) for i in range(0, F, 65536)])
            mx = v.amax(1, keepdim=True)
            x, E = ((v - mx) / p.T).exp(), (t / p.T).exp()
            s = x @ E[0].T if E.shape[0] == 1 else (E * x[:, None, :]).sum(2)
            return p.T * s.log() + mx
        z = pot[None, :] + v[:, cfg[:, 1 - side]]
        idx = cfg[:, side].expand(F, -1)
        out = torch.full((F, K), -math.inf, dtype=torch.float64, device="cuda").scatter_reduce_(1, idx, z, "amax")
        if p.T == 0:
            return out
        return out + p.T * torch.zeros_like(out).scatter_add_(1, idx, ((z - out.gather(1, idx)) / p.T).exp()).log()

    def norm(t):
        return t - t.amax(-1, keepdim=True)

    for _ in range(p.n_iters):
        b = beliefs()
        v0, v1 = b[vars_[:, 0]] - m[:, 0], b[vars_[:, 1]] - m[:, 1]
        new = torch.stack([norm(lse(v1, 0)), norm(lse(v0, 1))], 1)
        m = norm(DAMPING * m + (1 - DAMPING) * new)
    b = beliefs()
    return m.reshape(-1), (b - torch.logsumexp(b, 1, keepdim=True)).reshape(-1)


def _exact_grad(p, cot):
    """Beliefs and gradients of a binary grid in log-ratios, by torch's own autograd."""
    e = p.graph.enum_groups[0]
    a, b = (torch.from_numpy(e.vars[:, j].astype(np.int64)).cuda() for j in (0, 1))
    lp, ev = _d(p.log_pot).requires_grad_(True), _d(p.evidence).requires_grad_(True)
    t, h = lp.reshape(-1, 4), ev.reshape(-1, 2)
    h = h[:, 1] - h[:, 0]
    lae = torch.logaddexp
    da = db = torch.zeros(e.n_fac, dtype=torch.float64, device="cuda")
    for _ in range(p.n_iters):
        D = h.index_add(0, a, da).index_add(0, b, db)
        la, lb = D[a] - da, D[b] - db
        na = lae(t[:, 2], t[:, 3] + lb) - lae(t[:, 0], t[:, 1] + lb)
        nb = lae(t[:, 1], t[:, 3] + la) - lae(t[:, 0], t[:, 2] + la)
        da, db = DAMPING * da + (1 - DAMPING) * na, DAMPING * db + (1 - DAMPING) * nb
    D = h.index_add(0, a, da).index_add(0, b, db)
    out = torch.stack([torch.nn.functional.logsigmoid(-D), torch.nn.functional.logsigmoid(D)], 1).reshape(-1)
    return (out.detach(), *torch.autograd.grad(out, (lp, ev), _d(cot)))


def _exact_deconv(p):
    """Max-product over AND (two parents) and OR factors, as log-odds."""
    ga, go = p.graph.logic_groups
    V = p.graph.n_vars
    dev = dict(dtype=torch.float64, device="cuda")
    e = _d(p.evidence).reshape(V, 2)
    h = e[:, 1] - e[:, 0]
    par = torch.from_numpy(ga.parents.astype(np.int64).reshape(-1, 2)).cuda()
    va = torch.cat([par, torch.from_numpy(ga.child.astype(np.int64)).cuda()[:, None]], 1)  # [F, 3]
    off = go.par_off.astype(np.int64)
    seg = torch.from_numpy(np.repeat(np.arange(go.n_fac), np.diff(off))).cuda()
    vp, vc = torch.from_numpy(go.parents.astype(np.int64)).cuda(), torch.from_numpy(go.child.astype(np.int64)).cuda()
    ma, mp, mc = torch.zeros(va.shape, **dev), torch.zeros(vp.shape, **dev), torch.zeros(vc.shape, **dev)

    def total():
        return h.index_add(0, va.reshape(-1), ma.reshape(-1)).index_add(0, vp, mp).index_add(0, vc, mc)

    def to_parent(xc, S, M):  # S, M over the other parents
        return xc + S - (xc + S + M.clamp(max=0)).clamp(min=0)

    for _ in range(p.n_iters):
        D = total()
        x = -(D[va] - ma)  # AND is OR of the negations
        x0, x1, xc = x[:, 0], x[:, 1], x[:, 2]
        r0, r1 = x0.clamp(min=0), x1.clamp(min=0)
        na = -torch.stack([to_parent(xc, r1, x1), to_parent(xc, r0, x0), r0 + r1 + torch.maximum(x0, x1).clamp(max=0)], 1)
        x, xc = D[vp] - mp, D[vc] - mc
        r = x.clamp(min=0)
        S = torch.zeros(vc.shape, **dev).index_add_(0, seg, r)
        M1 = torch.full(vc.shape, -math.inf, **dev).scatter_reduce_(0, seg, x, "amax")
        at = torch.full(vc.shape, x.numel(), dtype=torch.int64, device="cuda").scatter_reduce_(
            0, seg, torch.where(x == M1[seg], torch.arange(x.numel(), device="cuda"), x.numel()), "amin")
        first = torch.arange(x.numel(), device="cuda") == at[seg]
        M2 = torch.full(vc.shape, -math.inf, **dev).scatter_reduce_(0, seg, torch.where(first, -math.inf, x), "amax")
        np_ = to_parent(xc[seg], S[seg] - r, torch.where(first, M2[seg], M1[seg]))
        nc = S + M1.clamp(max=0)
        ma, mp, mc = (DAMPING * o + (1 - DAMPING) * n for o, n in ((ma, na), (mp, np_), (mc, nc)))
    D = total()
    # the OR group's edges: each factor's parents, then its child
    mo = torch.empty(vp.numel() + vc.numel(), **dev)
    mo[torch.arange(vp.numel(), device="cuda") + seg] = mp
    mo[torch.from_numpy(off[1:] + np.arange(go.n_fac)).cuda()] = mc
    d = torch.cat([ma.reshape(-1), mo])
    ls = torch.nn.functional.logsigmoid
    return torch.stack([(-d).clamp(max=0), d.clamp(max=0)], 1).reshape(-1), torch.stack([ls(-D), ls(D)], 1).reshape(-1)


def exact(case, seed):
    k, ps = case["kind"], _problems(case, seed)
    p = ps[0]
    if k == "deconv":
        return _exact_deconv(p)
    if k == "grad":
        return _exact_grad(p, _extra(case, seed, p))
    if k == "multi":
        out = []
        for ev in _extra(case, seed, p):
            p.evidence = ev
            out.append(_exact_pairs(p)[0])
        return torch.stack(out)
    if k == "serve":  # the dense K = 16 maximum in 64 bits takes too long on large grids
        return [None if q.T == 0 and q.graph.num_states[0] > 4 and q.graph.n_vars > 40000 else _exact_pairs(q)[1] for q in ps]
    if k == "batch":
        both = [_exact_pairs(q) for q in ps]
        return tuple(torch.cat([b[i] for b in both]) for i in (0, 1))
    m, nb = _exact_pairs(p)
    return nb if k == "host" else (m, nb, None) if k == "grid" else (m, nb)
