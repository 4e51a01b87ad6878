"""Workloads for timing the library through its public entry points.

A case names a random-graph family with its size, a number of vector pairs and the
call a program makes on them; ``prepare`` builds the graph handle and the input
vectors on the GPU from a seed, ``run`` makes the call once.  The families are the
synthetic models the package is tested and benchmarked on (Erdos-Renyi,
Barabasi-Albert, Watts-Strogatz, power-law configuration model), generated here with
torch so that a graph of a million nodes takes well under a second.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2310_11222_gb300 as nvd

DEV = "cuda"
F64 = torch.float64


# ----------------------------------------------------------------- the cases

def listed():
    return [
        # one distance between two node vectors on a small social-network-sized graph: the
        # smallest call, where launches and round trips count
        dict(name="pair_ba_2k", call="distance", graph="ba", n=2000, degree=6, weights="unit", k=1, support=0.10,
             mode="fp64", rtol=1e-10),
        # the plain small workload: 16 pairs on a BA graph of 2,000 nodes
        dict(name="pairs_ba_2k", call="distance", graph="ba", n=2000, degree=6, weights="unit", k=16, support=0.10,
             mode="fp64", rtol=1e-10),
        # one point of a size sweep (one pair per graph) on the slowest topology, odd size
        dict(name="sweep_ws_20k", call="distance", graph="ws", n=20011, degree=8, weights="unit", k=1, support=0.10,
             mode="fp64", rtol=1e-10),
        # a few distances with their potentials z on a mid-sized graph; five pairs do not fill a tile
        dict(name="potentials_er_100k", call="distance_z", graph="er", n=100003, degree=10, weights="uniform", k=5,
             support=0.01, mode="fp64", rtol=1e-10),
        # the plain method at scale: 8 pairs, one right-hand side at a time
        dict(name="single_er_1m", call="distance_single", graph="er", n=1000000, degree=10, weights="uniform", k=8,
             support=0.01, mode="fp64", rtol=1e-10),
        # the same pairs in mixed precision, the mode meant for throughput
        dict(name="mixed_er_1m", call="distance", graph="er", n=1000000, degree=10, weights="uniform", k=8,
             support=0.01, mode="mixed", rtol=1e-4),
        # heavy-tailed degrees in mixed precision: the largest working set (block vectors
        # of 256 MB), graph stored by degree as a throughput run would
        dict(name="mixed_powerlaw_2m", call="distance", graph="powerlaw", n=2000000, degree=6, weights="lognormal",
             k=32, support=0.001, mode="mixed", rtol=5e-5),
        # many graphs of uneven size in one call, FP32, half BA and half WS
        dict(name="batch_uneven_32", call="batched", graph="mix", count=32, n=1000, n_max=100000, degree=10,
             weights="unit", k=32, support=1.0, mode="fp32", rtol=1e-6),
        # many small networks (one per subject, text or time step) compared pair by pair
        dict(name="batch_small_96", call="batched", graph="mix", count=96, n=24, n_max=500, degree=6,
             weights="unit", k=4, support=0.25, mode="fp64", rtol=1e-9),
        # a training step: distances, then gradients for both vectors and all edge weights
        dict(name="train_ba_200k", call="train", graph="ba", n=200000, degree=10, weights="lognormal_f32", k=16,
             support=0.10, mode="fp64", rtol=1e-10),
        # effective resistances between node pairs given by id
        dict(name="resistance_er_30k", call="resistance", graph="er", n=30011, degree=10, weights="uniform", k=96,
             support=0.0, mode="fp64", rtol=1e-10),
        # the operator alone on several vectors
        dict(name="apply_ws_300k", call="apply", graph="ws", n=300007, degree=10, weights="uniform", k=6,
             support=1.0, mode="fp64", rtol=0.0),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    call = rng.choice(["distance", "distance", "distance_z", "distance_single", "mixed", "powerlaw", "batched",
                       "batched_small", "train", "resistance", "apply"])
    c = dict(call=call, graph=rng.choice(["er", "ba", "ws"]), degree=rng.choice([6, 8, 10, 12]),
             weights=rng.choice(["unit", "uniform"]), support=rng.choice([0.01, 0.1]), mode="fp64", rtol=1e-10)
    if call == "distance":
        c.update(n=_log(rng, 2000, 300000), k=_log(rng, 1, 40))
    elif call == "distance_z":
        c.update(n=_log(rng, 2000, 200000), k=_log(rng, 1, 20), weights=rng.choice(["uniform", "lognormal_f32"]))
    elif call == "distance_single":
        c.update(n=_log(rng, 50000, 1000000), k=rng.randint(1, 8), graph=rng.choice(["er", "ba"]))
    elif call == "mixed":
        c.update(call="distance", n=_log(rng, 100000, 1000000), k=_log(rng, 2, 32), graph="er", weights="uniform",
                 mode="mixed", rtol=1e-4)
    elif call == "powerlaw":
        c.update(call="distance", n=_log(rng, 300000, 2000000), k=_log(rng, 8, 32), graph="powerlaw", degree=6,
                 weights="lognormal", support=0.001, mode="mixed", rtol=5e-5)
    elif call == "batched":
        c.update(graph="mix", count=_log(rng, 4, 32), n=1000, n_max=_log(rng, 10000, 100000), weights="unit",
                 k=_log(rng, 4, 32), support=1.0, mode="fp32", rtol=1e-6)
    elif call == "batched_small":
        c.update(call="batched", graph="mix", count=_log(rng, 16, 96), n=24, n_max=_log(rng, 100, 2000),
                 weights="unit", k=_log(rng, 1, 8), support=0.25, rtol=1e-9)
    elif call == "train":
        c.update(n=_log(rng, 20000, 200000), k=_log(rng, 2, 16), graph="ba", weights="lognormal_f32", support=0.1)
    elif call == "resistance":
        c.update(n=_log(rng, 2000, 100000), k=_log(rng, 4, 96), graph=rng.choice(["er", "ba"]), support=0.0)
    else:
        c.update(n=_log(rng, 3000, 300000), k=_log(rng, 1, 16), support=1.0, rtol=0.0)
    return c


# ----------------------------------------------------------------- graphs

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 12345)
    return g


def _simple(n, u, v):
    """Distinct undirected edges (a < b) of a multigraph without its self-loops."""
    a, b = torch.minimum(u, v), torch.maximum(u, v)
    key = torch.unique((a * n + b)[a != b])
    return key // n, key % n


def _er(n, degree, gen):
    m = n * degree // 2
    e = torch.randint(0, n, (2, m + m // 50 + 16), device=DEV, generator=gen)
    a, b = _simple(n, e[0], e[1])
    keep = torch.randperm(a.numel(), device=DEV, generator=gen)[:m]
    return a[keep], b[keep]


def _ba(n, degree, gen):
    """Preferential attachment: edge e of node t ends at a uniform endpoint of the edges
    of earlier nodes (repeats merged); endpoints that are themselves copies are followed
    until they name a node."""
    m = max(1, min(degree // 2, n - 2))
    t = torch.arange(m + 1, n, device=DEV).repeat_interleave(m)
    src = torch.cat([torch.arange(1, m + 1, device=DEV), t])        # edges 0..m-1: the seed star on node 0
    first = m + (t - (m + 1)) * m                                   # edges before node t's
    ptr = (torch.rand(t.numel(), dtype=F64, device=DEV, generator=gen) * (2 * first)).long()
    ptr = torch.cat([torch.full((m,), -1, device=DEV, dtype=torch.long), ptr])
    cur = ptr.clone()
    while True:                                                     # slot 2e: src[e]; slot 2e+1: edge e's target
        odd = (cur >= 0) & (cur % 2 == 1)
        if not bool(odd.any()):
            break
        cur = torch.where(odd, ptr[cur.clamp(min=0) // 2], cur)
    dst = torch.where(cur < 0, torch.zeros_like(cur), src[cur.clamp(min=0) // 2])
    return _simple(n, src, dst)


def _ws(n, degree, gen):
    h = max(1, min(degree // 2, (n - 1) // 2))
    u = torch.arange(n, device=DEV).repeat_interleave(h)
    v = (u + torch.arange(1, h + 1, device=DEV).repeat(n)) % n
    far = torch.randint(0, n, v.shape, device=DEV, generator=gen)
    v = torch.where(torch.rand(v.shape, device=DEV, generator=gen) < 0.1, far, v)
    return _simple(n, u, v)


def _powerlaw(n, degree, gen):
    """Erased configuration model, P(d) ~ d^-2.3 on [2, min(10,000, n / 10)]."""
    d = torch.arange(2, max(5, min(10000, n // 10)) + 1, dtype=F64, device=DEV)
    cdf = torch.cumsum(d ** -2.3, 0)
    cdf = cdf / cdf[-1]
    deg = torch.searchsorted(cdf, torch.rand(n, dtype=F64, device=DEV, generator=gen)).clamp(max=d.numel() - 1) + 2
    stubs = torch.arange(n, device=DEV).repeat_interleave(deg)
    stubs = stubs[torch.randperm(stubs.numel(), device=DEV, generator=gen)]
    m = stubs.numel() // 2
    return _simple(n, stubs[:m], stubs[m:2 * m])


def _components(n, a, b):
    """Smallest node id of every node's component."""
    lab = torch.arange(n, device=DEV)
    while True:
        new = lab.clone()
        new.scatter_reduce_(0, a, lab[b], "amin")
        new.scatter_reduce_(0, b, lab[a], "amin")
        new = torch.minimum(new, new[new])
        new = new[new]
        if torch.equal(new, lab):
            return lab
        lab = new


def _largest_component(n, a, b):
    lab = _components(n, a, b)
    keep = lab == torch.argmax(torch.bincount(lab, minlength=n))
    new = torch.cumsum(keep.long(), 0) - 1
    sel = keep[a]
    return int(keep.sum()), new[a[sel]], new[b[sel]]


def _csr(family, n, degree, weights, gen, whole=False, edges=0):
    """(n, rowptr, colidx, w) of one graph; ER and power-law graphs are cut to their
    largest component, as their workloads are, unless the whole graph is asked for.
    edges: that many of the edges, at random (0: all)."""
    a, b = {"er": _er, "ba": _ba, "ws": _ws, "powerlaw": _powerlaw}[family](n, degree, gen)
    if edges:
        keep = torch.randperm(a.numel(), device=DEV, generator=gen)[:edges]
        a, b = a[keep], b[keep]
    if family in ("er", "powerlaw") and not whole:
        n, a, b = _largest_component(n, a, b)
    m = a.numel()
    if weights == "unit":
        w = torch.ones(m, dtype=F64, device=DEV)
    elif weights == "uniform":
        w = torch.rand(m, dtype=F64, device=DEV, generator=gen) * 1.5 + 0.5
    else:
        s = 1.0 if weights == "lognormal" else 0.5
        w = torch.exp(s * torch.randn(m, dtype=F64, device=DEV, generator=gen)).float()
    u, v = torch.cat([a, b]), torch.cat([b, a])
    order = torch.argsort(u * n + v)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rowptr[1:] = torch.cumsum(torch.bincount(u, minlength=n), 0)
    return n, rowptr, v[order].int(), torch.cat([w, w])[order]


def _vectors(n, k, support, gen):
    """k node vectors: Uniform[0,1) values on a random share of the nodes, sum 1."""
    if support >= 1.0:
        x = torch.rand(k, n, dtype=F64, device=DEV, generator=gen)
    else:
        s = max(1, int(round(support * n)))
        x = torch.zeros(k, n, dtype=F64, device=DEV)
        for j in range(k):
            at = torch.randperm(n, device=DEV, generator=gen)[:s]
            x[j, at] = torch.rand(s, dtype=F64, device=DEV, generator=gen) + 1e-9
    return x / x.sum(1, keepdim=True)


# ----------------------------------------------------------------- inputs

def _sizes(case):
    """Node counts of a batched case, log-uniform in [n, n_max], the same for every seed."""
    r = np.random.default_rng([case["count"], case["n"], case["n_max"]])
    return [int(round(v)) for v in np.exp(r.uniform(np.log(case["n"]), np.log(case["n_max"]), case["count"]))]


def _inputs(case, seed):
    """The plain inputs of a case: CSR arrays and vectors (or node ids, or gbar)."""
    gen = _gen(seed)
    k = case["k"]
    if case["call"] == "batched":
        out = []
        for i, n in enumerate(_sizes(case)):
            n, rp, ci, w = _csr("ba" if i % 2 == 0 else "ws", n, case["degree"], case["weights"], gen)
            if case["mode"] == "fp32":
                # indicator pairs and diffuse pairs in equal parts
                x, y = _vectors(n, k, 1.0, gen), _vectors(n, k, 1.0, gen)
                h = k // 2
                x[:h], y[:h] = 0.0, 0.0
                at = torch.randint(0, n, (h,), device=DEV, generator=gen)
                step = torch.randint(1, n, (h,), device=DEV, generator=gen)
                rows = torch.arange(h, device=DEV)
                x[rows, at] = 1.0
                y[rows, (at + step) % n] = 1.0
            else:
                x, y = _vectors(n, k, case["support"], gen), _vectors(n, k, case["support"], gen)
            out.append((n, rp, ci, w, x, y))
        return out
    # calls that return a value per node or edge keep every node, and the same number of edges
    # for every seed (merging repeated BA edges leaves a few fewer than n * degree / 2)
    whole = case["call"] in ("distance_z", "train", "apply")
    edges = int(0.98 * (case["n"] * case["degree"] // 2)) if case["call"] == "train" else 0
    n, rp, ci, w = _csr(case["graph"], case["n"], case["degree"], case["weights"], gen, whole, edges)
    if case["call"] == "resistance":
        u = torch.randint(0, n, (k,), device=DEV, generator=gen)
        v = (u + torch.randint(1, n, (k,), device=DEV, generator=gen)) % n
        return n, rp, ci, w, u.cpu().numpy().astype(np.int32), v.cpu().numpy().astype(np.int32)
    if case["call"] == "apply":
        return n, rp, ci, w, torch.randn(k, n, dtype=F64, device=DEV, generator=gen), None
    x, y = _vectors(n, k, case["support"], gen), _vectors(n, k, case["support"], gen)
    return n, rp, ci, w, x, y


_MODE = {"fp64": nvd.MODE_FP64, "fp32": nvd.MODE_FP32, "mixed": nvd.MODE_MIXED}


def prepare(case, seed):
    call = case["call"]
    got = _inputs(case, seed)
    state = {"case": case}
    if call == "batched":
        state["graphs"] = [nvd.Graph(rp, ci, w) for _, rp, ci, w, _, _ in got]
        state["x"] = [g[4] for g in got]
        state["y"] = [g[5] for g in got]
        return state
    n, rp, ci, w, x, y = got
    state["x"], state["y"] = x, y
    state["graph"] = nvd.Graph(rp, ci, w, reorder=case["graph"] == "powerlaw")
    if call == "train":
        state["x"].requires_grad_(True)
        state["y"].requires_grad_(True)
        state["w"] = w.requires_grad_(True)
        state["gbar"] = torch.rand(case["k"], dtype=F64, device=DEV, generator=_gen(seed + 500009)) + 0.5
    return state


def run(state):
    case = state["case"]
    call = case["call"]
    opts = dict(mode=_MODE[case["mode"]], rtol=case["rtol"])
    if call == "batched":
        return nvd.ge_distance_batched(state["graphs"], state["x"], state["y"], **opts)
    g, x, y = state["graph"], state["x"], state["y"]
    if call == "distance":
        return nvd.ge_distance(g, x, y, **opts)
    if call == "distance_single":
        return nvd.ge_distance(g, x, y, single_rhs=True, **opts)
    if call == "distance_z":
        return nvd.ge_distance(g, x, y, return_z=True, **opts)
    if call == "resistance":
        return nvd.effective_resistance(g, x, y, **opts)
    if call == "apply":
        return nvd.laplacian_apply(g, x)
    d2 = nvd.ge_distance_autograd(g, x, y, state["w"], **opts)
    return (d2.detach(),) + torch.autograd.grad(d2, (x, y, state["w"]), grad_outputs=state["gbar"])


# ----------------------------------------------------------------- work

# CG iterations to the tolerances above, by family (measured; ~ constant in n and k)
_ITERS = {"er": 24, "ba": 23, "ws": 66, "powerlaw": 70, "mix": 45}


def work(case):
    """Each input read once and each result written once; the multiply-adds of Jacobi-PCG
    (one product with L and the vector updates per iteration)."""
    k, deg = case["k"], case["degree"]
    n = sum(_sizes(case)) if case["call"] == "batched" else case["n"]
    nnz = n * deg
    wsz = 4 if case["weights"].startswith("lognormal") else 8
    byts = 8 * (n + 1) + nnz * (4 + wsz)
    if case["call"] == "apply":
        return {"bytes": byts + 16 * n * k, "flops": 2 * (nnz + n) * k}
    flops = _ITERS[case["graph"]] * k * (2 * nnz + 12 * n)
    if case["call"] != "resistance":
        byts += 16 * n * k
    if case["call"] == "distance_z":
        byts += 8 * n * k
    if case["call"] == "train":
        byts += 16 * n * k + nnz * wsz
        flops += 3 * nnz * k
    return {"bytes": byts, "flops": flops}


# ----------------------------------------------------------------- exact values

def _solve(n, rp, ci, w, delta):
    """z = L^+ delta ([n, k], 64 bits) by Jacobi-PCG far below the rounding of the results."""
    w = w.detach().double()
    rows = torch.arange(n, device=DEV).repeat_interleave(rp[1:] - rp[:-1])
    A = torch.sparse_csr_tensor(rp, ci.long(), w, (n, n))
    deg = torch.zeros(n, dtype=F64, device=DEV).index_add_(0, rows, w)
    lab = _components(n, rows, ci.long())
    size = torch.bincount(lab, minlength=n).double().clamp(min=1)

    def project(v):
        s = torch.zeros_like(v).index_add_(0, lab, v) / size[:, None]
        return v - s[lab]

    dinv = torch.where(deg > 0, 1 / deg, torch.zeros_like(deg))[:, None]
    b = project(delta)
    z, r = torch.zeros_like(b), b.clone()
    u = dinv * r
    p, rho = u.clone(), (r * u).sum(0)
    stop = 1e-14 * b.norm(dim=0)
    going = torch.ones(b.shape[1], dtype=torch.bool, device=DEV)
    for it in range(5000):
        q = deg[:, None] * p - A @ p
        pq = (p * q).sum(0)
        # a column that is done stays as it is: what is left of its p is rounding
        alpha = torch.where(going & (pq > 0), rho / pq, torch.zeros_like(pq))
        z += alpha * p
        r -= alpha * q
        going &= r.norm(dim=0) > stop
        if it % 8 == 7 and not bool(going.any()):
            break
        u = dinv * r
        new = (r * u).sum(0)
        p = u + torch.where(rho > 0, new / rho, torch.zeros_like(rho)) * p
        rho = new
    z = project(z)
    d2 = 2 * (b * z).sum(0) - (z * (deg[:, None] * z - A @ z)).sum(0)
    return z, d2


def exact(case, seed):
    call = case["call"]
    got = _inputs(case, seed)
    if call == "batched":
        return torch.cat([_solve(n, rp, ci, w, (x - y).T.contiguous())[1] for n, rp, ci, w, x, y in got]).cpu()
    n, rp, ci, w, x, y = got
    if call == "apply":
        A = torch.sparse_csr_tensor(rp, ci.long(), w, (n, n))
        rows = torch.arange(n, device=DEV).repeat_interleave(rp[1:] - rp[:-1])
        deg = torch.zeros(n, dtype=F64, device=DEV).index_add_(0, rows, w)
        return (deg[:, None] * x.T - A @ x.T.contiguous()).T.contiguous()
    if call == "resistance":
        k = len(x)
        delta = torch.zeros(n, k, dtype=F64, device=DEV)
        cols = torch.arange(k, device=DEV)
        delta[torch.from_numpy(x).long().to(DEV), cols] += 1.0
        delta[torch.from_numpy(y).long().to(DEV), cols] -= 1.0
        return _solve(n, rp, ci, w, delta)[1].cpu().numpy()
    z, d2 = _solve(n, rp, ci, w, (x - y).T.contiguous())
    if call == "distance_z":
        return d2, z.T.contiguous()
    if call != "train":
        return d2
    gbar = torch.rand(case["k"], dtype=F64, device=DEV, generator=_gen(seed + 500009)) + 0.5
    gx = (2 * gbar[:, None] * z.T).contiguous()
    rows = torch.arange(n, device=DEV).repeat_interleave(rp[1:] - rp[:-1])
    gw = torch.zeros(ci.numel(), dtype=F64, device=DEV)
    for j in range(case["k"]):
        gw -= 0.5 * gbar[j] * (z[rows, j] - z[ci.long(), j]) ** 2
    return d2, gx, -gx, gw
