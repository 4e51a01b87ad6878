"""FP64 solves by one thread-block cluster per (component, pair): sizes at the edges of its
layout (rows per warp item, rows per CTA, CTAs per cluster, p replicated, published through
L2 or gathered from L2) against the oracle, and the same call forms as the tiled solve."""
import numpy as np
import pytest
import torch

import synth
from oracle import cg as ocg
from oracle import dense

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def nvd():
    import paper_2310_11222_gb300 as m
    m.load_library()
    return m


def on(x):
    return torch.as_tensor(x, dtype=torch.float64, device=DEV)


def rel(a, b):
    return np.max(np.abs(a - b) / np.maximum(np.abs(b), 1e-300))


def graph(kind, n, seed=0):
    rng = np.random.default_rng([n, seed])
    if kind == "path":
        eu, ev = synth.path_graph(n)
    elif kind == "star":
        eu, ev = synth.star_graph(n - 1)
    elif kind == "ba":
        eu, ev = synth.barabasi_albert(n, 4, rng)
    else:
        eu, ev = synth.watts_strogatz(n, 8, 0.1, rng)
    return synth.csr_from_edges(n, eu, ev, rng.uniform(0.5, 2.0, len(eu)))


def solve(nvd, G, X, Y, **kw):
    """d^2, z, stats and the kernels launched (the tiled solve launches three per iteration)."""
    l0 = nvd.kernel_launches()
    d2, z, st = nvd.ge_distance(G, on(X), on(Y), rtol=1e-12, return_z=True, return_stats=True, **kw)
    return d2.cpu().numpy(), z.cpu().numpy(), st, nvd.kernel_launches() - l0


# d^2 = delta^T z is second order in the residual (1e-12), so 1e-10 leaves room for rounding
# only; z is first order: its error is at most cond * 1e-12 (cond < 1e5 for the path of 257)
@pytest.mark.parametrize("kind,n", [("path", 2), ("path", 3), ("path", 257), ("star", 33), ("star", 130),
                                    ("star", 1500), ("ba", 31), ("ba", 32), ("ba", 127), ("ba", 128), ("ba", 129),
                                    ("ba", 500), ("ws", 1024), ("ws", 2049), ("ba", 2047)])
@pytest.mark.parametrize("k", [1, 5])
def test_small_graphs_match_the_dense_oracle(nvd, kind, n, k):
    g = graph(kind, n)
    X, Y = synth.diffuse_uniform_pairs(g.n, k, 11)
    d2, z, st, launches = solve(nvd, nvd.Graph.from_csr(g), X, Y)
    assert launches <= 3 and all(s["status"] == 0 and s["rel_resid"] <= 1e-12 for s in st)
    assert rel(d2, dense.ge_d2_eig(g.n, g.rowptr, g.colidx, g.w, X, Y)) < 1e-10
    L = dense.laplacian_dense(g.n, g.rowptr, g.colidx, g.w)
    delta = X - Y - (X - Y).mean(1, keepdims=True)
    want = np.linalg.lstsq(L, delta.T, rcond=None)[0].T
    want -= want.mean(1, keepdims=True)
    assert np.linalg.norm(z - want) <= 1e-7 * np.linalg.norm(want)


# one slot per thread ends at 16 x 1,024 rows, p replicated at about 24,000, p from L2 goes on
@pytest.mark.parametrize("kind,n", [("ba", 5200), ("ws", 16300), ("ba", 16500), ("ws", 23000), ("ba", 26001)])
def test_larger_graphs_match_the_oracle(nvd, kind, n):
    g = graph(kind, n)
    X, Y = synth.sparse_uniform_pairs(g.n, 9, 0.05, 3)
    d2, z, st, launches = solve(nvd, nvd.Graph.from_csr(g), X, Y)
    assert launches <= 3 and all(s["status"] == 0 for s in st)
    want, _, _ = ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, X, Y, rtol=1e-13)
    assert rel(d2, want) < 1e-10


def test_components_isolated_nodes_and_call_forms(nvd):
    """Interleaved components of different sizes with isolated nodes: device and host inputs,
    FP32 inputs, node-id pairs, new weights and repeated calls."""
    parts = [graph("ba", 700), graph("path", 2), graph("ws", 150), synth.csr_from_edges(
        1, np.empty(0, np.int64), np.empty(0, np.int64), np.empty(0)), graph("star", 300)]
    gu, _ = synth.disjoint_union(parts)
    rng = np.random.default_rng(4)
    perm = rng.permutation(gu.n)
    g = synth.csr_from_edges(gu.n, perm[gu.eu], perm[gu.ev], gu.ew)
    X, Y = rng.random((6, g.n)), rng.random((6, g.n))
    G = nvd.Graph.from_csr(g)
    d2, z, st, launches = solve(nvd, G, X, Y)
    assert launches <= 8
    want = dense.ge_d2_eig(g.n, g.rowptr, g.colidx, g.w, X, Y)
    assert rel(d2, want) < 1e-10
    again = solve(nvd, G, X, Y)
    assert np.array_equal(d2, again[0]) and np.array_equal(z, again[1])
    h, zh = nvd.ge_distance(G, X, Y, rtol=1e-12, return_z=True)
    assert np.array_equal(d2, h.numpy()) and np.array_equal(z, zh.numpy())
    X32, Y32 = X.astype(np.float32), Y.astype(np.float32)
    f = nvd.ge_distance(G, torch.as_tensor(X32, device=DEV), torch.as_tensor(Y32, device=DEV), rtol=1e-12)
    assert rel(f.cpu().numpy(), dense.ge_d2_eig(g.n, g.rowptr, g.colidx, g.w, X32.astype(float),
                                                Y32.astype(float))) < 1e-10
    u, v = rng.integers(0, g.n, 12), rng.integers(0, g.n, 12)
    R = nvd.effective_resistance(G, u, v, rtol=1e-12)
    want_r = np.array([dense.effective_resistance(g.n, g.rowptr, g.colidx, g.w, [a], [b])[0] for a, b in zip(u, v)])
    assert np.array_equal(np.isinf(R), np.isinf(want_r))
    ok = np.isfinite(R) & (want_r > 0)
    assert rel(R[ok], want_r[ok]) < 1e-10
    w2 = synth.csr_from_edges(g.n, g.eu, g.ev, rng.uniform(0.5, 2.0, g.m))
    G.set_weights(w2.w)
    assert rel(solve(nvd, G, X, Y)[0], dense.ge_d2_eig(g.n, g.rowptr, g.colidx, w2.w, X, Y)) < 1e-10


def test_statuses_and_d2_stop(nvd):
    g = graph("ba", 1000)
    X, Y = synth.sparse_uniform_pairs(g.n, 4, 0.1, 5)
    X[2] = Y[2]                                            # delta = 0: nothing to solve
    G = nvd.Graph.from_csr(g)
    d2, z, st, _ = solve(nvd, G, X, Y)
    assert d2[2] == 0.0 and st[2]["iters"] == 0 and not z[2].any()
    _, st = nvd.ge_distance(G, on(X[:2]), on(Y[:2]), rtol=1e-12, max_iter=3, return_stats=True,
                            allow_not_converged=True)
    assert [s["status"] for s in st] == [6, 6] and [s["iters"] for s in st] == [3, 3]
    stopped, ss = nvd.ge_distance(G, on(X), on(Y), rtol=1e-14, d2_stop=True, d2_rtol=1e-6, return_stats=True)
    keep = [0, 1, 3]
    assert rel(stopped.cpu().numpy()[keep], d2[keep]) <= 1e-6
    assert all(ss[j]["iters"] < 30 for j in keep)
    Xn = X.copy()
    Xn[1, 7] = np.inf
    with pytest.raises(nvd.NvdError) as e:
        nvd.ge_distance(G, on(Xn), on(Y), rtol=1e-12)
    assert e.value.status == 7


def test_batches_of_uneven_graphs(nvd):
    gs = [graph("ba", n, i) if i % 2 else graph("ws", n, i) for i, n in enumerate([20, 33, 150, 700, 2500, 64])]
    ks = [1, 4, 3, 2, 4, 0]
    pairs = [synth.diffuse_uniform_pairs(g.n, k, 7 + i) for i, (g, k) in enumerate(zip(gs, ks))]
    l0 = nvd.kernel_launches()
    d2, st = nvd.ge_distance_batched([nvd.Graph.from_csr(g) for g in gs], [on(x) for x, _ in pairs],
                                     [on(y) for _, y in pairs], mode=nvd.MODE_FP64, rtol=1e-12, return_stats=True)
    assert nvd.kernel_launches() - l0 <= 8 and all(s["status"] == 0 for s in st)
    want = np.concatenate([dense.ge_d2_eig(g.n, g.rowptr, g.colidx, g.w, x, y) for g, (x, y) in zip(gs, pairs)])
    assert rel(d2.numpy(), want) < 1e-10
