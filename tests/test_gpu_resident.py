"""FP64 solves by one persistent kernel with the vectors on chip: every tile width with ragged
last tiles, rows split over several warps, x in shared or global memory, and the call forms,
against the oracle and the tiled solve."""
import ctypes

import numpy as np
import pytest
import torch

import synth
from oracle import cg as ocg

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


def hub_graph(n, hubs, seed):
    """Watts-Strogatz ring plus `hubs` nodes joined to many others (rows from a few dozen to
    thousands of entries), with three isolated nodes, in a random node order."""
    rng = np.random.default_rng([n, seed])
    eu, ev = synth.watts_strogatz(n, 6, 0.1, rng)
    key = [np.minimum(eu, ev) * n + np.maximum(eu, ev)]
    for h, d in enumerate(hubs):
        v = rng.choice(np.arange(len(hubs), n), size=d, replace=False)
        key.append(np.int64(h) * n + v)
    key = np.unique(np.concatenate(key))
    u, v = key // n, key % n
    w = rng.uniform(0.5, 2.0, len(u))
    perm = rng.permutation(n + 3)
    return synth.csr_from_edges(n + 3, perm[u], perm[v], w)


@pytest.fixture(scope="module")
def case():
    g = hub_graph(31000, [33, 40, 200, 700, 3000, 9001], 1)
    X, Y = synth.sparse_uniform_pairs(g.n, 21, 0.02, 9)
    want = ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, X, Y, rtol=1e-13)[0]
    return g, X, Y, want


# d^2 is second order in the residual (1e-11): 1e-10 leaves room for rounding only; z against
# the tiled solve, both first order in it (condition number below 1e4)
@pytest.mark.parametrize("k", [2, 4, 7, 11, 16, 21])
def test_every_tile_width(nvd, case, k):
    g, X, Y, want = case
    G = nvd.Graph.from_csr(g)
    l0 = nvd.kernel_launches()
    d2, z, st = nvd.ge_distance(G, on(X[:k]), on(Y[:k]), rtol=1e-11, return_z=True, return_stats=True)
    assert nvd.kernel_launches() - l0 <= 6              # one launch per tile
    assert all(s["status"] == 0 and s["rel_resid"] <= 1e-11 for s in st)
    assert rel(d2.cpu().numpy(), want[:k]) < 1e-10
    t, zt = nvd.ge_distance(G, on(X[:k]), on(Y[:k]), rtol=1e-11, return_z=True, kt=4)
    assert rel(t.cpu().numpy(), want[:k]) < 1e-10
    assert float((z - zt).norm() / zt.norm()) < 1e-7
    again, z2 = nvd.ge_distance(G, on(X[:k]), on(Y[:k]), rtol=1e-11, return_z=True)
    assert torch.equal(d2, again) and torch.equal(z, z2)


def test_x_in_global_memory(nvd):
    g = hub_graph(70001, [500], 2)
    X, Y = synth.sparse_uniform_pairs(g.n, 16, 0.02, 5)
    G = nvd.Graph.from_csr(g)
    l0 = nvd.kernel_launches()
    d2 = nvd.ge_distance(G, on(X), on(Y), rtol=1e-11).cpu().numpy()
    assert nvd.kernel_launches() - l0 <= 4
    pick = [0, 9, 15]
    want = ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, X[pick], Y[pick], rtol=1e-13)[0]
    assert rel(d2[pick], want) < 1e-10


def test_call_forms(nvd, case):
    g, X, Y, want = case
    k = 6
    G = nvd.Graph.from_csr(g)
    d2, z = nvd.ge_distance(G, on(X[:k]), on(Y[:k]), rtol=1e-11, return_z=True)
    h, zh = nvd.ge_distance(G, X[:k], Y[:k], rtol=1e-11, return_z=True)
    assert np.array_equal(d2.cpu().numpy(), h.numpy()) and np.array_equal(z.cpu().numpy(), zh.numpy())
    X32, Y32 = X[:k].astype(np.float32), Y[:k].astype(np.float32)
    f, zf = nvd.ge_distance(G, torch.as_tensor(X32, device=DEV), torch.as_tensor(Y32, device=DEV), rtol=1e-11,
                            return_z=True)
    assert zf.dtype == torch.float32
    w32 = ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, X32.astype(float), Y32.astype(float), rtol=1e-13)[0]
    assert rel(f.cpu().numpy(), w32) < 1e-10
    lonely = int(np.flatnonzero(np.diff(g.rowptr) == 0)[0])
    u = np.array([0, 5, 7, lonely, 9, 11, 13, 15])
    v = np.array([1, 6, 7, 3, 99, 30000, 14, 16])
    keep = np.diff(g.rowptr)[u] * np.diff(g.rowptr)[v] > 0
    R = nvd.effective_resistance(G, u, v, rtol=1e-11)
    assert np.isinf(R[3]) and R[2] == 0.0
    E = np.zeros((len(u), g.n))
    F = np.zeros((len(u), g.n))
    E[np.arange(len(u)), u] = 1.0
    F[np.arange(len(u)), v] = 1.0
    sel = keep & (u != v)
    wr = ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, E[sel], F[sel], rtol=1e-13)[0]
    assert rel(R[sel], wr) < 1e-10
    # fewer iterations than needed, the d^2 stop, a non-finite column among good ones
    _, st = nvd.ge_distance(G, on(X[:k]), on(Y[:k]), rtol=1e-11, max_iter=4, return_stats=True,
                            allow_not_converged=True)
    assert all(s["status"] == 6 and s["iters"] == 4 for s in st)
    s2 = nvd.ge_distance(G, on(X[:k]), on(Y[:k]), rtol=1e-14, d2_stop=True, d2_rtol=1e-6)
    assert rel(s2.cpu().numpy(), want[:k]) <= 1e-6
    Xn = X[:k].copy()
    Xn[1, 17] = np.nan
    with pytest.raises(nvd.NvdError) as e:
        nvd.ge_distance(G, on(Xn), on(Y[:k]), rtol=1e-11)
    assert e.value.status == 7
    # new weights reach the plan
    w2 = np.random.default_rng(3).uniform(0.5, 2.0, g.m)
    g2 = synth.csr_from_edges(g.n, g.eu, g.ev, w2)
    G.set_weights(g2.w)
    got = nvd.ge_distance(G, on(X[:k]), on(Y[:k]), rtol=1e-11).cpu().numpy()
    assert rel(got, ocg.ge_d2_cg(g2.n, g2.rowptr, g2.colidx, g2.w, X[:k], Y[:k], rtol=1e-13)[0]) < 1e-10


@pytest.mark.parametrize("kt", [4, 8, 16])
def test_tiled_rows_over_all_lane_groups(nvd, case, kt):
    """The tiled FP64 SpMM gives rows of more than 32 entries a whole warp (and the longest a
    CTA): both against the oracle, with FP32 weights too (exact integer conversion)."""
    g, X, Y, want = case
    G = nvd.Graph.from_csr(g)
    d2 = nvd.ge_distance(G, on(X[:9]), on(Y[:9]), rtol=1e-11, kt=kt).cpu().numpy()
    assert rel(d2, want[:9]) < 1e-10
    w32 = np.float32(g.w)
    w32[w32 == 0] = 1.0
    d32 = nvd.ge_distance(nvd.Graph(g.rowptr, g.colidx, w32), on(X[:9]), on(Y[:9]), rtol=1e-11, kt=kt).cpu().numpy()
    ref = ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, w32.astype(np.float64), X[:9], Y[:9], rtol=1e-13)[0]
    assert rel(d32, ref) < 1e-10


# device d^2 and no stats: nobody asks for the pairs' statuses, in either form of the solve
@pytest.mark.parametrize("kt", [0, 4])
def test_device_result_without_statuses(nvd, case, kt):
    g, X, Y, _ = case
    k = 6
    G = nvd.Graph.from_csr(g)
    x, y = on(X[:k]), on(Y[:k])
    d2 = torch.full((k,), np.nan, dtype=torch.float64, device=DEV)
    o = nvd.default_opts(nvd.MODE_FP64, max_iter=3, kt=kt)
    o.flags |= nvd.SOLVE_D2_DEVICE
    rc = nvd.load_library().nvd_ge_distance(G.handle, k, x.data_ptr(), y.data_ptr(), nvd.F64, ctypes.byref(o),
                                            d2.data_ptr(), None, None, torch.cuda.current_stream().cuda_stream)
    assert rc == 0 and bool(torch.isfinite(d2).all())
