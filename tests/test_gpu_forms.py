"""Every kernel variant of the on-chip FP64 solves, forced through the handle and read back from
it, so that what runs here does not depend on the estimates that choose a form: every tile
width of the one-kernel form with several tiles and a ragged last one, every kernel of the
cluster form, new weights, and the call forms, against the oracle."""
import ctypes
import time

import numpy as np
import pytest
import torch

import synth
from oracle import cg as ocg

pytestmark = pytest.mark.gpu
DEV = "cuda"
TILES, CLUSTER, RESIDENT = 1, 2, 3
GLOBAL_P, MATRIX, ONE_SLOT, VIA_L2 = 1, 2, 4, 8


@pytest.fixture(scope="module")
def nvd():
    import paper_2310_11222_gb300 as m
    m.load_library()
    return m


def force(nvd, G, form, width):
    assert nvd.load_library().nvd_diag_force_form(G.handle, form, width) == 0


def last(nvd, G):
    v = [ctypes.c_int32() for _ in range(3)]
    assert nvd.load_library().nvd_diag_last_form(G.handle, *[ctypes.byref(c) for c in v]) == 0
    return tuple(c.value for c in v)


def on(x):
    return torch.as_tensor(x, dtype=torch.float64, device=DEV)


def rel(a, b):
    return np.max(np.abs(a - b) / np.maximum(np.abs(b), 1e-300))


def hub_graph(n, degrees, seed):
    """Watts-Strogatz ring plus nodes of the given degrees and three isolated nodes, in a random
    node order."""
    rng = np.random.default_rng([n, seed])
    eu, ev = synth.watts_strogatz(n, 6, 0.1, rng)
    key = [np.minimum(eu, ev) * n + np.maximum(eu, ev)]
    for h, d in enumerate(degrees):
        key.append(np.int64(h) * n + rng.choice(np.arange(len(degrees), n), size=d, replace=False))
    key = np.unique(np.concatenate(key))
    perm = rng.permutation(n + 3)
    return synth.csr_from_edges(n + 3, perm[key // n], perm[key % n], rng.uniform(0.5, 2.0, len(key)))


@pytest.fixture(scope="module")
def case():
    g = hub_graph(8000, [33, 40, 200, 700, 2100, 4999], 1)
    X, Y = synth.sparse_uniform_pairs(g.n, 21, 0.02, 9)
    return g, X, Y, ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, X, Y, rtol=1e-13)[0]


# d^2 is second order in the residual (1e-11): 1e-10 leaves room for rounding only; z against
# the tiled solve, both first order in it (condition number below 1e4)
@pytest.mark.parametrize("form,width,k", [(RESIDENT, 1, 1), (RESIDENT, 1, 3), (RESIDENT, 4, 21), (RESIDENT, 8, 21),
                                          (RESIDENT, 16, 21), (CLUSTER, 16, 21)])
def test_call_forms_and_weights(nvd, case, form, width, k):
    g, X, Y, want = case
    X, Y, want = X[:k], Y[:k], want[:k]
    G = nvd.Graph.from_csr(g)
    t, zt = nvd.ge_distance(G, on(X), on(Y), rtol=1e-11, return_z=True, kt=4)
    assert last(nvd, G) == (TILES, 4, 0)
    force(nvd, G, form, width)
    d2, z, st = nvd.ge_distance(G, on(X), on(Y), rtol=1e-11, return_z=True, return_stats=True)
    assert last(nvd, G)[:2] == (form, width)
    assert all(s["status"] == 0 and s["rel_resid"] <= 1e-11 for s in st)
    assert rel(d2.cpu().numpy(), want) < 1e-10
    assert float((z - zt).norm() / zt.norm()) < 1e-7
    lonely = np.flatnonzero(np.diff(g.rowptr) == 0)
    assert not z[:, lonely].any()
    h, zh = nvd.ge_distance(G, X, Y, rtol=1e-11, return_z=True)              # host buffers
    assert np.array_equal(d2.cpu().numpy(), h.numpy()) and np.array_equal(z.cpu().numpy(), zh.numpy())
    X32, Y32 = X.astype(np.float32), Y.astype(np.float32)
    f = nvd.ge_distance(G, torch.as_tensor(X32, device=DEV), torch.as_tensor(Y32, device=DEV), rtol=1e-11)
    assert rel(f.cpu().numpy(), ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, X32.astype(float), Y32.astype(float),
                                             rtol=1e-13)[0]) < 1e-10
    ids = np.flatnonzero(np.diff(g.rowptr) > 0)
    u, v = ids[:k], ids[100:100 + k]                                         # node-id pairs
    E, F = np.zeros((k, g.n)), np.zeros((k, g.n))
    E[np.arange(k), u] = 1.0
    F[np.arange(k), v] = 1.0
    R = nvd.effective_resistance(G, u, v, rtol=1e-11)
    assert last(nvd, G)[:2] == (form, width)
    assert rel(R, ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, E, F, rtol=1e-13)[0]) < 1e-10
    _, st = nvd.ge_distance(G, on(X), on(Y), rtol=1e-11, max_iter=4, return_stats=True, allow_not_converged=True)
    assert all(s["status"] == 6 and s["iters"] == 4 for s in st)
    s2 = nvd.ge_distance(G, on(X), on(Y), rtol=1e-14, d2_stop=True, d2_rtol=1e-6)
    assert rel(s2.cpu().numpy(), want) <= 1e-6
    Xn = X.copy()
    Xn[k - 1, ids[5]] = np.nan                                               # the last pair alone fails
    with pytest.raises(nvd.NvdError) as e:
        nvd.ge_distance(G, on(Xn), on(Y), rtol=1e-11)
    assert e.value.status == 7
    g2 = synth.csr_from_edges(g.n, g.eu, g.ev, np.random.default_rng(3).uniform(0.5, 2.0, g.m))
    G.set_weights(g2.w)
    got = nvd.ge_distance(G, on(X), on(Y), rtol=1e-11).cpu().numpy()
    assert last(nvd, G)[:2] == (form, width)
    assert rel(got, ocg.ge_d2_cg(g2.n, g2.rowptr, g2.colidx, g2.w, X, Y, rtol=1e-13)[0]) < 1e-10


def test_one_kernel_with_x_in_global_memory(nvd):
    g = hub_graph(70001, [500], 2)
    X, Y = synth.sparse_uniform_pairs(g.n, 18, 0.02, 5)
    G = nvd.Graph.from_csr(g)
    force(nvd, G, RESIDENT, 16)
    d2 = nvd.ge_distance(G, on(X), on(Y), rtol=1e-11).cpu().numpy()
    assert last(nvd, G) == (RESIDENT, 16, 1)
    pick = [0, 15, 17]
    assert rel(d2[pick], ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, X[pick], Y[pick], rtol=1e-13)[0]) < 1e-10


# 224 KB of shared memory per CTA, S slots a CTA: p replicated takes 8 S C of them (C CTAs), the
# matrix about 12 bytes per stored entry, r, x, q and scratch 8 S each and 16 KB (r and x in
# registers up to 1,024 slots); p goes through L2 from 40 KB on
@pytest.mark.parametrize("kind,n,width,cs,variant", [
    ("ws", 500, 16, 1, MATRIX | ONE_SLOT), ("ws", 2000, 4, 4, MATRIX | ONE_SLOT),
    ("ws", 6000, 16, 16, MATRIX | ONE_SLOT | VIA_L2), ("ws8", 15000, 16, 16, ONE_SLOT | VIA_L2),
    ("ws", 1100, 1, 1, MATRIX), ("ws8", 4000, 2, 2, 0), ("ws8", 6000, 2, 2, VIA_L2),
    ("ws", 26001, 16, 16, GLOBAL_P | VIA_L2)])
def test_every_cluster_kernel(nvd, kind, n, width, cs, variant):
    rng = np.random.default_rng(n)
    eu, ev = synth.watts_strogatz(n, 8 if kind == "ws8" else 4, 0.2, rng)
    g = synth.csr_from_edges(n, eu, ev, rng.uniform(0.5, 2.0, len(eu)))
    X, Y = synth.sparse_uniform_pairs(g.n, 5, 0.05, 3)
    G = nvd.Graph.from_csr(g)
    force(nvd, G, CLUSTER, width)
    d2, st = nvd.ge_distance(G, on(X), on(Y), rtol=1e-12, return_stats=True)
    assert last(nvd, G) == (CLUSTER, cs, variant)
    assert all(s["status"] == 0 for s in st)
    assert rel(d2.cpu().numpy(), ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, X, Y, rtol=1e-13)[0]) < 1e-10


def test_open_calls_take_the_estimated_form(nvd, case):
    """Small graphs the cluster form, explicit widths the tiles, and a form that cannot hold the
    graph is refused."""
    g, X, Y, want = case
    small = synth.csr_from_edges(500, *synth.barabasi_albert(500, 3, np.random.default_rng(1)), np.ones(1491))
    G = nvd.Graph.from_csr(small)
    x, y = torch.rand(4, 500, dtype=torch.float64, device=DEV), torch.rand(4, 500, dtype=torch.float64, device=DEV)
    nvd.ge_distance(G, x, y)
    assert last(nvd, G)[0] == CLUSTER
    nvd.ge_distance(G, x, y, kt=16)
    assert last(nvd, G) == (TILES, 16, 0)
    force(nvd, G, RESIDENT, 2)
    with pytest.raises(nvd.NvdError) as e:
        nvd.ge_distance(G, x, y)
    assert e.value.status == 9
    force(nvd, G, 0, 0)
    nvd.ge_distance(G, x, y)
    assert last(nvd, G)[0] == CLUSTER


def test_one_kernel_wait_that_gives_up(nvd, case):
    """The grid meeting waits for one arrival more than the grid has, so its bounded wait (2 s)
    runs out in the first of three tiles: one NVD_ERR_TIMEOUT for the call, the later tiles leave
    at once, and the next solve on the handle is right."""
    g, X, Y, want = case
    G = nvd.Graph.from_csr(g)
    force(nvd, G, RESIDENT, 8)
    d2 = nvd.ge_distance(G, on(X), on(Y), rtol=1e-11)
    t0 = time.perf_counter()
    with pytest.raises(nvd.NvdError) as e:
        nvd.ge_distance(G, on(X), on(Y), rtol=1e-11, test_timeout=True)
    dt = time.perf_counter() - t0
    assert e.value.status == 8 and last(nvd, G)[:2] == (RESIDENT, 8)
    assert 1.5 < dt < 3.5                                # one wait of 2 s, not one per tile
    again = nvd.ge_distance(G, on(X), on(Y), rtol=1e-11)
    assert torch.equal(d2, again) and rel(again.cpu().numpy(), want) < 1e-10
    # an open call with the flag keeps the tiles, which have no such wait
    force(nvd, G, 0, 0)
    t = nvd.ge_distance(G, on(X), on(Y), rtol=1e-11, test_timeout=True).cpu().numpy()
    assert last(nvd, G)[0] == TILES and rel(t, want) < 1e-10


# 5 pairs: tiles of 4 and of 8 columns are both estimated to beat the host-driven ones; 16 pairs: 8 and 16
@pytest.mark.parametrize("n,k", [(100003, 5), (70001, 16), (31003, 16), (2000, 16)])
def test_only_the_plan_that_is_used_is_built(nvd, n, k):
    rng = np.random.default_rng(n)
    eu, ev = synth.watts_strogatz(n, 10, 0.3, rng)
    g = synth.csr_from_edges(n, eu, ev, rng.uniform(0.5, 2.0, len(eu)))
    x, y = torch.rand(k, n, dtype=torch.float64, device=DEV), torch.rand(k, n, dtype=torch.float64, device=DEV)
    G = nvd.Graph.from_csr(g)
    d2 = nvd.ge_distance(G, x, y, rtol=1e-10)
    form, width, _ = last(nvd, G)
    H = nvd.Graph.from_csr(g)
    force(nvd, H, form, 16 if form == CLUSTER else width)
    assert torch.equal(d2, nvd.ge_distance(H, x, y, rtol=1e-10))
    assert last(nvd, H)[:2] == (form, width)
    assert G.info()["device_bytes"] == H.info()["device_bytes"]


def test_a_cluster_plan_that_does_not_fit_holds_no_memory(nvd):
    """Hubs take so much of some CTAs' time that the others' rows exceed their shared memory: the
    form is refused when asked for, and an open call takes another."""
    n = 100000
    g = hub_graph(n, [60000] * 8, 4)
    X, Y = synth.sparse_uniform_pairs(g.n, 3, 0.02, 5)
    G = nvd.Graph.from_csr(g)
    before = G.info()["device_bytes"]
    force(nvd, G, CLUSTER, 16)
    with pytest.raises(nvd.NvdError) as e:
        nvd.ge_distance(G, on(X), on(Y), rtol=1e-11)
    assert e.value.status == 9 and G.info()["device_bytes"] == before
    G.set_weights(g.w)
    force(nvd, G, 0, 0)
    d2 = nvd.ge_distance(G, on(X), on(Y), rtol=1e-11).cpu().numpy()
    assert last(nvd, G)[0] != CLUSTER
    assert rel(d2, ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, X, Y, rtol=1e-13)[0]) < 1e-10
