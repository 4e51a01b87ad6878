"""Scratch memory of the on-chip FP64 solves: bounded by more than the call's size, and where
it cannot be had the solve takes fewer tasks at a time or the tiles, with the same result."""
import ctypes

import numpy as np
import pytest
import torch

import synth
from oracle import cg as ocg
from oracle import dense

pytestmark = pytest.mark.gpu
DEV = "cuda"
TILES, CLUSTER, RESIDENT = 1, 2, 3


@pytest.fixture(scope="module")
def nvd():
    import paper_2310_11222_gb300 as m
    m.load_library()
    return m


def on(x):
    return torch.as_tensor(x, dtype=torch.float64, device=DEV)


def rel(a, b):
    return np.max(np.abs(a - b) / np.maximum(np.abs(b), 1e-300))


def last_form(nvd, G):
    v = [ctypes.c_int32() for _ in range(3)]
    nvd.load_library().nvd_diag_last_form(G.handle, *[ctypes.byref(c) for c in v])
    return v[0].value


def limit(nvd, G, nbytes):
    assert nvd.load_library().nvd_diag_alloc_limit(G.handle, ctypes.c_int64(nbytes)) == 0


def force(nvd, G, form, width):
    assert nvd.load_library().nvd_diag_force_form(G.handle, form, width) == 0


def test_many_components_and_pairs(nvd):
    """Results per (component, pair) are kept for so many pairs at a time: 20,001 components and
    1,500 node-id pairs would be 960 MB of them."""
    rng = np.random.default_rng(2)
    eu, ev = synth.barabasi_albert(400, 4, rng)
    a = 400 + 2 * np.arange(20000)
    u, v = np.concatenate([eu, a]), np.concatenate([ev, a + 1])
    w = rng.uniform(0.5, 2.0, len(u))
    g = synth.csr_from_edges(40400, u, v, w)
    G = nvd.Graph.from_csr(g)
    k = 1500
    s, t = rng.integers(0, 400, k), rng.integers(0, 399, k)
    t = np.where(t >= s, t + 1, t)
    s[7], t[7] = a[5], a[5] + 1
    R, st = nvd.effective_resistance(G, s, t, rtol=1e-12, return_stats=True)
    assert G.info()["device_bytes"] < 300 << 20
    assert all(x["status"] == 0 for x in st)
    sub = synth.csr_from_edges(400, eu, ev, w[:len(eu)])
    L = np.linalg.pinv(dense.laplacian_dense(sub.n, sub.rowptr, sub.colidx, sub.w))
    keep = np.arange(k) != 7
    i, j = s[keep], t[keep]
    assert rel(R[keep], L[i, i] - 2 * L[i, j] + L[j, j]) < 1e-10
    assert abs(R[7] * w[len(eu) + 5] - 1.0) < 1e-12


@pytest.fixture(scope="module")
def ring():
    rng = np.random.default_rng(5)
    eu, ev = synth.watts_strogatz(20011, 6, 0.2, rng)
    g = synth.csr_from_edges(20011, eu, ev, rng.uniform(0.5, 2.0, len(eu)))
    X, Y = synth.sparse_uniform_pairs(g.n, 40, 0.05, 3)
    pick = [0, 15, 16, 39]
    return g, X, Y, pick, ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, X[pick], Y[pick], rtol=1e-13)[0]


# d^2 is second order in the residual (1e-11): 1e-10 leaves room for rounding only.  One column of
# p is 160 KB, all 40 are 6.4 MB, a tile vector of 16 columns 2.6 MB.
def test_fewer_tasks_at_a_time(nvd, ring):
    g, X, Y, pick, want = ring
    G = nvd.Graph.from_csr(g)
    force(nvd, G, CLUSTER, 16)
    limit(nvd, G, 1 << 20)
    d2 = nvd.ge_distance(G, on(X), on(Y), rtol=1e-11)
    assert last_form(nvd, G) == CLUSTER and G.info()["device_bytes"] < 16 << 20
    limit(nvd, G, 0)
    H = nvd.Graph.from_csr(g)
    force(nvd, H, CLUSTER, 16)
    assert torch.equal(d2, nvd.ge_distance(H, on(X), on(Y), rtol=1e-11))
    assert rel(d2.cpu().numpy()[pick], want) < 1e-10


@pytest.mark.parametrize("form,width", [(CLUSTER, 16), (RESIDENT, 16)])
@pytest.mark.parametrize("host", [False, True])
def test_without_memory_the_tiles(nvd, ring, form, width, host):
    """Device inputs: the tiles' workspaces are there, the on-chip ones are refused.  Host inputs:
    room for a tile's staging, not for that of the whole call."""
    g, X, Y, pick, want = ring
    G = nvd.Graph.from_csr(g)
    args = (X, Y) if host else (on(X), on(Y))
    if not host:
        nvd.ge_distance(G, *args, rtol=1e-2, kt=16)
    force(nvd, G, form, width)
    limit(nvd, G, 3 << 20 if host else 100 << 10)
    d2, z, st = nvd.ge_distance(G, *args, rtol=1e-11, return_z=True, return_stats=True)
    assert last_form(nvd, G) == TILES and all(s["status"] == 0 for s in st)
    assert rel(d2.cpu().numpy()[pick], want) < 1e-10
    assert nvd.load_library().nvd_last_error() == b""
    limit(nvd, G, 0)
    again, z2 = nvd.ge_distance(G, *args, rtol=1e-11, return_z=True)
    assert last_form(nvd, G) == form
    assert rel(again.cpu().numpy()[pick], want) < 1e-10
    assert float((z - z2).norm() / z.norm()) < 1e-7


def test_batches_without_memory(nvd):
    rng = np.random.default_rng(9)
    gs, pairs = [], []
    for n in (64, 500, 6001):
        eu, ev = synth.barabasi_albert(n, 3, rng)
        gs.append(synth.csr_from_edges(n, eu, ev, rng.uniform(0.5, 2.0, len(eu))))
        pairs.append(synth.sparse_uniform_pairs(n, 3, 0.2, n))
    G = [nvd.Graph.from_csr(g) for g in gs]
    xs, ys = [on(x) for x, _ in pairs], [on(y) for _, y in pairs]

    def call(rtol):
        l0 = nvd.kernel_launches()
        d2 = nvd.ge_distance_batched(G, xs, ys, mode=nvd.MODE_FP64, rtol=rtol).numpy()
        return d2, nvd.kernel_launches() - l0

    nvd.ge_distance_batched(G, xs, ys, mode=nvd.MODE_FP64, rtol=1e-2, fold_direction=True)   # the tiles' workspaces
    limit(nvd, G[0], 64)            # nothing that is not there yet
    d2, launches = call(1e-12)
    assert launches > 20            # host-driven
    limit(nvd, G[0], 0)
    d2c, launches = call(1e-12)
    assert launches <= 8            # clusters
    want = np.concatenate([ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, x, y, rtol=1e-13)[0]
                           for g, (x, y) in zip(gs, pairs)])
    assert rel(d2, want) < 1e-10 and rel(d2c, want) < 1e-10


# One direction of every pair only: the 130,816 entries are an edge each, 16 bytes of places and 8
# of nodes.  z tile 512 nodes x 32 columns x 8 bytes = 131 KB; with several tiles or unsorted columns
# the gradient of every entry, 8 bytes (1,046,528 in all).
@pytest.mark.parametrize("k", [1, 4, 7, 16, 32, 40])
@pytest.mark.parametrize("zt,wt", [(np.float64, np.float64), (np.float32, np.float32), (np.float64, np.float32)])
def test_weight_gradient_without_an_edge_list(nvd, k, zt, wt):
    rng = np.random.default_rng([k, 4])
    n = 512
    rows, cols = np.triu_indices(n, 1)
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))])
    if k >= 16:                                  # unsorted columns: entries reach the handle by a map
        cols[[0, 1]] = cols[[1, 0]]
    G = nvd.Graph(rowptr, cols.astype(np.int32), np.ones(len(rows), wt), skip_sym_check=True)
    z = rng.standard_normal((k, n)).astype(zt)
    gbar = rng.uniform(-1.0, 1.0, k)
    args = (torch.as_tensor(z, device=DEV), torch.as_tensor(gbar, device=DEV))
    limit(nvd, G, 1100000)
    before = G.info()["device_bytes"]
    gw = nvd.ge_grad(G, *args)[0].cpu().numpy()
    assert G.info()["device_bytes"] - before < 1300000
    d = z.astype(np.float64)[:, rows] - z.astype(np.float64)[:, cols]
    want, size = -0.5 * (gbar[:, None] * d * d).sum(0), 0.5 * (np.abs(gbar)[:, None] * d * d).sum(0)
    # FP64 sums of k terms; rounded once to the weights' type
    tol = 1e-13 * size + (1e-7 * np.abs(want) if wt == np.float32 else 0.0)
    assert np.all(np.abs(gw - want) <= tol + 1e-300)
    limit(nvd, G, 0)
    full = nvd.ge_grad(G, *args)[0].cpu().numpy()
    assert G.info()["device_bytes"] - before > 3000000
    assert np.all(np.abs(full - want) <= tol + 1e-300)
