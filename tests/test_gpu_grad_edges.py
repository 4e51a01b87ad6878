"""The weight gradient over the undirected edge list: every tile width, ragged widths and
several tiles, FP64 and FP32 z and weights, repeated entries and self-loops, and a pattern with
entries whose mirror is not stored, against the formula per stored entry."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def nvd():
    import paper_2310_11222_gb300 as m
    m.load_library()
    return m


def csr(n, rows, cols, vals):
    order = np.lexsort((np.arange(len(rows)), rows))
    ptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(rows, minlength=n), out=ptr[1:])
    return ptr, cols[order].astype(np.int32), vals[order], rows[order]


def entries(rng, n, m):
    """A hub, random pairs (some repeated) and self-loops, both directions of every pair."""
    u = np.concatenate([np.zeros(n // 2, np.int64), rng.integers(0, n, m)])
    v = np.concatenate([rng.permutation(np.arange(1, n))[:n // 2], rng.integers(0, n, m)])
    u, v = u[u != v], v[u != v]
    loops = rng.integers(0, n, 7)
    w = rng.uniform(0.5, 2.0, len(u))
    return (np.concatenate([u, v, loops]), np.concatenate([v, u, loops]),
            np.concatenate([w, w, np.ones(len(loops))]))


@pytest.mark.parametrize("k", [1, 3, 4, 7, 8, 13, 16, 31, 32, 40])
@pytest.mark.parametrize("zt,wt", [(np.float64, np.float64), (np.float32, np.float32), (np.float64, np.float32)])
def test_every_width_and_type(nvd, k, zt, wt):
    rng = np.random.default_rng([k, 3])
    n = 531
    ptr, cols, w, rows = csr(n, *entries(rng, n, 1200))
    G = nvd.Graph(ptr, cols, w.astype(wt))
    z = rng.standard_normal((k, n)).astype(zt)
    gbar = rng.uniform(-1.0, 1.0, k)
    gw, _, _ = nvd.ge_grad(G, torch.as_tensor(z, device=DEV), torch.as_tensor(gbar, device=DEV))
    d = z.astype(np.float64)[:, rows] - z.astype(np.float64)[:, cols]
    want, size = -0.5 * (gbar[:, None] * d * d).sum(0), 0.5 * (np.abs(gbar)[:, None] * d * d).sum(0)
    # FP64 sums of k terms; rounded once to the weights' type
    tol = 1e-13 * size + (1e-7 * np.abs(want) if wt == np.float32 else 0.0)
    assert np.all(np.abs(gw.cpu().numpy() - want) <= tol + 1e-300)


def test_entries_without_a_mirror(nvd):
    rng = np.random.default_rng(8)
    n = 300
    u, v = rng.integers(0, n, 900), rng.integers(0, n, 900)
    u, v = u[u != v], v[u != v]
    key = np.unique(u * n + v)                       # one direction of most pairs only
    ptr, cols, w, rows = csr(n, key // n, key % n, np.ones(len(key)))
    G = nvd.Graph(ptr, cols, w, skip_sym_check=True)
    z = rng.standard_normal((5, n))
    gbar = rng.uniform(0.5, 1.0, 5)
    gw, _, _ = nvd.ge_grad(G, torch.as_tensor(z, device=DEV), torch.as_tensor(gbar, device=DEV))
    d = z[:, rows] - z[:, cols]
    want = -0.5 * (gbar[:, None] * d * d).sum(0)
    assert np.max(np.abs(gw.cpu().numpy() - want) / np.maximum(np.abs(want), 1e-300)) < 1e-12
