"""Blocks of one to four waves per launch on graphs of several components of equal size, against
the oracle on one component."""
import numpy as np
import pytest
import torch

import synth
from oracle import cg as ocg

pytestmark = pytest.mark.gpu
DEV = "cuda"
K = 16


@pytest.fixture(scope="module")
def nvd():
    import paper_2310_11222_gb300 as m
    m.load_library()
    return m


@pytest.fixture(scope="module")
def base():
    rng = np.random.default_rng(3)
    n = 60000
    eu, ev = synth.watts_strogatz(n, 6, 0.1, rng)
    g = synth.csr_from_edges(n, eu, ev, rng.uniform(0.5, 2.0, len(eu)))
    X, Y = synth.sparse_uniform_pairs(n, K, 0.05, 8)
    return g, X, Y, ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, X, Y, rtol=1e-13)[0]


# copies x 60,000 rows x 16 columns x 8 bytes: 15 and 23 MB (one wave), 46 (two), 69 (three), 100 (four).
# d^2 is second order in the residual (1e-11): 1e-10 leaves room for rounding only
@pytest.mark.parametrize("copies", [2, 3, 6, 9, 13])
def test_components_of_equal_size(nvd, base, copies):
    g, X, Y, want = base
    u, off = synth.disjoint_union([g] * copies)
    G = nvd.Graph.from_csr(u)
    x = torch.zeros((K, u.n), dtype=torch.float64, device=DEV)
    y = torch.zeros_like(x)
    for j in range(K):
        o = int(off[j % copies])
        x[j, o:o + g.n] = torch.as_tensor(X[j], device=DEV)
        y[j, o:o + g.n] = torch.as_tensor(Y[j], device=DEV)
    for kw in (dict(kt=16), dict(kt=16, persistent=True)):
        d2 = nvd.ge_distance(G, x, y, rtol=1e-11, **kw).cpu().numpy()
        assert np.max(np.abs(d2 - want) / want) < 1e-10, kw
