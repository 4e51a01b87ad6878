"""Block counts of the tiled launches: settings below one wave are one plan with one wave, more
waves and row limits on graphs of one and of several components match the oracle."""
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


@pytest.fixture(scope="module")
def cases():
    """A ring with hubs around the light-row limits, alone and beside three other components."""
    rng = np.random.default_rng(6)
    n = 9000
    eu, ev = synth.watts_strogatz(n, 6, 0.1, rng)
    key = [np.minimum(eu, ev) * n + np.maximum(eu, ev)]
    for h, d in enumerate((60, 130, 300, 700, 3000)):
        key.append(np.int64(h) * n + rng.choice(np.arange(5, n), size=d, replace=False))
    key = np.unique(np.concatenate(key))
    one = synth.csr_from_edges(n, key // n, key % n, rng.uniform(0.5, 2.0, len(key)))
    more = [one]
    for m in (2500, 7000, 300):
        u, v = synth.barabasi_albert(m, 4, rng)
        more.append(synth.csr_from_edges(m, u, v, rng.uniform(0.5, 2.0, len(u))))
    several, _ = synth.disjoint_union(more)
    out = []
    for g in (one, several):
        X, Y = rng.random((9, g.n)), rng.random((9, g.n))
        out.append((g, X, Y, ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, X, Y, rtol=1e-13)[0]))
    return out


# d^2 is second order in the residual (1e-12): 1e-10 leaves room for rounding only
@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("blocks_pct", [150, 200, 400, 1000])
@pytest.mark.parametrize("row_max_pct", [50, 100, 200])
def test_more_waves(nvd, cases, which, blocks_pct, row_max_pct):
    g, X, Y, want = cases[which]
    G = nvd.Graph.from_csr(g)
    G.set_tuning(mode=nvd.MODE_FP64, row_max_pct=row_max_pct, blocks_pct=blocks_pct)
    for kt in (1, 4, 16):
        d2 = nvd.ge_distance(G, on(X), on(Y), rtol=1e-12, kt=kt).cpu().numpy()
        assert np.max(np.abs(d2 - want) / want) < 1e-10, kt


def test_less_than_a_wave_is_one_plan(nvd, cases):
    g, X, Y, _ = cases[0]
    G = nvd.Graph.from_csr(g)
    got = []
    for pct in (100, 50, 10):
        G.set_tuning(mode=nvd.MODE_FP64, blocks_pct=pct)
        got.append((nvd.ge_distance(G, on(X), on(Y), rtol=1e-12, kt=4), G.info()["device_bytes"]))
    for d2, nbytes in got[1:]:
        assert torch.equal(d2, got[0][0]) and nbytes == got[0][1]
