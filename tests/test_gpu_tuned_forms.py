"""What a tuning, or one applied again from its result, leaves the form of later FP64 solves at."""
import ctypes

import numpy as np
import pytest
import torch

import synth
from oracle import cg as ocg

pytestmark = pytest.mark.gpu
DEV = "cuda"
TILES, CLUSTER, RESIDENT = 1, 2, 3


@pytest.fixture(scope="module")
def nvd():
    import paper_2310_11222_gb300 as m
    m.load_library()
    return m


def last(nvd, G):
    v = [ctypes.c_int32() for _ in range(3)]
    nvd.load_library().nvd_diag_last_form(G.handle, *[ctypes.byref(c) for c in v])
    return v[0].value, v[1].value


def graph(n, seed):
    rng = np.random.default_rng(seed)
    eu, ev = synth.watts_strogatz(n, 10, 0.3, rng)
    return synth.csr_from_edges(n, eu, ev, rng.uniform(0.5, 2.0, len(eu)))


def pairs(n, k):
    return synth.sparse_uniform_pairs(n, k, 0.1, 7)


def on(x):
    return torch.as_tensor(x, dtype=torch.float64, device=DEV)


KEYS = ("kt", "row_max_pct", "blocks_pct", "persistent", "fold_direction", "gather", "l2_hot")


@pytest.mark.parametrize("n", [2000, 40000])
def test_single_tuning_and_its_result_take_the_same_form(nvd, n):
    """The one-launch forms are several times faster here than any tiles."""
    g = graph(n, 1)
    X, Y = pairs(n, 3)
    want = ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, X, Y, rtol=1e-13)[0]
    G, H, U = (nvd.Graph.from_csr(g) for _ in range(3))
    r = G.tune(mode=nvd.MODE_FP64, k=3, single_rhs=True)
    H.set_tuning(mode=nvd.MODE_FP64, **{f: r[f] for f in KEYS})
    forms = []
    for K in (G, H, U):
        d2 = nvd.ge_distance(K, on(X), on(Y), rtol=1e-11, single_rhs=True).cpu().numpy()
        assert np.max(np.abs(d2 - want) / want) < 1e-10
        forms.append(last(nvd, K))
        nvd.ge_distance(K, on(X[0]), on(Y[0]), rtol=1e-11)
        forms.append(last(nvd, K))
    assert forms[0:2] == forms[2:4] == forms[4:6] and TILES not in [f for f, _ in forms]


def test_tiles_that_won_are_taken(nvd):
    """An open form made slow (90,000 rows on one cluster of 16 CTAs, about twice the tiles'
    time): later open calls take the tiles, on the tuned handle and on one set from its result."""
    n = 90000
    g = graph(n, 2)
    X, Y = pairs(n, 1)
    want = ocg.ge_d2_cg(g.n, g.rowptr, g.colidx, g.w, X, Y, rtol=1e-13)[0]
    lib = nvd.load_library()
    G, H, U = (nvd.Graph.from_csr(g) for _ in range(3))
    for K in (G, H, U):
        assert lib.nvd_diag_force_form(K.handle, CLUSTER, 16) == 0
    nvd.ge_distance(U, on(X), on(Y), rtol=1e-11)
    assert last(nvd, U) == (CLUSTER, 16)
    r = G.tune(mode=nvd.MODE_FP64, k=1, single_rhs=True)
    assert r["persistent"] or r["fold_direction"]
    H.set_tuning(mode=nvd.MODE_FP64, **{f: r[f] for f in KEYS})
    for K in (G, H):
        d2 = nvd.ge_distance(K, on(X), on(Y), rtol=1e-11).cpu().numpy()
        assert last(nvd, K) == (TILES, 1)
        assert np.max(np.abs(d2 - want) / want) < 1e-10


def test_settings_and_forms(nvd):
    """Which settings leave a call of one and of several right-hand sides its on-chip form."""
    g = graph(2000, 3)
    X, Y = pairs(2000, 12)
    table = [  # setting, form of one right-hand side, form of twelve
        (dict(), CLUSTER, CLUSTER), (dict(kt=1), CLUSTER, TILES), (dict(kt=16), TILES, TILES),
        (dict(persistent=-1), TILES, CLUSTER), (dict(kt=1, persistent=-1), TILES, TILES),
        (dict(persistent=True), TILES, TILES), (dict(fold_direction=True), TILES, TILES)]
    for setting, one, several in table:
        G = nvd.Graph.from_csr(g)
        G.set_tuning(mode=nvd.MODE_FP64, **setting)
        nvd.ge_distance(G, on(X[:1]), on(Y[:1]))
        assert last(nvd, G)[0] == one, setting
        nvd.ge_distance(G, on(X), on(Y), single_rhs=True)
        assert last(nvd, G)[0] == one, setting
        nvd.ge_distance(G, on(X), on(Y))
        assert last(nvd, G)[0] == several, setting
    with pytest.raises(nvd.NvdError):
        r = nvd.TuneResult(kt=1, row_max_pct=100, blocks_pct=100, persistent=-2)
        nvd._check(nvd.load_library().nvd_graph_set_tuning(G.handle, 0, ctypes.byref(r)), "nvd_graph_set_tuning")
