"""Kernel timing of a batched FP64 solve: the host-driven launches run and are counted while it
is on, and the result is that of the call without it."""
import numpy as np
import pytest
import torch

import synth
from oracle import dense

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def nvd():
    import paper_2310_11222_gb300 as m
    m.load_library()
    return m


def test_batched_launches_are_timed(nvd):
    rng = np.random.default_rng(5)
    gs, pairs = [], []
    for n in (60, 300, 900):
        eu, ev = synth.barabasi_albert(n, 3, rng)
        gs.append(synth.csr_from_edges(n, eu, ev, rng.uniform(0.5, 2.0, len(eu))))
        pairs.append(synth.diffuse_uniform_pairs(n, 3, n))
    G = [nvd.Graph.from_csr(g) for g in gs]
    xs = [torch.as_tensor(x, device=DEV) for x, _ in pairs]
    ys = [torch.as_tensor(y, device=DEV) for _, y in pairs]

    def call():
        return nvd.ge_distance_batched(G, xs, ys, mode=nvd.MODE_FP64, rtol=1e-12, return_stats=True)

    plain, _ = call()
    nvd.profile_enable(True)
    try:
        nvd.profile_read(0)
        timed, st = call()
        launches, ms, _ = nvd.profile_read(0)
    finally:
        nvd.profile_enable(False)
    assert launches >= max(s["iters"] for s in st) and ms > 0.0
    want = np.concatenate([dense.ge_d2_eig(g.n, g.rowptr, g.colidx, g.w, x, y) for g, (x, y) in zip(gs, pairs)])
    # d^2 is second order in the residual (1e-12): 1e-10 leaves room for rounding only
    for got in (plain.numpy(), timed.numpy()):
        assert np.max(np.abs(got - want) / want) < 1e-10
