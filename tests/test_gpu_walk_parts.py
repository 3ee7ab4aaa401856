"""One-walk interaction lists cut into parts per target: parts longer than
their scratch (walked again into place), parts without entries, trees of one
cell, an emitter tree whose targets sit at its first and last leaves, a batch
(each problem's tree a range of the forest).  Rays, evaluations and Gamma of
the memoised march against the per-ray march, which walks each target once
and uncut; the opening tests decided in FP64 are counted once per target.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def run(S, mode, theta, pos, h, src, L, V=None, walk_warp=0):
    n = len(h)
    ctx = S.Context(march_mode=mode, link_counts=mode, tau_cut=1e30, walk_warp=walk_warp)
    ctx.build_trees(pos, h, src, L, V, diffuse=V is not None)
    rng = np.random.default_rng(n)
    ctx.set_state(rng.uniform(0, 2e-4, n).astype(np.float32), rng.uniform(0.1, 1.0, n))
    g = np.zeros(n, np.float32)
    ctx.rt_solve(theta, gamma_out=g)
    return g.astype(np.float64), ctx.stats()


@pytest.mark.parametrize("n_p,n_s,theta,diffuse", [
    (1, 1, 0.5, False), (37, 2, 0.5, False), (200, 3, 1.0, False), (300, 4500, 0.0, False),
    (129, 9000, 0.3, False), (2, 0, 0.7, True), (33, 1, 0.7, True), (5000, 3, 0.0, True),
    (5000, 40, 0.8, True)])
def test_cut_walks_give_the_uncut_rows(n_p, n_s, theta, diffuse):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1005_5312_gb300 as S
    S.build()
    rng = np.random.default_rng(n_p + n_s)
    pos = rng.uniform(0.0, 2.0, (3, n_p)).astype(np.float32)
    h = np.full(n_p, 0.5 * 2.0 * (30.0 / (4.2 * max(n_p, 30))) ** (1 / 3), np.float32)
    src = rng.uniform(0.0, 2.0, (3, n_s)).astype(np.float32)
    L = rng.lognormal(0.0, 1.0, n_s) * 1e48
    V = np.full(n_p, 8.0 / n_p) if diffuse else None
    g1, s1 = run(S, 1, theta, pos, h, src, L, V)
    g0, s0 = run(S, 0, theta, pos, h, src, L, V)
    gw, sw = run(S, 1, theta, pos, h, src, L, V, walk_warp=1)   # not cut
    assert s1["rays"] == s0["rays"] and s1["hops"] == s0["hops"]
    assert s1["walk_fallbacks"] == s0["walk_fallbacks"]
    assert np.array_equal(g1, gw) and s1["evals"] == sw["evals"]
    # compensated sums of the same links either way
    np.testing.assert_allclose(g1, g0, rtol=2e-5)
