"""Chains followed by the Gamma sum beyond the last pointer-jumping round.

Particles on a line away from one source give chains of every length up to
the line's; isolated particles (no neighbours, chains of one link) beside them
set how many slots a round leaves open, so that short lines are followed from
the first round on, long ones past every block size, and a line alone takes
further rounds.  The counting form (compensated double-float sums of the same
links) is the reference: FP32 sums of L links differ from it by at most
log4(L) levels of three additions each, u (3 log4 L + 4) tau in Gamma.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24


def line(n, isolated, seed):
    """n particles spaced 1 along x with a small offset, their smoothing
    length reaching two spacings; isolated particles 50 apart."""
    rng = np.random.default_rng(seed)
    m = int(np.ceil(np.sqrt(max(isolated, 1))))
    k = np.arange(isolated)
    x = np.concatenate([np.arange(1, n + 1) + rng.uniform(-0.2, 0.2, n), 50.0 * (k // m)])
    y = np.concatenate([rng.uniform(-0.05, 0.05, n), 50.0 * (k % m) + 100.0])
    z = np.concatenate([rng.uniform(-0.05, 0.05, n), np.full(isolated, 300.0)])
    h = np.concatenate([np.full(n, 1.05), np.full(isolated, 1.0)]).astype(np.float32)
    return np.stack([x, y, z]).astype(np.float32), h


@pytest.mark.parametrize("n,isolated", [(3, 100), (4, 100), (5, 300), (16, 600), (17, 600),
                                        (63, 9000), (65, 9000), (257, 20000), (1023, 60000),
                                        (5000, 200000), (40, 0), (1500, 0)])
def test_open_chains_match_the_counting_form(n, isolated):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1005_5312_gb300 as S
    S.build()
    pos, h = line(n, isolated, n + isolated)
    n_p = pos.shape[1]
    out = {}
    for counts in (0, 1):
        ctx = S.Context(link_counts=counts, sigma_cm2=1.0, len_unit_cm=1.0)
        ctx.build_trees(pos, h, np.zeros((3, 1), np.float32), np.array([1e48]))
        g = np.zeros(n_p, np.float32)
        # the line is 4 deep in all; the isolated particles are transparent
        n_HI = np.concatenate([np.full(n, 4.0 / n), np.full(isolated, 1e-9)]).astype(np.float32)
        ctx.rt_solve(1.0, n_HI=n_HI, gamma_out=g)
        out[counts] = (g.astype(np.float64), ctx.stats())
    st = out[1][1]
    assert st["max_hops"] > 0.4 * n
    tol = U32 * (3 * np.log2(max(st["max_hops"], 2)) / 2 + 4) * 6.0 + 4 * U32
    np.testing.assert_allclose(out[0][0], out[1][0], rtol=tol)
    rounds = out[0][1]["jump_rounds"]
    assert rounds == 1 if isolated else rounds >= 1
    if (n, isolated) == (1500, 0):
        assert rounds > 1
