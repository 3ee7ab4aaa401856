"""The first hop's row search and candidate scan at the sizes where they
change shape.

At theta = 0 every particle lists every source, so a row holds n_s entries and
every link's upstream pair is in its row: a missed entry would be claimed as a
link outside the lists and show as an evaluation more than there are rays.
Chain lengths and Gamma are compared with the per-ray march, which shares
neither the search nor the staged scan.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def workload(n_p, n_s, neighbours, seed):
    rng = np.random.default_rng(seed)
    pos = rng.uniform(0.0, 3.0, (3, n_p)).astype(np.float32)
    d = np.sort(np.sqrt(((pos[:, :, None] - pos[:, None, :]).astype(np.float64) ** 2).sum(0)), 1)
    two_h = 0.5 * (d[:, neighbours] + d[:, neighbours + 1])   # d[:, 0] is the particle itself
    src = rng.uniform(0.0, 3.0, (3, n_s)).astype(np.float32)
    return pos, (0.5 * two_h).astype(np.float32), src, rng.lognormal(0.0, 1.0, n_s) * 1e48


@pytest.mark.parametrize("n_s", [1, 2, 7, 8, 9, 10, 11, 31, 32, 33, 34, 35, 143, 257])
@pytest.mark.parametrize("neighbours,row_bins", [(1, 4), (4, 0), (5, 4), (32, 4), (63, 4), (64, 0),
                                                 (65, 4)])
def test_every_link_of_a_full_row_is_found(n_s, neighbours, row_bins):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1005_5312_gb300 as S
    S.build()
    pos, h, src, L = workload(311, n_s, neighbours, 100 * n_s + neighbours)
    n_HI = np.random.default_rng(n_s).uniform(0.0, 2e-4, 311).astype(np.float32)
    out = []
    for mode in (1, 0):
        ctx = S.Context(march_mode=mode, link_counts=mode, row_bins=row_bins, tau_cut=1e30)
        ctx.build_trees(pos, h, src, L)
        g = np.zeros(311, np.float32)
        ctx.rt_solve(0.0, n_HI=n_HI, gamma_out=g)
        out.append((g.astype(np.float64), ctx.stats()))
    (gm, sm), (gr, sr) = out
    assert sm["rays"] == sr["rays"] == 311 * n_s
    assert sm["evals"] == sm["rays"]
    assert sm["hops"] == sr["hops"] and sm["max_hops"] == sr["max_hops"]
    # compensated sums of the same links both ways: a few roundings of tau (below
    # 30) and of each contribution
    np.testing.assert_allclose(gm, gr, rtol=2e-5)
