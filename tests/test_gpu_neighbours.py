"""The neighbour search where its shapes change: groups of 32 targets cut
short, one particle, lists beyond the 48 kept by the counting walk, groups
that straddle the box (wide), widely different smoothing lengths, leaves of
one and of many members, duplicates.  Sets are compared with a 64-bit
brute-force search.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 33, 129, 1000])
@pytest.mark.parametrize("leaf", [1, 16, 200])
@pytest.mark.parametrize("spread", ["uniform", "clumps", "mixed_h", "duplicates"])
def test_neighbour_sets_match_brute_force(n, leaf, spread):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1005_5312_gb300 as S
    S.build()
    rng = np.random.default_rng(n + leaf)
    pos = rng.uniform(0.0, 1.0, (3, n))
    h = np.full(n, 0.5 * (40.0 / max(n, 40)) ** (1.0 / 3.0))
    if spread == "clumps":   # eight far clumps: Morton neighbours a box apart
        pos = 0.02 * pos + np.round(rng.uniform(0.0, 1.0, (3, n)))
        h = np.full(n, 0.01)
    elif spread == "mixed_h":
        h = h * 10.0 ** rng.uniform(-1.0, 0.4, n)
    elif spread == "duplicates":
        pos[:, 1::2] = pos[:, 0:-1:2] if n % 2 else pos[:, 0::2]
    pos, h = pos.astype(np.float32), h.astype(np.float32)
    ctx = S.Context(ptree_leaf=leaf)
    ctx.build_trees(pos, h, np.zeros((3, 0), np.float32), np.zeros(0))
    off, idx = ctx.neighbors()
    p, r = pos.astype(np.float64), 2.0 * h.astype(np.float64)
    for i in range(n):
        d2 = ((p - p[:, i:i + 1]) ** 2).sum(0)
        want = np.nonzero(d2 < r[i] * r[i])[0]
        want = want[want != i]
        assert np.array_equal(np.sort(idx[off[i]:off[i + 1]]), want), i
