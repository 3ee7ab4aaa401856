"""The neighbour search at the sizes where the lanes per target change: every row's
count, sum and sum of squares of its indices against a 64-bit brute-force search."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [12288, 12289, 40960, 40961, 200000, 200003])
@pytest.mark.parametrize("spread", ["uniform", "mixed_h"])
def test_rows_match_brute_force(n, spread):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1005_5312_gb300 as S
    S.build()
    rng = np.random.default_rng(n)
    pos = rng.uniform(0.0, 1.0, (3, n)).astype(np.float32)
    h = np.full(n, 0.985 * n ** (-1.0 / 3.0))
    if spread == "mixed_h":   # rows of none to some hundreds
        h = h * 10.0 ** rng.uniform(-1.0, 0.3, n)
    h = h.astype(np.float32)
    ctx = S.Context()
    ctx.build_trees(pos, h, np.zeros((3, 0), np.float32), np.zeros(0))
    off, idx = ctx.neighbors()
    off, idx = off.astype(np.int64), idx.astype(np.int64)
    rows = np.repeat(np.arange(n), np.diff(off))
    got = [np.diff(off)] + [np.bincount(rows, weights=(idx ** e).astype(np.float64), minlength=n)
                            for e in (1, 2)]   # below 2^53: exact
    p = torch.from_numpy(pos).cuda().double()
    r2 = (2.0 * torch.from_numpy(h).cuda().double()) ** 2
    k = torch.arange(n, device="cuda", dtype=torch.float64)
    want = [[], [], []]
    for a in range(0, n, 2048):
        b = min(a + 2048, n)
        d2 = sum((p[c][None, :] - p[c][a:b, None]) ** 2 for c in range(3))
        m = d2 < r2[a:b, None]
        m[torch.arange(b - a), torch.arange(a, b)] = False
        want[0].append(m.sum(1).cpu())
        m = m.double()
        want[1].append((m @ k).cpu())
        want[2].append((m @ (k * k)).cpu())
    for g, w in zip(got, want):
        assert np.array_equal(g, torch.cat(w).numpy())
