"""The implicit temperature step over its whole range of states, against the
oracle's bisection: no sources, so the gas only cools (collisional and
recombination cooling from 10 K to 1e8.5 K, neutral to ionised)."""
import numpy as np
import pytest

import oracle
from start_inputs import ALPHA_A, ALPHA_B, KPC_CM, SIGMA_CM2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt,n_max", [(0.0, 1e2), (1e6, 1e2), (1e10, 1.0), (1e12, 1e-1),
                                      (3e13, 1e-3)])
def test_cooling_step_matches_bisection(dt, n_max):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1005_5312_gb300 as S
    S.build()
    n = 4001
    rng = np.random.default_rng(int(dt) % 1000 + 7)
    pos = rng.uniform(0.0, 1.0, (3, n)).astype(np.float32)
    h = np.full(n, 1e-4, np.float32)
    n_H = (n_max * 10.0 ** rng.uniform(-6, 0, n)).astype(np.float32)
    y0 = 10.0 ** rng.uniform(-6, 0, n)
    T0 = 10.0 ** rng.uniform(1.0, 8.5, n)
    T0[:3] = [10.0, 1e9, 1e4]
    src, L = np.full((3, 1), 0.5, np.float32), np.zeros(1)
    ctx = S.Context(thermal=1)
    ctx.build_trees(pos, h, src, L)
    ctx.set_state(n_H, y0)
    ctx.set_temperature(T0)
    ctx.rt_solve(1.0)
    y = np.zeros(n)
    ctx.ionize(dt, y_out=y)
    T = ctx.temperature()
    orc = oracle.Oracle(pos, h, src, L, sigma_cm2=SIGMA_CM2, len_unit_cm=KPC_CM, alpha_A=ALPHA_A,
                        alpha_B=ALPHA_B)
    y_ref, T_ref = orc.ionize_thermal(np.zeros(n), None, n_H, y0, T0, dt)
    np.testing.assert_allclose(y, y_ref, rtol=1e-12)
    # both solve the same equation to rounding; the residual's terms cancel to
    # u0 / (e1 T1) <= T0 / T1, which amplifies a few FP64 roundings
    tol = 1e-12 + 64 * 2.0 ** -53 * T0 / T_ref
    assert np.all(np.abs(T / T_ref - 1.0) <= tol), np.max(np.abs(T / T_ref - 1.0) / tol)
