"""The band averages of the self terms around the widths where their panels
change, against adaptive quadrature: emitters alone in the dark (far apart,
transparent to each other), so that the heating is each particle's own."""
import math

import numpy as np
import pytest

from start_inputs import ALPHA_A, ALPHA_B, KPC_CM, SIGMA_CM2

pytestmark = pytest.mark.gpu

HNU_L, K_B = 13.6 * 1.602176634e-12, 1.380649e-16


@pytest.mark.parametrize("T_rec", [100.0, 1e4, 12620.0, 12640.0, 18900.0, 19000.0, 47300.0,
                                   47400.0, 1e5])
def test_self_heating_is_the_band_average(T_rec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from scipy.integrate import quad
    import paper_1005_5312_gb300 as S
    S.build()
    n = 40
    rng = np.random.default_rng(3)
    pos = np.stack([1e9 * np.arange(n), np.zeros(n), np.zeros(n)]).astype(np.float32)
    h = np.full(n, 1.0, np.float32)
    n_H = (10.0 ** rng.uniform(-5, 0, n)).astype(np.float32)
    y = 10.0 ** rng.uniform(-3, -0.1, n)
    V = np.full(n, 0.1 ** 3)
    ctx = S.Context(T_rec=T_rec)
    ctx.build_trees(pos, h, np.zeros((3, 0), np.float32), np.zeros(0), V, diffuse=True)
    ctx.set_state(n_H, y)
    ctx.rt_solve(1.0)
    heat = ctx.heating().astype(np.float64)
    D = K_B * T_rec / HNU_L
    R = (3.0 * V[0] / (4.0 * math.pi)) ** (1 / 3) * KPC_CM
    for i in range(n):
        ne, ts = (1.0 - y[i]) * float(n_H[i]), SIGMA_CM2 * y[i] * float(n_H[i]) * R

        def f(x):
            u3 = (1.0 + x) ** -3
            return x * u3 * -math.expm1(-ts * u3) / (ts * u3)
        own = (ALPHA_A - ALPHA_B) * ne * ne * SIGMA_CM2 * R * HNU_L * quad(
            f, 0.0, D, epsabs=0.0, epsrel=1e-11)[0] / D
        # float32 result; the other emitters, 1e9 kpc away, add below 1e-12 of it
        assert abs(heat[i] / own - 1.0) < 3e-7, (i, heat[i], own)
