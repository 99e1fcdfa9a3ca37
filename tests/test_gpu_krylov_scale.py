"""Scheme I in complex64 with time steps far beyond the fastest mode's period, where the squares
of the Krylov vectors before their normalisation leave the FP32 range.

Flat space, no mass: the middle step multiplies a mode of wave number k by the Cayley factors
(1 -+ i k dt/2) / (1 +- i k dt/2), which are -1 to within 2 / (k dt) < 1e-19 here. Tolerance:
the initial state has modes of one |k| only, on which a relative residual of 1e-6 is a relative
error of 1e-6; the Krylov vectors hold the other modes at the FP32 rounding level with
coefficients of order one. 1e-5 is the complex64 tolerance of the parity tests. |k| is a quarter
of the largest wave number, so FP32 rounding (6e-8 per value, amplified by at most 4) leaves
residuals below 1e-6. n = 256 runs the two-pass operator, n = 64 the general one.
"""
import numpy as np
import pytest

import paper_1909_02894_gb300 as D
from paper_1909_02894_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dt", [1e10, 1e20, 1e22, 1e30])
@pytest.mark.parametrize("n", [64, 256])
def test_large_time_steps_flip_the_sign_of_every_mode(n, dt):
    D.build()
    a = 10.0
    X, Y = W.mesh(n, n, a, a)
    k = np.pi / a * (n // 8)
    psi = np.stack([np.exp(1j * k * X) + 0.5 * np.exp(-1j * k * Y),
                    0.3 * np.exp(1j * k * Y) + 0.7 * np.exp(-1j * k * X)])
    psi /= np.linalg.norm(psi)
    one = np.ones((n, n))
    w = W.Workload("waves", n, n, a, a, one, one, one, mass=0.0, c=1.0, pml_width_x=0,
                   pml_width_y=0, pml_type=1, sigma0=1.0, theta=0.0, psi0=psi, dt=dt, steps=1)
    with D.Simulation(w, precision=D.DIRAC_C64, conn=D.DIRAC_CONN_NONE,
                      scheme=D.DIRAC_SCHEME_CRANK_NICOLSON) as s:
        D.dirac_set_krylov(s.ctx, 1e-6, 20, 100)
        s.set_state(psi)
        s.step(1, dt)
        got = s.get_state()
    assert np.linalg.norm(got + psi) <= 1e-5
