"""Bounded waits of the unsplit operator's passes that run out: reported, nothing iterates on
what the stopped passes left, and the context works again. No fault, trap or hang is
involved: the waits expect bytes that no copy delivers and give up after their bound.
"""
import numpy as np
import pytest

import paper_1909_02894_gb300 as D
from paper_1909_02894_gb300 import workloads as W

pytestmark = pytest.mark.gpu
CN = D.DIRAC_SCHEME_CRANK_NICOLSON
CHEB = D.DIRAC_SCHEME_POLY_CHEBYSHEV


def grid(nx, ny):
    ax, ay = 0.1 * nx, 0.1 * ny
    X, Y = W.mesh(nx, ny, ax, ay)
    g11 = 1.0 + 0.2 * np.exp(-(X ** 2 + Y ** 2) / (0.2 * ax * ay))
    psi0 = W.wave_packet(nx, ny, ax, ay, 0.1 * min(ax, ay) + 0.5, (1.0, -0.7))
    return W.Workload("wait", nx, ny, ax, ay, np.ones((ny, nx)), g11, np.ones((ny, nx)),
                      mass=0.4, c=1.0, pml_width_x=0, pml_width_y=0, pml_type=1, sigma0=0.5,
                      theta=0.0, psi0=psi0, dt=0.03, steps=2)


@pytest.mark.parametrize("scheme,nx,ny", [(CHEB, 256, 512), (CHEB, 1024, 1024), (CN, 256, 256),
                                          (CN, 1024, 1024)],
                         ids=["chebyshev-staged", "chebyshev-pairs", "cn-staged", "cn-pairs"])
def test_timeout_in_the_unsplit_operator_is_reported_and_the_context_recovers(scheme, nx, ny):
    D.build()
    w = grid(nx, ny)
    with D.Simulation(w, precision=D.DIRAC_C64, scheme=scheme) as s:
        s.set_state(w.psi0)
        s.step(2, w.dt)
        want = s.get_state()
    with D.Simulation(w, precision=D.DIRAC_C64, scheme=scheme) as s:
        s.set_state(w.psi0)
        D.dirac_test_timeout_next_step(s.ctx)
        with pytest.raises(D.DiracError) as e:
            s.step(1, w.dt)
            assert scheme == CHEB, "Scheme I waits for its inner products and must see it"
            D.dirac_synchronize(s.ctx)
        assert e.value.status == D.DIRAC_ETIMEOUT
        D.dirac_synchronize(s.ctx)  # reported once
        s.set_state(w.psi0)
        s.step(2, w.dt)
        assert np.array_equal(s.get_state(), want)


def test_the_hook_does_not_outlive_a_step_without_bounded_waits():
    """A 256 x 64 polynomial step has none; the later Scheme II step, whose x pass has, is not
    touched."""
    D.build()
    w = grid(256, 64)
    with D.Simulation(w, precision=D.DIRAC_C64, scheme=CHEB) as s:
        s.set_state(w.psi0)
        D.dirac_test_timeout_next_step(s.ctx)
        s.step(1, w.dt)
        D.dirac_synchronize(s.ctx)
        D.dirac_set_scheme(s.ctx, D.DIRAC_SCHEME_II)
        s.step(1, w.dt)
        D.dirac_synchronize(s.ctx)
