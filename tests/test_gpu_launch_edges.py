"""Launch shapes that the other parity tests do not reach, against the oracle (1e-5, the
complex64 tolerance of the parity tests): 16 lines of 1024..4096 points in the team pass, the
unsplit operator on lines of 2048 and 4096 points, and a batch whose class grows over the
paired shape's threshold while its contexts are under way.
"""
import numpy as np
import pytest

import oracle
import paper_1909_02894_gb300 as D
from paper_1909_02894_gb300 import workloads as W
from parity_util import assert_parity

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _built():
    D.build()
    oracle.build()


def grid(nx, ny):
    ax, ay = 0.1 * nx, 0.1 * ny
    X, Y = W.mesh(nx, ny, ax, ay)
    g11 = 1.0 + 0.2 * np.exp(-((X - 0.1 * ax) ** 2 + Y ** 2) / (0.2 * ax * ay))
    psi0 = W.wave_packet(nx, ny, ax, ay, 0.1 * min(ax, ay) + 0.5, (1.0, -0.7))
    return W.Workload("edge", nx, ny, ax, ay, np.ones((ny, nx)), g11, 1.0 + 0.5 * (g11 - 1.0),
                      mass=0.4, c=1.0, pml_width_x=nx // 16, pml_width_y=ny // 16, pml_type=1,
                      sigma0=0.5, theta=0.0, psi0=psi0, dt=0.03, steps=3)


@pytest.mark.parametrize("nx,ny", [(1024, 16), (2048, 16), (4096, 16), (16, 4096)])
def test_sixteen_long_lines(nx, ny):
    w = grid(nx, ny)
    with D.Simulation(w, precision=D.DIRAC_C64) as s:
        D.dirac_set_launch(s.ctx, 1024, 1024)
        s.set_state(w.psi0)
        s.step(3, w.dt)
        assert_parity(s.get_state(),
                      oracle.run(oracle.Problem.from_workload(w), w.psi0, w.dt, 3), w, TOL)


@pytest.mark.parametrize("scheme,family,degree",
                         [(D.DIRAC_SCHEME_POLY_TAYLOR, oracle.POLY_TAYLOR, 3),
                          (D.DIRAC_SCHEME_POLY_CHEBYSHEV, oracle.POLY_CHEBYSHEV, 8)])
@pytest.mark.parametrize("nx,ny", [(2048, 256), (256, 2048), (4096, 256), (256, 4096)])
def test_unsplit_operator_on_long_lines(nx, ny, scheme, family, degree):
    w = grid(nx, ny)
    ref = oracle.run_poly(oracle.Problem.from_workload(w), w.psi0, w.dt, 3, family=family,
                          order=degree)
    with D.Simulation(w, precision=D.DIRAC_C64, scheme=scheme, poly_degree=degree) as s:
        s.set_state(w.psi0)
        s.step(3, w.dt)
        assert_parity(s.get_state(), ref, w, TOL)


def test_a_class_that_grows_over_the_pair_threshold_between_ticks():
    """512^2 instances: a table of 4 holds 2^20 points (staged output), of 8 2^21 (line pairs,
    and the branch the large classes share). The first four are half way when the fifth joins;
    all equal their alone runs bit for bit."""
    w = grid(512, 512)
    rng = np.random.default_rng(3)
    states = [w.psi0 * np.exp(2j * np.pi * rng.random()) for _ in range(5)]
    want = []
    for psi in states:
        with D.Simulation(w, precision=D.DIRAC_C64) as s:
            s.set_state(psi)
            s.step(8, w.dt)
            want.append(s.get_state())
    sims = [D.Simulation(w, precision=D.DIRAC_C64) for _ in states]
    batch = D.dirac_batch_create(1 << 34, D.DIRAC_C64, steps_per_tick=4)
    try:
        for i, (s, psi) in enumerate(zip(sims, states)):
            s.set_state(psi)
            if i == 4:
                D.dirac_batch_run(batch, 1)
            D.dirac_batch_submit(batch, s.ctx, 8, w.dt)
        while D.dirac_batch_active(batch):
            D.dirac_batch_run(batch, 1)
        D.dirac_batch_synchronize(batch)
        for slot in range(5):
            assert D.dirac_batch_poll(batch, slot)
            D.dirac_batch_release(batch, slot)
        for s, ref in zip(sims, want):
            assert np.array_equal(s.get_state(), ref)
    finally:
        D.dirac_batch_destroy(batch)
        for s in sims:
            s.close()
