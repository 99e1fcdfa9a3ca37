"""The radix-16 team pass and the unsplit operator built on it (complex64, axes of 256..4096
points) against the oracle, at the edges of their launch rules: small CTAs up to 2^18 points,
staged output up to 2^20, line pairs above; 16 lines of every length; odd and even polynomial
degrees (the terms alternate between the two layouts); more than four Krylov vectors.

Tolerance: 1e-5 (rel-L2 and layer maximum), the complex64 tolerance of the other parity tests.
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


def grid(nx, ny, noise=0.01, steps=3):
    ax, ay = 0.1 * nx, 0.1 * ny
    X, Y = W.mesh(nx, ny, ax, ay)
    g11 = 1.0 + 0.2 * np.exp(-((X - 0.1 * ax) ** 2 + Y ** 2) / (0.2 * ax * ay))
    g22 = 1.0 + 0.1 * np.exp(-(X ** 2 + (Y + 0.1 * ay) ** 2) / (0.3 * ax * ay))
    psi0 = W.wave_packet(nx, ny, ax, ay, 0.1 * min(ax, ay) + 0.5, (1.0, -0.7))
    psi0 += noise * W.random_state(nx, ny, nx + 3 * ny)
    return W.Workload("team", nx, ny, ax, ay, np.ones((ny, nx)), g11, g22, mass=0.4, c=1.0,
                      pml_width_x=nx // 16, pml_width_y=ny // 16, pml_type=1, sigma0=0.5,
                      theta=0.0, psi0=psi0, dt=0.03, steps=steps)


@pytest.mark.parametrize("scheme", [D.DIRAC_SCHEME_II, D.DIRAC_SCHEME_II_SYMMETRIC],
                         ids=["printed", "symmetric"])
@pytest.mark.parametrize("nx,ny", [(256, 16), (512, 16), (512, 512), (1024, 256), (512, 1024),
                                   (1024, 1024), (256, 4096), (2048, 512)])
def test_step_matches_oracle_in_every_launch_shape(nx, ny, scheme):
    w = grid(nx, ny)
    osch = oracle.SCHEME_II if scheme == D.DIRAC_SCHEME_II else oracle.SCHEME_II_SYMMETRIC
    ref = oracle.run(oracle.Problem.from_workload(w), w.psi0, w.dt, 3, scheme=osch)
    with D.Simulation(w, precision=D.DIRAC_C64, scheme=scheme) as s:
        D.dirac_set_launch(s.ctx, 1024, 1024)
        s.set_state(w.psi0)
        s.step(3, w.dt)
        assert_parity(s.get_state(), ref, w, TOL)


@pytest.mark.parametrize("scheme,family", [(D.DIRAC_SCHEME_POLY_TAYLOR, oracle.POLY_TAYLOR),
                                           (D.DIRAC_SCHEME_POLY_CHEBYSHEV, oracle.POLY_CHEBYSHEV)])
@pytest.mark.parametrize("nx,ny,degree", [(256, 512, 1), (256, 512, 2), (256, 512, 3),
                                          (256, 512, 8), (1024, 1024, 3), (1024, 1024, 8)])
def test_polynomial_schemes_on_the_team_operator(nx, ny, scheme, family, degree):
    w = grid(nx, ny, noise=0.0)
    ref = oracle.run_poly(oracle.Problem.from_workload(w), w.psi0, w.dt, 3, family=family,
                          order=degree)
    with D.Simulation(w, precision=D.DIRAC_C64, scheme=scheme, poly_degree=degree) as s:
        s.set_state(w.psi0)
        s.step(2, w.dt)
        s.step(1, w.dt)
        assert_parity(s.get_state(), ref, w, TOL)


@pytest.mark.parametrize("prec", [D.DIRAC_C64, D.DIRAC_C128], ids=["c64", "c128"])
def test_krylov_solver_beyond_four_vectors(prec):
    """White noise at a larger time step needs more than four basis vectors per solve: the
    Gram-Schmidt sweeps beyond the fused one, in chunks of four."""
    w = grid(256, 256, noise=0.5, steps=2)
    ref, _ = oracle.run_cn(oracle.Problem.from_workload(w), w.psi0, 0.06, 2, tol=1e-14)
    with D.Simulation(w, precision=prec, scheme=D.DIRAC_SCHEME_CRANK_NICOLSON) as s:
        D.dirac_set_krylov(s.ctx, 0.0, 30, 100)
        s.set_state(w.psi0)
        s.step(2, 0.06)
        got = s.get_state()
        assert D.dirac_krylov_iterations(s.ctx) >= 2 * 6
    assert_parity(got, ref, w, 1e-11 if prec == D.DIRAC_C128 else TOL)


def test_krylov_norms_keep_the_state_s_scale():
    """States whose squared amplitudes leave the FP32 range are solved as accurately."""
    w = grid(256, 256, noise=0.0)
    for scale in (1e-24, 1e22):
        psi0 = w.psi0 * scale
        ref, _ = oracle.run_cn(oracle.Problem.from_workload(w), psi0, w.dt, 1, tol=1e-14)
        with D.Simulation(w, precision=D.DIRAC_C64, scheme=D.DIRAC_SCHEME_CRANK_NICOLSON) as s:
            s.set_state(psi0)
            s.step(1, w.dt)
            assert_parity(s.get_state(), ref, w, TOL)


@pytest.mark.parametrize("scheme", [D.DIRAC_SCHEME_II, D.DIRAC_SCHEME_II_SYMMETRIC],
                         ids=["printed", "symmetric"])
@pytest.mark.parametrize("nx,ny", [(512, 256), (128, 512), (256, 128), (1024, 1024)])
def test_potentials_inside_the_team_pass(nx, ny, scheme):
    """The general half step in the last pass's store (axes of team-pass length, both layouts)
    and by its own kernel (the other axes), over two calls and a change of dt."""
    w = grid(nx, ny)
    X, Y = W.mesh(nx, ny, w.ax, w.ay)
    V = 0.8 * np.exp(-(X ** 2 + Y ** 2) / (0.1 * w.ax * w.ay))
    Ax, Ay = 0.15 * np.sin(np.pi * Y / w.ay), -0.1 * np.sin(np.pi * X / w.ax)
    prob = oracle.Problem.from_workload(w)
    prob.V, prob.Ax, prob.Ay = V, Ax, Ay
    osch = oracle.SCHEME_II if scheme == D.DIRAC_SCHEME_II else oracle.SCHEME_II_SYMMETRIC
    ref = oracle.run(prob, w.psi0, w.dt, 3, scheme=osch)
    ref = oracle.run(prob, ref, 0.5 * w.dt, 2, scheme=osch)
    with D.Simulation(w, precision=D.DIRAC_C64, scheme=scheme) as s:
        D.dirac_set_potentials(s.ctx, V, Ax, Ay, shape=(ny, nx))
        s.set_state(w.psi0)
        s.step(2, w.dt)
        s.step(1, w.dt)
        s.step(2, 0.5 * w.dt)
        assert_parity(s.get_state(), ref, w, TOL)


@pytest.mark.parametrize("prec", [D.DIRAC_C64, D.DIRAC_C128], ids=["c64", "c128"])
@pytest.mark.parametrize("nx,ny", [(16, 1024), (32, 1024), (64, 1024), (128, 1024), (128, 512),
                                   (64, 16), (32, 32)])
def test_short_lines_with_two_and_four_points_per_thread(nx, ny, prec):
    """The small shape of lines of 128 points or fewer around its rule (512 lines), in the step
    and in the derivative mode (the energy's derivatives), against the oracle."""
    w = grid(nx, ny, noise=0.0)
    prob = oracle.Problem.from_workload(w)
    ref = oracle.run(prob, w.psi0, w.dt, 3)
    with D.Simulation(w, precision=prec) as s:
        D.dirac_set_launch(s.ctx, 256, 256)
        s.set_state(w.psi0)
        s.step(3, w.dt)
        got, obs = s.get_state(), s.observables()
    assert_parity(got, ref, w, 1e-11 if prec == D.DIRAC_C128 else TOL)
    want = oracle.observables(prob, got)
    tol = 1e-12 if prec == D.DIRAC_C128 else 1e-6
    for k in ("norm", "norm_gamma", "energy"):
        assert abs(obs[k] - want[k]) <= tol * max(1.0, abs(want[k])), k


@pytest.mark.parametrize("mass,conn", [(0.4, D.DIRAC_CONN_COVARIANT), (0.0, D.DIRAC_CONN_NONE)],
                         ids=["curved", "no-half-step"])
@pytest.mark.parametrize("nx,ny", [(64, 64), (64, 128), (128, 64), (128, 128)])
def test_whole_steps_in_one_launch(nx, ny, mass, conn):
    """Default complex64 steps of grids of 64- and 128-point axes (one launch for all steps of a
    call) equal, bit for bit, the two passes per step of the larger shape, over several calls,
    a change of dt and more steps than one launch takes, and match the oracle."""
    w = grid(nx, ny)
    w.mass = mass

    def run(shape):
        with D.Simulation(w, precision=D.DIRAC_C64, conn=conn) as s:
            D.dirac_set_launch(s.ctx, shape, shape)
            s.set_state(w.psi0)
            n0 = D.dirac_launch_count(s.ctx)
            for n, dt in ((1, w.dt), (2, w.dt), (5, 0.5 * w.dt), (1100, 0.5 * w.dt)):
                s.step(n, dt)
                if n == 5:
                    mid = s.get_state()
            return mid, s.get_state(), D.dirac_launch_count(s.ctx) - n0

    mid, end, launches = run(0)
    mid2, end2, launches2 = run(512)
    assert np.array_equal(mid, mid2) and np.array_equal(end, end2)
    assert launches < 40 < 2 * 1108 <= launches2
    prob = oracle.Problem.from_workload(w, conn=conn)
    ref = oracle.run(prob, w.psi0, w.dt, 3)
    assert_parity(mid, oracle.run(prob, ref, 0.5 * w.dt, 5), w, TOL)
