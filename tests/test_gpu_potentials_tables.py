"""The half-step matrices of contexts with static potentials: one pair of arrays (U and U^2, 32
bytes per point each in complex64), in the layout the launch shape reads, remade when the shape
changes. Tolerance 1e-5: the complex64 tolerance of the parity tests.
"""
import numpy as np
import pytest

import oracle
import paper_1909_02894_gb300 as D
from paper_1909_02894_gb300 import workloads as W
from parity_util import assert_parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    D.build()
    oracle.build()


def case(nx, ny):
    ax, ay = 0.1 * nx, 0.1 * ny
    X, Y = W.mesh(nx, ny, ax, ay)
    g11 = 1.0 + 0.2 * np.exp(-(X ** 2 + Y ** 2) / (0.2 * ax * ay))
    w = W.Workload("pot", nx, ny, ax, ay, np.ones((ny, nx)), g11, np.ones((ny, nx)), mass=0.4,
                   c=1.0, pml_width_x=0, pml_width_y=0, pml_type=1, sigma0=0.5, theta=0.0,
                   psi0=W.wave_packet(nx, ny, ax, ay, 0.1 * min(ax, ay) + 0.5, (1.0, -0.7)),
                   dt=0.03, steps=2)
    V = 0.8 * np.exp(-(X ** 2 + (Y - 0.2 * ay) ** 2) / (0.1 * ax * ay))
    return w, V, 0.15 * np.sin(np.pi * Y / ay), -0.1 * np.sin(np.pi * X / ax)


@pytest.mark.parametrize("shape", [0, 512], ids=["in-the-y-pass", "own-kernel"])
def test_potentials_take_64_bytes_per_point(shape):
    torch = pytest.importorskip("torch")
    w, V, Ax, Ay = case(512, 2048)

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    with D.Simulation(w, precision=D.DIRAC_C64) as s:
        D.dirac_set_launch(s.ctx, shape, shape)
        s.set_state(w.psi0)
        D.dirac_set_potentials(s.ctx, V, Ax, Ay)
        s.step(1, w.dt)  # also loads the kernels that come first with it
        s.get_state()
        with D.Simulation(w, precision=D.DIRAC_C64) as t:
            D.dirac_set_launch(t.ctx, shape, shape)
            t.set_state(w.psi0)
            D.dirac_set_potentials(t.ctx, V, Ax, Ay)
            before = free()
            t.step(1, w.dt)
            # allocations are rounded up to 2 MiB
            assert before - free() <= 64 * w.nx * w.ny + 2 * (2 << 20)


@pytest.mark.parametrize("nx,ny", [(16, 256), (128, 512), (1024, 1024)])
def test_layout_follows_the_launch_shape(nx, ny):
    w, V, Ax, Ay = case(nx, ny)
    prob = oracle.Problem.from_workload(w)
    prob.V, prob.Ax, prob.Ay = V, Ax, Ay
    ref = oracle.run(prob, w.psi0, w.dt, 8)
    with D.Simulation(w, precision=D.DIRAC_C64) as s:
        D.dirac_set_potentials(s.ctx, V, Ax, Ay, shape=(ny, nx))
        s.set_state(w.psi0)
        for shape in (0, 256, 1024, 512):
            D.dirac_set_launch(s.ctx, shape, shape)
            s.step(2, w.dt)
        assert_parity(s.get_state(), ref, w, 1e-5)
