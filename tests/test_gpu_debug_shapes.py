"""The bounds-checked debug build (see test_gpu_debug_build.py) through the launch shapes that
grids above 2^16 points, other schemes, batches and the one-launch small grids take: small,
staged and paired team passes, rows and general-U output, batched instances, both phases of
the unsplit operator, the whole-step kernel. Every result must match the oracle to the
complex64 tolerance of the parity tests, 1e-5, with no index check failing.
"""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu

SCRIPT = r'''
import json
import numpy as np
import oracle
import paper_1909_02894_gb300 as D
from paper_1909_02894_gb300 import workloads as W
oracle.build()
out = []


def case(nx, ny):
    ax, ay = 0.1 * nx, 0.1 * ny
    X, Y = W.mesh(nx, ny, ax, ay)
    g11 = 1.0 + 0.2 * np.exp(-((X - 0.1 * ax) ** 2 + Y ** 2) / (0.2 * ax * ay))
    psi0 = W.wave_packet(nx, ny, ax, ay, 0.1 * min(ax, ay) + 0.5, (1.0, -0.7))
    w = W.Workload("dbg", nx, ny, ax, ay, np.ones((ny, nx)), g11, 1.0 + 0.5 * (g11 - 1.0),
                   mass=0.4, c=1.0, pml_width_x=nx // 16, pml_width_y=ny // 16, pml_type=1,
                   sigma0=0.5, theta=0.0, psi0=psi0, dt=0.03, steps=3)
    V = 0.8 * np.exp(-(X ** 2 + Y ** 2) / (0.1 * ax * ay))
    return w, V, 0.15 * np.sin(np.pi * Y / ay), -0.1 * np.sin(np.pi * X / ax)


def note(what, w, got, ref):
    out.append({"what": what, "grid": [w.nx, w.ny], "rel_l2": W.rel_l2(got, ref)})


SYM = D.DIRAC_SCHEME_II_SYMMETRIC
for nx, ny in ((512, 512), (256, 2048), (1024, 1024), (64, 64), (64, 128), (128, 64), (128, 128)):
    w, V, Ax, Ay = case(nx, ny)
    for scheme, osch in ((D.DIRAC_SCHEME_II, oracle.SCHEME_II), (SYM, oracle.SCHEME_II_SYMMETRIC)):
        for pot in (False, True):
            prob = oracle.Problem.from_workload(w)
            with D.Simulation(w, precision=D.DIRAC_C64, scheme=scheme) as s:
                if pot:
                    prob.V, prob.Ax, prob.Ay = V, Ax, Ay
                    D.dirac_set_potentials(s.ctx, V, Ax, Ay)
                s.set_state(w.psi0)
                s.step(3, w.dt)
                note(["step", scheme, pot], w, s.get_state(),
                     oracle.run(prob, w.psi0, w.dt, 3, scheme=osch))

for nx, ny in ((256, 512), (1024, 1024), (2048, 256), (256, 2048), (4096, 256), (256, 4096)):
    w = case(nx, ny)[0]
    for scheme, fam in ((D.DIRAC_SCHEME_POLY_TAYLOR, oracle.POLY_TAYLOR),
                        (D.DIRAC_SCHEME_POLY_CHEBYSHEV, oracle.POLY_CHEBYSHEV)):
        for deg in (3, 8):
            with D.Simulation(w, precision=D.DIRAC_C64, scheme=scheme, poly_degree=deg) as s:
                s.set_state(w.psi0)
                s.step(2, w.dt)
                note(["poly", scheme, deg], w, s.get_state(),
                     oracle.run_poly(oracle.Problem.from_workload(w), w.psi0, w.dt, 2,
                                     family=fam, order=deg))

# one class each of the small, staged and paired batch shapes (their capacity is 4), short lines
ws = [case(n, n)[0] for n in (128, 256, 512, 1024, 1024)]
sims = [D.Simulation(w, precision=D.DIRAC_C64) for w in ws]
batch = D.dirac_batch_create(1 << 34, D.DIRAC_C64, steps_per_tick=2)
for s, w in zip(sims, ws):
    s.set_state(w.psi0)
    D.dirac_batch_submit(batch, s.ctx, 3, w.dt)
while D.dirac_batch_active(batch):
    D.dirac_batch_run(batch, 1)
D.dirac_batch_synchronize(batch)
D.dirac_batch_destroy(batch)
for s, w in zip(sims, ws):
    note(["batch"], w, s.get_state(), oracle.run(oracle.Problem.from_workload(w), w.psi0, w.dt, 3))
    s.close()
print(json.dumps(out))
'''


def test_every_launch_shape_passes_its_index_checks():
    env = dict(os.environ, DIRAC_NVCC_EXTRA="-DDIRAC_DEBUG=1", DIRAC_BUILD_TAG="debug")
    subprocess.run([sys.executable, "-c",
                    "import paper_1909_02894_gb300._build as b; b.build()"],
                   env=env, cwd=ROOT, check=True, timeout=900)
    lib = os.path.join(ROOT, "paper_1909_02894_gb300", "libdirac_debug.so")
    env = dict(os.environ, DIRAC_LIB=lib)
    env.pop("DIRAC_NVCC_EXTRA", None)
    r = subprocess.run([sys.executable, "-c", SCRIPT], env=env, cwd=ROOT, capture_output=True,
                       text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    res = json.loads(r.stdout.strip().splitlines()[-1])
    assert len(res) == 7 * 4 + 6 * 4 + 5
    for x in res:
        assert x["rel_l2"] <= 1e-5, x
