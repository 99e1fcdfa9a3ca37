"""The autotuner's cache returns a shape only to the device, library build, grid, precision,
scheme and potentials it was measured with (a fake library, no GPU)."""
import json
from types import SimpleNamespace

import numpy as np
import pytest

import paper_1909_02894_gb300 as D
from paper_1909_02894_gb300 import autotune


class FakeLib:
    """Accepts every call; dirac_create hands out handles."""

    def __init__(self):
        self.handles = 0

    def __getattr__(self, name):
        def call(*args):
            if name == "dirac_create":
                self.handles += 1
                args[-1]._obj.value = self.handles
            return 0
        return call


@pytest.fixture
def tuner(monkeypatch, tmp_path):
    fake = FakeLib()
    monkeypatch.setattr(D, "lib", lambda: fake)
    so = tmp_path / "lib.so"
    so.write_bytes(b"build 1")
    monkeypatch.setattr(autotune, "LIB_PATH", str(so), raising=False)
    monkeypatch.setattr(autotune, "_device_name", lambda: "device")
    measured, applied = [], []

    def measure(ctx, reps):
        measured.append(ctx)
        return 100 + len(measured), 200

    monkeypatch.setattr(autotune, "dirac_autotune", measure)
    monkeypatch.setattr(autotune, "dirac_set_launch", lambda *a: applied.append(a))
    return SimpleNamespace(so=so, measured=measured, applied=applied,
                           cache=str(tmp_path / "c" / "cache.json"))


def sim(n=128, scheme=D.DIRAC_SCHEME_II):
    ctx = D.dirac_create(n, n, 1.0, 1.0)
    if scheme != D.DIRAC_SCHEME_II:
        D.dirac_set_scheme(ctx, scheme)
    return SimpleNamespace(ctx=ctx, nx=n, ny=n)


def test_a_hit_needs_the_same_scheme_potentials_and_build(tuner):
    def tune(s, prec=0):
        return autotune.tune(s, prec, cache_path=tuner.cache)

    a = sim()
    first = tune(a)
    assert first == (101, 200) and not tuner.applied
    b = sim()
    assert tune(b) == list(first) or tune(b) == first  # same in every respect: no measurement
    assert len(tuner.measured) == 1 and tuner.applied[-1] == (b.ctx, 101, 200)
    others = [sim(scheme=D.DIRAC_SCHEME_II_SYMMETRIC), sim(), sim(n=64)]
    D.dirac_set_potentials(others[1].ctx, V=np.zeros((128, 128)))
    for i, s in enumerate(others):
        assert tuple(tune(s)) == (102 + i, 200)
    assert tuple(tune(sim(), prec=1)) == (105, 200)
    D.dirac_set_potentials(others[1].ctx)  # removed again: as the first
    assert tuple(tune(others[1])) == (101, 200)
    tuner.so.write_bytes(b"another build")
    assert tuple(tune(sim())) == (106, 200)


def test_an_entry_of_an_older_build_is_not_applied(tuner):
    import os

    os.makedirs(os.path.dirname(tuner.cache))
    with open(tuner.cache, "w") as f:
        json.dump({"device|128x128|c64": [512, 512]}, f)
    assert tuple(autotune.tune(sim(), 0, cache_path=tuner.cache)) == (101, 200)
    assert not tuner.applied


def test_a_handle_used_again_starts_as_scheme_ii(tuner):
    s = sim(scheme=D.DIRAC_SCHEME_II_SYMMETRIC)
    key = autotune.cache_key(s, 0)
    D.dirac_destroy(s.ctx)
    assert autotune.cache_key(s, 0) == key.replace("scheme1", "scheme0")
