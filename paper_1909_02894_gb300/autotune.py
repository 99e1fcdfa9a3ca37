"""Autotuner cache: the fastest CTA shape of each pass per (device, library build, grid,
precision, scheme, static potentials or none), measured on the device by dirac_autotune and
kept in a JSON file. A shape of another build or scheme is not reused: the same number may
name another kernel there, and any shape but 0 takes a small grid off the one-launch path."""
from __future__ import annotations

import functools
import hashlib
import json
import os

from . import DIRAC_SCHEME_II, LIB_PATH, _routes, dirac_autotune, dirac_set_launch

DEFAULT_CACHE = os.path.join(os.path.expanduser("~"), ".cache", "dirac_gb300_autotune.json")


def _device_name():
    try:
        import torch

        return torch.cuda.get_device_name()
    except Exception:
        return "cuda"


@functools.lru_cache(maxsize=4)
def _build_id(path, mtime_ns, size):
    h = hashlib.sha256()
    with open(path, "rb") as f:
        for block in iter(lambda: f.read(1 << 20), b""):
            h.update(block)
    return h.hexdigest()[:16]


def cache_key(sim, precision):
    st = os.stat(LIB_PATH)
    scheme, potentials = _routes.get(sim.ctx, (DIRAC_SCHEME_II, False))
    return "|".join((_device_name(), _build_id(LIB_PATH, st.st_mtime_ns, st.st_size),
                     f"{sim.nx}x{sim.ny}", "c64" if precision == 0 else "c128",
                     f"scheme{scheme}", "potentials" if potentials else "free"))


def tune(sim, precision, cache_path: str = DEFAULT_CACHE, reps: int = 20, refresh: bool = False):
    """Apply the cached (or newly measured) launch shapes to a Simulation's context."""
    key = cache_key(sim, precision)
    cache = {}
    if os.path.exists(cache_path):
        try:
            cache = json.load(open(cache_path))
        except (OSError, ValueError):
            cache = {}
    if key in cache and not refresh:
        tx, ty = cache[key]
        dirac_set_launch(sim.ctx, tx, ty)
        return tx, ty
    tx, ty = dirac_autotune(sim.ctx, reps)
    cache[key] = [tx, ty]
    os.makedirs(os.path.dirname(cache_path), exist_ok=True)
    tmp = cache_path + f".tmp{os.getpid()}"
    with open(tmp, "w") as f:
        json.dump(cache, f, indent=1, sort_keys=True)
    os.replace(tmp, cache_path)
    return tx, ty
