"""Loads through the read-only path name tables only.

Kernels launched with programmatic stream serialization can be resident while the kernel
before them still writes its results, and ld.global.nc (and __ldg) needs memory that nobody
writes for the whole lifetime of the loading kernel. So the helpers that use that path may
be called on coefficients, twiddles, multipliers and instance pointers, never on a state, a
polynomial term or another array that a kernel of the chain writes. Read from the sources.
"""
import glob
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1909_02894_gb300", "csrc")
# local names and members that hold tables: twiddles, multipliers, b - 1, half-step matrices
TABLES = {"tw", "tw1", "tw2", "twk", "mt", "mult", "beta", "u_load", "u_store", "ug", "ip"}


def strip_comments(s):
    return re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", s, flags=re.S))


def helpers_of(src):
    """Names of the device functions whose body takes the read-only path."""
    out = set()
    for m in re.finditer(r"__forceinline__\s+[\w<>:\s*&]*?[\s*&](\w+)\(([^()]*)\)\s*\{", src):
        depth, i = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(src[i], 0)
            i += 1
        if re.search(r"ld\.global\.nc|__ldg\(", src[m.end():i]):
            out.add(m.group(1))
    return out


def test_the_read_only_path_loads_tables_only():
    srcs = {p: strip_comments(open(p).read())
            for p in sorted(glob.glob(os.path.join(CSRC, "*.cu*")))}
    helpers = set().union(*(helpers_of(s) for s in srcs.values()))
    assert {"ldg_q4", "ldg_cx", "ld_stream", "ld_stream_q4", "ld_ptr"} <= helpers
    # no kernel takes the path other than through a helper
    direct = [p for p, s in srcs.items()
              for _ in re.finditer(r"__ldg\((?!reinterpret_cast<const (?:float|double)[24]\*>\(p\))", s)]
    assert not direct, direct
    calls = 0
    for p, s in srcs.items():
        for m in re.finditer(r"\b(%s)\(\s*&?([\w.>-]+)" % "|".join(sorted(helpers)), s):
            arg = re.split(r"\.|->", m.group(2))
            if arg[0] in ("const", "P"):
                continue  # the helper's own declaration
            name = arg[0] if arg[0] == "ip" else arg[-1]
            assert name in TABLES, f"{os.path.basename(p)}: {m.group(0)} is not a table"
            calls += 1
    assert calls >= 20
