"""Loads of the kernels that start while the one before them still runs.

A kernel that calls depend_wait() is alive while its predecessor writes.  CUDA
allows read-only loads (__ldg, ld.global.nc) and `__restrict__` only for data
that nothing else writes during the kernel's life, and the compiler may move
such a load above the wait.  So in these kernels `__restrict__` stands on
nothing but the tables of set-up, __ldg reads nothing but the material, and
nothing that a kernel writes is read ahead of the wait."""

import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1402_6297_gb300", "csrc")
TABLES = {"lam", "twx", "twy", "twz", "basis"}  # written when a context is set up
OWN = {"smem_raw", "tw", "tz", "ty", "ws", "cs", "x"}  # shared memory and registers
CALLS = {"for", "if", "min", "__align__", "static_assert", "tw_entry"}
MATERIAL = {"t + (long long)k * c.n3", "s + (long long)k * c.n3"}  # pmat, pmu


def sources():
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = re.sub(r"//[^\n]*", "", open(f).read())
        yield os.path.basename(f), text


def closing(text, at, pair):
    depth = 0
    for i in range(at, len(text)):
        depth += (text[i] == pair[0]) - (text[i] == pair[1])
        if depth == 0:
            return i
    raise AssertionError("unbalanced " + pair)


def kernels(text):
    """(name, parameters, body) of every kernel that is defined in text."""
    for m in re.finditer(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(", text):
        end = closing(text, m.end() - 1, "()")
        body = text.index("{", end)
        yield m.group(1), text[m.end():end], text[body:closing(text, body, "{}") + 1]


def test_overlapping_kernels_keep_read_only_loads_for_tables():
    seen = []
    for name, text in sources():
        for kernel, params, body in kernels(text):
            if "depend_wait()" not in body:
                continue
            seen.append(kernel)
            restricted = set(re.findall(r"__restrict__\s+(\w+)", params))
            assert restricted <= TABLES, (name, kernel, restricted - TABLES)
            assert not re.findall(r"__restrict__|__ldg|ldg_c|__ldc[gsv]", body), (name, kernel)
            # ahead of the wait: tables and what the kernel itself holds, no calls that load
            ahead = re.sub(r"auto \w+ = \[&\].*?\n  };", "", body[:body.index("depend_wait()")], flags=re.S)
            assert set(re.findall(r"(\w+)\s*\[", ahead)) <= TABLES | OWN, (name, kernel)
            assert set(re.findall(r"(\w+)\(", ahead)) <= CALLS, (name, kernel)
    assert {"k_rows_in", "k_columns", "k_rows_out", "k_gs_dots", "k_gs_update", "k_gs_finish",
            "k_gmres_columns"} <= set(seen)


def test_read_only_loads_of_the_material_step():
    """The steps that the column kernel calls: __ldg of the material alone."""
    text = dict(sources())["matvec_kernels.cuh"]
    for m in re.finditer(r"\b(__ldg|ldg_c)\(", text):
        arg = text[m.end():closing(text, m.end() - 1, "()")]
        assert arg in MATERIAL, arg
