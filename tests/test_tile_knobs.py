"""The tile knobs that the autotuner tries, at every plane edge.  The workspace
holds the x slots of a row in runs of XL, one after the other: a run that does
not divide the edge would overlap the next row's and leave the workspace at its
end.  A column CTA's X slots have to lie within one run."""

import concurrent.futures as cf
import itertools
import subprocess

import pytest

from paper_1402_6297_gb300 import autotune, build

CHECK = """
#include "dfloat.cuh"
#include "matvec_impl.cuh"
template <typename R, int N> constexpr bool fits() {
  using S = nfs::PlaneSplit<R, N>;
  return N % S::XL == 0 && S::XL % S::X == 0 && S::XL >= 1 && N == S::N1 * S::N2;
}
#define NFS_CASE(N) static_assert(fits<float, N>() && fits<double, N>() && fits<nfs::df, N>(), "runs of x slots");
NFS_FOR_EACH_SIZE(NFS_CASE)
"""


def test_runs_of_x_slots_divide_every_edge(tmp_path):
    src = tmp_path / "tiles.cu"
    src.write_text(CHECK)
    knobs = {k: v for k, v in autotune.KNOBS.items() if k in ("NFS_X", "NFS_XL")}
    combos = [dict(zip(knobs, v)) for v in itertools.product(*knobs.values())]

    def check(c):
        cmd = [build.nvcc_path(), "-std=c++17", "-c", str(src), "-I", build.CSRC, "-I", build.ROOT + "/include",
               "-o", str(tmp_path / ("_".join(map(str, c.values())) + ".o"))] + build.ARCH
        r = subprocess.run(cmd + [f"-D{k}={v}" for k, v in c.items()], capture_output=True, text=True)
        return None if r.returncode == 0 else (c, r.stderr[-500:])
    with cf.ThreadPoolExecutor(3) as ex:
        bad = [b for b in ex.map(check, combos) if b]
    assert not bad, bad


def test_a_variant_that_does_not_build_is_passed_over(monkeypatch, tmp_path):
    """A candidate that fails to compile counts as no candidate; the run goes on."""
    def fail_other_runs(defines, workdir):
        if defines["NFS_XL"] != autotune.KNOBS["NFS_XL"][0]:
            raise RuntimeError("nvcc failed")
        return "lib"
    monkeypatch.setattr(autotune, "build_variant", fail_other_runs)
    monkeypatch.setattr(autotune, "time_variant", lambda lib, size: {"ms": 1.0, "err": 1e-7, "cg_res": 1e-12})
    monkeypatch.setattr(autotune, "TUNING_H", str(tmp_path / "tuning.h"))
    monkeypatch.setattr("sys.argv", ["autotune", "--sizes", "48", "--knobs", "NFS_XL"])
    autotune.main()
    assert "#define NFS_XL 4" in (tmp_path / "tuning.h").read_text()
