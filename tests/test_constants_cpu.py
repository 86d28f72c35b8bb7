"""Constants of the solvers that depend on one another: a change that would break the
problem tables, the per-lane shift recurrences or the rings does not compile."""
import pathlib
import re
import shutil
import subprocess

import pytest

CSRC = pathlib.Path(__file__).resolve().parents[1] / "paper_2212_06635_gb300" / "csrc"
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


def _compile(tmp_path, edits):
    (tmp_path / "include").mkdir()
    shutil.copy(CSRC.parents[1] / "include" / "tm.h", tmp_path / "include")
    tmp_path = tmp_path / "package" / "csrc"   # (the headers include ../../include/tm.h)
    tmp_path.mkdir(parents=True)
    for h in CSRC.glob("*.h"):
        src = h.read_text()
        for name, value in edits.items():
            src = re.sub(r"(constexpr int %s = )[^;]+;" % name, r"\g<1>%s;" % value, src)
        (tmp_path / h.name).write_text(src)
    (tmp_path / "t.cu").write_text('''#include "tm_internal.h"
#include "tm_kernels.h"
static_assert(sizeof(tmk::SolverCtl::alpha_ring) == sizeof(double) * tmk::RING, "control word");
static_assert(sizeof(tmk::MsCtl::alpha_ring) == sizeof(double) * tmk::RING * tmk::MAX_SHIFTS, "multishift state");
''')
    cmd = [NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "--expt-relaxed-constexpr",
           "-c", str(tmp_path / "t.cu"), "-o", str(tmp_path / "t.o")]
    return subprocess.run(cmd, capture_output=True, text=True)


@pytest.mark.skipif(not pathlib.Path(NVCC).exists(), reason="needs nvcc")
@pytest.mark.parametrize("edits,compiles", [({}, True), ({"RING": 8}, True), ({"MAX_SHIFTS": 32}, False),
                                            ({"MAX_SHIFTS": 33}, False), ({"MAX_SHIFTS": 1}, False)],
                         ids=["as they are", "a longer ring", "group like a batch", "more shifts than lanes",
                              "group like one problem"])
def test_dependent_constants(tmp_path, edits, compiles):
    r = _compile(tmp_path, edits)
    assert (r.returncode == 0) == compiles, r.stderr[-2000:]
    if not compiles:
        assert "static assertion failed" in r.stderr
