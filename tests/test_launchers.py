"""The Jacobian apply's internal launchers: an arithmetic without dot products takes no basis."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

HEAD = """#include "mca_internal.cuh"
using namespace mca;
void f(const Grid& gr, const double* D, const float* z, double* w, const double* V, double* part,
       const VecCtl* ctl, unsigned int* cnt, double* h, cudaStream_t s) {
"""


def _compiles(tmp_path, body):
    src = tmp_path / "f.cu"
    src.write_text(HEAD + body + "}\n")
    return subprocess.run(
        [NVCC, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
         os.path.join(ROOT, "include"), "-I",
         os.path.join(ROOT, "paper_2109_07929_gb300", "csrc"), "-c", str(src), "-o",
         str(tmp_path / "f.o")], capture_output=True, text=True).returncode == 0


@pytest.mark.skipif(not os.path.exists(NVCC), reason="needs nvcc")
def test_no_basis_where_the_apply_has_no_dots(tmp_path):
    """FP32 z with a basis is offered for the arithmetics that form dot products only: any other
    would have to launch nothing."""
    assert _compiles(tmp_path, "launch_spmv_dots(gr, D, z, 2, w, V, 2, 1, part, 1, 1, ctl, cnt, h, s);")
    assert _compiles(tmp_path, "launch_apply(gr, D, z, w, 1, 1, kApplyF32, s);")
    for mode in ("kApplyF32", "kApplyF64"):
        assert not _compiles(tmp_path, "launch_spmv_dots(gr, D, z, 2, w, V, 2, 1, part, 1, 1, ctl, "
                                       f"cnt, h, s, {mode});")
