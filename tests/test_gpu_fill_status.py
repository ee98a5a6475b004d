"""Status of the fill's launches.  The far kernels' launchers take the error from the runtime
and return it, so a fill that drops their result reports success for a matrix without
its far pairs.  Two launches that the runtime or the launcher refuses on the host, with one
element of zeros and every buffer large enough for the kernels before them: an FP32 form
without a kernel, and an FP64 table block beyond the shared memory.  (A mesh with more
elements than a grid has rows, 65,535, is refused in the same way.)"""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1809_05334_gb300")

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "fill.h"
using namespace vie;
template <typename T> T *zeros() {   // 1 MB, far more than one element takes
    void *p = nullptr;
    if (cudaMalloc(&p, 1 << 20) != cudaSuccess || cudaMemset(p, 0, 1 << 20) != cudaSuccess) exit(3);
    return static_cast<T *>(p);
}
int main(int argc, char **argv) {
    const bool fp64 = !strcmp(argv[1], "fp64");
    DevMesh m{};
    m.nt = 1;
    m.N = 4;
    m.tv = m.cen = m.vol = m.far64 = zeros<double>();
    m.far32 = zeros<float>();
    m.mk_tt = zeros<uint16_t>();
    DevReq q{};
    q.row = zeros<int32_t>();
    q.coef = q.wt = q.kap = q.ieps = zeros<double>();
    q.ptet = zeros<float4>();
    q.etet = zeros<float4>();
    q.ph64 = zeros<double>();
    q.fp.mode = FAR_NORMAL;
    q.fp.nq = 7;                 // no such kernel
    q.f64.n_blob = 100000000;    // 800 MB of shared memory
    void *Z = zeros<char>();
    const cudaError_t e = fp64 ? launch_fill<double>(m, q, static_cast<double *>(Z), 4, nullptr, 0)
                               : launch_fill<float>(m, q, static_cast<float *>(Z), 4, nullptr, 0);
    if (cudaDeviceSynchronize() != cudaSuccess) return 4;
    printf("%d\n", (int)e);
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    pytest.importorskip("paper_1809_05334_gb300.vie").load()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = tmp_path_factory.mktemp("status")
    (d / "h.cu").write_text(HARNESS)
    subprocess.run([nvcc, "-O1", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", os.path.join(PKG, "csrc"),
                    str(d / "h.cu"), os.path.join(PKG, "libvie.so"), "-Xlinker", "-rpath=" + PKG, "-o", str(d / "h")], check=True)
    return str(d / "h")


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_a_refused_far_launch_is_reported(harness, prec):
    out = subprocess.run([harness, prec], capture_output=True, text=True)
    assert out.returncode == 0, (out.returncode, out.stderr)
    assert int(out.stdout) != 0
