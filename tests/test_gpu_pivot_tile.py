"""Inverse of one 64 x 64 pivot tile (gj_invert_tc at n = 64) with condition 1e5: its residual is
that of a rounded inverse, not of an elimination without pivoting.  An entry of A X is a sum
of 64 products whose factors carry a rounding or two each: 16 u max|A| max|X| bounds it
(sqrt(64) of them in quadrature, twice u); elimination in FP32 alone leaves 100 u and more of
it (the growth of its pivots)."""
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1809_05334_gb300")

HARNESS = r"""
#include <cstdio>
#include <vector>
#include "linalg.h"
using namespace vie;
int main(int argc, char **argv) {
    const int n = 64;
    std::vector<float> a(2 * n * n);
    FILE *f = fopen(argv[1], "rb");
    if (!f || fread(a.data(), 4, a.size(), f) != a.size()) return 2;
    fclose(f);
    float *A = nullptr;
    int *status = nullptr, bad = -1;
    void *pack = nullptr;
    cudaStream_t st, aux;
    if (cudaMalloc(&A, 4 * a.size()) || cudaMalloc(&status, sizeof(int)) || cudaMalloc(&pack, gj_pack_bytes(n)) ||
        cudaStreamCreate(&st) || cudaStreamCreate(&aux) || cudaMemset(status, 0, sizeof(int)) ||
        cudaMemcpy(A, a.data(), 4 * a.size(), cudaMemcpyHostToDevice) || cudaDeviceSynchronize()) return 3;
    if (gj_invert_tc(A, n, n, status, pack, st, aux, nullptr, 512, n) || cudaStreamSynchronize(st)) return 4;
    if (cudaMemcpy(a.data(), A, 4 * a.size(), cudaMemcpyDeviceToHost) ||
        cudaMemcpy(&bad, status, sizeof(int), cudaMemcpyDeviceToHost)) return 5;
    f = fopen(argv[1], "wb");
    if (!f || fwrite(a.data(), 4, a.size(), f) != a.size() || fclose(f)) return 6;
    return bad ? 7 : 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    pytest.importorskip("paper_1809_05334_gb300.vie").load()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = tmp_path_factory.mktemp("tile")
    (d / "h.cu").write_text(HARNESS)
    subprocess.run([nvcc, "-O1", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", os.path.join(PKG, "csrc"),
                    str(d / "h.cu"), os.path.join(PKG, "libvie.so"), "-Xlinker", "-rpath=" + PKG, "-o", str(d / "h")], check=True)
    return d


@pytest.mark.parametrize("seed", [3, 4, 5])
def test_residual_of_an_ill_conditioned_tile(harness, seed):
    rng = np.random.default_rng(seed)

    def unitary():
        return np.linalg.qr(rng.standard_normal((64, 64)) + 1j * rng.standard_normal((64, 64)))[0]
    A = (unitary() @ np.diag(np.logspace(0, -5, 64)) @ unitary()).astype(np.complex64)
    path = harness / "a.bin"
    A.tofile(path)
    out = subprocess.run([str(harness / "h"), str(path)], capture_output=True, text=True)
    assert out.returncode == 0, (out.returncode, out.stderr)
    X = np.fromfile(path, np.complex64).reshape(64, 64).astype(complex)
    A = A.astype(complex)
    res = np.max(np.abs(np.eye(64) - A @ X)) / (2.0 ** -24 * np.max(np.abs(A)) * np.max(np.abs(X)))
    assert res <= 16.0, res
