"""The near-pair lists that vie_set_mesh builds on the device (mesh.cu) against those of
build_topology (topology.cpp, checked against the oracle on the CPU): for all four
kinds of pairs the dense masks, the entries of the elements that do not touch and of those
that do, in their order, and the partner of every touching entry, one by one.  Cells:
structured (exact ties of the distance), jittered, three domains, unequal periods, element
counts on both sides of the 256 that a pass takes at a time."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import cellgen

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1809_05334_gb300")
CSRC = os.path.join(PKG, "csrc")

HARNESS = r"""
#include <cstdio>
#include <cmath>
#include <cstdlib>
#include <vector>
#include "mesh.h"
#include "vie_internal.h"
using namespace vie;
template <typename T> T *dev(const std::vector<T> &v) {
    T *p = nullptr;
    if (cudaMalloc(&p, sizeof(T) * (v.size() + 1)) != cudaSuccess) exit(4);
    if (!v.empty() && cudaMemcpy(p, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice) != cudaSuccess) exit(4);
    return p;
}
template <typename T> std::vector<T> host(const T *p, size_t n) {
    std::vector<T> v(n);
    if (n && cudaMemcpy(v.data(), p, sizeof(T) * n, cudaMemcpyDeviceToHost) != cudaSuccess) exit(4);
    return v;
}
int main(int argc, char **argv) {
    FILE *f = fopen(argv[1], "rb");
    int hdr[4];
    double ab[2];
    if (!f || fread(hdr, sizeof(int), 4, f) != 4 || fread(ab, sizeof(double), 2, f) != 2) return 2;
    const int nv = hdr[0], nt = hdr[1];
    std::vector<double> v(3 * (size_t)nv);
    std::vector<int32_t> t(4 * (size_t)nt), d(nt);
    if (fread(v.data(), sizeof(double), v.size(), f) != v.size() || fread(t.data(), 4, t.size(), f) != t.size() ||
        fread(d.data(), 4, d.size(), f) != d.size()) return 3;
    fclose(f);
    Topology T;
    if (!build_topology(v.data(), nv, t.data(), nt, d.data(), hdr[2], ab[0], ab[1], hdr[3], T, true).empty()) return 5;
    const int nf = (int)T.cf.size(), nh = (int)T.hf.size();
    std::vector<double> hc, hr, hv;
    for (int h : T.hf) {
        hc.insert(hc.end(), &T.fcen[3 * (size_t)h], &T.fcen[3 * (size_t)h] + 3);
        hr.push_back(T.frad[h]);
        hv.insert(hv.end(), &T.fv[9 * (size_t)h], &T.fv[9 * (size_t)h] + 9);
    }
    double reach = 0;
    for (double x : v) reach = std::max(reach, std::fabs(x));
    const ElementSet tet{dev(T.cen), dev(T.rad), dev(T.tv), nt, 4}, face{dev(T.fcen), dev(T.frad), dev(T.fv), nf, 3},
        half{dev(hc), dev(hr), dev(hv), nh, 3};
    const ElementSet sx[4] = {tet, tet, half, half}, sy[4] = {tet, face, tet, face};
    const std::vector<NearPair> *lists[4] = {&T.near_tt, &T.near_tf, &T.near_ft, &T.near_ff};
    long bad = 0, pairs = 0, touching = 0;
    for (int i = 0; i < 4; ++i) {
        const ElementSet &x = sx[i], &y = sy[i];
        if (!x.n || !y.n) continue;
        std::vector<uint16_t> mk((size_t)x.n * y.n, 0);
        std::vector<NearEntry> pr, to;
        for (auto &p : *lists[i]) {
            mk[(size_t)p.x * y.n + p.y] = p.mask;
            for (int k = 0; k < 9; ++k)
                if ((p.mask >> k) & 1u) ((p.touch >> k) & 1u ? to : pr).push_back({p.x, p.y, k, 0});
        }
        uint16_t *dm = dev(std::vector<uint16_t>(mk.size(), 0));
        unsigned *work = dev(std::vector<unsigned>(near_work_words(x.n), 0));
        if (near_count(x, y, T.a, T.b, reach, dm, work, 0) != cudaSuccess) return 6;
        const std::vector<unsigned> tot = host(work + 6 * (size_t)x.n, 3);
        if (tot[0] != pr.size() || tot[1] != to.size() || tot[2] != lists[i]->size()) { ++bad; continue; }
        NearEntry *dp = dev(std::vector<NearEntry>(pr.size())), *dt = dev(std::vector<NearEntry>(to.size()));
        if (near_emit(x, y, T.a, T.b, reach, dm, work, dp, dt, 0) != cudaSuccess) return 7;
        if (host(dm, mk.size()) != mk) ++bad;
        auto differ = [](const NearEntry &p, const NearEntry &q) { return p.x != q.x || p.y != q.y || p.k != q.k; };
        const std::vector<NearEntry> gp = host(dp, pr.size()), gt = host(dt, to.size());
        for (size_t e = 0; e < pr.size(); ++e) bad += differ(gp[e], pr[e]);
        for (size_t e = 0; e < to.size(); ++e) bad += differ(gt[e], to[e]);
        if (i == 0) {
            int32_t *part = dev(std::vector<int32_t>(to.size(), -1));
            int *flag = dev(std::vector<int>(1, 0));
            if (near_partner(dt, (int)to.size(), x.n, work, part, flag, 0) != cudaSuccess) return 8;
            bad += host(flag, 1)[0];
            const std::vector<int32_t> q = host(part, to.size());
            for (size_t e = 0; e < to.size(); ++e)
                bad += q[e] < 0 || q[e] >= (int)to.size() || differ(to[q[e]], NearEntry{to[e].y, to[e].x, 8 - to[e].k, 0});
        }
        pairs += (long)pr.size();
        touching += (long)to.size();
    }
    if (cudaDeviceSynchronize() != cudaSuccess) return 9;
    printf("%ld %ld %ld %d %d %d\n", bad, pairs, touching, nt, nf, nh);
}
"""

CELLS = {"ties": lambda: cellgen.slab_cell(3, 3, 1, 200.0, 200.0, 40.0, (4.0, 0.5)),
         "252": lambda: cellgen.slab_cell(7, 6, 1, 210.0, 150.0, 30.0, (4.0, 0.5)),
         "258": lambda: cellgen.slab_cell(43, 1, 1, 860.0, 20.0, 20.0, (4.0, 0.5)),
         "jitter": lambda: cellgen.slab_cell(6, 5, 3, 180.0, 120.0, 90.0, (4.0, 0.5), jitter=0.15, seed=4),
         "three domains": lambda: cellgen.small_cells()["plasmonic_tiny"],
         "sphere": lambda: cellgen.layered_cell(200.0, 160.0, [(40.0, "buffer"), (100.0, "active")],
                                                spheres=[(100.0, 80.0, 90.0, 20.0, "ag")], h_coarse=40.0, h_fine=16.7,
                                                h_z=40.0, jitter=0.1, seed=3, lateral_fine=False)}


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    pytest.importorskip("paper_1809_05334_gb300.vie").load()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = tmp_path_factory.mktemp("near")
    (d / "h.cu").write_text(HARNESS)
    subprocess.run([nvcc, "-O1", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, str(d / "h.cu"),
                    os.path.join(PKG, "libvie.so"), "-Xlinker", "-rpath=" + PKG, "-o", str(d / "h")], check=True)
    return d


@pytest.mark.parametrize("name", sorted(CELLS))
def test_device_lists_equal_the_host_lists(harness, name):
    cell = CELLS[name]()
    path = harness / "mesh.bin"
    with open(path, "wb") as f:
        np.array([len(cell.verts), len(cell.tets), cell.n_domains, cell.active_domain], np.int32).tofile(f)
        np.array([cell.period_a, cell.period_b], np.float64).tofile(f)
        np.ascontiguousarray(cell.verts, np.float64).tofile(f)
        np.ascontiguousarray(cell.tets, np.int32).tofile(f)
        np.ascontiguousarray(cell.tet_domain, np.int32).tofile(f)
    out = subprocess.run([str(harness / "h"), str(path)], capture_output=True, text=True)
    assert out.returncode == 0, (out.returncode, out.stderr)
    bad, pairs, touching, nt, nf, nh = (int(v) for v in out.stdout.split())
    assert touching >= nt and pairs + touching > nt      # every element touches itself
    assert bad == 0
