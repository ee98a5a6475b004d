// Matrix fill of the periodic SWG VIE (Eq. (2)) on the GPU.
//
// Z_mn = int f_m.f_n/eps_r - k0^2 int int f_m . kappa' f_n g_p + int int div f_m q_n g_p
// (lengths in nm, scaled by eps0), with q_n = div'(kappa f_n) including the
// surface charge (kappa- - kappa+) on face n and the surface term -delta of a
// half test function.  Every Z entry is a sum over element pairs (tetrahedra
// and charge-carrying faces); each element pair is integrated once and its
// contributions are added into Z with atomics.
//
//  far pairs : degree-2 product rules (4 points per tetrahedron, 3 per
//              triangle), g_p by the Ewald series, precision T (FP32 or FP64).
//  near pairs: the static part exp(j k_par.R)/(4 pi R) of every near image is
//              integrated in closed form over one element at the degree-5
//              points of the other, averaged over both orders, plus the
//              remainder of g_p with the degree-2 product rules.  The closed
//              forms run in FP64 when the elements touch, in T otherwise.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "device_math.cuh"
#include "far_poly.cuh"
#include "fill.h"

namespace vie {

__constant__ double c_w5tet[14];
__constant__ double c_w5tri[7];

// ---------------------------------------------------------------------------
// host set-up of the constant tables
// ---------------------------------------------------------------------------
static void weideman_coeffs(int N, double &L, std::vector<double> &a) {
    L = std::sqrt(N / std::sqrt(2.0));
    const int M = 16 * N;
    a.assign(N + 1, 0.0);
    for (int k = 0; k < M; ++k) {
        double th = -M_PI + (k + 0.5) * 2.0 * M_PI / M;
        double t = L * std::tan(0.5 * th);
        double F = std::exp(-t * t) * (L * L + t * t);
        for (int n = 0; n <= N; ++n) a[n] += F * std::cos(n * th) / M;
    }
}

cudaError_t upload_constants() {
    WeidemanTables w{};
    std::vector<double> a;
    double L;
    weideman_coeffs(NW64, L, a);
    w.L64 = L;
    for (int n = 0; n <= NW64; ++n) w.a64[n] = a[n];
    weideman_coeffs(NW32, L, a);
    w.L32 = (float)L;
    for (int n = 0; n <= NW32; ++n) w.a32[n] = (float)a[n];
    cudaError_t e = cudaMemcpyToSymbol(c_weid, &w, sizeof(w));
    if (e != cudaSuccess) return e;
    e = upload_far64_constants(&w);   // far64.cu's own copy of c_weid
    if (e != cudaSuccess) return e;
    double w5t[14], w5f[7];
    tet_rule5(nullptr, w5t);
    tri_rule5(nullptr, w5f);
    e = cudaMemcpyToSymbol(c_w5tet, w5t, sizeof(w5t));
    if (e != cudaSuccess) return e;
    return cudaMemcpyToSymbol(c_w5tri, w5f, sizeof(w5f));
}

cudaError_t upload_ewald(EwaldTables *dev, const EwaldTables &t, cudaStream_t st) {
    return cudaMemcpyAsync(dev, &t, sizeof(t), cudaMemcpyHostToDevice, st);
}

// ---------------------------------------------------------------------------
// per-request tables of the FP32 path (built in FP64 from the Ewald series):
// cubic Hermite coefficients per interval, in the local variable u in [0, 1)
// ---------------------------------------------------------------------------
__device__ void hermite(double f0, double d0, double f1, double d1, double h, double c[4]) {
    c[0] = f0;
    c[1] = h * d0;
    c[2] = 3.0 * (f1 - f0) - h * (2.0 * d0 + d1);
    c[3] = 2.0 * (f0 - f1) + h * (d0 + d1);
}

__device__ void spatial_node(const EwaldTables *ew, double x, double &F, double &dF) {
    // F(x) = exp(-x^2) Re erfcx(x + j b),  F'(x) = -exp(-x^2) (2 b Im erfcx(x + j b) + 2/sqrt(pi))
    const double b = ew->bb;
    cx<double> w = erfcx_c<double>(cx<double>{x, b});
    const double g = exp(-x * x);
    F = g * w.re;
    dF = -g * (2.0 * b * w.im + 2.0 * rsqrt_pi<double>());
}

__device__ void spectral_node(const EwaldTables *ew, int tb, double z, cx<double> &G, cx<double> &dG) {
    // G(z) = (t1 + t2)/(4ab gamma), G'(z) = gamma (t1 - t2)/(4ab gamma)
    const double E = ew->E;
    const cx<double> g = {ew->tab_gamma[tb][0], ew->tab_gamma[tb][1]};
    const cx<double> ig = {ew->tab_ig[tb][0], ew->tab_ig[tb][1]};
    const double pre = ew->tab_pre[tb] * exp(-(z * E) * (z * E));
    cx<double> t1, t2;
    if (g.im == 0.0) {
        const double gr = g.re;
        t1 = {pre * erfcx_r<double>(gr / (2 * E) + z * E), 0.0};
        const double u = gr / (2 * E) - z * E;
        t2 = {(u >= 0) ? pre * erfcx_r<double>(u) : 2.0 * exp(-gr * z) - pre * erfcx_r<double>(-u), 0.0};
    } else {
        const double gi = g.im;
        cx<double> e1 = erfcx_c<double>(cx<double>{z * E, gi / (2 * E)});
        double sg, cg;
        sincos(gi * z, &sg, &cg);
        t1 = pre * e1;
        t2 = cx<double>{2.0 * cg - pre * e1.re, -2.0 * sg + pre * e1.im};
    }
    G = (t1 + t2) * ig;
    dG = (g * (t1 - t2)) * ig;
}

__global__ void k_build_tables(const EwaldTables *__restrict__ ew, float *stab, float2 *ztab, int n_tab,
                               float4 *rtab) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < NSPAT) {
        const double h = ew->xs_h;
        double F0, D0, F1, D1, c[4];
        spatial_node(ew, i * h, F0, D0);
        spatial_node(ew, (i + 1) * h, F1, D1);
        hermite(F0, D0, F1, D1, h, c);
        for (int k = 0; k < 4; ++k) stab[4 * i + k] = float(c[k]);
        return;
    }
    const int j = i - NSPAT;
    const int tb = j / NZTAB, iz = j % NZTAB;
    if (rtab && tb == n_tab) {   // the zero table after the real tables
        rtab[(size_t)n_tab * NZTAB + iz] = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    if (tb >= n_tab) return;
    const double h = double(ew->z_max) / NZTAB;
    cx<double> G0, D0, G1, D1;
    spectral_node(ew, tb, iz * h, G0, D0);
    spectral_node(ew, tb, (iz + 1) * h, G1, D1);
    double cr[4], ci[4];
    hermite(G0.re, D0.re, G1.re, D1.re, h, cr);
    hermite(G0.im, D0.im, G1.im, D1.im, h, ci);
    for (int k = 0; k < 4; ++k) ztab[((size_t)tb * NZTAB + iz) * 4 + k] = make_float2(float(cr[k]), float(ci[k]));
    // the real and the imaginary parts apart, 16 bytes per interval each
    if (rtab) {
        rtab[(size_t)tb * NZTAB + iz] = make_float4(float(cr[0]), float(cr[1]), float(cr[2]), float(cr[3]));
        rtab[(size_t)(n_tab + 1 + tb) * NZTAB + iz] = make_float4(float(ci[0]), float(ci[1]), float(ci[2]), float(ci[3]));
    }
}

cudaError_t launch_build_tables(const EwaldTables *ew, float *stab, float2 *ztab, int n_tab, cudaStream_t st,
                                float4 *rtab) {
    const int n = NSPAT + (n_tab + (rtab ? 1 : 0)) * NZTAB;
    k_build_tables<<<(n + 127) / 128, 128, 0, st>>>(ew, stab, ztab, n_tab, rtab); ++g_launches;
    return cudaGetLastError();
}

// near-image mask of the reversed pair: image (m,n) <-> (-m,-n), i.e. bit k <-> bit 8-k
__device__ __forceinline__ unsigned mirror_mask(unsigned sub) {
    unsigned r = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k)
        if ((sub >> k) & 1u) r |= 1u << (8 - k);
    return r;
}

// g_p for the fill kernels: FP64 by the Ewald series, FP32 from the tables
template <typename T> struct Green;
// eval2 returns g_p(d) and g_p(-d) (the same near-image mask applies to both)
template <> struct Green<double> {
    template <bool SYM = false>
    __device__ static cx<double> eval(double dx, double dy, double dz, unsigned sub, const float *, const float2 *,
                                      const EwaldTables *ew, const EwaldF32 &, const float4 * = nullptr,
                                      unsigned long long = ~0ull) {
        return green_p<double>(dx, dy, dz, sub, ew);
    }
    template <bool SYM = false>
    __device__ static void eval2(double dx, double dy, double dz, unsigned sub, const float *, const float2 *,
                                 const EwaldTables *ew, const EwaldF32 &, cx<double> &gp, cx<double> &gm,
                                 const float4 * = nullptr, unsigned long long = ~0ull) {
        gp = green_p<double>(dx, dy, dz, sub, ew);
        gm = green_p<double>(-dx, -dy, -dz, mirror_mask(sub), ew);
    }
};
template <> struct Green<float> {
    template <bool SYM = false>
    __device__ static cx<float> eval(float dx, float dy, float dz, unsigned sub, const float *stab,
                                     const float2 *ztab, const EwaldTables *, const EwaldF32 &ef,
                                     const float4 *rtab = nullptr, unsigned long long imask = ~0ull) {
        cx<float> g, unused;
        green_tab_impl<false, SYM>(dx, dy, dz, sub, stab, ztab, ef, g, unused, rtab, imask);
        return g;
    }
    template <bool SYM = false>
    __device__ static void eval2(float dx, float dy, float dz, unsigned sub, const float *stab, const float2 *ztab,
                                 const EwaldTables *, const EwaldF32 &ef, cx<float> &gp, cx<float> &gm,
                                 const float4 *rtab = nullptr, unsigned long long imask = ~0ull) {
        green_tab_impl<true, SYM>(dx, dy, dz, sub, stab, ztab, ef, gp, gm, rtab, imask);
    }
};

// stage the spatial table in shared memory (FP32 path only)
template <typename T>
__device__ __forceinline__ const float *stage_stab(const DevReq &q, float *smem) {
    if (sizeof(T) == 8) return nullptr;
    for (int i = threadIdx.x; i < 4 * NSPAT; i += blockDim.x) smem[i] = q.stab[i];
    __syncthreads();
    return smem;
}

template <typename T> constexpr size_t stab_bytes() { return sizeof(T) == 4 ? 4 * NSPAT * sizeof(float) : 0; }

// ---------------------------------------------------------------------------
// helpers
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void atomic_add_c(T *Z, size_t idx, cx<T> v) {
    if constexpr (sizeof(T) == 4) {
        red_c(Z, idx, v.re, v.im);
    } else {
        atomicAdd(Z + 2 * idx, v.re);
        atomicAdd(Z + 2 * idx + 1, v.im);
    }
}

__device__ __forceinline__ cx<double> ld2(const double *p) { return {p[0], p[1]}; }

// scatter the 16 face-pair contributions of one tetrahedron pair
template <typename T>
__device__ void scatter_tt(const DevMesh &m, const DevReq &q, T *Z, size_t N, int t, int s,
                           const Mom<T> &mo) {
    if constexpr (sizeof(T) == 4) {
        scatter_rec<false>(Z, N, float(q.k0 * q.k0), load_tet_rec(q.etet, m.nt, t), load_tet_rec(q.etet, m.nt, s), mo, mo.S,
                           false);
        return;
    }
    const T *ft = m.far<T>(t);
    const T *fs = m.far<T>(s);
    const T k2 = T(q.k0 * q.k0);
    cx<T> kap = {T(q.kap[2 * s]), T(q.kap[2 * s + 1])};
    cx<T> kS = kap * mo.S;
    for (int i = 0; i < 4; ++i) {
        const T wi[3] = {ft[15 + 3 * i], ft[16 + 3 * i], ft[17 + 3 * i]};
        const T ci = T(q.coef[4 * t + i]);
        cx<T> wti = {T(q.wt[2 * (4 * t + i)]), T(q.wt[2 * (4 * t + i) + 1])};
        size_t row = (size_t)q.row[4 * t + i];
        cx<T> wB = wi[0] * mo.B[0] + wi[1] * mo.B[1] + wi[2] * mo.B[2];
        for (int j = 0; j < 4; ++j) {
            const T wj[3] = {fs[15 + 3 * j], fs[16 + 3 * j], fs[17 + 3 * j]};
            const T cj = T(q.coef[4 * s + j]);
            cx<T> wsj = {T(q.wt[2 * (4 * s + j)]), -T(q.wt[2 * (4 * s + j) + 1])};
            size_t col = (size_t)q.row[4 * s + j];
            cx<T> M = mo.C - (wj[0] * mo.A[0] + wj[1] * mo.A[1] + wj[2] * mo.A[2]) - wB +
                      (wi[0] * wj[0] + wi[1] * wj[1] + wi[2] * wj[2]) * mo.S;
            cx<T> val = (-k2 * ci * cj) * (kap * M) + (T(9) * ci * cj) * kS;
            val = (wti * wsj) * val;
            atomic_add_c(Z, row * N + col, val);
        }
    }
}

// ---------------------------------------------------------------------------
// all tetrahedron pairs: degree-2 product rule of g_p; for the near images of a
// pair the static part is removed here and integrated by k_pr_tt / k_touch_tt
// ---------------------------------------------------------------------------
// Each unordered pair {t, s} (s >= t) is evaluated once: one pass over the 16
// point pairs gives g_p(x_a - y_b) for the block (t, s) and g_p(y_b - x_a) for
// the block (s, t) (the reversed pair's moments swap the roles of the offsets).
// SYM: normal incidence (the tabulated path's symmetric mode sum, gm = gp).
// Eight CTAs per SM for the FP32 tables (64 registers; the kernel is
// issue-bound and its fixed-latency waits need the extra warps), six for FP64.
template <typename T, bool SYM>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 8 : 6)
    k_far_tt(DevMesh m, const __grid_constant__ DevReq q, T *Z, size_t N) {
    extern __shared__ float smem_tab[];
    const int t = blockIdx.y;
    if ((int)(blockIdx.x * blockDim.x + blockDim.x) <= t) return;   // the whole block is below the diagonal
    const float *stab = stage_stab<T>(q, smem_tab);
    const int s0 = blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = s0 < m.nt && s0 >= t;   // lanes off the pair range stay until the warp's image mask is formed
    const int s = live ? s0 : t;
    // near images of this pair: their static part is integrated separately
    const unsigned sub = m.mk_tt[(size_t)t * m.nt + s];
    const T *ft = m.far<T>(t);
    const T *fs = m.far<T>(s);
    Mom<T> mo, mr;   // blocks (t, s) and (s, t)
    mo.zero();
    mr.zero();
    const T wgt = ft[27] * fs[27];
    // images that can reach the cut from some point pair of {t, s}, decided once
    // for the 16 point pairs (FP32 tables only): every point pair lies within
    // rt + rs of the centroid offset
    unsigned long long imask = ~0ull;
    if (sizeof(T) == 4) {
        float rt = 0.f, rs = 0.f;
        for (int a = 0; a < 4; ++a) {
            const float ux = float(ft[3 * a] - ft[12]), uy = float(ft[3 * a + 1] - ft[13]), uz = float(ft[3 * a + 2] - ft[14]);
            const float vx = float(fs[3 * a] - fs[12]), vy = float(fs[3 * a + 1] - fs[13]), vz = float(fs[3 * a + 2] - fs[14]);
            rt = fmaxf(rt, sqrtf(ux * ux + uy * uy + uz * uz));
            rs = fmaxf(rs, sqrtf(vx * vx + vy * vy + vz * vz));
        }
        imask = image_mask(q.ef, float(ft[12] - fs[12]), float(ft[13] - fs[13]), float(ft[14] - fs[14]), rt + rs);
        // one image list for the whole warp (the union of its pairs' lists): the
        // image index is warp-uniform, so the image loop runs on the uniform
        // datapath and its table entries are broadcast loads
        if (!live) imask = 0ull;
        const unsigned lo = __reduce_or_sync(0xffffffffu, (unsigned)imask);
        const unsigned hi = __reduce_or_sync(0xffffffffu, (unsigned)(imask >> 32));
        imask = ((unsigned long long)hi << 32) | lo;
    }
    if (!live) return;
    for (int a = 0; a < 4; ++a) {
        const T xa[3] = {ft[3 * a], ft[3 * a + 1], ft[3 * a + 2]};
        const T ra[3] = {xa[0] - ft[12], xa[1] - ft[13], xa[2] - ft[14]};
        for (int b = 0; b < 4; ++b) {
            const T yb[3] = {fs[3 * b], fs[3 * b + 1], fs[3 * b + 2]};
            const T rb[3] = {yb[0] - fs[12], yb[1] - fs[13], yb[2] - fs[14]};
            cx<T> g, gr;
            Green<T>::template eval2<SYM>(xa[0] - yb[0], xa[1] - yb[1], xa[2] - yb[2], sub, stab, q.ztab, q.ew,
                                          q.ef, g, gr, q.rtab, imask);
            g = wgt * g;
            const T rr = ra[0] * rb[0] + ra[1] * rb[1] + ra[2] * rb[2];
            mo.S = mo.S + g;
            for (int d = 0; d < 3; ++d) {
                mo.A[d] = mo.A[d] + ra[d] * g;
                mo.B[d] = mo.B[d] + rb[d] * g;
            }
            mo.C = mo.C + rr * g;
            if (!SYM) {
                gr = wgt * gr;
                mr.S = mr.S + gr;
                for (int d = 0; d < 3; ++d) {
                    mr.A[d] = mr.A[d] + rb[d] * gr;
                    mr.B[d] = mr.B[d] + ra[d] * gr;
                }
                mr.C = mr.C + rr * gr;
            }
        }
    }
    if (SYM) {   // g_p(-d) = g_p(d): the reversed pair's moments swap A and B
        mr.S = mo.S;
        mr.C = mo.C;
        for (int d = 0; d < 3; ++d) { mr.A[d] = mo.B[d]; mr.B[d] = mo.A[d]; }
    }
    scatter_tt<T>(m, q, Z, N, t, s, mo);
    if (s != t) scatter_tt<T>(m, q, Z, N, s, t, mr);
}

// ---------------------------------------------------------------------------
// near tetrahedron pairs: one warp per pair
// ---------------------------------------------------------------------------
__device__ __forceinline__ float inv_sqrt(float x) { return rsqrt_ftz(x); }
__device__ __forceinline__ double inv_sqrt(double x) { return rsqrt(x); }

// near image of a pair, elements not touching: degree-5 x degree-5 product
// rule of exp(j k_par.R)/(4 pi R), one thread per (pair, image); 3.3 ms of the
// bench cell's fill with the loops exchanged (every load of the inner loop a
// gather, L1 87% busy)
template <typename T>
__global__ void __launch_bounds__(128) k_pr_tt(DevMesh m, const __grid_constant__ DevReq q, T *Z, size_t N, const NearEntry *list, int n) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const NearEntry en = list[e];
    const int t = en.x, s = en.y, k = en.k;
    const double R[3] = {(k / 3 - 1) * m.a, (k % 3 - 1) * m.b, 0.0};
    const double *ct = m.cen + 3 * (size_t)t, *cs = m.cen + 3 * (size_t)s;
    const T *nx = m.nrel<T>(t), *ny = m.nrel<T>(s);
    const T dc[3] = {T(ct[0] - cs[0] + R[0]), T(ct[1] - cs[1] + R[1]), T(ct[2] - cs[2])};
    // the source points (another element per lane) in the outer loop, the test
    // points (the entries are sorted by test element: mostly one per warp, a
    // broadcast load) in the inner one
    T s0 = 0, sA[3] = {0, 0, 0}, sB[3] = {0, 0, 0}, sC = 0;
#pragma unroll 1
    for (int b = 0; b < 14; ++b) {
        const T yb[4] = {ny[4 * b], ny[4 * b + 1], ny[4 * b + 2], ny[4 * b + 3]};
        const T o[3] = {dc[0] - yb[0], dc[1] - yb[1], dc[2] - yb[2]};
        T f0 = 0, fa[3] = {0, 0, 0};
#pragma unroll
        for (int a = 0; a < 14; ++a) {
            const T xa[4] = {nx[4 * a], nx[4 * a + 1], nx[4 * a + 2], nx[4 * a + 3]};
            const T dx = xa[0] + o[0], dy = xa[1] + o[1], dz = xa[2] + o[2];
            const T f = xa[3] * inv_sqrt(dx * dx + dy * dy + dz * dz);
            f0 += f;
            fa[0] += f * xa[0];
            fa[1] += f * xa[1];
            fa[2] += f * xa[2];
        }
        f0 *= yb[3];
        s0 += f0;
        for (int d = 0; d < 3; ++d) {
            fa[d] *= yb[3];
            sA[d] += fa[d];
            sB[d] += f0 * yb[d];
            sC += fa[d] * yb[d];
        }
    }
    const cx<T> pt = {T(q.img_ph[2 * k]), T(q.img_ph[2 * k + 1])};
    Mom<T> mo;
    mo.S = s0 * pt;
    mo.C = sC * pt;
    for (int d = 0; d < 3; ++d) {
        mo.A[d] = sA[d] * pt;
        mo.B[d] = sB[d] * pt;
    }
    scatter_tt<T>(m, q, Z, N, t, s, mo);
}

// Touching images, exploiting the symmetry of the two integration orders:
// order (ii) of the entry (t, s, k) is order (i) of its partner (s, t, 8-k)
// with the test and source polynomial moments exchanged.  k_touch_half
// computes order (i) of every entry once (phase-free real moments, FP64;
// half a warp per entry, lane q = degree-5 point q of the test element);
// k_touch_combine averages each entry with its partner and scatters.
// Bound by the FP64 pipe: the source's geometry comes from its record, the
// arctangents of a face are one solid angle (6 logarithms, 4 arctangents and 4
// square roots per point; 12 arctangents, 10 square roots and 25 divisions before).
__global__ void k_geom(DevMesh m, TetGeom *tet, TriGeom *tri) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < m.nt) tet_geom(m.tv + 12 * (size_t)e, tet[e]);
    else if (e - m.nt < m.nf) tri_geom(m.fv + 9 * (size_t)(e - m.nt), tri[e - m.nt]);
}

__global__ void __launch_bounds__(128) k_touch_half(DevMesh m, const TetGeom *geom, const NearEntry *list, int n, double *out) {
    const int e = (blockIdx.x * blockDim.x + threadIdx.x) >> 4;
    const int hl = threadIdx.x & 15;
    double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    if (e < n && hl < 14) {
        const NearEntry en = list[e];
        const int t = en.x, s = en.y, k = en.k;
        const double R[3] = {(k / 3 - 1) * m.a, (k % 3 - 1) * m.b, 0.0};
        const double *r5 = m.q5 + (size_t)t * 42 + 3 * hl;
        const double w = m.vol[t] * c_w5tet[hl];
        const double *src = m.tv + 12 * (size_t)s;
        const double *ct = m.cen + 3 * (size_t)t, *cs = m.cen + 3 * (size_t)s;
        double rel[12];
        for (int j = 0; j < 4; ++j)
            for (int d = 0; d < 3; ++d) rel[3 * j + d] = (src[3 * j + d] - R[d]) - r5[d];
        double I, vec[3];
        tet_integrals<true>(geom[s], rel, I, vec);
        double f[3], rho[3];
        for (int d = 0; d < 3; ++d) {
            f[d] = vec[d] + (r5[d] - (cs[d] - R[d])) * I;   // int (r' - c_s)/R over the image source
            rho[d] = r5[d] - ct[d];
        }
        acc[0] = w * I;
        for (int d = 0; d < 3; ++d) {
            acc[1 + d] = w * rho[d] * I;   // test polynomial
            acc[4 + d] = w * f[d];         // source polynomial
        }
        acc[7] = w * (rho[0] * f[0] + rho[1] * f[1] + rho[2] * f[2]);
    }
    for (int i = 0; i < 8; ++i)
        for (int o = 8; o > 0; o >>= 1) acc[i] += __shfl_down_sync(0xffffffffu, acc[i], o, 16);
    if (e < n && hl == 0)
        for (int i = 0; i < 8; ++i) out[8 * (size_t)e + i] = acc[i];
}

template <typename T>
__global__ void __launch_bounds__(128) k_touch_combine(DevMesh m, const __grid_constant__ DevReq q, T *Z, size_t N, const NearEntry *list,
                                                       const int32_t *partner, const double *half, int n) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const NearEntry en = list[e];
    const double *a = half + 8 * (size_t)e;
    const double *b = half + 8 * (size_t)partner[e];
    const double pr = 0.5 * q.img_ph[2 * en.k], pi = 0.5 * q.img_ph[2 * en.k + 1];
    // moments of this entry: S and C symmetric, test/source polynomials exchanged in the partner
    double v[8];
    v[0] = a[0] + b[0];
    for (int d = 0; d < 3; ++d) {
        v[1 + d] = a[1 + d] + b[4 + d];
        v[4 + d] = a[4 + d] + b[1 + d];
    }
    v[7] = a[7] + b[7];
    Mom<T> mo;
    mo.S = {T(pr * v[0]), T(pi * v[0])};
    mo.C = {T(pr * v[7]), T(pi * v[7])};
    for (int d = 0; d < 3; ++d) {
        mo.A[d] = {T(pr * v[1 + d]), T(pi * v[1 + d])};
        mo.B[d] = {T(pr * v[4 + d]), T(pi * v[4 + d])};
    }
    scatter_tt<T>(m, q, Z, N, en.x, en.y, mo);
}

// ---------------------------------------------------------------------------
// scalar element pairs involving charge faces:
//   TF: test tet t, source charge face f   -> Z[row(t,i), frow(f)] += wt 3c qs_f S
//   FT: test half face h, source tet s     -> Z[frow(hf h), row(s,j)] -= conj(wt) kappa_s 3c S
//   FF: test half face h, source face f    -> Z[frow(hf h), frow(f)] -= qs_f S
// ---------------------------------------------------------------------------
enum PairKind { PK_TF = 0, PK_FT = 1, PK_FF = 2 };

template <int PK> struct PKTraits;
template <> struct PKTraits<PK_TF> { static constexpr bool xtet = true, ytet = false; };
template <> struct PKTraits<PK_FT> { static constexpr bool xtet = false, ytet = true; };
template <> struct PKTraits<PK_FF> { static constexpr bool xtet = false, ytet = false; };

template <typename T, int PK>
__device__ void scatter_scalar(const DevMesh &m, const DevReq &q, T *Z, size_t N, int x, int y, cx<T> S) {
    if (PK == PK_TF) {
        cx<T> qs = {T(q.qs[2 * y]), T(q.qs[2 * y + 1])};
        size_t col = (size_t)q.frow[y];
        cx<T> qS = qs * S;
        for (int i = 0; i < 4; ++i) {
            cx<T> wti = {T(q.wt[2 * (4 * x + i)]), T(q.wt[2 * (4 * x + i) + 1])};
            T di = T(3) * T(q.coef[4 * x + i]);
            atomic_add_c(Z, (size_t)q.row[4 * x + i] * N + col, di * (wti * qS));
        }
    } else if (PK == PK_FT) {
        size_t row = (size_t)q.frow[m.hf[x]];
        cx<T> kap = {T(q.kap[2 * y]), T(q.kap[2 * y + 1])};
        cx<T> kS = kap * S;
        for (int j = 0; j < 4; ++j) {
            cx<T> wsj = {T(q.wt[2 * (4 * y + j)]), -T(q.wt[2 * (4 * y + j) + 1])};
            T dj = T(3) * T(q.coef[4 * y + j]);
            atomic_add_c(Z, row * N + (size_t)q.row[4 * y + j], (-dj) * (wsj * kS));
        }
    } else {
        size_t row = (size_t)q.frow[m.hf[x]];
        cx<T> qs = {T(q.qs[2 * y]), T(q.qs[2 * y + 1])};
        atomic_add_c(Z, row * N + (size_t)q.frow[y], T(-1) * (qs * S));
    }
}

template <typename T, bool TET>
__device__ __forceinline__ const T *far_el(const DevMesh &m, int e) {
    return TET ? m.far<T>(e) : m.ffar<T>(e);
}

// SYM: normal incidence (the tabulated path's symmetric mode sum).
template <typename T, int PK, bool SYM>
__global__ void __launch_bounds__(128) k_far_scalar(DevMesh m, const __grid_constant__ DevReq q, T *Z, size_t N, int nx, int ny,
                                                    const uint16_t *mk) {
    extern __shared__ float smem_tab[];
    const float *stab = stage_stab<T>(q, smem_tab);
    const int y = blockIdx.x * blockDim.x + threadIdx.x;
    const int x = blockIdx.y;
    if (y >= ny) return;
    const unsigned sub = mk[(size_t)x * ny + y];
    constexpr bool XT = PKTraits<PK>::xtet, YT = PKTraits<PK>::ytet;
    // a test face is addressed by its half-function index; geometry by charge-face index
    const T *fx = far_el<T, XT>(m, XT ? x : m.hf[x]);
    const T *fy = far_el<T, YT>(m, y);
    const int qx = XT ? 4 : 3, qy = YT ? 4 : 3;
    const T wgt = fx[XT ? 27 : 9] * fy[YT ? 27 : 9];
    // images that can reach the cut from some point pair, decided once per
    // element pair (FP32 tables only): centres and radii of the two point sets
    unsigned long long imask = ~0ull;
    if (sizeof(T) == 4) {
        float c1[3] = {0.f, 0.f, 0.f}, c2[3] = {0.f, 0.f, 0.f};
        for (int a = 0; a < qx; ++a)
            for (int d = 0; d < 3; ++d) c1[d] += float(fx[3 * a + d]) / qx;
        for (int b = 0; b < qy; ++b)
            for (int d = 0; d < 3; ++d) c2[d] += float(fy[3 * b + d]) / qy;
        float r1 = 0.f, r2 = 0.f;
        for (int a = 0; a < qx; ++a) {
            const float ux = float(fx[3 * a]) - c1[0], uy = float(fx[3 * a + 1]) - c1[1], uz = float(fx[3 * a + 2]) - c1[2];
            r1 = fmaxf(r1, sqrtf(ux * ux + uy * uy + uz * uz));
        }
        for (int b = 0; b < qy; ++b) {
            const float ux = float(fy[3 * b]) - c2[0], uy = float(fy[3 * b + 1]) - c2[1], uz = float(fy[3 * b + 2]) - c2[2];
            r2 = fmaxf(r2, sqrtf(ux * ux + uy * uy + uz * uz));
        }
        imask = image_mask(q.ef, c1[0] - c2[0], c1[1] - c2[1], c1[2] - c2[2], r1 + r2);
    }
    cx<T> S = {0, 0};
    for (int a = 0; a < qx; ++a)
        for (int b = 0; b < qy; ++b) {
            cx<T> g = Green<T>::template eval<SYM>(fx[3 * a] - fy[3 * b], fx[3 * a + 1] - fy[3 * b + 1],
                                                   fx[3 * a + 2] - fy[3 * b + 2], sub, stab, q.ztab, q.ew, q.ef,
                                                   q.rtab, imask);
            S = S + g;
        }
    S = wgt * S;
    scatter_scalar<T, PK>(m, q, Z, N, x, y, S);
}

template <typename T, int PK>
__global__ void __launch_bounds__(128) k_pr_scalar(DevMesh m, const __grid_constant__ DevReq q, T *Z, size_t N, const NearEntry *list,
                                                   int n) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    constexpr bool XT = PKTraits<PK>::xtet, YT = PKTraits<PK>::ytet;
    const NearEntry en = list[e];
    const int x = en.x, y = en.y, k = en.k;
    const int xf = XT ? x : m.hf[x];
    constexpr int nqx = XT ? 14 : 7, nqy = YT ? 14 : 7;
    const double R[3] = {(k / 3 - 1) * m.a, (k % 3 - 1) * m.b, 0.0};
    const T *nx = XT ? m.nrel<T>(xf) : m.fnrel<T>(xf);
    const T *ny = YT ? m.nrel<T>(y) : m.fnrel<T>(y);
    const double *cxp = XT ? m.cen + 3 * (size_t)xf : m.fcen + 3 * (size_t)xf;
    const double *cyp = YT ? m.cen + 3 * (size_t)y : m.fcen + 3 * (size_t)y;
    const T dc[3] = {T(cxp[0] - cyp[0] + R[0]), T(cxp[1] - cyp[1] + R[1]), T(cxp[2] - cyp[2])};
    T s0 = 0;
    for (int a = 0; a < nqx; ++a) {
        const T *xa = nx + 4 * a;
        T f0 = 0;
        for (int b = 0; b < nqy; ++b) {
            const T *yb = ny + 4 * b;
            const T dx = xa[0] - yb[0] + dc[0], dy = xa[1] - yb[1] + dc[1], dz = xa[2] - yb[2] + dc[2];
            f0 += yb[3] * rsqrt(dx * dx + dy * dy + dz * dz);
        }
        s0 += xa[3] * f0;
    }
    scatter_scalar<T, PK>(m, q, Z, N, x, y, s0 * cx<T>{T(q.img_ph[2 * k]), T(q.img_ph[2 * k + 1])});
}

// Touching face entries: the static integral, both integration orders averaged,
// summed over the degree-5 points (phase-free, FP64, request independent).  One
// launch per order, so that the lanes of a warp integrate over the same kind of
// element: OX: the outer points are those of x, else of y (then added to the
// first order's sum); 16 lanes per entry for a tetrahedron's 14 points, 8 for a
// face's 7.
template <int PK, bool OX>
__global__ void __launch_bounds__(128) k_touch_scalar(DevMesh m, const TetGeom *tet, const TriGeom *tri,
                                                      const NearEntry *list, int n, double *out) {
    constexpr bool XT = PKTraits<PK>::xtet, YT = PKTraits<PK>::ytet;
    constexpr bool OT = OX ? XT : YT, ST = OX ? YT : XT;   // outer and source element are tetrahedra
    constexpr int G = OT ? 16 : 8, NP = OT ? 14 : 7;
    const int e = (blockIdx.x * blockDim.x + threadIdx.x) / G, q = threadIdx.x % G;
    double acc = 0;
    if (e < n && q < NP) {
        const NearEntry en = list[e];
        const int xf = XT ? en.x : m.hf[en.x], yf = en.y, k = en.k;
        const int o = OX ? xf : yf, s = OX ? yf : xf;
        const double sg = OX ? -1.0 : 1.0;   // the source's image as the outer element sees it
        const double R[3] = {sg * (k / 3 - 1) * m.a, sg * (k % 3 - 1) * m.b, 0.0};
        const double *r5 = (OT ? m.q5 + (size_t)o * 42 : m.f5 + (size_t)o * 21) + 3 * q;
        const double w = OT ? m.vol[o] * c_w5tet[q] : m.farea[o] * c_w5tri[q];
        const double *v = ST ? m.tv + 12 * (size_t)s : m.fv + 9 * (size_t)s;
        double rel[ST ? 12 : 9];
        for (int j = 0; j < (ST ? 4 : 3); ++j)
            for (int d = 0; d < 3; ++d) rel[3 * j + d] = (v[3 * j + d] + R[d]) - r5[d];
        double I;
        if constexpr (ST) tet_integrals<false>(tet[s], rel, I, nullptr);
        else I = tri_inv(tri[s], rel);
        acc = 0.5 * w * I;
    }
    for (int h = G / 2; h > 0; h >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, h, G);
    if (e < n && q == 0) out[e] = OX ? acc : out[e] + acc;
}

// scatter the cached static integral of every touching face entry with the
// request's image phase exp(j k_par.R)/(4 pi)
template <typename T, int PK>
__global__ void __launch_bounds__(128) k_touch_apply(DevMesh m, const __grid_constant__ DevReq q, T *Z, size_t N,
                                                     const NearEntry *list, const double *sc, int n) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const NearEntry en = list[e];
    const double v = sc[e];
    scatter_scalar<T, PK>(m, q, Z, N, en.x, en.y,
                          cx<T>{T(v * q.img_ph[2 * en.k]), T(v * q.img_ph[2 * en.k + 1])});
}

// ---------------------------------------------------------------------------
// local (Gram) term and right-hand side, per tetrahedron
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_gram(DevMesh m, const __grid_constant__ DevReq q, T *Z, size_t N) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m.nt) return;
    const double *P = m.tv + 12 * (size_t)t;
    const double *c = m.cen + 3 * (size_t)t;
    double d[4][3], sq = 0;
    for (int i = 0; i < 4; ++i)
        for (int k = 0; k < 3; ++k) {
            d[i][k] = P[3 * i + k] - c[k];
            sq += d[i][k] * d[i][k];
        }
    const double V = m.vol[t];
    cx<double> ie = ld2(q.ieps + 2 * t);
    for (int i = 0; i < 4; ++i) {
        cx<double> wti = ld2(q.wt + 2 * (4 * t + i));
        for (int j = 0; j < 4; ++j) {
            cx<double> wsj = cconj(ld2(q.wt + 2 * (4 * t + j)));
            double G = V * (sq / 20.0 + d[i][0] * d[j][0] + d[i][1] * d[j][1] + d[i][2] * d[j][2]);
            cx<double> val = (q.coef[4 * t + i] * q.coef[4 * t + j] * G) * ((wti * wsj) * ie);
            atomic_add_c<T>(Z, (size_t)q.row[4 * t + i] * N + q.row[4 * t + j], cx<T>{T(val.re), T(val.im)});
        }
    }
}

__global__ void k_rhs(DevMesh m, const __grid_constant__ DevReq q, double *b) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= m.nt) return;
    const double *P = m.tv + 12 * (size_t)t;
    const double *c = m.cen + 3 * (size_t)t;
    const double V = m.vol[t];
    for (int pol = 0; pol < 2; ++pol) {
        const double *pv = q.pol + 3 * pol;
        cx<double> s0 = {0, 0}, s1 = {0, 0};   // sum w e^{..}, sum w ((x-c).p) e^{..}
        for (int k = 0; k < 14; ++k) {
            const double *x = m.q5 + (size_t)t * 42 + 3 * k;
            double ph = -(q.kinc[0] * x[0] + q.kinc[1] * x[1] + q.kinc[2] * x[2]);
            double sn, cs;
            sincos(ph, &sn, &cs);
            double w = V * c_w5tet[k];
            double xp = (x[0] - c[0]) * pv[0] + (x[1] - c[1]) * pv[1] + (x[2] - c[2]) * pv[2];
            s0.re += w * cs; s0.im += w * sn;
            s1.re += w * xp * cs; s1.im += w * xp * sn;
        }
        for (int i = 0; i < 4; ++i) {
            double vp = (P[3 * i] - c[0]) * pv[0] + (P[3 * i + 1] - c[1]) * pv[1] + (P[3 * i + 2] - c[2]) * pv[2];
            cx<double> integ = {s1.re - vp * s0.re, s1.im - vp * s0.im};
            cx<double> val = q.coef[4 * t + i] * (ld2(q.wt + 2 * (4 * t + i)) * integ);
            size_t r = (size_t)q.row[4 * t + i];
            atomicAdd(b + 4 * r + 2 * pol, val.re);
            atomicAdd(b + 4 * r + 2 * pol + 1, val.im);
        }
    }
}

// ---------------------------------------------------------------------------
// checks of the special functions
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_erfcx(const double *u, double *out, int n) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    cx<T> r = erfcx_c<T>(cx<T>{T(u[2 * i]), T(u[2 * i + 1])});
    out[2 * i] = double(r.re);
    out[2 * i + 1] = double(r.im);
}

template <typename T, bool SYM = false>
__global__ void k_green(const double *d, double *out, int n, const float *stab, const float2 *ztab,
                        const EwaldTables *ew, const __grid_constant__ EwaldF32 ef) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    cx<T> r = Green<T>::template eval<SYM>(T(d[3 * i]), T(d[3 * i + 1]), T(d[3 * i + 2]), 0u, stab, ztab, ew, ef);
    out[2 * i] = double(r.re);
    out[2 * i + 1] = double(r.im);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
template <typename T, int PK>
cudaError_t far_scalar(bool sym, dim3 grid, size_t sm, cudaStream_t st, const DevMesh &m, const DevReq &q, T *Z, size_t N,
                       int nx, int ny, const uint16_t *mk) {
    if constexpr (sizeof(T) == 4) {
        if (q.fp.mode != FAR_NONE) return launch_far_scalar(PK, m, q, Z, N, st);
        if (sym) k_far_scalar<T, PK, true><<<grid, 128, sm, st>>>(m, q, Z, N, nx, ny, mk);
        else k_far_scalar<T, PK, false><<<grid, 128, sm, st>>>(m, q, Z, N, nx, ny, mk);
    } else {
        if (q.f64.n_blob > 0) return launch_far64_scalar(PK, m, q, Z, N, st);
        k_far_scalar<T, PK, false><<<grid, 128, sm, st>>>(m, q, Z, N, nx, ny, mk);
    }
    ++g_launches;
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_fill(const DevMesh &m, const DevReq &q, T *Z, size_t ld, double *b, cudaStream_t st,
                        cudaEvent_t far0, cudaEvent_t far1) {
    // Z: N rows of ld complex entries (row stride ld >= N), domain-blocked order
    const size_t N = ld;
    // the first error of any part (the launchers take theirs from the runtime and return it)
    cudaError_t err = cudaSuccess;
    auto part = [&](cudaError_t e) { if (err == cudaSuccess) err = e; };
    part(cudaMemsetAsync(Z, 0, sizeof(T) * 2 * ld * (size_t)m.N, st));
    if (b) part(cudaMemsetAsync(b, 0, sizeof(double) * 4 * (size_t)m.N, st));
    dim3 blk(128);
    k_gram<T><<<(m.nt + 127) / 128, blk, 0, st>>>(m, q, Z, N); ++g_launches;
    if (b) { k_rhs<<<(m.nt + 127) / 128, blk, 0, st>>>(m, q, b); ++g_launches; }
    part(cudaGetLastError());
    if (sizeof(T) == 4) part(launch_far_prep(m, q, st));   // element records of the FP32 kernels
    else if (q.f64.n_blob > 0) part(launch_far64_prep(m, q, st));
    const size_t sm = stab_bytes<T>();
    if (far0) cudaEventRecord(far0, st);
    const bool sym = sizeof(T) == 4 && q.ef.sym;   // normal incidence: the symmetric tabulated path
    if constexpr (sizeof(T) == 4) {
        const dim3 gtt((m.nt + 127) / 128, m.nt);
        if (q.fp.mode != FAR_NONE) {
            part(launch_far_tt(m, q, Z, N, st));
        } else {
            if (sym) k_far_tt<T, true><<<gtt, blk, sm, st>>>(m, q, Z, N);
            else k_far_tt<T, false><<<gtt, blk, sm, st>>>(m, q, Z, N);
            ++g_launches;
        }
    } else if (q.f64.n_blob > 0) {
        part(launch_far64_tt(m, q, Z, N, st));
    } else {
        k_far_tt<T, false><<<dim3((m.nt + 127) / 128, m.nt), blk, sm, st>>>(m, q, Z, N);
        ++g_launches;
    }
    part(cudaGetLastError());
    if (far1) cudaEventRecord(far1, st);
    auto grid1 = [](int n) { return (unsigned)((n + 127) / 128); };
    if (m.npr[0]) { k_pr_tt<T><<<grid1(m.npr[0]), blk, 0, st>>>(m, q, Z, N, m.pr[0], m.npr[0]); ++g_launches; }
    if (m.nto[0]) {
        k_touch_combine<T><<<grid1(m.nto[0]), blk, 0, st>>>(m, q, Z, N, m.to[0], m.touch_partner, m.touch_half,
                                                            m.nto[0]); ++g_launches;
    }
    if (m.nf) {
        part(far_scalar<T, PK_TF>(sym, dim3((m.nf + 127) / 128, m.nt), sm, st, m, q, Z, N, m.nt, m.nf, m.mk_tf));
        if (m.npr[1]) { k_pr_scalar<T, PK_TF><<<grid1(m.npr[1]), blk, 0, st>>>(m, q, Z, N, m.pr[1], m.npr[1]); ++g_launches; }
        if (m.nto[1]) { k_touch_apply<T, PK_TF><<<grid1(m.nto[1]), blk, 0, st>>>(m, q, Z, N, m.to[1], m.touch_sc[1], m.nto[1]); ++g_launches; }
    }
    if (m.nh) {
        part(far_scalar<T, PK_FT>(sym, dim3((m.nt + 127) / 128, m.nh), sm, st, m, q, Z, N, m.nh, m.nt, m.mk_ft));
        if (m.npr[2]) { k_pr_scalar<T, PK_FT><<<grid1(m.npr[2]), blk, 0, st>>>(m, q, Z, N, m.pr[2], m.npr[2]); ++g_launches; }
        if (m.nto[2]) { k_touch_apply<T, PK_FT><<<grid1(m.nto[2]), blk, 0, st>>>(m, q, Z, N, m.to[2], m.touch_sc[2], m.nto[2]); ++g_launches; }
        part(far_scalar<T, PK_FF>(sym, dim3((m.nf + 127) / 128, m.nh), sm, st, m, q, Z, N, m.nh, m.nf, m.mk_ff));
        if (m.npr[3]) { k_pr_scalar<T, PK_FF><<<grid1(m.npr[3]), blk, 0, st>>>(m, q, Z, N, m.pr[3], m.npr[3]); ++g_launches; }
        if (m.nto[3]) { k_touch_apply<T, PK_FF><<<grid1(m.nto[3]), blk, 0, st>>>(m, q, Z, N, m.to[3], m.touch_sc[3], m.nto[3]); ++g_launches; }
    }
    part(cudaGetLastError());
    return err;
}

size_t static_geom_bytes(size_t nt, size_t nf) { return sizeof(TetGeom) * nt + sizeof(TriGeom) * (nf + 1); }

cudaError_t launch_static_cache(const DevMesh &m, double *touch_half, double *const touch_sc[4], void *geom,
                                cudaStream_t st) {
    TetGeom *tet = static_cast<TetGeom *>(geom);
    TriGeom *tri = reinterpret_cast<TriGeom *>(tet + m.nt);
    const dim3 blk(128);
    auto grid = [](int n, int lanes) { return (unsigned)(((size_t)n * lanes + 127) / 128); };
    k_geom<<<(m.nt + m.nf + 127) / 128, blk, 0, st>>>(m, tet, tri); ++g_launches;
    if (m.nto[0]) { k_touch_half<<<grid(m.nto[0], 16), blk, 0, st>>>(m, tet, m.to[0], m.nto[0], touch_half); ++g_launches; }
    if (m.nto[1]) {
        k_touch_scalar<PK_TF, true><<<grid(m.nto[1], 16), blk, 0, st>>>(m, tet, tri, m.to[1], m.nto[1], touch_sc[1]); ++g_launches;
        k_touch_scalar<PK_TF, false><<<grid(m.nto[1], 8), blk, 0, st>>>(m, tet, tri, m.to[1], m.nto[1], touch_sc[1]); ++g_launches;
    }
    if (m.nto[2]) {
        k_touch_scalar<PK_FT, true><<<grid(m.nto[2], 8), blk, 0, st>>>(m, tet, tri, m.to[2], m.nto[2], touch_sc[2]); ++g_launches;
        k_touch_scalar<PK_FT, false><<<grid(m.nto[2], 16), blk, 0, st>>>(m, tet, tri, m.to[2], m.nto[2], touch_sc[2]); ++g_launches;
    }
    if (m.nto[3]) {
        k_touch_scalar<PK_FF, true><<<grid(m.nto[3], 8), blk, 0, st>>>(m, tet, tri, m.to[3], m.nto[3], touch_sc[3]); ++g_launches;
        k_touch_scalar<PK_FF, false><<<grid(m.nto[3], 8), blk, 0, st>>>(m, tet, tri, m.to[3], m.nto[3], touch_sc[3]); ++g_launches;
    }
    return cudaGetLastError();
}

template cudaError_t launch_fill<float>(const DevMesh &, const DevReq &, float *, size_t, double *, cudaStream_t,
                                        cudaEvent_t, cudaEvent_t);
template cudaError_t launch_fill<double>(const DevMesh &, const DevReq &, double *, size_t, double *, cudaStream_t,
                                         cudaEvent_t, cudaEvent_t);

cudaError_t launch_erfcx(const double *u, double *out, int n, bool fp64, cudaStream_t st) {
    if (fp64) { k_erfcx<double><<<(n + 127) / 128, 128, 0, st>>>(u, out, n); ++g_launches; }
    else { k_erfcx<float><<<(n + 127) / 128, 128, 0, st>>>(u, out, n); ++g_launches; }
    return cudaGetLastError();
}

cudaError_t launch_green(const double *d, double *out, int n, bool fp64, const float *stab, const float2 *ztab,
                         const EwaldTables *ew, const EwaldF32 &ef, cudaStream_t st) {
    if (fp64) { k_green<double><<<(n + 127) / 128, 128, 0, st>>>(d, out, n, stab, ztab, ew, ef); ++g_launches; }
    else if (ef.sym) { k_green<float, true><<<(n + 127) / 128, 128, 0, st>>>(d, out, n, stab, ztab, ew, ef); ++g_launches; }
    else { k_green<float><<<(n + 127) / 128, 128, 0, st>>>(d, out, n, stab, ztab, ew, ef); ++g_launches; }
    return cudaGetLastError();
}

}  // namespace vie

// ===========================================================================
// Allocation-free evaluation of the periodic Green's function.
//
// Some callers cannot allocate device memory while they run: a host framework
// that reserves all of HBM up front through its own pool and forbids
// cudaMalloc/cudaFree afterwards (a long-running serving process, for
// example), or code that must not let an allocation synchronise the device.
// vie_green_noalloc serves them: the caller passes device buffers for the
// inputs and outputs, and the only scratch -- the FP32 interpolation tables of
// the Ewald series -- lives in the file-scope array below, which every GPU
// that loads this library holds until the process exits.
// ===========================================================================
#include <mutex>
#include <vector>

#include "../../include/vie.h"

namespace vie {


constexpr int NOALLOC_MAX_TAB = 96;   // distinct Floquet decay constants the scratch can hold
// whole 16-byte units: the spatial table after it is read with 16-byte loads
constexpr size_t NOALLOC_EW_FLOAT2 = (sizeof(EwaldTables) + 15) / 16 * 2;
constexpr size_t NOALLOC_FLOAT2 = NOALLOC_EW_FLOAT2 + 2 * NSPAT + (size_t)NOALLOC_MAX_TAB * NZTAB * 4;
// Ewald parameter block (~49 KB), spatial table (4*NSPAT floats), spectral tables
// (float2): about 0.85 MB in total
static __device__ __align__(256) float2 g_noalloc_scratch[NOALLOC_FLOAT2];

namespace {

constexpr int NOALLOC_MAX_DEVICES = 64;
std::mutex g_noalloc_mu;                                   // guards the per-device set-up below
float2 *g_scratch_ptr[NOALLOC_MAX_DEVICES] = {};           // device address of the array, per device

}  // namespace
}  // namespace vie

extern "C" int vie_green_noalloc(double lambda_nm, double theta, double phi, double period_a, double period_b,
                                 double z_extent, const double *d_dev, double *out_dev, int32_t n,
                                 int32_t precision, void *stream) {
    using namespace vie;
    if (n < 0 || (n > 0 && (!d_dev || !out_dev))) return VIE_EINVAL;
    if (!(lambda_nm > 0) || !(period_a > 0) || !(period_b > 0) || !(std::fabs(theta) < M_PI / 2) ||
        !(z_extent >= 0) || !std::isfinite(lambda_nm + period_a + period_b + z_extent))
        return VIE_EINVAL;
    if (precision != VIE_FP64 && precision != VIE_FP32) return VIE_EINVAL;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES) return VIE_ECUDA;
    float2 *base = nullptr;
    {
        // one-time set-up per device, with the device current, under one lock
        // across threads: the library's constant tables (the same once-per-device
        // upload that vie_create does, so a device whose solves are running is
        // never written again) and the device address of the scratch array
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        if (!g_scratch_ptr[dev]) {
            if (upload_device_constants(dev) != cudaSuccess) return VIE_ECUDA;
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return VIE_ECUDA;
            g_scratch_ptr[dev] = static_cast<float2 *>(p);
        }
        base = g_scratch_ptr[dev];
    }
    if (n == 0) return VIE_OK;
    static thread_local EwaldTables tabs;
    const double k0 = 2.0 * M_PI / lambda_nm;
    const char *why = "";
    const int rc = build_ewald_tables(period_a, period_b, k0, k0 * std::sin(theta) * std::cos(phi),
                                      k0 * std::sin(theta) * std::sin(phi), z_extent, precision == VIE_FP64, tabs,
                                      nullptr, &why, 0.0, false);   // results leave in FP64: the finest spacing
    if (rc != VIE_OK) return rc;
    if (precision == VIE_FP32 && tabs.n_tab > NOALLOC_MAX_TAB) return VIE_EINVAL;   // scratch too small
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    EwaldTables *ewd = reinterpret_cast<EwaldTables *>(base);
    if (upload_ewald(ewd, tabs, st) != cudaSuccess) return VIE_ECUDA;
    float *stab = reinterpret_cast<float *>(base + NOALLOC_EW_FLOAT2);
    float2 *ztab = base + NOALLOC_EW_FLOAT2 + 2 * NSPAT;
    if (precision == VIE_FP32 && launch_build_tables(ewd, stab, ztab, tabs.n_tab, st) != cudaSuccess) return VIE_ECUDA;
    if (launch_green(d_dev, out_dev, n, precision == VIE_FP64, stab, ztab, ewd, make_ewald_f32(tabs, false), st) !=
        cudaSuccess)
        return VIE_ECUDA;
    return VIE_OK;
}
