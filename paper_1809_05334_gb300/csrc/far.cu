// Far element pairs of the FP32 fill in the polynomial form (far_poly.cuh):
// tetrahedron pairs, pairs with charge-carrying faces, the per-request element
// records they read, and g_p at single displacements for the parity entry point.
#include <cuda_runtime.h>

#include "far_poly.cuh"

namespace vie {

// CTAs per SM of the tetrahedron-pair kernels (bench cell, 21,024 unknowns; compared
// before the image cut and the scatter took their present form): at normal incidence
// and in the fold 128 registers and four CTAs (18.4 / 24.9 ms; three 18.5 / 26.8,
// five 18.5 / 27.1, spilling); the full rectangle keeps the complex columns of four
// test points in 168 registers (31.9 ms; two points at a time in 128: 34.2)
#ifndef VIE_FAR_MINB
#define VIE_FAR_MINB 4
#endif
#ifndef VIE_FAR_MINB_FULL
#define VIE_FAR_MINB_FULL 3
#endif

// ---------------------------------------------------------------------------
// element records of one request
// ---------------------------------------------------------------------------
__device__ __forceinline__ void point_record(const EwaldF32 &ef, float4 *p, size_t n, const float *x, const float *c,
                                             float w) {
    p[(size_t)FPT_POS * n] = make_float4(ef.Eih * x[0], ef.Eih * x[1], ef.Eih * x[2], w);
    p[(size_t)FPT_REL * n] = make_float4(x[0] - c[0], x[1] - c[1], x[2] - c[2], 0.f);
    const float ip = 0.31830988618f;
    float s0, c0, s1, c1, s2, c2, s3, c3;
    sincospif(ef.step_x * ip * x[0], &s2, &c2);
    sincospif(ef.step_y * ip * x[1], &s3, &c3);
    if (ef.sym) {
        p[(size_t)FPT_PH0 * n] = make_float4(c2, c3, s2, s3);
        return;
    }
    sincospif(ef.ob_kx0 * ip * x[0], &s0, &c0);
    sincospif(ef.ob_ky0 * ip * x[1], &s1, &c1);
    p[(size_t)FPT_PH0 * n] = make_float4(c0, s0, c1, s1);
    p[(size_t)FPT_PH1 * n] = make_float4(c2, s2, c3, s3);
}

__global__ void __launch_bounds__(128) k_far_prep(DevMesh m, const __grid_constant__ DevReq q) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    const EwaldF32 &ef = q.ef;
    if (e < m.nt) {
        const float *f = m.far<float>(e);
        float rad = 0.f;
        for (int a = 0; a < 4; ++a) {
            point_record(ef, q.ptet + (size_t)a * FPT * m.nt + e, m.nt, f + 3 * a, f + 12, f[27]);
            const float u[3] = {f[3 * a] - f[12], f[3 * a + 1] - f[13], f[3 * a + 2] - f[14]};
            rad = fmaxf(rad, sqrtf(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]));
        }
        float4 *o = q.etet + e;
        const size_t n = m.nt;
        const double *c = q.coef + 4 * (size_t)e, *w = q.wt + 8 * (size_t)e;
        const int32_t *r = q.row + 4 * (size_t)e;
        o[FEL_CEN * n] = make_float4(ef.Eih * f[12], ef.Eih * f[13], ef.Eih * f[14], ef.Eih * rad);
        o[FEL_COEF * n] = make_float4(float(c[0]), float(c[1]), float(c[2]), float(c[3]));
        o[FEL_W01 * n] = make_float4(float(w[0]), float(w[1]), float(w[2]), float(w[3]));
        o[FEL_W23 * n] = make_float4(float(w[4]), float(w[5]), float(w[6]), float(w[7]));
        o[FEL_KAP * n] = make_float4(float(q.kap[2 * e]), float(q.kap[2 * e + 1]), 0.f, 0.f);
        o[FEL_VX * n] = make_float4(f[15], f[18], f[21], f[24]);
        o[FEL_VY * n] = make_float4(f[16], f[19], f[22], f[25]);
        o[FEL_VZ * n] = make_float4(f[17], f[20], f[23], f[26]);
        o[FEL_ROW * n] = make_float4(__int_as_float(r[0]), __int_as_float(r[1]), __int_as_float(r[2]), __int_as_float(r[3]));
    }
    const int fi = e - m.nt;
    if (fi >= 0 && fi < m.nf) {
        const float *f = m.ffar<float>(fi);
        float c[3], rad = 0.f;
        for (int d = 0; d < 3; ++d) c[d] = (f[d] + f[3 + d] + f[6 + d]) / 3.f;
        for (int a = 0; a < 3; ++a) {
            point_record(ef, q.pface + (size_t)a * FPT * m.nf + fi, m.nf, f + 3 * a, c, f[9]);
            const float u[3] = {f[3 * a] - c[0], f[3 * a + 1] - c[1], f[3 * a + 2] - c[2]};
            rad = fmaxf(rad, sqrtf(u[0] * u[0] + u[1] * u[1] + u[2] * u[2]));
        }
        q.eface[fi] = make_float4(ef.Eih * c[0], ef.Eih * c[1], ef.Eih * c[2], ef.Eih * rad);
        q.eface[(size_t)m.nf + fi] = make_float4(float(q.qs[2 * fi]), float(q.qs[2 * fi + 1]), __int_as_float(q.frow[fi]), 0.f);
    }
}

// ---------------------------------------------------------------------------
// Tetrahedron pairs: one thread per unordered pair {t, s}, s >= t, both ordered
// blocks from the same 16 evaluations.  Four test points against one source
// point per step: they share the coefficient and image loads, and the moments
// factor (sums over the test points first).  Bound by L1: the gathers of the
// spatial table, 83% busy, 56% of the issue slots (9,882 unknowns, normal incidence).
// Measured (ms, far tetrahedron pairs; per-lane spectral table entries, single
// points and scalar atomics before): 21,024 unknowns 37.3 -> 19.8 at normal
// incidence, 59.3 -> 28.7 in the fold, 82.6 -> 35.1 full rectangle (26.6 and 33.7 with
// the charge term in single roundings, far_poly.cuh); 48,678
// unknowns 223 -> 98.
// ---------------------------------------------------------------------------
template <int MODE, int NQ>
__global__ void __launch_bounds__(FAR_THREADS, MODE == FAR_FULL ? VIE_FAR_MINB_FULL : VIE_FAR_MINB)
    k_far_tt_p(DevMesh m, const __grid_constant__ DevReq q, float *Z, size_t N) {
    __shared__ FarShared S;
    extern __shared__ __align__(16) p2 s_coef[];
    const int t = blockIdx.y;
    if ((int)(blockIdx.x * blockDim.x + blockDim.x) <= t) return;   // the whole block is below the diagonal
    const EwaldF32 &ef = q.ef;
    far_stage<MODE, NQ>(q, S, s_coef);
    far_stage_points<MODE, 4>(q.ptet, m.nt, t, S);
    const int s0 = blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = s0 < m.nt && s0 >= t;   // lanes off the pair range stay until the warp's masks are formed
    const int s = live ? s0 : t;
    const unsigned sub = live ? (unsigned)m.mk_tt[(size_t)t * m.nt + s] : 0u;
    __syncthreads();
    const unsigned long long regm = far_regular(ef, sub);
    unsigned long long regany = 0ull;
    if (__any_sync(0xffffffffu, regm != 0ull))
        regany = (unsigned long long)__reduce_or_sync(0xffffffffu, (unsigned)regm) |
                 ((unsigned long long)__reduce_or_sync(0xffffffffu, (unsigned)(regm >> 32)) << 32);
    const int n_list = far_images(ef, S, q.etet[t], q.etet[s], live, regany);
    if (!live) return;
    Mom<float> mo, mc;
    mo.zero();
    mc.zero();
    constexpr int NP = 2;   // both pairs of test points at once
    const size_t nt = m.nt;
    float ws = 0.f;
    // oblique incidence: S and T as 16 times their first value plus the sum of the differences
    float ref[4] = {0.f, 0.f, 0.f, 0.f}, dif[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
    for (int b = 0; b < 4; ++b) {
        const float4 *p = q.ptet + (size_t)b * FPT * nt + s;
        const float4 yb = p[FPT_POS * nt], rb = p[FPT_REL * nt], pb = p[FPT_PH0 * nt];
        const float4 sb = MODE == FAR_NORMAL ? make_float4(0.f, 0.f, 0.f, 0.f) : p[FPT_PH1 * nt];
        ws = yb.w;
        // sums over the test points: of g, and of r_a g (T: the same of the correction)
        cx<float> s0c = {0.f, 0.f}, sA[3], t0 = {0.f, 0.f}, tA[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) sA[d] = tA[d] = {0.f, 0.f};
        {
            constexpr int h0 = 0;
            p2 gre[NP], gim[NP], tre[NP], tim[NP];
            far_eval<MODE, NQ, NP>(S, s_coef, q, h0, yb, pb, sb, n_list, regm, regany, gre, gim, tre, tim);
            auto sums = [&](const p2 (&re)[NP], const p2 (&im)[NP], cx<float> &z0, cx<float> (&zA)[3]) {
                p2 ar = re[0], ai = im[0];
#pragma unroll
                for (int h = 1; h < NP; ++h) { ar = add2(ar, re[h]); ai = add2(ai, im[h]); }
                z0.re += hsum(ar);
                z0.im += hsum(ai);
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    p2 xr = mul2(S.pt[h0][SP_R + d], re[0]), xi = mul2(S.pt[h0][SP_R + d], im[0]);
#pragma unroll
                    for (int h = 1; h < NP; ++h) {
                        xr = fma2(S.pt[h0 + h][SP_R + d], re[h], xr);
                        xi = fma2(S.pt[h0 + h][SP_R + d], im[h], xi);
                    }
                    zA[d].re += hsum(xr);
                    zA[d].im += hsum(xi);
                }
            };
            sums(gre, gim, s0c, sA);
            if constexpr (MODE != FAR_NORMAL) {
                sums(tre, tim, t0, tA);
                auto differences = [&](const p2 (&v)[NP], float &r, float &d) {
                    if (b == 0) r = upk(v[0]).x;
                    const p2 nr = dup(-r);
                    d += hsum(add2(add2(v[0], nr), add2(v[1], nr)));
                };
                differences(gre, ref[0], dif[0]);
                differences(gim, ref[1], dif[1]);
                differences(tre, ref[2], dif[2]);
                differences(tim, ref[3], dif[3]);
            }
        }
        const float r[3] = {rb.x, rb.y, rb.z};
        auto add = [&](Mom<float> &M, cx<float> z0, const cx<float> (&zA)[3]) {
            M.S = M.S + z0;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                M.A[d] = M.A[d] + zA[d];
                cfma(M.B[d], r[d], z0);
                cfma(M.C, r[d], zA[d]);
            }
        };
        add(mo, s0c, sA);
        if constexpr (MODE != FAR_NORMAL) add(mc, t0, tA);
    }
    const float wt = q.ptet[(size_t)FPT_POS * nt + t].w, wgt = wt * ws;
    const TetRec rt = load_tet_rec(q.etet, m.nt, t), rs = load_tet_rec(q.etet, m.nt, s);
    const float k2 = float(q.k0 * q.k0);
    if constexpr (MODE == FAR_NORMAL) {
        mo.S = wgt * mo.S;
        mo.C = wgt * mo.C;
#pragma unroll
        for (int d = 0; d < 3; ++d) { mo.A[d] = wgt * mo.A[d]; mo.B[d] = wgt * mo.B[d]; }
        const float w16 = 16.f * wgt;
        scatter_rec<true>(Z, N, k2, rt, rs, mo, {fmaf(w16, q.fp.k_re, mo.S.re), fmaf(w16, q.fp.k_im, mo.S.im)}, s != t);
    } else {
        // g_p(-d) = conj(g_p(d)) + 2 j conj(T): the reversed pair's moments, A and B exchanged
        auto rev = [&](cx<float> g, cx<float> c) { return cx<float>{wgt * fmaf(2.f, c.im, g.re), wgt * fmaf(2.f, c.re, -g.im)}; };
        Mom<float> mr;
        mr.S = rev(mo.S, mc.S);
        mr.C = rev(mo.C, mc.C);
#pragma unroll
        for (int d = 0; d < 3; ++d) { mr.A[d] = rev(mo.B[d], mc.B[d]); mr.B[d] = rev(mo.A[d], mc.A[d]); }
        mo.S = wgt * mo.S;
        mo.C = wgt * mo.C;
#pragma unroll
        for (int d = 0; d < 3; ++d) { mo.A[d] = wgt * mo.A[d]; mo.B[d] = wgt * mo.B[d]; }
        const W2 sr = {16.f * ref[0], dif[0]}, si = {16.f * ref[1], dif[1]}, tr = {32.f * ref[2], 2.f * dif[2]},
                 ti = {32.f * ref[3], 2.f * dif[3]};   // T twice
        scatter_w2(Z, N, k2, rt, rs, mo, charge_base({sr, si}, rs.kap, wt, ws, 9.f));
        if (s != t) scatter_w2(Z, N, k2, rs, rt, mr, charge_base({w2_add(sr, ti), w2_add(tr, {-si.h, -si.l})}, rt.kap, wt, ws, 9.f));
    }
}

// ---------------------------------------------------------------------------
// pairs with charge faces: one thread per (x, y), x = blockIdx.y
//   PK 0: test tetrahedron x, source charge face y   -> Z[row(x,i), frow(y)] += 3 c_i w_i qs_y S
//   PK 1: test half face x, source tetrahedron y     -> Z[frow(x), row(y,j)] -= 3 c_j conj(w_j) kappa_y S
//   PK 2: test half face x, source charge face y     -> Z[frow(x), frow(y)] -= qs_y S
// ---------------------------------------------------------------------------
template <int MODE, int NQ, int PK>
__global__ void __launch_bounds__(FAR_THREADS) k_far_scalar_p(DevMesh m, const __grid_constant__ DevReq q, float *Z,
                                                              size_t N, int ny, const uint16_t *mk) {
    __shared__ FarShared S;
    extern __shared__ __align__(16) p2 s_coef[];
    constexpr bool XT = PK == 0, YT = PK == 1;
    constexpr int qx = XT ? 4 : 3, qy = YT ? 4 : 3;
    const EwaldF32 &ef = q.ef;
    const int x = blockIdx.y;
    const int xe = XT ? x : m.hf[x];   // a test face is addressed by its half-function index
    far_stage<MODE, NQ>(q, S, s_coef);
    far_stage_points<MODE, qx>(XT ? q.ptet : q.pface, XT ? m.nt : m.nf, xe, S);
    const int y0 = blockIdx.x * blockDim.x + threadIdx.x;
    const bool live = y0 < ny;
    const int y = live ? y0 : ny - 1;
    const unsigned sub = live ? (unsigned)mk[(size_t)x * ny + y] : 0u;
    __syncthreads();
    const float4 *ex = XT ? q.etet : q.eface, *ey = YT ? q.etet : q.eface;
    const unsigned long long regm = far_regular(ef, sub);
    unsigned long long regany = 0ull;
    if (__any_sync(0xffffffffu, regm != 0ull))
        regany = (unsigned long long)__reduce_or_sync(0xffffffffu, (unsigned)regm) |
                 ((unsigned long long)__reduce_or_sync(0xffffffffu, (unsigned)(regm >> 32)) << 32);
    const int n_list = far_images(ef, S, ex[xe], ey[y], live, regany);
    if (!live) return;
    constexpr int NP = 2;   // both pairs of test points at once
    const size_t n = YT ? m.nt : m.nf;
    const float4 *py = (YT ? q.ptet : q.pface) + y;
    cx<float> Sm = {0.f, 0.f};
    float wy = 0.f, ref[2] = {0.f, 0.f}, dif[2] = {0.f, 0.f};   // oblique incidence: as k_far_tt_p
#pragma unroll 1
    for (int b = 0; b < qy; ++b) {
        const float4 *p = py + (size_t)b * FPT * n;
        const float4 yb = p[FPT_POS * n], pb = p[FPT_PH0 * n];
        const float4 sb = MODE == FAR_NORMAL ? make_float4(0.f, 0.f, 0.f, 0.f) : p[FPT_PH1 * n];
        wy = yb.w;
        {
            constexpr int h0 = 0;
            p2 gre[NP], gim[NP], tre[NP], tim[NP];
            far_eval<MODE, NQ, NP>(S, s_coef, q, h0, yb, pb, sb, n_list, regm, regany, gre, gim, tre, tim);
#pragma unroll
            for (int h = 0; h < NP; ++h) {
                const float2 re = upk(gre[h]), im = upk(gim[h]);
                const bool both = qx == 4 || h0 + h == 0;   // a face has no fourth point
                if (MODE == FAR_NORMAL) {
                    Sm.re += both ? re.x + re.y : re.x;
                    Sm.im += both ? im.x + im.y : im.x;
                } else {
                    if (b == 0 && h == 0) { ref[0] = re.x; ref[1] = im.x; }
                    dif[0] += both ? (re.x - ref[0]) + (re.y - ref[0]) : re.x - ref[0];
                    dif[1] += both ? (im.x - ref[1]) + (im.y - ref[1]) : im.x - ref[1];
                }
            }
        }
    }
    const float wx = (XT ? q.ptet : q.pface)[(XT ? (size_t)FPT_POS * m.nt : (size_t)FPT_POS * m.nf) + xe].w;
    // S times the weights and c: at normal incidence Sm, else both parts of the value
    const float c = PK == 0 ? 3.f : (PK == 1 ? -3.f : -1.f);
    const float np = float(qx * qy);   // 9, 12: np ref is rounded, the rest of it goes with the differences
    auto two = [&](int k) { const float h = np * ref[k]; return W2{h, fmaf(np, ref[k], -h) + dif[k]}; };
    auto base = [&](cx<float> f) -> CW2 {
        if (MODE == FAR_NORMAL) {
            const cx<float> v = f * ((wx * wy) * Sm);
            return {{c * v.re, 0.f}, {c * v.im, 0.f}};
        }
        return charge_base({two(0), two(1)}, f, wx, wy, c);
    };
    auto times = [](CW2 v, float f) { return CW2{w2_mul(v.re, f), w2_mul(v.im, f)}; };
    const cx<float> none = {0.f, 0.f};
    if constexpr (PK == 0) {
        const float4 fr = q.eface[(size_t)m.nf + y];
        const TetRec r = load_tet_rec(q.etet, m.nt, x);
        const CW2 qS = base({fr.x, fr.y});
        const size_t col = (size_t)__float_as_int(fr.z);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const cx<float> v = charge_value(times(qS, r.coef[i]), r.w[i], none);
            red_c(Z, (size_t)r.row[i] * N + col, v.re, v.im);
        }
    } else if constexpr (PK == 1) {
        const size_t row = (size_t)__float_as_int(q.eface[(size_t)m.nf + xe].z);
        const TetRec r = load_tet_rec(q.etet, m.nt, y);
        const CW2 kS = base(r.kap);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const cx<float> v = charge_value(times(kS, r.coef[j]), cconj(r.w[j]), none);
            red_c(Z, row * N + (size_t)r.row[j], v.re, v.im);
        }
    } else {
        const size_t row = (size_t)__float_as_int(q.eface[(size_t)m.nf + xe].z);
        const float4 fr = q.eface[(size_t)m.nf + y];
        const cx<float> v = charge_value(base({fr.x, fr.y}), {1.f, 0.f}, none);
        red_c(Z, row * N + (size_t)__float_as_int(fr.z), v.re, v.im);
    }
}

// g_p at single displacements: the displacement as the test point, the source
// at the origin, every image visited
template <int MODE, int NQ>
__global__ void __launch_bounds__(FAR_THREADS) k_green_p(const double *d, double *out, int n,
                                                         const __grid_constant__ DevReq q) {
    __shared__ FarShared S;
    extern __shared__ __align__(16) p2 s_coef[];
    const EwaldF32 &ef = q.ef;
    far_stage<MODE, NQ>(q, S, s_coef);
    if (threadIdx.x < 2 * 14) (&S.pt[0][0])[threadIdx.x] = 0ull;
    __syncthreads();
    if (threadIdx.x < 2) {   // test points at the origin: unit phases
        p2 *P = &S.pt[threadIdx.x][SP_P];
        if (MODE == FAR_NORMAL) { P[0] = P[1] = dup(2.f); }
        else { P[0] = P[2] = P[4] = P[6] = dup(1.f); }
    }
    __syncthreads();
    // every image, in every warp's list
    for (int k = threadIdx.x & 31; k <= ef.n_img; k += 32) {
        float4 *l = &S.list[threadIdx.x >> 5][2 * k];
        l[0] = k < ef.n_img ? S.img[2 * k] : make_float4(1e15f, 1e15f, 1e15f, 1e15f);
        l[1] = k < ef.n_img ? S.img[2 * k + 1] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncwarp();
    const int n_list = (ef.n_img + 1) & ~1;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    // the source point at -d: x_a - y_b = d
    const float x[3] = {-float(d[3 * i]), -float(d[3 * i + 1]), -float(d[3 * i + 2])};
    float4 rec[FPT];
    const float zero[3] = {0.f, 0.f, 0.f};
    point_record(ef, rec, 1, x, zero, 1.f);
    p2 gre[1], gim[1], tre[1], tim[1];
    far_eval<MODE, NQ, 1>(S, s_coef, q, 0, rec[FPT_POS], rec[FPT_PH0], MODE == FAR_NORMAL ? rec[FPT_PH0] : rec[FPT_PH1],
                          n_list, 0ull, 0ull, gre, gim, tre, tim);
    out[2 * i] = double(upk(gre[0]).x + q.fp.k_re);
    out[2 * i + 1] = double(upk(gim[0]).x + q.fp.k_im);
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// f(mode, columns) for the request's form
template <typename F>
static cudaError_t far_dispatch(const FarPoly &fp, F &&f) {
    using std::integral_constant;
#define FAR_CASE(M, Q) if (fp.mode == M && fp.nq == Q) { f(integral_constant<int, M>{}, integral_constant<int, Q>{}); return cudaGetLastError(); }
    FAR_CASE(FAR_NORMAL, 3) FAR_CASE(FAR_NORMAL, 4) FAR_CASE(FAR_NORMAL, 5)
    FAR_CASE(FAR_FOLD, 3) FAR_CASE(FAR_FOLD, 4) FAR_CASE(FAR_FOLD, 5)
    FAR_CASE(FAR_FULL, 4) FAR_CASE(FAR_FULL, 5) FAR_CASE(FAR_FULL, 6) FAR_CASE(FAR_FULL, 8)
#undef FAR_CASE
    return cudaErrorInvalidValue;
}

cudaError_t launch_far_prep(const DevMesh &m, const DevReq &q, cudaStream_t st) {
    k_far_prep<<<(m.nt + m.nf + 127) / 128, 128, 0, st>>>(m, q); ++g_launches;
    return cudaGetLastError();
}

cudaError_t launch_far_tt(const DevMesh &m, const DevReq &q, float *Z, size_t N, cudaStream_t st) {
    const dim3 grid((m.nt + FAR_THREADS - 1) / FAR_THREADS, m.nt);
    ++g_launches;
    return far_dispatch(q.fp, [&](auto mode, auto nq) {
        k_far_tt_p<mode(), nq()><<<grid, FAR_THREADS, sizeof(p2) * q.fp.n_coef, st>>>(m, q, Z, N);
    });
}

cudaError_t launch_far_scalar(int pk, const DevMesh &m, const DevReq &q, float *Z, size_t N, cudaStream_t st) {
    const int nx = pk == 0 ? m.nt : m.nh, ny = pk == 1 ? m.nt : m.nf;
    const uint16_t *mk = pk == 0 ? m.mk_tf : (pk == 1 ? m.mk_ft : m.mk_ff);
    const dim3 grid((ny + FAR_THREADS - 1) / FAR_THREADS, nx);
    const size_t sm = sizeof(p2) * q.fp.n_coef;
    ++g_launches;
    return far_dispatch(q.fp, [&](auto mode, auto nq) {
        if (pk == 0) k_far_scalar_p<mode(), nq(), 0><<<grid, FAR_THREADS, sm, st>>>(m, q, Z, N, ny, mk);
        else if (pk == 1) k_far_scalar_p<mode(), nq(), 1><<<grid, FAR_THREADS, sm, st>>>(m, q, Z, N, ny, mk);
        else k_far_scalar_p<mode(), nq(), 2><<<grid, FAR_THREADS, sm, st>>>(m, q, Z, N, ny, mk);
    });
}

cudaError_t launch_green_poly(const double *d, double *out, int n, const DevReq &q, cudaStream_t st) {
    ++g_launches;
    return far_dispatch(q.fp, [&](auto mode, auto nq) {
        k_green_p<mode(), nq()><<<(n + FAR_THREADS - 1) / FAR_THREADS, FAR_THREADS, sizeof(p2) * q.fp.n_coef, st>>>(d, out, n, q);
    });
}

}  // namespace vie
