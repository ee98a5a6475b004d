// Far element pairs of the FP32 fill: the Ewald-summed g_p of Sec. 2.2 at the
// degree-2 product-rule points, four test points against one source point per
// step.
//
//   g_p(d) = sum_ij X_i Y_j G_ij(|z|) + sum_i ph_i F(R_i E) / R_i
//
// Spectral part: each order is a polynomial in t = 2 (z / z_max)^2 - 1
// (FarPoly, ewald_params.h) whose coefficients are the same for every lane, so
// they are shared-memory broadcasts and the whole sum is fused multiply-adds.
// The form with per-lane table entries that this replaces was bound by L1: 16
// gathers of 16 bytes per evaluation at ~11.5 wavefronts each.  The rows of
// orders are a run-time loop (small code: the unrolled rectangle missed the
// instruction cache), the columns unrolled.
// Spatial part: one cubic of F per image and lane from the table in shared
// memory, coordinates pre-scaled to table units (x = Eih d, Eih a power of two,
// so R is the table abscissa itself and nothing is rounded).  The image list is
// warp-uniform.
// Arithmetic on pairs of test points uses the packed FP32 instructions
// (fma.rn.f32x2): the kernels are bound by instruction issue.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "device_math.cuh"
#include "fill.h"

namespace vie {

// ---------------------------------------------------------------------------
// pairs of FP32 values
// ---------------------------------------------------------------------------
using p2 = unsigned long long;
__device__ __forceinline__ p2 pk(float a, float b) {
    p2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ p2 dup(float a) { return pk(a, a); }
__device__ __forceinline__ float2 upk(p2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ p2 fma2(p2 a, p2 b, p2 c) {
    p2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ p2 mul2(p2 a, p2 b) {
    p2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ p2 add2(p2 a, p2 b) {
    p2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ p2 add2_rm(p2 a, p2 b) {   // rounded towards minus infinity
    p2 r;
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float hsum(p2 v) {
    const float2 f = upk(v);
    return f.x + f.y;
}

// ---------------------------------------------------------------------------
// per-request element records (k_far_prep), structure of arrays: field f of
// element e at [f * n + e]
// ---------------------------------------------------------------------------
// point records: field (point * FPT + k)
constexpr int FPT_POS = 0;    // Eih x, Eih y, Eih z, rule weight
constexpr int FPT_REL = 1;    // position relative to the centroid (tetrahedra)
constexpr int FPT_PH0 = 2;    // normal: (cos, cos, sin, sin) of 2 pi (x/a, y/b); oblique: (cos, sin) of kx0 x, ky0 y
constexpr int FPT_PH1 = 3;    // oblique: (cos, sin) of 2 pi x/a, 2 pi y/b
constexpr int FPT = 4;
// element records
constexpr int FEL_CEN = 0;    // Eih times the centre of the points, Eih times their largest distance from it
constexpr int FEL_COEF = 1;   // tetrahedra: coefficient of the four local faces; faces: (qs.re, qs.im, row bits, 0)
constexpr int FEL_W01 = 2;    // test phases (re, im) of local faces 0, 1
constexpr int FEL_W23 = 3;
constexpr int FEL_KAP = 4;    // kappa (re, im)
constexpr int FEL_VX = 5;     // v_i - c of the four vertices, x, y, z
constexpr int FEL_VY = 6;
constexpr int FEL_VZ = 7;
constexpr int FEL_ROW = 8;    // matrix rows of the four local faces (bits)
constexpr int FEL_TET = 9;
constexpr int FEL_FACE = 2;

// ---------------------------------------------------------------------------
// shared state of a CTA
// ---------------------------------------------------------------------------
constexpr int FAR_THREADS = 128;
constexpr int FAR_MAX_IMG = 64;
struct FarShared {
    float4 tab[NSPAT + 1];          // cubic of F per interval; the last entry is zero (beyond the cut)
    float4 img[2 * FAR_MAX_IMG];    // (ox, ox, oy, oy) and (pr, pr, pi, pi) of every image
    float4 list[FAR_THREADS / 32][2 * (FAR_MAX_IMG + 1)];   // each warp's images, records as in img, an even number
    p2 pt[2][14];                   // the test element's points in pairs: x y z, rx ry rz, phases
};
// fields of FarShared::pt
constexpr int SP_X = 0, SP_R = 3, SP_P = 6;

template <int MODE, int NQ>
__device__ __forceinline__ void far_stage(const DevReq &q, FarShared &S, p2 *coef) {
    const EwaldF32 &ef = q.ef;
    const float4 *gtab = reinterpret_cast<const float4 *>(q.stab);
    for (int i = threadIdx.x; i <= NSPAT; i += blockDim.x)
        S.tab[i] = i < NSPAT ? gtab[i] : make_float4(0.f, 0.f, 0.f, 0.f);
    // order (0, 0) without its value at z = 0 (a rounding of this difference is a constant)
    constexpr int NS = (NQ + 1) & ~1;
    const int kr = q.fp.off[0] + q.fp.deg[0] * NS, ki = q.fp.im_deg[0] >= 0 ? q.fp.im_off[0] + q.fp.im_deg[0] * NS : -1;
    for (int i = threadIdx.x; i < q.fp.n_coef; i += blockDim.x)
        coef[i] = dup(MODE != FAR_NORMAL ? q.fcoef[i] : q.fcoef[i] - (i == kr ? q.fp.k_re : i == ki ? q.fp.k_im : 0.f));
    // F / R in table units: 1 / R = Eih / |x|, the factor goes into the image phases
    for (int i = threadIdx.x; i < ef.n_img; i += blockDim.x) {
        const float ox = ef.Eih * ef.img[i][0], oy = ef.Eih * ef.img[i][1];
        const float pr = ef.Eih * ef.img[i][2], pi = ef.Eih * ef.img[i][3];
        S.img[2 * i] = make_float4(ox, ox, oy, oy);
        S.img[2 * i + 1] = make_float4(pr, pr, pi, pi);
    }
}

// the test element's NPT points (4 or 3; a third point stands in for a missing fourth)
template <int MODE, int NPT>
__device__ __forceinline__ void far_stage_points(const float4 *__restrict__ pts, int n, int e, FarShared &S) {
    if (threadIdx.x < 4) {
        const int a = threadIdx.x, src = a < NPT ? a : NPT - 1;
        const float4 *p = pts + (size_t)src * FPT * n + e;
        const float4 x = p[(size_t)FPT_POS * n], r = p[(size_t)FPT_REL * n], c = p[(size_t)FPT_PH0 * n];
        float *o = reinterpret_cast<float *>(&S.pt[a >> 1][0]) + (a & 1);
        o[2 * (SP_X + 0)] = x.x; o[2 * (SP_X + 1)] = x.y; o[2 * (SP_X + 2)] = x.z;
        o[2 * (SP_R + 0)] = r.x; o[2 * (SP_R + 1)] = r.y; o[2 * (SP_R + 2)] = r.z;
        if (MODE == FAR_NORMAL) {
            o[2 * (SP_P + 0)] = 2.f * c.x; o[2 * (SP_P + 1)] = 2.f * c.y;
            o[2 * (SP_P + 2)] = 2.f * c.z; o[2 * (SP_P + 3)] = 2.f * c.w;
        } else {
            const float4 s = p[(size_t)FPT_PH1 * n];
            o[2 * (SP_P + 0)] = c.x; o[2 * (SP_P + 1)] = c.y; o[2 * (SP_P + 2)] = c.z; o[2 * (SP_P + 3)] = c.w;
            o[2 * (SP_P + 4)] = s.x; o[2 * (SP_P + 5)] = s.y; o[2 * (SP_P + 6)] = s.z; o[2 * (SP_P + 7)] = s.w;
        }
    }
}

// Images that can reach the cut from some point pair of the two elements (every
// point pair lies within ra + rb of the centre offset), the union over the warp;
// those in `out` (their static part is removed: a loop of their own) left out.
// Their records go to the warp's list, padded with one too far away to count to
// an even number; returns that number.
__device__ __forceinline__ int far_images(const EwaldF32 &ef, FarShared &S, float4 ca, float4 cb, bool live,
                                          unsigned long long out) {
    const float cx = ca.x - cb.x, cy = ca.y - cb.y, cz = ca.z - cb.z;
    // the table's cut (xs_max), in table units: the ring up to it from FP32_XCUT is 2e-8 an
    // image, all of one sign, which an ill-conditioned cell lifts to 2e-5 of its solution
    const float rc = (ef.xs_max * ef.xs_inv_h + ca.w + cb.w) * 1.0001f +
                     1e-6f * (fabsf(ca.x) + fabsf(ca.y) + fabsf(ca.z) + fabsf(cb.x) + fabsf(cb.y) + fabsf(cb.z));
    const float lim = live ? rc * rc - cz * cz : -1.f;
    const int n = ef.n_img, lane = threadIdx.x & 31;
    float4 *list = S.list[threadIdx.x >> 5];
    int count = 0;
    for (int i0 = 0; i0 < n; i0 += 32) {
        unsigned m = 0u;
        const int k = min(32, n - i0);
        for (int i = 0; i < k; ++i) {
            const float4 o = S.img[2 * (i0 + i)];
            const float x = cx + o.x, y = cy + o.z;
            if (fmaf(x, x, y * y) <= lim) m |= 1u << i;
        }
        m = __reduce_or_sync(0xffffffffu, m) & ~(unsigned)(out >> i0);
        if ((m >> lane) & 1u) {
            const int at = count + __popc(m & ((1u << lane) - 1u));
            list[2 * at] = S.img[2 * (i0 + lane)];
            list[2 * at + 1] = S.img[2 * (i0 + lane) + 1];
        }
        count += __popc(m);
    }
    if ((count & 1) && lane == 0) {
        list[2 * count] = make_float4(1e15f, 1e15f, 1e15f, 1e15f);
        list[2 * count + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncwarp();
    return (count + 1) & ~1;
}

// images whose static part is removed from this pair (9-bit mask over (m, n) in {-1, 0, 1}^2)
__device__ __forceinline__ unsigned long long far_regular(const EwaldF32 &ef, unsigned sub) {
    unsigned long long regm = 0ull;
    if (sub) {
#pragma unroll
        for (int k = 0; k < 9; ++k)
            if ((sub >> k) & 1u) regm |= 1ull << ef.near_img[k];
    }
    return regm;
}

// e^{-j th_a} conj(e^{-j th_b}) of a pair of test points and one source point
__device__ __forceinline__ void phase_diff2(p2 ca, p2 sa, p2 cb, p2 sb, p2 ncb, p2 &re, p2 &im) {
    re = fma2(ca, cb, mul2(sa, sb));
    im = fma2(ca, sb, mul2(sa, ncb));
}

// One source point against NP pairs of test points: gre + j gim = g_p(x_a - y_b);
// tre + j tim = sum over the propagating orders of X_i Y_j Im G_ij (the
// correction of the reversed pair at oblique incidence).
template <int MODE, int NQ, int NP>
__device__ __forceinline__ void far_eval(const FarShared &S, const p2 *__restrict__ coef, const DevReq &q, int h0,
                                         float4 yb, float4 pb, float4 sb, int n_list, unsigned long long regm,
                                         unsigned long long regany, p2 (&gre)[NP], p2 (&gim)[NP], p2 (&tre)[NP], p2 (&tim)[NP]) {
    const FarPoly &fp = q.fp;
    p2 dx[NP], dy[NP], dz[NP], t[NP];
    const p2 ny0 = dup(-yb.x), ny1 = dup(-yb.y), ny2 = dup(-yb.z);
    const p2 ts = dup(fp.t_scale), m1 = dup(-1.f);
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        dx[h] = add2(S.pt[h0 + h][SP_X + 0], ny0);
        dy[h] = add2(S.pt[h0 + h][SP_X + 1], ny1);
        dz[h] = add2(S.pt[h0 + h][SP_X + 2], ny2);
        dz[h] = mul2(dz[h], dz[h]);   // dz^2 from here on
        t[h] = fma2(dz[h], ts, m1);
    }
    // ---- spectral series ----
    p2 Yr[NQ][NP], Yi[NQ][NP];           // column weights (Yi: FAR_FULL only; NORMAL, FOLD: Yr[0] is 1)
    p2 Xr[NP], Xi[NP], Sxr[NP], Sxi[NP];   // row weight and its step (NORMAL: D_i, -D_{i-1}, D_1)
#pragma unroll
    for (int h = 0; h < NP; ++h) {
        const p2 *P = &S.pt[h0 + h][SP_P];
        if (MODE == FAR_NORMAL) {
            Xr[h] = fma2(P[0], dup(pb.x), mul2(P[2], dup(pb.z)));     // 2 cos 2 pi (x_a - y_b)/a
            Yr[1][h] = fma2(P[1], dup(pb.y), mul2(P[3], dup(pb.w)));
            Sxr[h] = Xr[h];
            Xi[h] = dup(-2.f);
        } else {
            phase_diff2(P[0], P[1], dup(pb.x), dup(pb.y), dup(-pb.x), Xr[h], Xi[h]);
            phase_diff2(P[4], P[5], dup(sb.x), dup(sb.y), dup(-sb.x), Sxr[h], Sxi[h]);
            if (MODE == FAR_FOLD) {
                const p2 c = fma2(P[6], dup(sb.z), mul2(P[7], dup(sb.w)));
                Yr[1][h] = add2(c, c);
            } else {
                p2 sr, si;
                phase_diff2(P[2], P[3], dup(pb.z), dup(pb.w), dup(-pb.z), Yr[0][h], Yi[0][h]);
                phase_diff2(P[6], P[7], dup(sb.z), dup(sb.w), dup(-sb.z), sr, si);
                const p2 nsi = mul2(si, m1);
#pragma unroll
                for (int j = 1; j < NQ; ++j) {
                    Yr[j][h] = fma2(Yr[j - 1][h], sr, mul2(Yi[j - 1][h], nsi));
                    Yi[j][h] = fma2(Yr[j - 1][h], si, mul2(Yi[j - 1][h], sr));
                }
            }
        }
        if (MODE != FAR_FULL) {
#pragma unroll
            for (int j = 2; j < NQ; ++j)
                Yr[j][h] = fma2(Yr[1][h], Yr[j - 1][h], j == 2 ? dup(-2.f) : mul2(Yr[j - 2][h], m1));
        }
    }
    // all columns of one row at t, highest power first
    constexpr int NS = (NQ + 1) & ~1;   // row stride of the coefficients: whole 16-byte loads
    auto row_poly = [&](int off, int deg, p2 (&g)[NQ][NP]) {
        const ulonglong2 *c = reinterpret_cast<const ulonglong2 *>(coef + off);
#pragma unroll
        for (int j = 0; j < NQ; ++j) {
            const ulonglong2 cc = c[j >> 1];
#pragma unroll
            for (int h = 0; h < NP; ++h) g[j][h] = j & 1 ? cc.y : cc.x;
        }
#pragma unroll 1
        for (int n = 0; n < deg; n += 2, c += NS)   // degrees are even
#pragma unroll
            for (int u = 1; u <= 2; ++u)
#pragma unroll
                for (int j = 0; j < NQ; ++j) {
                    const ulonglong2 cc = c[u * (NS / 2) + (j >> 1)];
#pragma unroll
                    for (int h = 0; h < NP; ++h) g[j][h] = fma2(g[j][h], t[h], j & 1 ? cc.y : cc.x);
                }
    };
#pragma unroll
    for (int h = 0; h < NP; ++h) gre[h] = gim[h] = tre[h] = tim[h] = 0ull;
    if constexpr (MODE == FAR_NORMAL) {
        // the (0, 0) order's imaginary part, the only one (row 0, column 0)
        if (fp.im_deg[0] >= 0) {
            const p2 *c = coef + fp.im_off[0];
#pragma unroll
            for (int h = 0; h < NP; ++h) gim[h] = c[0];
#pragma unroll 1
            for (int n = 0; n < fp.im_deg[0]; ++n) {
                c += NS;
#pragma unroll
                for (int h = 0; h < NP; ++h) gim[h] = fma2(gim[h], t[h], c[0]);
            }
        }
    }
#pragma unroll 1
    for (int i = 0; i < fp.rows; ++i) {
        p2 g[NQ][NP];
        row_poly(fp.off[i], fp.deg[i], g);
        if constexpr (MODE == FAR_NORMAL) {
#pragma unroll
            for (int h = 0; h < NP; ++h) {
                p2 r = g[0][h];
#pragma unroll
                for (int j = 1; j < NQ; ++j) r = fma2(Yr[j][h], g[j][h], r);
                if (i == 0) {
                    gre[h] = r;
                } else {   // D_i, then D_{i+1} = D_1 D_i - D_{i-1}
                    gre[h] = fma2(Xr[h], r, gre[h]);
                    const p2 nx = fma2(Sxr[h], Xr[h], Xi[h]);
                    Xi[h] = mul2(Xr[h], m1);
                    Xr[h] = nx;
                }
            }
        } else {
            const int imd = fp.im_deg[i];
#pragma unroll
            for (int part = 0; part < 2; ++part) {
                if (part == 1) {
                    if (imd < 0) break;
                    row_poly(fp.im_off[i], imd, g);
                }
#pragma unroll
                for (int h = 0; h < NP; ++h) {
                    p2 &ar = part ? tre[h] : gre[h], &ai = part ? tim[h] : gim[h];
                    if constexpr (MODE == FAR_FOLD) {
                        p2 r = g[0][h];
#pragma unroll
                        for (int j = 1; j < NQ; ++j) r = fma2(Yr[j][h], g[j][h], r);
                        ar = fma2(Xr[h], r, ar);
                        ai = fma2(Xi[h], r, ai);
                    } else {
                        p2 rr = mul2(Yr[0][h], g[0][h]), ri = mul2(Yi[0][h], g[0][h]);
#pragma unroll
                        for (int j = 1; j < NQ; ++j) {
                            rr = fma2(Yr[j][h], g[j][h], rr);
                            ri = fma2(Yi[j][h], g[j][h], ri);
                        }
                        const p2 nri = mul2(ri, m1);
                        ar = fma2(Xr[h], rr, fma2(Xi[h], nri, ar));
                        ai = fma2(Xr[h], ri, fma2(Xi[h], rr, ai));
                    }
                }
            }
#pragma unroll
            for (int h = 0; h < NP; ++h) {   // next row's phase
                const p2 nsi = mul2(Sxi[h], m1);
                const p2 xr = fma2(Xr[h], Sxr[h], mul2(Xi[h], nsi));
                Xi[h] = fma2(Xr[h], Sxi[h], mul2(Xi[h], Sxr[h]));
                Xr[h] = xr;
            }
        }
    }
    if constexpr (MODE != FAR_NORMAL) {   // + j T
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            gre[h] = fma2(tim[h], m1, gre[h]);
            gim[h] = add2(gim[h], tre[h]);
        }
    }
    // ---- lattice images ----
    const p2 magic = dup(8388608.f), nmagic = dup(-8388608.f);
    const unsigned tab_s = static_cast<unsigned>(__cvta_generic_to_shared(&S.tab[0])) - (0x4B000000u << 4);
    p2 sv[NP];
#pragma unroll
    for (int h = 0; h < NP; ++h) sv[h] = 0ull;
    // one image, one pair of test points: F and 1/R, both in table units.  REG:
    // the static part is removed on the lanes whose pair asks for it
    auto image = [&](p2 ox, p2 oy, int h, auto reg_form, bool reg, p2 &f, p2 &ri) {
        constexpr bool REG = decltype(reg_form)::value;
        const p2 x = add2(dx[h], ox), y = add2(dy[h], oy);
        const p2 r2 = fma2(x, x, fma2(y, y, dz[h]));
        const float2 R2 = upk(r2);
        float i0 = rsqrt_ftz(R2.x), i1 = rsqrt_ftz(R2.y);
        if (REG) {   // R = 0 only on an image whose static part is removed
            i0 = R2.x > 0.f ? i0 : 0.f;
            i1 = R2.y > 0.f ? i1 : 0.f;
        }
        ri = pk(i0, i1);
        float2 xu = upk(mul2(r2, ri));
        xu.x = fminf(xu.x, float(NSPAT));   // beyond the table: its zero entry
        xu.y = fminf(xu.y, float(NSPAT));
        // floor(x) in the low mantissa bits of x + 2^23 rounded down
        const p2 xp = pk(xu.x, xu.y), tt = add2_rm(xp, magic);
        const float2 v = upk(fma2(add2(tt, nmagic), m1, xp));
        const float2 tf = upk(tt);
        float4 c0, c1;
        asm("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(c0.x), "=f"(c0.y), "=f"(c0.z), "=f"(c0.w)
            : "r"(tab_s + (__float_as_uint(tf.x) << 4)));
        asm("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(c1.x), "=f"(c1.y), "=f"(c1.z), "=f"(c1.w)
            : "r"(tab_s + (__float_as_uint(tf.y) << 4)));
        const float q0 = fmaf(v.x, fmaf(v.x, c0.w, c0.z), c0.y), q1 = fmaf(v.y, fmaf(v.y, c1.w, c1.z), c1.y);
        float f0 = fmaf(v.x, q0, c0.x), f1 = fmaf(v.y, q1, c1.x);
        if (REG && reg) {   // (F(x) - F(0)) / R; in the first interval from its slope
            if (xu.x < 1.f) { f0 = q0; i0 = 1.f; } else f0 -= q.ef.e_mb2;
            if (xu.y < 1.f) { f1 = q1; i1 = 1.f; } else f1 -= q.ef.e_mb2;
            ri = pk(i0, i1);
        }
        f = pk(f0, f1);
    };
    auto accumulate = [&](const ulonglong2 *rec, int h, p2 f, p2 ri) {
        if constexpr (MODE == FAR_NORMAL) {
            sv[h] = fma2(f, ri, sv[h]);
        } else {
            const ulonglong2 ph = rec[1];
            const p2 val = mul2(f, ri);
            gre[h] = fma2(val, ph.x, gre[h]);
            gim[h] = fma2(val, ph.y, gim[h]);
        }
    };
    {
        const ulonglong2 *rec = reinterpret_cast<const ulonglong2 *>(&S.list[threadIdx.x >> 5][0]);
#pragma unroll 1
        for (int k = 0; k < n_list; k += 2, rec += 4) {   // two images at a time
            p2 f[2][NP], ri[2][NP];
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int h = 0; h < NP; ++h)
                    image(rec[2 * u].x, rec[2 * u].y, h, std::false_type{}, false, f[u][h], ri[u][h]);
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int h = 0; h < NP; ++h) accumulate(rec + 2 * u, h, f[u][h], ri[u][h]);
        }
    }
    // images whose static part some lane's pair removes (warp-uniform list), near the cut or not
#pragma unroll 1
    for (unsigned long long mk = regany; mk; mk &= mk - 1ull) {
        const int i = __ffsll((long long)mk) - 1;
        const ulonglong2 *rec = reinterpret_cast<const ulonglong2 *>(&S.img[2 * i]);
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            p2 f, ri;
            image(rec[0].x, rec[0].y, h, std::true_type{}, (regm >> i) & 1ull, f, ri);
            accumulate(rec, h, f, ri);
        }
    }
    if constexpr (MODE == FAR_NORMAL) {
        const p2 fac = reinterpret_cast<const ulonglong2 *>(&S.img[1])->x;   // every image carries the same real factor
#pragma unroll
        for (int h = 0; h < NP; ++h) gre[h] = fma2(fac, sv[h], gre[h]);
    }
}

// Records of one tetrahedron for the scatter.
struct TetRec {
    float coef[4];
    cx<float> w[4], kap;
    float v[4][3];   // v_i - c
    int row[4];
};
__device__ __forceinline__ TetRec load_tet_rec(const float4 *__restrict__ el, int n, int e) {
    TetRec r;
    const float4 *p = el + e;
    const float4 c = p[(size_t)FEL_COEF * n], w0 = p[(size_t)FEL_W01 * n], w1 = p[(size_t)FEL_W23 * n],
                 kp = p[(size_t)FEL_KAP * n], vx = p[(size_t)FEL_VX * n], vy = p[(size_t)FEL_VY * n],
                 vz = p[(size_t)FEL_VZ * n], rw = p[(size_t)FEL_ROW * n];
    r.coef[0] = c.x; r.coef[1] = c.y; r.coef[2] = c.z; r.coef[3] = c.w;
    r.w[0] = {w0.x, w0.y}; r.w[1] = {w0.z, w0.w}; r.w[2] = {w1.x, w1.y}; r.w[3] = {w1.z, w1.w};
    r.kap = {kp.x, kp.y};
    const float x[4] = {vx.x, vx.y, vx.z, vx.w}, y[4] = {vy.x, vy.y, vy.z, vy.w}, z[4] = {vz.x, vz.y, vz.z, vz.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) { r.v[i][0] = x[i]; r.v[i][1] = y[i]; r.v[i][2] = z[i]; }
    r.row[0] = __float_as_int(rw.x); r.row[1] = __float_as_int(rw.y);
    r.row[2] = __float_as_int(rw.z); r.row[3] = __float_as_int(rw.w);
    return r;
}

// Complex FP32 entry added with one 8-byte reduction (the two scalar ones it
// replaces sent every sector twice).
__device__ __forceinline__ void red_c(float *Z, size_t idx, float re, float im) {
    atomicAdd(reinterpret_cast<float2 *>(Z) + idx, make_float2(re, im));
}

// The 16 entries of the ordered tetrahedron pair (test t, source s) from its moments,
//   Z_ij += c_i w_i c_j conj(w_j) kappa [9 S - k0^2 (C - v_j.A - v_i.B + v_i.v_j Sv)],
// Sv: S with the constant that the charge term leaves out (FarPoly::k_re; it drops out
// of A, B and C, whose points sum to zero).  The charge term stays a product of its own,
// with one rounding on every face of the pair: folded into a base value with the k0^2
// terms it costs less (far pairs at 21,024 unknowns 18.9 against 19.8 ms), but the
// matrix error of a cube cell is 7.1e-9 of max|Z| against 6.1e-9.
__device__ __forceinline__ void scatter_one(float *Z, size_t N, float k2, const TetRec &t, const TetRec &s,
                                            const Mom<float> &mo, cx<float> Sv) {
    const cx<float> kS = s.kap * mo.S;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const cx<float> wB = t.v[i][0] * mo.B[0] + t.v[i][1] * mo.B[1] + t.v[i][2] * mo.B[2];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const cx<float> wsj = cconj(s.w[j]);
            const cx<float> M = mo.C - (s.v[j][0] * mo.A[0] + s.v[j][1] * mo.A[1] + s.v[j][2] * mo.A[2]) - wB +
                                (t.v[i][0] * s.v[j][0] + t.v[i][1] * s.v[j][1] + t.v[i][2] * s.v[j][2]) * Sv;
            cx<float> val = (-k2 * t.coef[i] * s.coef[j]) * (s.kap * M) + (9.f * t.coef[i] * s.coef[j]) * kS;
            val = (t.w[i] * wsj) * val;
            red_c(Z, (size_t)t.row[i] * N + (size_t)s.row[j], val.re, val.im);
        }
    }
}
// ---------------------------------------------------------------------------
// The charge term at double length (oblique incidence)
// ---------------------------------------------------------------------------
// There g_p carries a large near-constant, K exp(-j k_par.d) of the (0, 0) order, that has to
// cancel between the elements of a basis function: every rounding between the sum of the 16
// values and Z is of its size, and the roundings of one pair are common to its 16 entries.
// Unevaluated sums h + l in FP32 leave the last one, into Z.  With single roundings the
// converged FP32 solutions of 150 drawn cells were 1.11 (k_y = 0) and 1.08 (conical) times as
// far from FP64 as those of the per-lane form before.
struct W2 {
    float h, l;
};
struct CW2 {
    W2 re, im;
};
__device__ __forceinline__ W2 w2_mul(W2 a, float b) {
    const float h = a.h * b;
    return {h, fmaf(a.l, b, fmaf(a.h, b, -h))};
}
__device__ __forceinline__ W2 w2_add(W2 a, W2 b) {
    const float h = __fadd_rn(a.h, b.h), t = __fsub_rn(h, a.h);
    return {h, __fadd_rn(__fadd_rn(__fsub_rn(a.h, __fsub_rn(h, t)), __fsub_rn(b.h, t)), __fadd_rn(a.l, b.l))};
}
// c wx wy kappa S (wx, wy: the weights of the two rules; their product is not rounded either)
__device__ __forceinline__ CW2 charge_base(CW2 S, cx<float> kap, float wx, float wy, float c) {
    auto scaled = [&](W2 v) { return w2_mul(w2_mul(w2_mul(v, wx), wy), c); };
    return {scaled(w2_add(w2_mul(S.re, kap.re), w2_mul(S.im, -kap.im))),
            scaled(w2_add(w2_mul(S.re, kap.im), w2_mul(S.im, kap.re)))};
}
// w (v + add), w the phase of functions across the walls (else 1), rounded once
__device__ __forceinline__ cx<float> charge_value(CW2 v, cx<float> w, cx<float> add) {
    const float lr = v.re.l + add.re, li = v.im.l + add.im;
    return {fmaf(w.re, v.re.h, fmaf(-w.im, v.im.h, fmaf(w.re, lr, -w.im * li))),
            fmaf(w.re, v.im.h, fmaf(w.im, v.re.h, fmaf(w.re, li, w.im * lr)))};
}
// scatter_one with the charge term c_i c_j kS, kS as charge_base
__device__ __forceinline__ void scatter_w2(float *Z, size_t N, float k2, const TetRec &t, const TetRec &s,
                                           const Mom<float> &mo, CW2 kS) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const cx<float> wB = t.v[i][0] * mo.B[0] + t.v[i][1] * mo.B[1] + t.v[i][2] * mo.B[2];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const cx<float> M = mo.C - (s.v[j][0] * mo.A[0] + s.v[j][1] * mo.A[1] + s.v[j][2] * mo.A[2]) - wB +
                                (t.v[i][0] * s.v[j][0] + t.v[i][1] * s.v[j][1] + t.v[i][2] * s.v[j][2]) * mo.S;
            const float f = t.coef[i] * s.coef[j], fl = fmaf(t.coef[i], s.coef[j], -f);
            const cx<float> m = (-k2 * f) * (s.kap * M);
            const float hr = kS.re.h * f, hi = kS.im.h * f;
            const CW2 v = {{hr, fmaf(kS.re.h, fl, fmaf(kS.re.l, f, fmaf(kS.re.h, f, -hr)))},
                           {hi, fmaf(kS.im.h, fl, fmaf(kS.im.l, f, fmaf(kS.im.h, f, -hi)))}};
            const cx<float> z = charge_value(v, t.w[i] * cconj(s.w[j]), m);
            red_c(Z, (size_t)t.row[i] * N + (size_t)s.row[j], z.re, z.im);
        }
    }
}
// SYM (normal incidence): the reversed pair's entries too when `both`, from its moments S, B, A, C
template <bool SYM>
__device__ __forceinline__ void scatter_rec(float *Z, size_t N, float k2, const TetRec &t, const TetRec &s,
                                            const Mom<float> &mo, cx<float> Sv, bool both) {
    scatter_one(Z, N, k2, t, s, mo, Sv);
    if (SYM && both) {
        Mom<float> mr = mo;
        for (int d = 0; d < 3; ++d) { mr.A[d] = mo.B[d]; mr.B[d] = mo.A[d]; }
        scatter_one(Z, N, k2, s, t, mr, Sv);
    }
}

}  // namespace vie
