// Device math for the fill: complex helpers, Faddeeva function, Ewald-summed
// 2D periodic Green's function (Eq. (3)-(4), Sec. 2.2) and closed-form
// integrals of 1/R and R over triangles and tetrahedra.
#pragma once
#include <cuda_runtime.h>
#include <math_constants.h>

#include "ewald_params.h"

namespace vie {

template <typename T> struct cx { T re, im; };

template <typename T> __device__ __forceinline__ cx<T> mk(T r, T i) { return {r, i}; }
template <typename T> __device__ __forceinline__ cx<T> operator+(cx<T> a, cx<T> b) { return {a.re + b.re, a.im + b.im}; }
template <typename T> __device__ __forceinline__ cx<T> operator-(cx<T> a, cx<T> b) { return {a.re - b.re, a.im - b.im}; }
template <typename T> __device__ __forceinline__ cx<T> operator*(cx<T> a, cx<T> b) {
    return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
template <typename T> __device__ __forceinline__ cx<T> operator*(T s, cx<T> a) { return {s * a.re, s * a.im}; }
template <typename T> __device__ __forceinline__ cx<T> cconj(cx<T> a) { return {a.re, -a.im}; }
template <typename T> __device__ __forceinline__ cx<T> crecip(cx<T> a) {
    // 1/a with scaling to avoid overflow of |a|^2
    T s = fmax(fabs(a.re), fabs(a.im));
    T ar = a.re / s, ai = a.im / s;
    T d = s * (ar * ar + ai * ai);
    return {ar / d, -ai / d};
}
template <typename T> __device__ __forceinline__ void cfma(cx<T> &acc, T s, cx<T> a) {
    acc.re = fma(s, a.re, acc.re);
    acc.im = fma(s, a.im, acc.im);
}

// Moments of one ordered element pair: sums of g, r_x g, r_y g and (r_x.r_y) g
// (r relative to the elements' centroids).
template <typename T> struct Mom {
    cx<T> S, A[3], B[3], C;
    __device__ void zero() {
        S = {0, 0}; C = {0, 0};
        for (int d = 0; d < 3; ++d) { A[d] = {0, 0}; B[d] = {0, 0}; }
    }
};

// ---------------------------------------------------------------------------
// Faddeeva function w(z) = exp(-z^2) erfc(-j z) for Im z >= 0 by Weideman's
// rational expansion (SIAM J. Numer. Anal. 31, 1994):
//   w(z) = 2 p(Zz) / (L - j z)^2 + 1 / (sqrt(pi) (L - j z)),  Zz = (L + j z)/(L - j z),
// p(Zz) = sum_{n=1}^{NW} a_n Zz^(n-1), a_n the Fourier coefficients of
// (L^2 + t^2) exp(-t^2) in the variable theta, t = L tan(theta/2).  The
// coefficients are computed on the host in FP64 and stored here.
constexpr int NW64 = 40;
constexpr int NW32 = 20;
struct WeidemanTables {
    double a64[NW64 + 1];
    float a32[NW32 + 1];
    double L64;
    float L32;
};
static __constant__ WeidemanTables c_weid;   // filled by upload_constants() (fill.cu)

template <typename T> struct WTraits;
template <> struct WTraits<double> {
    static constexpr int N = NW64;
    __device__ static double L() { return c_weid.L64; }
    __device__ static double a(int n) { return c_weid.a64[n]; }
};
template <> struct WTraits<float> {
    static constexpr int N = NW32;
    __device__ static float L() { return c_weid.L32; }
    __device__ static float a(int n) { return c_weid.a32[n]; }
};

template <typename T> __device__ __forceinline__ T rsqrt_pi() { return T(0.56418958354775628695); }

// erfcx(u) = exp(u^2) erfc(u) = w(j u), complex u with Re u >= 0.
template <typename T> __device__ __forceinline__ cx<T> erfcx_c(cx<T> u) {
    const T L = WTraits<T>::L();
    // z = j u: L - j z = L + u, L + j z = L - u
    cx<T> dm = {L + u.re, u.im};
    cx<T> dp = {L - u.re, -u.im};
    cx<T> inv = crecip(dm);
    cx<T> Z = dp * inv;
    cx<T> p = {WTraits<T>::a(WTraits<T>::N), T(0)};
#pragma unroll
    for (int n = WTraits<T>::N - 1; n >= 1; --n) {
        p = p * Z;
        p.re += WTraits<T>::a(n);
    }
    cx<T> t = inv * p;
    t.re = fma(T(2), t.re, rsqrt_pi<T>());
    t.im = T(2) * t.im;
    return inv * t;
}

// erfcx(x) for real x >= 0 (the expansion at z = j x stays real).
template <typename T> __device__ __forceinline__ T erfcx_r(T x) {
    const T L = WTraits<T>::L();
    T inv = T(1) / (L + x);
    T Z = (L - x) * inv;
    T p = WTraits<T>::a(WTraits<T>::N);
#pragma unroll
    for (int n = WTraits<T>::N - 1; n >= 1; --n) p = fma(p, Z, WTraits<T>::a(n));
    return inv * fma(T(2) * p, inv, rsqrt_pi<T>());
}

// Ewald parameter blocks (EwaldTables, EwaldF32): ewald_params.h

template <typename T> struct ETraits;
template <> struct ETraits<double> {
    __device__ static const double *img(const EwaldTables *ew, int i) { return ew->img64[i]; }
    __device__ static const double *mode(const EwaldTables *ew, int i) { return ew->mode64[i]; }
    __device__ static double xcut(const EwaldTables *ew) { return ew->xcut64; }
};
template <> struct ETraits<float> {
    __device__ static const float *img(const EwaldTables *ew, int i) { return ew->img32[i]; }
    __device__ static const float *mode(const EwaldTables *ew, int i) { return ew->mode32[i]; }
    __device__ static float xcut(const EwaldTables *ew) { return ew->xcut32; }
};

// g_p(d) for an in-cell difference d; images whose bit is set in `sub`
// (9-bit mask over (m,n) in {-1,0,1}^2) have their static part
// phase/(4 pi R) removed.
template <typename T>
__device__ cx<T> green_p(T dx, T dy, T dz, unsigned sub, const EwaldTables *__restrict__ ew) {
    const T E = T(ew->E);
    const T bb = T(ew->bb);
    const T xc = ETraits<T>::xcut(ew) + T(0.5);
    cx<T> acc = {T(0), T(0)};
    // spectral series
    const T z = fabs(dz);
    const T ez = exp(-(z * E) * (z * E));
    const T inv2E = T(0.5) / E;
    for (int i = 0; i < ew->n_mode; ++i) {
        const T *md = ETraits<T>::mode(ew, i);
        T s, c;
        sincos(-(md[0] * dx + md[1] * dy), &s, &c);
        cx<T> ph = {c, s};
        cx<T> br;
        if (md[3] == T(0)) {                       // evanescent: gamma real
            T g = md[2];
            T pre = md[4] * ez;
            T t1 = pre * erfcx_r(g * inv2E + z * E);
            T u = g * inv2E - z * E;
            T t2 = (u >= T(0)) ? pre * erfcx_r(u) : T(2) * exp(-g * z) - pre * erfcx_r(-u);
            br = {t1 + t2, T(0)};
        } else {                                    // propagating: gamma = j gi
            T gi = md[3];
            T pre = md[4] * ez;
            cx<T> e1 = erfcx_c(cx<T>{z * E, gi * inv2E});
            // erfcx(zE - j gi/2E) = conj(e1)
            T sg, cg;
            sincos(gi * z, &sg, &cg);
            // t1 = pre e1; t2 = 2 e^{-j gi z} - pre conj(e1)
            br = {pre * e1.re + T(2) * cg - pre * e1.re, pre * e1.im - T(2) * sg + pre * e1.im};
        }
        cx<T> ig = {md[5], md[6]};
        acc = acc + ph * (br * ig);
    }
    // spatial series
    for (int i = 0; i < ew->n_img; ++i) {
        const T *im = ETraits<T>::img(ew, i);
        T x = dx + im[0], y = dy + im[1];
        T R2 = x * x + y * y + dz * dz;
        T R = sqrt(R2);
        bool regular = false;
        if (sub) {
#pragma unroll
            for (int k = 0; k < 9; ++k)
                if (((sub >> k) & 1u) && ew->near_img[k] == i) regular = true;
        }
        const bool beyond = R * E > xc;   // nothing of the image term itself left
        if (beyond && !regular) continue;
        if (regular && R * E < T(1e-6)) {
            // continuous limit at R = 0 of (image term - static term):
            // reg0 = (E/4pi)[2 b erfi(b) - (2/sqrt pi) exp(b^2)]; the table
            // phase carries exp(b^2)/(4 pi), undone here
            cx<T> ph = {im[2], im[3]};
            T unscale = T(4.0 * CUDART_PI) * exp(-bb * bb) * T(ew->reg0_re);
            acc = acc + unscale * ph;
            continue;
        }
        T val = beyond ? T(0) : exp(-R2 * E * E) * erfcx_c(cx<T>{R * E, bb}).re / R;
        if (regular) val -= exp(-bb * bb) / R;   // static part phase/(4 pi R) in table units
        cx<T> ph = {im[2], im[3]};
        acc = acc + val * ph;
    }
    return acc;
}

// FP32 g_p from per-request tables (same series, same truncation as green_p):
//  spectral: sum_pq exp(-j k_t,pq . rho) G_pq(|z|), G = [e^{gz}erfc(..) + e^{-gz}erfc(..)]/(4ab g)
//            tabulated per distinct gamma; phases by recurrence over the (p, q) rectangle
//  spatial:  phase_mn exp(b^2)/(4 pi) F(R E)/R with F(x) = exp(-x^2) Re erfcx(x + j b);
//            the regularised near image uses (F(RE) - F(0))/R, formed without
//            cancellation in the first interval
// stab: [NSPAT][4] cubic coefficients (shared memory); ztab: [n_tab][NZTAB][4] complex
// With PAIR the same pass also returns gm = g_p(-d): the spectral terms of -d
// carry the conjugate phases, and the spatial term of image -R_mn at -d is the
// table value of image R_mn at d with the conjugate lattice phase (the image
// list and the near-image masks are symmetric under (m,n) -> (-m,-n)).
// rtab (may be null): the real parts of the tables as one float4 per
// interval; used for the tables flagged TAB_REAL (their imaginary parts are 0)
// SYM (normal incidence, k_par = 0, mode rectangle symmetric about (0, 0)):
// G_pq = G_-p-q, so the orders pair up into 2 G_pq cos(k_t,pq . rho) over the
// half plane p > 0 or (p = 0, q > 0), plus G_00; g_p is even in d, so gm = gp.
template <bool PAIR, bool SYM = false>
__device__ __forceinline__ void green_tab_impl(float dx, float dy, float dz, unsigned sub, const float *stab,
                                               const float2 *__restrict__ ztab, const EwaldF32 &ew,
                                               cx<float> &gp, cx<float> &gm,
                                               const float4 *__restrict__ rtab = nullptr,
                                               unsigned long long imask = ~0ull) {
    cx<float> acc = {0.f, 0.f}, acc2 = {0.f, 0.f};
    const float z = fabsf(dz);
    float zu = fminf(z * ew.z_inv_h, float(NZTAB));
    int iz = min((int)zu, NZTAB - 1);
    const float u = zu - iz;
    // G of the mode table `code` at |z| (real tables: one 16-byte load)
    auto table = [&](int code, float &gr, float &gi) {
        const int tb = code & TAB_INDEX;
        if (rtab && (code & TAB_REAL)) {
            const float4 c = __ldg(rtab + (size_t)tb * NZTAB + iz);
            gr = fmaf(u, fmaf(u, fmaf(u, c.w, c.z), c.y), c.x);
            gi = 0.f;
            return true;
        }
        const float2 *cf = ztab + ((size_t)tb * NZTAB + iz) * 4;
        const float2 c0 = __ldg(cf), c1 = __ldg(cf + 1), c2 = __ldg(cf + 2), c3 = __ldg(cf + 3);
        gr = fmaf(u, fmaf(u, fmaf(u, c3.x, c2.x), c1.x), c0.x);
        gi = fmaf(u, fmaf(u, fmaf(u, c3.y, c2.y), c1.y), c0.y);
        return false;
    };
    const int np = ew.np, nq = ew.nq;
    float s, c;
    if constexpr (SYM) {
        if (np > 0) {
            // G_pq depends on |k_t,pq| alone, so it is even in p and in q separately:
            // sum_pq G_pq exp(-j k_t,pq . rho) = sum_{p,q >= 0} w_p w_q G_pq cos(k_p x) cos(k_q y)
            // (w_0 = 1, w_>0 = 2; the sine products cancel), one table evaluation per
            // order of the quadrant; D_q = 2 cos(k_q y) and D_p by Chebyshev recurrence
            const int P = (np - 1) / 2, Q = (nq - 1) / 2;
            const float d1x = 2.f * cospif(ew.step_x * dx * 0.31830988618f);
            const float d1y = 2.f * cospif(ew.step_y * dy * 0.31830988618f);
            float dp_prev = 2.f, dp = d1x;   // D_0, D_1 in x
            for (int p = 0; p <= P; ++p) {
                const int row = (P + p) * nq + Q;
                float rr = 0.f, ri = 0.f, gr, gi;
                const int c0 = ew.rect_tab[row];
                if (c0 >= 0) { table(c0, rr, ri); }
                float dq_prev = 2.f, dq = d1y;   // D_0, D_1 in y
                for (int q = 1; q <= Q; ++q) {
                    const int code = ew.rect_tab[row + q];
                    if (code >= 0) {
                        if (table(code, gr, gi)) rr = fmaf(dq, gr, rr);
                        else { rr = fmaf(dq, gr, rr); ri = fmaf(dq, gi, ri); }
                    }
                    const float dn = fmaf(d1y, dq, -dq_prev);
                    dq_prev = dq;
                    dq = dn;
                }
                const float wp = p == 0 ? 1.f : dp;
                acc.re = fmaf(wp, rr, acc.re);
                acc.im = fmaf(wp, ri, acc.im);
                if (p >= 1) {   // D_{p+1} = d1x D_p - D_{p-1}
                    const float dn = fmaf(d1x, dp, -dp_prev);
                    dp_prev = dp;
                    dp = dn;
                }
            }
        }
    } else {
        sincospif(-(ew.kx + ew.p0 * ew.step_x) * dx * 0.31830988618f, &s, &c);
        cx<float> ex = {c, s};
        sincospif(-ew.step_x * dx * 0.31830988618f, &s, &c);
        const cx<float> sx = {c, s};
        sincospif(-(ew.ky + ew.q0 * ew.step_y) * dy * 0.31830988618f, &s, &c);
        const cx<float> ey0 = {c, s};
        sincospif(-ew.step_y * dy * 0.31830988618f, &s, &c);
        const cx<float> sy = {c, s};
        for (int p = 0; p < np; ++p) {
            cx<float> inner = {0.f, 0.f}, inner2 = {0.f, 0.f};
            cx<float> ey = ey0;
            for (int q = 0; q < nq; ++q) {
                const int code = ew.rect_tab[p * nq + q];
                if (code >= 0) {
                    float gr, gi;
                    if (table(code, gr, gi)) {   // real G: real products
                        inner.re = fmaf(ey.re, gr, inner.re);
                        inner.im = fmaf(ey.im, gr, inner.im);
                        if (PAIR) {
                            inner2.re = fmaf(ey.re, gr, inner2.re);
                            inner2.im = fmaf(-ey.im, gr, inner2.im);
                        }
                    } else {
                        const cx<float> g = {gr, gi};
                        inner = inner + ey * g;
                        if (PAIR) inner2 = inner2 + cconj(ey) * g;
                    }
                }
                ey = ey * sy;
            }
            acc = acc + ex * inner;
            if (PAIR) acc2 = acc2 + cconj(ex) * inner2;
            ex = ex * sx;
        }
    }
    const float E = ew.Ef;
    const float xmax = ew.xs_max, ih = ew.xs_inv_h;
    const float r2max = (xmax / E) * (xmax / E) * 1.0001f;   // loose: the exact test follows
    float sv = 0.f;   // SYM: the sum of the image values before their common factor
    auto image = [&](int i) {
        const float *im = ew.img[i];
        const float x = dx + im[0], y = dy + im[1];
        const float R2 = x * x + y * y + dz * dz;
        bool regular = false;
        if (sub) {
#pragma unroll
            for (int k = 0; k < 9; ++k)
                if (((sub >> k) & 1u) && ew.near_img[k] == i) regular = true;
        }
        if (R2 > r2max && !regular) return;   // outside the cut: skip before the square root
        const float rinv = R2 > 0.f ? rsqrtf(R2) : 0.f;   // R = 0 only on a regularised image (no 1/R)
        const float R = R2 * rinv;
        const float xr = R * E;
        const bool beyond = xr > xmax;
        if (beyond && !regular) return;
        const float xu = xr * ih;
        const int ix = min((int)xu, NSPAT - 1);
        const float v = xu - ix;
        const float4 cs = *reinterpret_cast<const float4 *>(stab + 4 * ix);   // one 16-byte load
        float val;
        if (beyond) {   // F is zero there: what is left is the static part removed
            val = -ew.e_mb2 * rinv;
        } else if (regular) {
            if (ix == 0)   // (F(x) - F(0))/R = E (c1 + v (c2 + v c3)) / h
                val = E * ih * fmaf(v, fmaf(v, cs.w, cs.z), cs.y);
            else
                val = (fmaf(v, fmaf(v, fmaf(v, cs.w, cs.z), cs.y), cs.x) - ew.e_mb2) * rinv;
        } else {
            val = fmaf(v, fmaf(v, fmaf(v, cs.w, cs.z), cs.y), cs.x) * rinv;
        }
        if (SYM) {   // k_par = 0: every image carries the same real phase factor
            sv += val;
            return;
        }
        acc.re = fmaf(val, im[2], acc.re);
        acc.im = fmaf(val, im[3], acc.im);
        if (PAIR) {
            acc2.re = fmaf(val, im[2], acc2.re);
            acc2.im = fmaf(-val, im[3], acc2.im);
        }
    };
    // images 0..63 as the caller's mask selects them (it leaves out only images
    // beyond the cut) and those whose static part is removed, the rest one by one
    if (sub)
        for (int k = 0; k < 9; ++k)
            if (((sub >> k) & 1u) && ew.near_img[k] < 64) imask |= 1ull << ew.near_img[k];
    if (ew.n_img < 64) imask &= (1ull << ew.n_img) - 1ull;
    for (unsigned long long mk = imask; mk; mk &= mk - 1ull) image(__ffsll((long long)mk) - 1);
    for (int i = 64; i < ew.n_img; ++i) image(i);
    if (SYM) acc.re = fmaf(ew.img[0][2], sv, acc.re);
    gp = acc;
    gm = SYM ? acc : acc2;
}

// Images (of the first 64) that can lie inside the spatial cut for some
// displacement within `rad` of (cx, cy, cz): every image whose shifted centre
// distance exceeds the cut radius + rad is left out.
__device__ __forceinline__ unsigned long long image_mask(const EwaldF32 &ew, float cx, float cy, float cz,
                                                         float rad) {
    const float rc = ew.xs_max / ew.Ef * 1.0001f + rad * 1.0001f + 1e-6f * (fabsf(cx) + fabsf(cy) + fabsf(cz));
    const float rc2 = rc * rc;
    const int n = min(ew.n_img, 64);
    unsigned long long m = 0ull;
    for (int i = 0; i < n; ++i) {
        const float x = cx + ew.img[i][0], y = cy + ew.img[i][1];
        if (x * x + y * y + cz * cz <= rc2) m |= 1ull << i;
    }
    return m;
}

__device__ __forceinline__ cx<float> green_tab(float dx, float dy, float dz, unsigned sub, const float *stab,
                                               const float2 *__restrict__ ztab, const EwaldF32 &ew) {
    cx<float> g, unused;
    green_tab_impl<false>(dx, dy, dz, sub, stab, ztab, ew, g, unused);
    return g;
}

// ---------------------------------------------------------------------------
// Closed forms (divergence theorem, polygonal / polyhedral sources), observer at
// the origin:
//  triangle: int 1/R = sum_i t_i ln[(R+_i + s+_i)/(R-_i + s-_i)] - |h| Omega
//            int R   = ( h^2 int 1/R + 1/2 sum_i t_i (s+R+ - s-R- + R0^2 ln(..)) ) / 3
//  tetrahedron: int 1/R = 1/2 sum_f d_f int_f 1/R,  int (r'-r)/R = sum_f n_f int_f R
// t_i: signed in-plane distance to edge i, R0^2 = t^2 + h^2, Omega the solid angle
// of the triangle, from its vertices (van Oosterom and Strackee, IEEE Trans.
// Biomed. Eng. 30, 1983): tan(Omega/2) = |a.(b x c)| / (abc + (a.b)c + (a.c)b + (b.c)a).
// What depends on the source alone (edge directions, normals) is a record built
// once per element.
struct TriGeom {
    double lh[3][3], len[3];   // edge directions (vertex q to q + 1) and lengths
    double n[3], a2;           // unit normal, twice the area
    double u[3][3];            // in-plane outward normals of the edges
    double tiny;
};
struct TetGeom {
    double lh[6][3], len[6];   // edges (0,1) (0,2) (0,3) (1,2) (1,3) (2,3)
    double n[4][3], a2[4];     // outward unit normal and twice the area of the face opposite each vertex
    double u[4][3][3];         // in-plane outward normals of its edges
    double tiny;
};
__host__ __device__ __forceinline__ double dot3(const double *a, const double *b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; }
__host__ __device__ __forceinline__ void cross3(const double *a, const double *b, double *c) {
    c[0] = a[1] * b[2] - a[2] * b[1];
    c[1] = a[2] * b[0] - a[0] * b[2];
    c[2] = a[0] * b[1] - a[1] * b[0];
}
// edges of the face opposite vertex f and the face's third vertex per edge
__host__ __device__ __forceinline__ constexpr int tet_fe(int f, int q) {
    constexpr int FE[4][3] = {{3, 5, 4}, {1, 5, 2}, {0, 4, 2}, {0, 3, 1}};
    return FE[f][q];
}
__host__ __device__ __forceinline__ constexpr int tet_fc(int f, int q) {
    constexpr int FC[4][3] = {{3, 1, 2}, {3, 0, 2}, {3, 0, 1}, {2, 0, 1}};
    return FC[f][q];
}
__host__ __device__ __forceinline__ constexpr int tet_ea(int e) { return e < 3 ? 0 : (e < 5 ? 1 : 2); }
__host__ __device__ __forceinline__ constexpr int tet_eb(int e) { return e < 3 ? e + 1 : (e < 5 ? e - 1 : 3); }

__host__ __device__ inline void tri_geom(const double *v, TriGeom &g) {   // v: vertices [3][3]
    double e1[3], e2[3];
    for (int d = 0; d < 3; ++d) { e1[d] = v[3 + d] - v[d]; e2[d] = v[6 + d] - v[d]; }
    cross3(e1, e2, g.n);
    g.a2 = sqrt(dot3(g.n, g.n));
    for (int d = 0; d < 3; ++d) g.n[d] /= g.a2;
    double scale = 0;
    for (int q = 0; q < 3; ++q) {
        const double *pa = v + 3 * q, *pb = v + 3 * ((q + 1) % 3);
        double d[3] = {pb[0] - pa[0], pb[1] - pa[1], pb[2] - pa[2]};
        g.len[q] = sqrt(dot3(d, d));
        scale = fmax(scale, g.len[q]);
        for (int k = 0; k < 3; ++k) g.lh[q][k] = d[k] / g.len[q];
        cross3(g.lh[q], g.n, g.u[q]);
    }
    g.tiny = 1e-13 * scale;
}
__host__ __device__ inline void tet_geom(const double *v, TetGeom &g) {   // v: vertices [4][3]
    double scale = 0;
    for (int e = 0; e < 6; ++e) {
        const double *pa = v + 3 * tet_ea(e), *pb = v + 3 * tet_eb(e);
        double d[3] = {pb[0] - pa[0], pb[1] - pa[1], pb[2] - pa[2]};
        g.len[e] = sqrt(dot3(d, d));
        scale = fmax(scale, g.len[e]);
        for (int k = 0; k < 3; ++k) g.lh[e][k] = d[k] / g.len[e];
    }
    g.tiny = 1e-13 * scale;
    for (int f = 0; f < 4; ++f) {
        const int fv[3] = {f == 0 ? 1 : 0, f <= 1 ? 2 : 1, f <= 2 ? 3 : 2};
        const double *p0 = v + 3 * fv[0], *p1 = v + 3 * fv[1], *p2 = v + 3 * fv[2];
        double e1[3], e2[3], o[3];
        for (int d = 0; d < 3; ++d) { e1[d] = p1[d] - p0[d]; e2[d] = p2[d] - p0[d]; o[d] = p0[d] - v[3 * f + d]; }
        cross3(e1, e2, g.n[f]);
        g.a2[f] = sqrt(dot3(g.n[f], g.n[f]));
        const double sg = dot3(g.n[f], o) >= 0 ? 1.0 / g.a2[f] : -1.0 / g.a2[f];
        for (int d = 0; d < 3; ++d) g.n[f][d] *= sg;
        for (int q = 0; q < 3; ++q) {   // outward: away from the face's third vertex
            const int e = tet_fe(f, q);
            cross3(g.lh[e], g.n[f], g.u[f][q]);
            const double *pa = v + 3 * tet_ea(e), *pc = v + 3 * tet_fc(f, q);
            const double w[3] = {pa[0] - pc[0], pa[1] - pc[1], pa[2] - pc[2]};
            if (dot3(g.u[f][q], w) < 0)
                for (int d = 0; d < 3; ++d) g.u[f][q][d] = -g.u[f][q][d];
        }
    }
}
// ln[(Rb + sb)/(Ra + sa)] along an edge, with R + s = d2/(R - s) for s < 0 (d2: squared
// distance to the edge line)
__host__ __device__ __forceinline__ double edge_log(const double *pa, const double *lh, double sa, double sb, double Ra,
                                                    double Rb) {
    if (sa >= 0) return log((Rb + sb) / (Ra + sa));
    if (sb <= 0) return log((Ra - sa) / (Rb - sb));
    double c[3];
    cross3(pa, lh, c);
    const double d2 = dot3(c, c);
    return d2 > 0 ? log((Rb + sb) * (Ra - sa) / d2) : 0.0;
}
// int 1/R over a triangle; v: its vertices relative to the observer
__host__ __device__ inline double tri_inv(const TriGeom &g, const double *v) {
    const double R[3] = {sqrt(dot3(v, v)), sqrt(dot3(v + 3, v + 3)), sqrt(dot3(v + 6, v + 6))};
    const double ah = fabs(dot3(g.n, v));
    double slog = 0;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const double *pa = v + 3 * q;
        const double t = dot3(g.u[q], pa);
        if (fabs(t) <= g.tiny) continue;
        const double sa = dot3(g.lh[q], pa);
        slog += t * edge_log(pa, g.lh[q], sa, sa + g.len[q], R[q], R[(q + 1) % 3]);
    }
    if (ah > g.tiny) {
        const double den = R[0] * R[1] * R[2] + dot3(v, v + 3) * R[2] + dot3(v, v + 6) * R[1] + dot3(v + 3, v + 6) * R[0];
        slog -= ah * 2.0 * atan2(g.a2 * ah, den);
    }
    return slog;
}
// int 1/R and (VEC) int (r' - r)/R over a tetrahedron; v: its vertices relative to the observer
template <bool VEC>
__host__ __device__ inline void tet_integrals(const TetGeom &g, const double *v, double &inv, double *vec) {
    double R[4], L[6], sR[6], dt[6];
#pragma unroll
    for (int k = 0; k < 4; ++k) R[k] = sqrt(dot3(v + 3 * k, v + 3 * k));
#pragma unroll
    for (int e = 0; e < 6; ++e) {
        const double *pa = v + 3 * tet_ea(e), *pb = v + 3 * tet_eb(e);
        const double sa = dot3(g.lh[e], pa), sb = sa + g.len[e], Ra = R[tet_ea(e)], Rb = R[tet_eb(e)];
        L[e] = edge_log(pa, g.lh[e], sa, sb, Ra, Rb);
        if (VEC) sR[e] = sb * Rb - sa * Ra;
        dt[e] = dot3(pa, pb);
    }
    inv = 0;
    if (VEC) vec[0] = vec[1] = vec[2] = 0;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        const double d = dot3(g.n[f], v + 3 * (f == 0 ? 1 : 0));   // signed distance of the face
        const double ah = fabs(d);
        double slog = 0, sr = 0;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const int e = tet_fe(f, q);
            const double t = dot3(g.u[f][q], v + 3 * tet_ea(e));
            if (fabs(t) <= g.tiny) continue;
            slog += t * L[e];
            if (VEC) sr += t * (sR[e] + (t * t + d * d) * L[e]);
        }
        if (ah > g.tiny) {
            const int i = f == 0 ? 1 : 0, j = f <= 1 ? 2 : 1, k = f <= 2 ? 3 : 2;
            double den = R[i] * R[j] * R[k];
#pragma unroll
            for (int q = 0; q < 3; ++q) den += dt[tet_fe(f, q)] * R[tet_fc(f, q)];
            slog -= ah * 2.0 * atan2(g.a2[f] * ah, den);
        }
        inv += 0.5 * d * slog;
        if (VEC) {
            const double fr = (d * d * slog + 0.5 * sr) / 3.0;
            for (int q = 0; q < 3; ++q) vec[q] += g.n[f][q] * fr;
        }
    }
}

}  // namespace vie
