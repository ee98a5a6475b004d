// Far element pairs of the FP64 fill: the Ewald series of green_p with the orders
// as polynomials and the spatial kernel from a table of polynomials (Far64,
// ewald_params.h), both fitted on the host in extended precision: against 32-digit
// values of g_p at six cells its rms error is 0.29 to 0.67 of the series' own (fitted in
// FP64: up to 3.6).  6 x 6 x 2 slab, FP64: 273 -> 27 ms a solve.  Bound by the
// FP64 pipe (1/64 of the FP32 rate): what counts is FP64 instructions per
// evaluation.  Summed term by term (green_p) each Floquet order takes two
// 40-term Faddeeva expansions, an exponential and a sincos, each image one complex
// expansion, an exponential and a square root, and the reversed pair everything
// again; here an order takes one fused multiply-add per degree (~18), an image 28
// instructions with the square root from an FP32 seed, the phases come from
// per-point records and the reversed pair's value from the same pass.
#include <cuda_runtime.h>

#include "device_math.cuh"
#include "fill.h"

namespace vie {

namespace {

__global__ void k_prep64(DevMesh m, const __grid_constant__ DevReq q) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int nt4 = 4 * m.nt;
    if (i >= nt4 + 3 * m.nf) return;
    const double *x = i < nt4 ? m.far64 + 28 * (size_t)(i / 4) + 3 * (i % 4) : m.ffar64 + 12 * (size_t)((i - nt4) / 3) + 3 * ((i - nt4) % 3);
    double *o = q.ph64 + 8 * (size_t)i;
    sincos(q.f64.kx * x[0], o + 1, o);
    sincos(q.f64.ky * x[1], o + 3, o + 2);
    sincos(q.f64.sx * x[0], o + 5, o + 4);
    sincos(q.f64.sy * x[1], o + 7, o + 6);
}

// e^{-j th_a} conj(e^{-j th_b}) from (cos, sin) of th_a and th_b
__device__ __forceinline__ cx<double> phase_diff(const double *a, const double *b) {
    return {fma(a[0], b[0], a[1] * b[1]), fma(a[0], b[1], -a[1] * b[0])};
}

__device__ __forceinline__ double horner(const double *c, int d, double t) {
    double s = c[0];
    for (int n = 1; n <= d; ++n) s = fma(s, t, c[n]);
    return s;
}

// g_p(d) and (PAIR) g_p(-d) of one point pair with phase records pa, pb; the same
// near-image mask applies to both (mirrored)
template <bool PAIR>
__device__ __forceinline__ void green64(const Far64 &f, const double *blob, double dx, double dy, double dz,
                                        const double *pa, const double *pb, unsigned sub, cx<double> &gp, cx<double> &gm) {
    const double dz2 = dz * dz, t = fma(f.t_scale, dz2, -1.0);
    const int4 *dir = reinterpret_cast<const int4 *>(blob + f.dir);
    cx<double> S = {0, 0}, T = {0, 0};   // sums with Re G and Im G
    if (f.sym) {
        const double c1x = 2.0 * fma(pa[4], pb[4], pa[5] * pb[5]), c1y = 2.0 * fma(pa[6], pb[6], pa[7] * pb[7]);
        double xp = 2.0, xc = 1.0;   // D_{i-1}, weight of row i
        for (int i = 0; i < f.rows; ++i) {
            double r = 0, ri = 0, yp = 2.0, yc = 1.0;
            for (int j = 0; j < f.cols; ++j) {
                const int4 e = dir[i * f.cols + j];
                if (e.y >= 0) r = fma(yc, horner(blob + e.x, e.y, t), r);
                if (e.w >= 0) ri = fma(yc, horner(blob + e.z, e.w, t), ri);
                const double yn = j == 0 ? c1y : fma(c1y, yc, -yp);
                yp = j == 0 ? 2.0 : yc;
                yc = yn;
            }
            S.re = fma(xc, r, S.re);
            T.re = fma(xc, ri, T.re);
            const double xn = i == 0 ? c1x : fma(c1x, xc, -xp);
            xp = i == 0 ? 2.0 : xc;
            xc = xn;
        }
    } else {
        // outwards from order (0, 0), the largest: up from it, then down (from the first
        // row its phase came out of -p0 products and carried their rounding)
        const cx<double> X0 = phase_diff(pa, pb), Y0 = phase_diff(pa + 2, pb + 2);
        cx<double> sx = phase_diff(pa + 4, pb + 4), sy0 = phase_diff(pa + 6, pb + 6), X = X0;
        const int iu = f.rows - f.i0, ju = f.cols - f.j0;
        for (int k = 0; k < f.rows; ++k) {
            if (k == iu) {
                sx.im = -sx.im;
                X = X0 * sx;
            }
            const int i = k < iu ? f.i0 + k : f.rows - 1 - k;
            cx<double> r = {0, 0}, ri = {0, 0}, Y = Y0, sy = sy0;
            for (int l = 0; l < f.cols; ++l) {
                if (l == ju) {
                    sy.im = -sy.im;
                    Y = Y0 * sy;
                }
                const int4 e = dir[i * f.cols + (l < ju ? f.j0 + l : f.cols - 1 - l)];
                if (e.y >= 0) cfma(r, horner(blob + e.x, e.y, t), Y);
                if (e.w >= 0) cfma(ri, horner(blob + e.z, e.w, t), Y);
                Y = Y * sy;
            }
            S = S + X * r;
            T = T + X * ri;
            X = X * sx;
        }
    }
    gp = {S.re - T.im, S.im + T.re};
    // images: at -d the image -R carries the same value and the conjugate phase
    cx<double> im = {0, 0};
    for (int i = 0; i < f.n_img; ++i) {
        const double *R = blob + f.img + 4 * i;
        const double x = dx + R[0], y = dy + R[1];
        const double R2 = fma(x, x, fma(y, y, dz2));
        // 1/R from an FP32 seed by one third-order step (error ~ 1e-21 of it)
        const double r0 = (double)rsqrtf((float)R2);
        const double e = fma(-R2 * r0, r0, 1.0);
        const double ri = fma(r0, e * fma(0.375, e, 0.5), r0);
        const double xu = R2 * ri * f.xs;
        const float xf = (float)xu;
        bool reg = false;
        if (sub) {
#pragma unroll
            for (int k = 0; k < 9; ++k)
                if (((sub >> k) & 1u) && f.near_img[k] == i) reg = true;
        }
        if (!(xf < (float)F64_SPAT) && R2 > 0.0 && !reg) continue;   // beyond the cut
        const int ix = R2 > 0.0 ? min((int)xf, F64_SPAT) : 0;
        const double *c = blob + (F64_DEG + 1) * ix;
        const double v = R2 > 0.0 ? xu - (double)ix : 0.0;
        double val;
        if (reg) {
            // (F(x) - F(0)) / R of near pairs: the difference would lift the table's
            // rounding by F / (F - F(0)) (3e-14 of max|Z|), so F itself, as green_p
            const double R = R2 * ri, x = R * f.E;
            if (!(x >= 1e-6)) val = f.reg0;
            else val = ((ix == F64_SPAT ? 0.0 : exp(-x * x) * erfcx_c(cx<double>{x, f.bb}).re) - f.e_mb2) / R;
        } else {
            double s = c[F64_DEG];
#pragma unroll
            for (int n = F64_DEG - 1; n >= 0; --n) s = fma(s, v, c[n]);
            val = s * ri;
        }
        im.re = fma(val, R[2], im.re);
        im.im = fma(val, R[3], im.im);
    }
    gp = gp + im;
    // the spectral part at -d: conj(S) + j conj(T)
    if (PAIR) gm = {S.re + T.im + im.re, -S.im + T.re - im.im};
}

__device__ __forceinline__ void red2(double *Z, size_t idx, cx<double> v) {
    atomicAdd(Z + 2 * idx, v.re);
    atomicAdd(Z + 2 * idx + 1, v.im);
}

// the 16 entries of the ordered pair (test t, source s)
__device__ void scatter64(const DevMesh &m, const DevReq &q, double *Z, size_t N, int t, int s, const Mom<double> &mo) {
    const double *ft = m.far64 + 28 * (size_t)t, *fs = m.far64 + 28 * (size_t)s;
    const double k2 = q.k0 * q.k0;
    const cx<double> kap = {q.kap[2 * s], q.kap[2 * s + 1]};
    const cx<double> base = {9.0 * mo.S.re - k2 * mo.C.re, 9.0 * mo.S.im - k2 * mo.C.im};
    cx<double> A[4], F[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const double *w = fs + 15 + 3 * j;
        A[j] = k2 * (w[0] * mo.A[0] + w[1] * mo.A[1] + w[2] * mo.A[2]);
        F[j] = q.coef[4 * s + j] * (kap * cx<double>{q.wt[2 * (4 * s + j)], -q.wt[2 * (4 * s + j) + 1]});
    }
    for (int i = 0; i < 4; ++i) {
        const double *w = ft + 15 + 3 * i;
        const cx<double> P = base + k2 * (w[0] * mo.B[0] + w[1] * mo.B[1] + w[2] * mo.B[2]);
        const cx<double> E = q.coef[4 * t + i] * cx<double>{q.wt[2 * (4 * t + i)], q.wt[2 * (4 * t + i) + 1]};
        const size_t row = (size_t)q.row[4 * t + i];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const double *u = fs + 15 + 3 * j;
            cx<double> Q = P + A[j];
            cfma(Q, -k2 * (w[0] * u[0] + w[1] * u[1] + w[2] * u[2]), mo.S);
            red2(Z, row * N + (size_t)q.row[4 * s + j], E * (F[j] * Q));
        }
    }
}

__device__ __forceinline__ void stage64(const DevReq &q, double *blob) {
    for (int i = threadIdx.x; i < q.f64.n_blob; i += blockDim.x) blob[i] = q.blob64[i];
    __syncthreads();
}

// one thread per unordered pair {t, s}, s >= t
__global__ void __launch_bounds__(128) k_far_tt64(DevMesh m, const __grid_constant__ DevReq q, double *Z, size_t N) {
    extern __shared__ __align__(16) double blob[];
    const int t = blockIdx.y;
    if ((int)(blockIdx.x * blockDim.x + blockDim.x) <= t) return;   // the whole block is below the diagonal
    stage64(q, blob);
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= m.nt || s < t) return;
    const unsigned sub = m.mk_tt[(size_t)t * m.nt + s];
    const double *ft = m.far64 + 28 * (size_t)t, *fs = m.far64 + 28 * (size_t)s;
    Mom<double> mo, mr;   // blocks (t, s) and (s, t)
    mo.zero();
    mr.zero();
    for (int b = 0; b < 4; ++b) {
        const double *yb = fs + 3 * b;
        cx<double> z0 = {0, 0}, y0 = {0, 0}, zA[3], yA[3];
        for (int d = 0; d < 3; ++d) zA[d] = yA[d] = {0, 0};
        for (int a = 0; a < 4; ++a) {
            const double *xa = ft + 3 * a;
            cx<double> g, gr;
            green64<true>(q.f64, blob, xa[0] - yb[0], xa[1] - yb[1], xa[2] - yb[2], q.ph64 + 8 * (4 * (size_t)t + a),
                          q.ph64 + 8 * (4 * (size_t)s + b), sub, g, gr);
            z0 = z0 + g;
            y0 = y0 + gr;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                cfma(zA[d], xa[d] - ft[12 + d], g);
                cfma(yA[d], xa[d] - ft[12 + d], gr);
            }
        }
        mo.S = mo.S + z0;
        mr.S = mr.S + y0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {   // in the reversed block the test polynomial is s's
            const double r = yb[d] - fs[12 + d];
            mo.A[d] = mo.A[d] + zA[d];
            cfma(mo.B[d], r, z0);
            cfma(mo.C, r, zA[d]);
            mr.B[d] = mr.B[d] + yA[d];
            cfma(mr.A[d], r, y0);
            cfma(mr.C, r, yA[d]);
        }
    }
    const double w = ft[27] * fs[27];
    auto scale = [&](Mom<double> &M) {
        M.S = w * M.S;
        M.C = w * M.C;
        for (int d = 0; d < 3; ++d) { M.A[d] = w * M.A[d]; M.B[d] = w * M.B[d]; }
    };
    scale(mo);
    scatter64(m, q, Z, N, t, s, mo);
    if (s != t) {
        scale(mr);
        scatter64(m, q, Z, N, s, t, mr);
    }
}

// pairs with charge faces, kinds as k_far_scalar_p (far.cu)
template <int PK>
__global__ void __launch_bounds__(128) k_far_scalar64(DevMesh m, const __grid_constant__ DevReq q, double *Z, size_t N, int ny,
                                                      const uint16_t *mk) {
    extern __shared__ __align__(16) double blob[];
    constexpr bool XT = PK == 0, YT = PK == 1;
    constexpr int qx = XT ? 4 : 3, qy = YT ? 4 : 3;
    stage64(q, blob);
    const int x = blockIdx.y, y = blockIdx.x * blockDim.x + threadIdx.x;
    if (y >= ny) return;
    const int xe = XT ? x : m.hf[x];
    const unsigned sub = mk[(size_t)x * ny + y];
    const double *fx = XT ? m.far64 + 28 * (size_t)xe : m.ffar64 + 12 * (size_t)xe;
    const double *fy = YT ? m.far64 + 28 * (size_t)y : m.ffar64 + 12 * (size_t)y;
    const double *px = q.ph64 + 8 * (XT ? 4 * (size_t)xe : 4 * (size_t)m.nt + 3 * (size_t)xe);
    const double *py = q.ph64 + 8 * (YT ? 4 * (size_t)y : 4 * (size_t)m.nt + 3 * (size_t)y);
    cx<double> S = {0, 0};
    for (int b = 0; b < qy; ++b)
        for (int a = 0; a < qx; ++a) {
            cx<double> g, unused;
            green64<false>(q.f64, blob, fx[3 * a] - fy[3 * b], fx[3 * a + 1] - fy[3 * b + 1], fx[3 * a + 2] - fy[3 * b + 2],
                           px + 8 * a, py + 8 * b, sub, g, unused);
            S = S + g;
        }
    S = (fx[XT ? 27 : 9] * fy[YT ? 27 : 9]) * S;
    if constexpr (PK == 0) {
        const cx<double> qS = cx<double>{q.qs[2 * y], q.qs[2 * y + 1]} * S;
        const size_t col = (size_t)q.frow[y];
        for (int i = 0; i < 4; ++i)
            red2(Z, (size_t)q.row[4 * x + i] * N + col,
                 (3.0 * q.coef[4 * x + i]) * (cx<double>{q.wt[2 * (4 * x + i)], q.wt[2 * (4 * x + i) + 1]} * qS));
    } else if constexpr (PK == 1) {
        const size_t row = (size_t)q.frow[xe];
        const cx<double> kS = cx<double>{q.kap[2 * y], q.kap[2 * y + 1]} * S;
        for (int j = 0; j < 4; ++j)
            red2(Z, row * N + (size_t)q.row[4 * y + j],
                 (-3.0 * q.coef[4 * y + j]) * (cx<double>{q.wt[2 * (4 * y + j)], -q.wt[2 * (4 * y + j) + 1]} * kS));
    } else {
        red2(Z, (size_t)q.frow[xe] * N + (size_t)q.frow[y], -1.0 * (cx<double>{q.qs[2 * y], q.qs[2 * y + 1]} * S));
    }
}

}  // namespace

cudaError_t upload_far64_constants(const void *weideman) { return cudaMemcpyToSymbol(c_weid, weideman, sizeof(WeidemanTables)); }
cudaError_t launch_far64_prep(const DevMesh &m, const DevReq &q, cudaStream_t st) {
    k_prep64<<<(4 * m.nt + 3 * m.nf + 127) / 128, 128, 0, st>>>(m, q); ++g_launches;
    return cudaGetLastError();
}
cudaError_t launch_far64_tt(const DevMesh &m, const DevReq &q, double *Z, size_t N, cudaStream_t st) {
    k_far_tt64<<<dim3((m.nt + 127) / 128, m.nt), 128, sizeof(double) * q.f64.n_blob, st>>>(m, q, Z, N); ++g_launches;
    return cudaGetLastError();
}
cudaError_t launch_far64_scalar(int pk, const DevMesh &m, const DevReq &q, double *Z, size_t N, cudaStream_t st) {
    const int nx = pk == 0 ? m.nt : m.nh, ny = pk == 1 ? m.nt : m.nf;
    const uint16_t *mk = pk == 0 ? m.mk_tf : (pk == 1 ? m.mk_ft : m.mk_ff);
    const dim3 grid((ny + 127) / 128, nx);
    const size_t sm = sizeof(double) * q.f64.n_blob;
    if (pk == 0) k_far_scalar64<0><<<grid, 128, sm, st>>>(m, q, Z, N, ny, mk);
    else if (pk == 1) k_far_scalar64<1><<<grid, 128, sm, st>>>(m, q, Z, N, ny, mk);
    else k_far_scalar64<2><<<grid, 128, sm, st>>>(m, q, Z, N, ny, mk);
    ++g_launches;
    return cudaGetLastError();
}

}  // namespace vie
