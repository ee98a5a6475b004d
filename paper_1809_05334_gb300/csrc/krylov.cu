// Vector kernels of the block GMRES iteration (declared in linalg.h): TE and TM
// span one Krylov space, basis blocks of two columns.  One iteration is
//   matvec_rinv, the preconditioner's stages, dots, subtract, dots, subtract
// with no host wait in it: the coefficients, the Gram matrix and its Cholesky
// factor are formed by the last CTA of the kernel that completes their sums, and
// the last kernel sends the new column of the Hessenberg matrix to pinned host
// memory, where the host reads it while the next iteration runs.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "linalg.h"

namespace vie {

namespace {

// layout of the state (m = restart length)
struct State {
    double *dots;      // [2][m + 1][8]: raw w_j^H w, (a, p) = column a of w_j, column p of w: re, im at 4 a + 2 p
    double *gram;      // [2][4]: |c0|^2, |c1|^2, conj(c0) c1 (re, im)
    unsigned *count;   // [4] CTAs done: dots pass 0, 1, subtract pass 0, 1
    float *coef;       // [m + 1][8]: C_j, as dots
    float *ginv;       // [m + 2][4]: inverse Gram of block j
    float *rinv;       // [m + 2][4]: inverse Cholesky factor of block j
    float *applied;    // [2][m + 1][8]: coefficients of both passes, for the message
    float *tt;         // [2]: the coefficient that took column 0 out of column 1
};
__host__ __device__ inline State view(void *p, int m) {
    State s;
    const size_t k = m + 2;
    s.dots = static_cast<double *>(p);
    s.gram = s.dots + 16 * k;
    s.count = reinterpret_cast<unsigned *>(s.gram + 8);
    s.coef = reinterpret_cast<float *>(s.count + 4);
    s.ginv = s.coef + 8 * k;
    s.rinv = s.ginv + 4 * k;
    s.applied = s.rinv + 4 * k;
    s.tt = s.applied + 16 * k;
    return s;
}

// unevaluated sums S + C (TwoSum): the warp reductions keep more than FP32 without
// the FP64 pipe (1/64 of the FP32 rate)
struct DF {
    float s, c;
};
__device__ __forceinline__ DF df_add(DF a, DF b) {
    const float t = __fadd_rn(a.s, b.s), bp = __fsub_rn(t, a.s);
    const float e = __fadd_rn(__fsub_rn(a.s, __fsub_rn(t, bp)), __fsub_rn(b.s, bp));
    return {t, __fadd_rn(e, __fadd_rn(a.c, b.c))};
}
__device__ __forceinline__ DF df_xor(DF v, int o) {
    return {__shfl_xor_sync(0xffffffffu, v.s, o), __shfl_xor_sync(0xffffffffu, v.c, o)};
}

// true in every thread of the CTA that finishes last; *count ends at zero
__device__ __forceinline__ bool last_cta(unsigned *count, unsigned total) {
    __shared__ unsigned last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(count, 1u) == total - 1 ? 1u : 0u;
        if (last) *count = 0u;
    }
    __syncthreads();
    if (last) __threadfence();
    return last != 0u;
}

}  // namespace

size_t block_state_bytes(int m) {
    State s = view(nullptr, m);
    return reinterpret_cast<size_t>(s.tt + 2) + 64;
}
size_t block_message_doubles(int m) { return 16 * (size_t)(m + 1) + 8 + 2; }
const float *block_rinv(void *state, int m, int j) { return view(state, m).rinv + 4 * (size_t)j; }

// ---------------------------------------------------------------------------
// dots: grid (row chunks) x (groups of basis blocks); a CTA keeps its 1024 rows
// of w in registers and walks its basis blocks (read once; all of V stays in L2
// for the usual restart lengths).  Per thread FP32 over 4 rows, then compensated
// across the warp, FP64 across warps and CTAs.
// ---------------------------------------------------------------------------
constexpr int BD_ROWS = 4;
constexpr int BD_CHUNK = 256 * BD_ROWS;

__global__ void __launch_bounds__(256) k_bdots(const float *V, size_t vstride, int nv, const float *w, int n, int m,
                                               void *state, int pass) {
    __shared__ DF red[2][8][8];
    State S = view(state, m);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
    const int base = blockIdx.x * BD_CHUNK + threadIdx.x;
    float4 x[BD_ROWS];
#pragma unroll
    for (int u = 0; u < BD_ROWS; ++u) {
        const int i = base + 256 * u;
        x[u] = i < n ? *reinterpret_cast<const float4 *>(w + 4 * (size_t)i) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    int buf = 0;
    for (int j = blockIdx.y; j < nv; j += gridDim.y, buf ^= 1) {
        const float *v = V + (size_t)j * vstride;
        float a[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int u = 0; u < BD_ROWS; ++u) {
            const int i = base + 256 * u;
            if (i >= n) continue;
            const float4 b = *reinterpret_cast<const float4 *>(v + 4 * (size_t)i);
            const float vr[2] = {b.x, b.z}, vi[2] = {b.y, b.w}, xr[2] = {x[u].x, x[u].z}, xi[2] = {x[u].y, x[u].w};
#pragma unroll
            for (int c = 0; c < 2; ++c)
#pragma unroll
                for (int p = 0; p < 2; ++p) {   // conj(v) x
                    a[4 * c + 2 * p] = fmaf(vr[c], xr[p], fmaf(vi[c], xi[p], a[4 * c + 2 * p]));
                    a[4 * c + 2 * p + 1] = fmaf(vr[c], xi[p], fmaf(-vi[c], xr[p], a[4 * c + 2 * p + 1]));
                }
        }
        // eight sums over 32 lanes: halve the values per lane three times, then two more steps
        DF d[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) d[k] = {a[k], 0.f};
#pragma unroll
        for (int o = 16, k = 4; k >= 1; o >>= 1, k >>= 1) {
            const bool hi = lane & o;
#pragma unroll
            for (int q = 0; q < k; ++q) {
                const DF keep = hi ? d[q + k] : d[q], give = hi ? d[q] : d[q + k];
                d[q] = df_add(keep, df_xor(give, o));
            }
        }
        d[0] = df_add(d[0], df_xor(d[0], 2));
        d[0] = df_add(d[0], df_xor(d[0], 1));
        // lane 4 q holds value: bits 16, 8, 4 of the lane select 4, 2, 1
        if ((lane & 3) == 0) red[buf][warp][((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)] = d[0];
        __syncthreads();
        if (threadIdx.x < 8) {
            double s = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) s += (double)red[buf][q][threadIdx.x].s + (double)red[buf][q][threadIdx.x].c;
            atomicAdd(S.dots + 8 * ((size_t)pass * (m + 1) + j) + threadIdx.x, s);
        }
    }
    if (!last_cta(S.count + pass, gridDim.x * gridDim.y)) return;
    // C_j = Ginv_j D_j; the sums go back to zero
    for (int j = threadIdx.x; j < nv; j += blockDim.x) {
        double *D = S.dots + 8 * ((size_t)pass * (m + 1) + j);
        float d[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            d[k] = (float)__ldcg(D + k);
            D[k] = 0.0;
        }
        const float4 g = *reinterpret_cast<const float4 *>(S.ginv + 4 * (size_t)j);   // a, b, c: [[a, c], [conj(c), b]]
        float c[8];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            const float r0 = d[2 * p], i0 = d[2 * p + 1], r1 = d[4 + 2 * p], i1 = d[4 + 2 * p + 1];
            c[2 * p] = g.x * r0 + (g.z * r1 - g.w * i1);
            c[2 * p + 1] = g.x * i0 + (g.z * i1 + g.w * r1);
            c[4 + 2 * p] = g.y * r1 + (g.z * r0 + g.w * i0);
            c[4 + 2 * p + 1] = g.y * i1 + (g.z * i0 - g.w * r0);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            S.coef[8 * (size_t)j + k] = c[k];
            S.applied[8 * ((size_t)pass * (m + 1) + j) + k] = c[k];
        }
    }
}

// ---------------------------------------------------------------------------
// subtract: 32 rows per CTA (one per lane), the 8 warps split the basis blocks
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_bsub(const float *V, size_t vstride, int nv, float *w, int n, int m, void *state,
                                              int pass, double *message, unsigned long long seq) {
    __shared__ float4 part[8][32];
    State S = view(state, m);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i = blockIdx.x * 32 + lane;
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < n) {
#pragma unroll 4
        for (int j = warp; j < nv; j += 8) {
            const float4 v = *reinterpret_cast<const float4 *>(V + (size_t)j * vstride + 4 * (size_t)i);
            const float4 c0 = *reinterpret_cast<const float4 *>(S.coef + 8 * (size_t)j);        // column 0 of w_j
            const float4 c1 = *reinterpret_cast<const float4 *>(S.coef + 8 * (size_t)j + 4);    // column 1
            s.x = fmaf(v.x, c0.x, fmaf(-v.y, c0.y, fmaf(v.z, c1.x, fmaf(-v.w, c1.y, s.x))));
            s.y = fmaf(v.x, c0.y, fmaf(v.y, c0.x, fmaf(v.z, c1.y, fmaf(v.w, c1.x, s.y))));
            s.z = fmaf(v.x, c0.z, fmaf(-v.y, c0.w, fmaf(v.z, c1.z, fmaf(-v.w, c1.w, s.z))));
            s.w = fmaf(v.x, c0.w, fmaf(v.y, c0.z, fmaf(v.z, c1.w, fmaf(v.w, c1.z, s.w))));
        }
    }
    part[warp][lane] = s;
    __syncthreads();
    if (warp == 0) {
        float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i < n) {
            float4 t = part[0][lane];
#pragma unroll
            for (int q = 1; q < 8; ++q) {
                const float4 u = part[q][lane];
                t.x += u.x; t.y += u.y; t.z += u.z; t.w += u.w;
            }
            float4 *o = reinterpret_cast<float4 *>(w + 4 * (size_t)i);
            c = *o;
            c.x -= t.x; c.y -= t.y; c.z -= t.z; c.w -= t.w;
            if (pass == 1) {   // column 1 -= column 0 t
                const float tr = S.tt[0], ti = S.tt[1];
                c.z -= c.x * tr - c.y * ti;
                c.w -= c.x * ti + c.y * tr;
            }
            *o = c;
        }
        DF g[4] = {{c.x * c.x, 0.f}, {c.z * c.z, 0.f}, {c.x * c.z, 0.f}, {c.x * c.w, 0.f}};
        g[0] = df_add(g[0], {c.y * c.y, 0.f});
        g[1] = df_add(g[1], {c.w * c.w, 0.f});
        g[2] = df_add(g[2], {c.y * c.w, 0.f});
        g[3] = df_add(g[3], {-c.y * c.z, 0.f});
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) g[k] = df_add(g[k], df_xor(g[k], o));
        if (lane < 4) {
            const DF v = lane == 0 ? g[0] : (lane == 1 ? g[1] : (lane == 2 ? g[2] : g[3]));
            atomicAdd(S.gram + 4 * pass + lane, (double)v.s + (double)v.c);
        }
    }
    if (!last_cta(S.count + 2 + pass, gridDim.x)) return;
    double *G = S.gram + 4 * pass;
    if (pass == 0) {
        if (threadIdx.x == 0) {   // t = conj(c0) c1 / |c0|^2
            const double g11 = __ldcg(G), inv = g11 > 0.0 ? 1.0 / g11 : 0.0;
            S.tt[0] = (float)(__ldcg(G + 2) * inv);
            S.tt[1] = (float)(__ldcg(G + 3) * inv);
        }
        return;
    }
    // the message: coefficients as applied, Gram of this pass, t; then its sequence number
    double *msg = message;
    for (int k = threadIdx.x; k < 8 * nv; k += blockDim.x) {
        msg[k] = (double)S.applied[k];
        msg[8 * (size_t)(m + 1) + k] = (double)S.applied[8 * (size_t)(m + 1) + k];
    }
    double *tail = msg + 16 * (size_t)(m + 1);
    if (threadIdx.x < 4) tail[threadIdx.x] = __ldcg(G + threadIdx.x);
    if (threadIdx.x < 2) tail[4 + threadIdx.x] = (double)S.tt[threadIdx.x];
    __threadfence_system();
    __syncthreads();
    if (threadIdx.x == 0) {
        const double g11 = __ldcg(G), g22 = __ldcg(G + 1), cr = __ldcg(G + 2), ci = __ldcg(G + 3);
        // Cholesky of [[g11, c], [conj(c), g22]]: r11, r12 = c / r11, r22; a zero column stays zero
        const double i11 = g11 > 0.0 ? rsqrt(g11) : 0.0;
        const double sr = cr * i11, si = ci * i11;
        const double d22 = g22 - (sr * sr + si * si);
        const double i22 = d22 > 1e-12 * g22 ? rsqrt(d22) : 0.0;
        // R^-1 = [[i11, -r12 i11 i22], [0, i22]]
        const double tr = -sr * i11 * i22, ti = -si * i11 * i22;
        float *R = S.rinv + 4 * (size_t)nv, *I = S.ginv + 4 * (size_t)nv;
        R[0] = (float)i11; R[1] = (float)tr; R[2] = (float)ti; R[3] = (float)i22;
        // G^-1 = R^-1 R^-H
        I[0] = (float)(i11 * i11 + tr * tr + ti * ti);
        I[1] = (float)(i22 * i22);
        I[2] = (float)(tr * i22);
        I[3] = (float)(ti * i22);
#pragma unroll
        for (int k = 0; k < 8; ++k) S.gram[k] = 0.0;
        __threadfence_system();
        *reinterpret_cast<volatile unsigned long long *>(tail + 8) = seq;
    }
}

__global__ void k_bcombine(const float *V, size_t vstride, int nv, const double *Y, double *x, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double s[4] = {0, 0, 0, 0};
    for (int j = 0; j < nv; ++j) {
        const float4 v = *reinterpret_cast<const float4 *>(V + (size_t)j * vstride + 4 * (size_t)i);
        const double *c = Y + 8 * (size_t)j;
#pragma unroll
        for (int p = 0; p < 2; ++p) {
            s[2 * p] += double(v.x) * c[2 * p] - double(v.y) * c[2 * p + 1] + double(v.z) * c[4 + 2 * p] - double(v.w) * c[4 + 2 * p + 1];
            s[2 * p + 1] += double(v.x) * c[2 * p + 1] + double(v.y) * c[2 * p] + double(v.z) * c[4 + 2 * p + 1] + double(v.w) * c[4 + 2 * p];
        }
    }
    double *o = x + 4 * (size_t)i;
#pragma unroll
    for (int k = 0; k < 4; ++k) o[k] += s[k];
}

cudaError_t block_dots(const float *V, size_t vstride, int nv, const float *w, int n, int m, void *state, int pass,
                       cudaStream_t st) {
    if (nv <= 0) return cudaSuccess;
    const int gx = (n + BD_CHUNK - 1) / BD_CHUNK;
    const int gy = std::max(1, std::min(nv, 608 / gx));   // about four CTAs per SM
    return launch_pdl(k_bdots, dim3(gx, gy), 256, st, V, vstride, nv, w, n, m, state, pass);
}
cudaError_t block_subtract(const float *V, size_t vstride, int nv, float *w, int n, int m, void *state, int pass,
                           double *message, unsigned long long seq, cudaStream_t st) {
    return launch_pdl(k_bsub, dim3((n + 31) / 32), 256, st, V, vstride, nv, w, n, m, state, pass, message, seq);
}
cudaError_t block_combine(const float *V, size_t vstride, int nv, const double *Y, double *x, int n, cudaStream_t st) {
    k_bcombine<<<(n + 127) / 128, 128, 0, st>>>(V, vstride, nv, Y, x, n); ++g_launches;
    return cudaGetLastError();
}

}  // namespace vie
