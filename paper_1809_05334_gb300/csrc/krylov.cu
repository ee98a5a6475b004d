// Vector kernels of the GMRES iteration of the mixed paths (declared in linalg.h): TE
// and TM advance together, one Krylov space each, a basis vector of both stored as
// one [n][2] complex vector.  One iteration is
//   matvec_norm, the preconditioner's stages, dots, subtract, dots, subtract
// with no host wait in it: the coefficients are formed by the last CTA of the
// kernel that completes their sums, the norms of the new vector by the last CTA of the
// second subtraction, which sends the new column of the Hessenberg matrices to pinned
// host memory, where the host reads it while the next iteration runs.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "linalg.h"

namespace vie {

namespace {

// layout of the state (m = restart length)
struct State {
    double *dots;      // [2][m + 1][4]: raw w_j^H w of both passes, per right-hand side (re, im)
    double *norm2;     // [2]: |w|^2 of the new vector
    double *ginv;      // [m + 2][2]: 1 / |w_j|^2 (0 for a zero vector)
    unsigned *count;   // [4] CTAs done: dots pass 0, 1, subtract pass 1
    float *coef;       // [m + 1][4]: C_j of the pass under way, as dots
    float *applied;    // [2][m + 1][4]: coefficients of both passes, for the message
    float *rinv;       // [m + 2][2]: 1 / |w_j|
};
__host__ __device__ inline State view(void *p, int m) {
    State s;
    const size_t k = m + 2;
    s.dots = static_cast<double *>(p);
    s.norm2 = s.dots + 8 * k;
    s.ginv = s.norm2 + 2;
    s.count = reinterpret_cast<unsigned *>(s.ginv + 2 * k);
    s.coef = reinterpret_cast<float *>(s.count + 4);
    s.applied = s.coef + 4 * k;
    s.rinv = s.applied + 8 * k;
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

size_t krylov_state_bytes(int m) {
    State s = view(nullptr, m);
    return reinterpret_cast<size_t>(s.rinv + 2 * (m + 2)) + 64;
}
size_t krylov_message_doubles(int m) { return 8 * (size_t)(m + 1) + 4 + 4; }
const float *krylov_rinv(void *state, int m, int j) { return view(state, m).rinv + 2 * (size_t)j; }

// ---------------------------------------------------------------------------
// dots: grid (row chunks) x (groups of basis vectors); a CTA keeps its 1024 rows
// of w in registers and walks its basis vectors (read once; all of V stays in L2
// for the usual restart lengths).  Per thread FP32 over 4 rows, then compensated
// across the warp, FP64 across warps and CTAs.
// ---------------------------------------------------------------------------
constexpr int KD_ROWS = 4;
constexpr int KD_CHUNK = 256 * KD_ROWS;

__global__ void __launch_bounds__(256) k_kdots(const float *V, size_t vstride, int nv, const float *w, int n, int m,
                                               void *state, int pass) {
    __shared__ DF red[2][8][4];
    State S = view(state, m);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
    const int base = blockIdx.x * KD_CHUNK + threadIdx.x;
    float4 x[KD_ROWS];
#pragma unroll
    for (int u = 0; u < KD_ROWS; ++u) {
        const int i = base + 256 * u;
        x[u] = i < n ? *reinterpret_cast<const float4 *>(w + 4 * (size_t)i) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    int buf = 0;
    for (int j = blockIdx.y; j < nv; j += gridDim.y, buf ^= 1) {
        const float *v = V + (size_t)j * vstride;
        float a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int u = 0; u < KD_ROWS; ++u) {
            const int i = base + 256 * u;
            if (i >= n) continue;
            const float4 b = *reinterpret_cast<const float4 *>(v + 4 * (size_t)i);
            // conj(v) x
            a[0] = fmaf(b.x, x[u].x, fmaf(b.y, x[u].y, a[0]));
            a[1] = fmaf(b.x, x[u].y, fmaf(-b.y, x[u].x, a[1]));
            a[2] = fmaf(b.z, x[u].z, fmaf(b.w, x[u].w, a[2]));
            a[3] = fmaf(b.z, x[u].w, fmaf(-b.w, x[u].z, a[3]));
        }
        // four sums over 32 lanes: halve the values per lane twice, then three more steps
        DF d[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) d[k] = {a[k], 0.f};
#pragma unroll
        for (int o = 16, k = 2; k >= 1; o >>= 1, k >>= 1) {
            const bool hi = lane & o;
#pragma unroll
            for (int q = 0; q < k; ++q) {
                const DF keep = hi ? d[q + k] : d[q], give = hi ? d[q] : d[q + k];
                d[q] = df_add(keep, df_xor(give, o));
            }
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) d[0] = df_add(d[0], df_xor(d[0], o));
        // lane 8 q holds value: bits 16, 8 of the lane select 2, 1
        if ((lane & 7) == 0) red[buf][warp][lane >> 3] = d[0];
        __syncthreads();
        if (threadIdx.x < 4) {
            double s = 0;
#pragma unroll
            for (int q = 0; q < 8; ++q) s += (double)red[buf][q][threadIdx.x].s + (double)red[buf][q][threadIdx.x].c;
            atomicAdd(S.dots + 4 * ((size_t)pass * (m + 1) + j) + threadIdx.x, s);
        }
    }
    if (!last_cta(S.count + pass, gridDim.x * gridDim.y)) return;
    // C_j = D_j / |w_j|^2; the sums go back to zero
    for (int e = threadIdx.x; e < 4 * nv; e += blockDim.x) {
        double *D = S.dots + 4 * (size_t)pass * (m + 1) + e;
        const float c = (float)(__ldcg(D) * S.ginv[e >> 1]);   // e >> 1: vector e / 4, right-hand side (e / 2) % 2
        *D = 0.0;
        S.coef[e] = c;
        S.applied[4 * (size_t)pass * (m + 1) + e] = c;
    }
}

// ---------------------------------------------------------------------------
// subtract: 32 rows per CTA (one per lane), the 8 warps split the basis vectors
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_ksub(const float *V, size_t vstride, int nv, float *w, int n, int m, void *state,
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
            const float4 c = *reinterpret_cast<const float4 *>(S.coef + 4 * (size_t)j);
            s.x = fmaf(v.x, c.x, fmaf(-v.y, c.y, s.x));
            s.y = fmaf(v.x, c.y, fmaf(v.y, c.x, s.y));
            s.z = fmaf(v.z, c.z, fmaf(-v.w, c.w, s.z));
            s.w = fmaf(v.z, c.w, fmaf(v.w, c.z, s.w));
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
            *o = c;
        }
        if (pass == 1) {
            DF g[2] = {{c.x * c.x, 0.f}, {c.z * c.z, 0.f}};
            g[0] = df_add(g[0], {c.y * c.y, 0.f});
            g[1] = df_add(g[1], {c.w * c.w, 0.f});
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) g[k] = df_add(g[k], df_xor(g[k], o));
            if (lane < 2) {
                const DF v = lane == 0 ? g[0] : g[1];
                atomicAdd(S.norm2 + lane, (double)v.s + (double)v.c);
            }
        }
    }
    if (pass == 0 || !last_cta(S.count + 2, gridDim.x)) return;
    // the message: coefficients as applied, squared norms and 1 / norm as the next product
    // takes it; then its sequence number
    for (int k = threadIdx.x; k < 4 * nv; k += blockDim.x) {
        message[k] = (double)S.applied[k];
        message[4 * (size_t)(m + 1) + k] = (double)S.applied[4 * (size_t)(m + 1) + k];
    }
    double *tail = message + 8 * (size_t)(m + 1);
    if (threadIdx.x < 2) {
        const double g = __ldcg(S.norm2 + threadIdx.x);
        const float r = g > 0.0 ? (float)rsqrt(g) : 0.f;
        S.rinv[2 * (size_t)nv + threadIdx.x] = r;
        S.ginv[2 * (size_t)nv + threadIdx.x] = g > 0.0 ? 1.0 / g : 0.0;
        S.norm2[threadIdx.x] = 0.0;
        tail[threadIdx.x] = g;
        tail[2 + threadIdx.x] = (double)r;
    }
    __threadfence_system();
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence_system();
        *reinterpret_cast<volatile unsigned long long *>(tail + 4) = seq;
    }
}

cudaError_t krylov_dots(const float *V, size_t vstride, int nv, const float *w, int n, int m, void *state, int pass,
                        cudaStream_t st) {
    if (nv <= 0) return cudaSuccess;
    const int gx = (n + KD_CHUNK - 1) / KD_CHUNK;
    const int gy = std::max(1, std::min(nv, 608 / gx));   // about four CTAs per SM
    return launch_pdl(k_kdots, dim3(gx, gy), 256, st, V, vstride, nv, w, n, m, state, pass);
}
cudaError_t krylov_subtract(const float *V, size_t vstride, int nv, float *w, int n, int m, void *state, int pass,
                            double *message, unsigned long long seq, cudaStream_t st) {
    return launch_pdl(k_ksub, dim3((n + 31) / 32), 256, st, V, vstride, nv, w, n, m, state, pass, message, seq);
}

}  // namespace vie
