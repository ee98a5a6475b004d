// Near-pair lists of a mesh on the device (the criterion and the order of the
// entries are those of build_topology, csrc/topology.cpp): for every element pair
// the 9-bit mask of its near lattice images, and the (pair, image) entry lists of
// the elements that do not touch and of those that do, sorted by x, y, image.
//
// One CTA per x.  The first pass writes the dense mask row and counts; after a
// scan of the counts the second pass emits the entries in order (an ordered block
// scan per 256 y).  Distances are compared in FP64; an FP32 test with a margin for
// its own rounding decides most of the nine images without it (the FP64 pipe runs
// at 1/64 of the FP32 rate).  The host built the same lists with OpenMP, packed
// the dense masks and uploaded both (40 MB of masks and 200 MB of entries at 10,368
// tetrahedra).  vie_set_mesh with the static integrals: 103 -> 12 ms at 3,072
// tetrahedra, 545 -> 41 at 10,368, 1,350 -> 95 at 23,940.
#include <cuda_runtime.h>

#include <algorithm>

#include "fill.h"
#include "mesh.h"

namespace vie {

namespace {

struct NearArgs {
    ElementSet x, y;
    double a, b, tol;
    float slack;       // bound on the FP32 rounding of a coordinate difference
};

// Bits of the near images of (i, j).
__device__ __forceinline__ unsigned near_mask(const NearArgs &g, int i, int j) {
    const double *cx = g.x.cen + 3 * (size_t)i, *cy = g.y.cen + 3 * (size_t)j;
    const float rf = (float)(g.x.rad[i] + g.y.rad[j]);
    const float limf = (float)NEAR_FACTOR * rf * 1.0001f + 2.f * g.slack;
    const float fx = (float)cx[0] - (float)cy[0], fy = (float)cx[1] - (float)cy[1], fz = (float)cx[2] - (float)cy[2];
    const float af = (float)g.a, bf = (float)g.b;
    unsigned cand = 0u;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const float dx = fx + (float)(k / 3 - 1) * af, dy = fy + (float)(k % 3 - 1) * bf;
        if (dx * dx + dy * dy + fz * fz <= limf * limf) cand |= 1u << k;
    }
    if (!cand) return 0u;
    const double lim = NEAR_FACTOR * (g.x.rad[i] + g.y.rad[j]) * (1.0 + NEAR_MARGIN);
    const double d0 = cx[0] - cy[0], d1 = cx[1] - cy[1], d2 = cx[2] - cy[2];
    unsigned mask = 0u;
    for (unsigned c = cand; c; c &= c - 1u) {
        const int k = __ffs((int)c) - 1;
        const double e0 = d0 + (k / 3 - 1) * g.a, e1 = d1 + (k % 3 - 1) * g.b;
        if (sqrt(e0 * e0 + e1 * e1 + d2 * d2) < lim) mask |= 1u << k;
    }
    return mask;
}

// Of the near images `mask` of (i, j), those in which the elements share a vertex.  Both
// passes call it with the stored mask, the first to count the entries of a list, the
// second to write them, so the same bits have to come out: every operation is rounded by
// itself (nothing that the compiler may contract in one kernel and not in the other).
__device__ __forceinline__ unsigned touch_mask(const NearArgs &g, int i, int j, unsigned mask) {
    const double tol2 = __dmul_rn(g.tol, g.tol);
    // centroids further apart than both radii (FP32, with a margin for its rounding): no shared vertex
    const double *cx = g.x.cen + 3 * (size_t)i, *cy = g.y.cen + 3 * (size_t)j;
    const float rf = __fadd_rn((float)g.x.rad[i], (float)g.y.rad[j]);
    const float lim = __fadd_rn(__fmul_rn(rf, 1.0001f), __fmul_rn(2.f, g.slack)), lim2 = __fmul_rn(lim, lim);
    const float fx = __fsub_rn((float)cx[0], (float)cy[0]), fy = __fsub_rn((float)cx[1], (float)cy[1]),
                fz = __fsub_rn((float)cx[2], (float)cy[2]);
    unsigned touch = 0u;
    for (unsigned c = mask; c; c &= c - 1u) {
        const int k = __ffs((int)c) - 1;
        const float dx = __fadd_rn(fx, __fmul_rn((float)(k / 3 - 1), (float)g.a)),
                    dy = __fadd_rn(fy, __fmul_rn((float)(k % 3 - 1), (float)g.b));
        if (__fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(fz, fz)) > lim2) continue;
        const double R0 = __dmul_rn((double)(k / 3 - 1), g.a), R1 = __dmul_rn((double)(k % 3 - 1), g.b);
        bool t = false;
        for (int p = 0; p < g.x.kv && !t; ++p) {
            const double *u = g.x.verts + 3 * ((size_t)g.x.kv * i + p);
            for (int q = 0; q < g.y.kv; ++q) {
                const double *v = g.y.verts + 3 * ((size_t)g.y.kv * j + q);
                const double x = __dsub_rn(u[0], __dsub_rn(v[0], R0));
                if (fabs(x) >= g.tol) continue;
                const double y = __dsub_rn(u[1], __dsub_rn(v[1], R1)), z = __dsub_rn(u[2], v[2]);
                if (__dadd_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)), __dmul_rn(z, z)) < tol2) { t = true; break; }
            }
        }
        if (t) touch |= 1u << k;
    }
    return touch;
}

// exclusive ordered scan over the 256 threads of a CTA of two counts packed in one
// 64-bit word; *total: the CTA's sum
__device__ __forceinline__ unsigned long long block_scan(unsigned long long v, unsigned long long *total) {
    __shared__ unsigned long long warp_sum[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long s = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long u = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += u;
    }
    __syncthreads();
    if (lane == 31) warp_sum[warp] = s;
    __syncthreads();
    unsigned long long before = 0, all = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        if (q < warp) before += warp_sum[q];
        all += warp_sum[q];
    }
    *total = all;
    return before + s - v;
}

// EMIT 0: masks and counts [3][nx] (not touching, touching, near pairs); 1: entries
template <bool EMIT>
__global__ void __launch_bounds__(256) k_near(NearArgs g, uint16_t *mk, unsigned *counts, const unsigned *offsets,
                                              NearEntry *pr, NearEntry *to) {
    const int i = blockIdx.x, nx = g.x.n, ny = g.y.n;
    unsigned long long done = EMIT ? ((unsigned long long)offsets[nx + i] << 32) | offsets[i] : 0ull;
    unsigned n_pr = 0, n_to = 0, n_pair = 0;
    for (int j0 = 0; j0 < ny; j0 += 256) {
        const int j = j0 + threadIdx.x;
        unsigned mask = 0u, touch = 0u;
        if (j < ny) mask = EMIT ? (unsigned)mk[(size_t)i * ny + j] : near_mask(g, i, j);
        if (mask) touch = touch_mask(g, i, j, mask);
        if (!EMIT) {
            if (j < ny) mk[(size_t)i * ny + j] = (uint16_t)mask;
            n_pr += __popc(mask & ~touch);
            n_to += __popc(touch);
            n_pair += mask ? 1u : 0u;
        } else {
            unsigned long long total;
            const unsigned long long at = block_scan(((unsigned long long)__popc(touch) << 32) | __popc(mask & ~touch), &total);
            unsigned a = (unsigned)(done + at), b = (unsigned)((done + at) >> 32);
            for (unsigned c = mask; c; c &= c - 1u) {
                const int k = __ffs((int)c) - 1;
                const NearEntry e = {i, j, k, 0};
                if ((touch >> k) & 1u) to[b++] = e;
                else pr[a++] = e;
            }
            done += total;
        }
    }
    if (!EMIT) {
        for (int o = 16; o > 0; o >>= 1) {
            n_pr += __shfl_down_sync(0xffffffffu, n_pr, o);
            n_to += __shfl_down_sync(0xffffffffu, n_to, o);
            n_pair += __shfl_down_sync(0xffffffffu, n_pair, o);
        }
        __shared__ unsigned s[3][8];
        if ((threadIdx.x & 31) == 0) {
            s[0][threadIdx.x >> 5] = n_pr;
            s[1][threadIdx.x >> 5] = n_to;
            s[2][threadIdx.x >> 5] = n_pair;
        }
        __syncthreads();
        if (threadIdx.x < 3) {
            unsigned t = 0;
            for (int q = 0; q < 8; ++q) t += s[threadIdx.x][q];
            counts[(size_t)threadIdx.x * nx + i] = t;
        }
    }
}

// exclusive scan of the three count rows [3][nx] into offsets [3][nx], totals [3] behind them
__global__ void __launch_bounds__(256) k_scan_counts(const unsigned *counts, int nx, unsigned *offsets) {
    for (int r = 0; r < 3; ++r) {
        unsigned long long done = 0;
        for (int i0 = 0; i0 < nx; i0 += 256) {
            const int i = i0 + threadIdx.x;
            unsigned long long total;
            const unsigned long long at = block_scan(i < nx ? counts[(size_t)r * nx + i] : 0u, &total);
            if (i < nx) offsets[(size_t)r * nx + i] = (unsigned)(done + at);
            done += total;
            __syncthreads();
        }
        if (threadIdx.x == 0) offsets[3 * (size_t)nx + r] = (unsigned)done;
    }
}

// partner (y, x, 8 - k) of every touching tetrahedron entry, by bisection of row y
__global__ void k_partner(const NearEntry *to, int n, const unsigned *offsets, int nx, int32_t *partner, int *bad) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    const NearEntry en = to[e];
    const unsigned *row = offsets + nx;   // first touching entry of every x
    int lo = (int)row[en.y], hi = en.y + 1 < nx ? (int)row[en.y + 1] : n;
    const int key = 9 * en.x + (8 - en.k);
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (9 * to[mid].y + to[mid].k < key) lo = mid + 1;
        else hi = mid;
    }
    const bool ok = lo < n && to[lo].x == en.y && to[lo].y == en.x && to[lo].k == 8 - en.k;
    partner[e] = ok ? lo : 0;
    if (!ok) *bad = 1;
}

NearArgs args(const ElementSet &x, const ElementSet &y, double a, double b, double reach) {
    // FP32 rounding of a difference of two coordinates and a period: a few 2^-24 of their size
    return {x, y, a, b, 1e-9 * std::max(a, b), (float)(1e-6 * (reach + a + b))};
}

}  // namespace

cudaError_t near_count(const ElementSet &x, const ElementSet &y, double a, double b, double reach, uint16_t *mk,
                       unsigned *work, cudaStream_t st) {
    k_near<false><<<x.n, 256, 0, st>>>(args(x, y, a, b, reach), mk, work, nullptr, nullptr, nullptr); ++g_launches;
    k_scan_counts<<<1, 256, 0, st>>>(work, x.n, work + 3 * (size_t)x.n); ++g_launches;
    return cudaGetLastError();
}
cudaError_t near_emit(const ElementSet &x, const ElementSet &y, double a, double b, double reach, uint16_t *mk,
                      const unsigned *work, NearEntry *pr, NearEntry *to, cudaStream_t st) {
    k_near<true><<<x.n, 256, 0, st>>>(args(x, y, a, b, reach), mk, nullptr, work + 3 * (size_t)x.n, pr, to); ++g_launches;
    return cudaGetLastError();
}
cudaError_t near_partner(const NearEntry *to, int n, int nx, const unsigned *work, int32_t *partner, int *bad,
                         cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_partner<<<(n + 255) / 256, 256, 0, st>>>(to, n, work + 3 * (size_t)nx, nx, partner, bad); ++g_launches;
    return cudaGetLastError();
}

}  // namespace vie
