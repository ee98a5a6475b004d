// Dense complex linear algebra used by the solve (see linalg.cu).
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <cstddef>
#include <utility>
#include <vector>

#include "vie_internal.h"

namespace vie {

// y <- alpha Z x (+ y if accumulate) for FP32 Z and FP64 x, y, at double-length
// accuracy from FP32 arithmetic (x split into two FP32 parts, exact products,
// compensated sums); xs is device scratch of 8 cols floats
cudaError_t matvec_ds(const float *A, size_t ld, int rows, int cols, const double *x, float *xs, double *y,
                      double alpha, bool accumulate, cudaStream_t st);
// y <- alpha A x (+ y if accumulate) for two right-hand sides; grid_mult: row
// ranges per resident CTA (1: one; the autotuner may pick more)
template <typename TZ, typename TX, typename TA>
cudaError_t matvec(const TZ *A, size_t ld, int rows, int cols, const TX *x, TA *y, TA alpha, bool accumulate,
                   cudaStream_t st, int grid_mult = 1);
// Launch that may become resident before the kernel in front of it in the stream
// has finished (programmatic dependent launch); every kernel launched so waits
// (cudaGridDependencySynchronize) before it touches anything but constant data.
// The gap between dependent launches, 2-4 us each, is most of a GMRES iteration on
// small cells.
template <typename... KA, typename... A>
cudaError_t launch_pdl(void (*kernel)(KA...), dim3 grid, int block, cudaStream_t st, A... args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    ++g_launches;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KA>(args)...);
}
// y <- alpha A (x diag(rinv)), FP32 vectors (16-bit A: column-interleaved rows of ld
// entries, x zero up to pad_cols), rinv one
// factor per right-hand side (device); launched with launch_pdl
template <typename TZ>
cudaError_t matvec_norm(const TZ *A, size_t ld, int rows, int cols, const float *x, float *y, float alpha,
                        const float *rinv, cudaStream_t st, int grid_mult);

// ---- GMRES of the mixed paths (krylov.cu), FP32 vectors, both right-hand sides ----
// Basis vector j of both right-hand sides is one [n][2] complex vector w_j, orthogonal
// (per right-hand side) to the vectors before it but not normalised: v_j = w_j / |w_j|.
// `state`: device scratch of one solve, zeroed before the first vector
size_t krylov_state_bytes(int m);
// doubles of one message to the host (pinned): coefficients of both passes
// [m + 1][4] each (as applied, FP32 values), |w|^2 [2], the FP32 value of 1 / |w| that
// the next product takes [2], then one 64-bit sequence word
size_t krylov_message_doubles(int m);
// C_j = w_j^H w / |w_j|^2 for the nv vectors of V into pass `pass` of the state
cudaError_t krylov_dots(const float *V, size_t vstride, int nv, const float *w, int n, int m, void *state, int pass,
                        cudaStream_t st);
// w -= sum_j w_j C_j; pass 1: then the norms of vector nv, and the message with sequence number seq
cudaError_t krylov_subtract(const float *V, size_t vstride, int nv, float *w, int n, int m, void *state, int pass,
                            double *message, unsigned long long seq, cudaStream_t st);
const float *krylov_rinv(void *state, int m, int j);   // device address of 1 / |w_j| [2]

// CUDA-event timing of selected launches (optional)
struct KernelTimer {
    cudaEvent_t (*alloc)(void *) = nullptr;   // returns the next event of the caller's pool
    void *pool = nullptr;
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> ev;
    std::vector<double> work;    // algorithmic bytes of each timed launch
    std::vector<double> flops;   // and its algorithmic flops
    cudaEvent_t next() { return alloc ? alloc(pool) : nullptr; }
    void add(cudaEvent_t a, cudaEvent_t b, double w, double f = 0) {
        ev.push_back({a, b});
        work.push_back(w);
        flops.push_back(f);
    }
};
// In-place factorisation of an n x n complex FP32 block (no pivoting) by blocked
// Gauss-Jordan with 512-wide outer pivot blocks and the tcgen05 products
// (FP16 operands with power-of-two scales, FP32 accumulation); *status gets
// bit 0 for a zero or non-finite pivot and bit 1 for a bounded device wait
// that ran out;
// `pack` is device scratch of gj_pack_bytes(n) bytes (the packed operands and
// their scale words), aux a second stream of the caller (look-ahead); the work
// is complete on st when the last call returns on it.
// pivot: width of the outer pivot blocks, 512 (default) or 1024 (half the
// passes over the block).  group: columns per pivot group, a multiple of the
// pivot width; group >= n leaves the inverse in A, a smaller one the
// block-triangular factor that precond_step applies (linalg.cu).  regs: pivot blocks
// by 128-wide steps in registers (the FP64 path)
size_t gj_pack_bytes(int n);
cudaError_t gj_invert_tc(float *A, size_t ld, int n, int *status, void *pack, cudaStream_t st, cudaStream_t aux,
                         KernelTimer *kt, int pivot, int group, bool regs = false);
// columns per pivot group that vie_solve takes for a block of n unknowns
int gj_group(int n, int pivot);

// One step of an application of the preconditioner: the row group `row0` of one
// domain block times the columns [c0, c1) of its FP16 factor (column-interleaved
// rows of ld16 entries; c0 a multiple of 128), two right-hand sides.
//   forward (bwd 0):  y = in + alpha sum_c M x       backward (bwd 1): out = alpha sum_c M x,  z = zscale out
// x is the vector x1 for columns below split (a multiple of 128 or c1) and x2 from
// there on: 0 in, 1 y, 2 z.  All vector indices start at the block's offset voff.
struct PrecondJob {
    long long m;         // offset of entry (row0, c0) in the factor, complex entries
    long long pre;       // work units (4-row groups x 128-column chunks) of the step's jobs before this one
    int ld16, voff, row0, rows, c0, c1, split, x1, x2, bwd;
    double alpha, zscale;
};
inline long long precond_units(const PrecondJob &j) { return (long long)((j.rows + 3) / 4) * ((j.c1 - j.c0 + 127) / 128); }
// the njobs jobs of one step in one launch (on the host and as a device array: a few
// travel as kernel parameters); total: their work units.  in, y, z are readable and
// finite up to whole 128-column chunks of every block (pad_cols)
template <typename TV>
cudaError_t precond_step(const __half *M, const PrecondJob *host_jobs, const PrecondJob *jobs, int njobs, long long total,
                         const TV *in, TV *out, TV *y, TV *z, cudaStream_t st);
// columns of a vector that the 16-bit products read: whole 128-column chunks
inline size_t pad_cols(int n) { return ((size_t)n + 127) / 128 * 128 + 128; }
// out[0], out[1] (zeroed by the caller) <- the largest |Re|, |Im| of an n x n
// block inside and outside its diagonal groups, as float bits
cudaError_t absmax_groups(const float *A, size_t ld, int n, int group, unsigned *out, cudaStream_t st);
// FP16 copy of an n x n block (column-interleaved, rows of ld16(n)): entries
// inside the diagonal groups times sd, the others times sw
cudaError_t to_half_groups(const float *A, size_t ld, int n, int group, float sd, float sw, __half *B, cudaStream_t st);
// one bounded mbarrier wait of at most `polls` polls on a barrier that gets its
// arrival (arrive) or never does: bit 1 of *status (device) when it runs out
cudaError_t wait_check(bool arrive, long long polls, int *status, cudaStream_t st);
// one launch of the FMA-loop peak kernel (FP32 or FP64), events e0/e1 around
// it on st; *flops = its floating-point operations
cudaError_t fma_peak(bool fp64, int iters, cudaStream_t st, cudaEvent_t e0, cudaEvent_t e1, double *flops);
// *out (zeroed by the caller) <- max |A[i]| over count floats, as float bits
cudaError_t absmax(const float *A, size_t count, unsigned *out, cudaStream_t st);
// 16-bit copies of complex FP32 matrices in the column-interleaved layout the
// 16-bit products read: rows of ld16(cols) complex entries; inside each chunk
// of 128 columns, position p holds column (p % 4) * 32 + p / 4 of the chunk
// (zero past cols), so the four entries of one 16-byte load are columns
// j, j + 32, j + 64, j + 96 and the product's x loads are contiguous across a
// warp.  il_pos(c): the position of column c.
inline size_t ld16(int cols) { return ((size_t)cols + 127) / 128 * 128; }
__host__ __device__ inline size_t il_pos(size_t c) {
    const size_t j = c & 127;
    return (c - j) + (j & 31) * 4 + (j >> 5);
}
// B = scale A in FP16 (interleaved; A: rows x cols complex, row stride lda complex)
cudaError_t to_half_il(const float *A, size_t lda, int rows, int cols, float scale, __half *B, cudaStream_t st);
// B = A in BF16 (interleaved)
cudaError_t to_bf16_il(const float *A, size_t lda, int rows, int cols, __nv_bfloat16 *B, cudaStream_t st);
template <typename TS, typename TD>
cudaError_t copy_block(const TS *Z, size_t ldz, int off, int n, TD *B, size_t ldb, cudaStream_t st);
template <typename TV>
cudaError_t dots(const TV *V, size_t vstride, int nv, const TV *w, int n, double *h, cudaStream_t st);
template <typename TV>
cudaError_t subtract(const TV *V, size_t vstride, int nv, const double *h, TV *w, int n, cudaStream_t st);
template <typename TX, typename TY>
cudaError_t scale(const TX *x, TY *y, int n, const double s[4], cudaStream_t st);
template <typename TV>
cudaError_t combine(const TV *V, size_t vstride, int nv, const double *y, double *x, int n, cudaStream_t st);

}  // namespace vie
