// Near-pair lists on the device (mesh.cu).
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

#include "fill.h"

namespace vie {

// elements of one kind (device arrays): centroids [n][3], largest vertex distance
// from it [n], kv vertices [n][kv][3]
struct ElementSet {
    const double *cen, *rad, *verts;
    int n, kv;
};
inline size_t near_work_words(int nx) { return 6 * (size_t)nx + 4; }
// Masks mk [nx][ny] and the counts per x of the pairs (x, y): work (near_work_words)
// receives the counts [3][nx], their scans [3][nx] and the totals [3] (entries that do
// not touch, entries that touch, near pairs).  reach: the largest |coordinate|.
cudaError_t near_count(const ElementSet &x, const ElementSet &y, double a, double b, double reach, uint16_t *mk,
                       unsigned *work, cudaStream_t st);
// the entry lists, sorted by x, y, image (after near_count; the lists sized by its totals)
cudaError_t near_emit(const ElementSet &x, const ElementSet &y, double a, double b, double reach, uint16_t *mk,
                      const unsigned *work, NearEntry *pr, NearEntry *to, cudaStream_t st);
// partner[e] = index of the entry (y, x, 8 - k) of touching entry e; *bad set where there is none
cudaError_t near_partner(const NearEntry *to, int n, int nx, const unsigned *work, int32_t *partner, int *bad,
                         cudaStream_t st);

}  // namespace vie
