// Shared by the two tensor-core neighbour searches (affinity.cu, knn_scan.cu):
// the tiles' geometry and the launcher of the two-pass search.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

struct pxsne_ctx;

namespace pxsne {

constexpr int kTcRows = 128;     // query rows per CTA (MMA M)
constexpr int kTcCols = 128;     // candidates per tile (MMA N)
constexpr int kTcPolls = 1 << 22;
constexpr uint32_t kTcSleepNs = 2000u;  // suspend hint of the pipeline waits
// per candidate tile: h_j (128), g_j (128), then per 32-column chunk min h, max
// g and max rounding error (4 + 4 + 4): 268 floats, 1072 bytes (a multiple of
// 16 for the bulk copy)
constexpr int kHG = 2 * kTcCols + 12;

// What the searches read of a set of rows in locality order: the FP32 rows
// (ld floats each, a multiple of 4, zeros past D), the FP16 tile images, the
// rounded rows' norms and rounding errors, the tiles' filter data, and the
// tiles' centroids and radii.
struct KnnRows {
    int64_t n, T;          // rows, tiles
    const float *X;
    const uint8_t *img;
    const float *nrm, *rerr, *HG;
    const float *cent, *rad;
};

struct KnnScan {
    KnnRows q, s;          // the rows, and the sample of every kScanStride-th one
    int ld, Dp, k;
    float inv_s2, kappa, eps_abs;
    const uint32_t *order;  // ordered position -> row of X
    int32_t *out_idx;
    float *out_d2;
    unsigned *err;
    // exact distances, kept candidates, skipped tile pairs, tile products, query
    // tiles scanned again and left to the one-pass search (DevScalars::knn_*)
    unsigned long long *stats;
};

// The sample takes the ordered rows kScanPhase + i kScanStride.
constexpr int kScanStride = 8;
constexpr int kScanPhase = 3;
inline int64_t scan_sample_rows(int64_t n) {
    return n > kScanPhase ? (n - kScanPhase + kScanStride - 1) / kScanStride : 0;
}

// Whether the two-pass search takes this size (see knn_scan.cu).
bool knn_scan_takes(int64_t n, int k, int Dp, int smem_max);
// Lists of every row into out_idx / out_d2 (by row of X), except for the query
// tiles written to failed (room for q.T) and counted in *nfailed (device),
// whose lists are left to the one-pass search.  cudaErrorMemoryAllocation: nothing
// was launched (its scratch is the caller's to free).
cudaError_t launch_knn_scan(const pxsne_ctx *c, const KnnScan &a, int sms, uint32_t *failed,
                            uint32_t *nfailed, cudaStream_t st);

}  // namespace pxsne
