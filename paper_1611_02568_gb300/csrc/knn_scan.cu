// The exact neighbour search in two passes over the tensor-core tiles.
//
// The one-pass search (k_knn_tc, affinity.cu) tightens each row's k-th distance
// while it runs: at n = 1M every row took 616 exact distances and 533 heap
// insertions for its 90 neighbours, one CTA per SM (the heaps fill the shared
// memory), 247 ms.  Here a first pass over a sample of the rows (every
// kScanStride-th in the locality order, so every neighbourhood is sampled in
// proportion) finds, per row, the r-th smallest approximate distance to the
// sample: a threshold tau that with r = k / 8 + 3.75 sigma + 1 lies above the
// true k-th distance for all but two rows in 10^4 at most, and that about 8 r rows
// reach.  The second pass has that threshold from its first tile on: it keeps
// no list, every candidate whose rigorous bound (below) does not exceed tau is
// appended to the row's buffer in global memory, and two CTAs fit on an SM.
// k_knn_pick then forms the exact FP32 distances of a row's candidates and
// sorts them.  tau need not be right: every row at an exact distance of at most
// tau is among the candidates, so if at least k candidates have one, the k
// nearest of them are the row's k nearest.  Where fewer have, or a buffer
// overflowed, the row gets a wider or narrower threshold and its tile a second scan,
// and where that does not do either, the tile goes to the one-pass search.
//
//   k_knn_scan<0>  the sample pass: tau
//   k_knn_scan<1>  the candidates of every row
//   k_knn_pick     exact distances, the k nearest in order
//
// The bound is that of the one-pass search: with x~ the FP16-rounded rows and
// E = |x~ - x| known per row, a candidate is dropped only if the lower bound
// on |q~ - c~|^2 exceeds (sqrt(tau) + E_q + E_c)^2.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "knn.cuh"
#include "sort.cuh"
#include "tc.cuh"

namespace pxsne {
namespace {

// Candidate-tile stages in shared memory, and slots of the tiles' norms: four
// where two CTAs still fit on an SM with them, else two.  (D = 128, n = 1M, one
// CTA of four stages: 60 ms for the second pass, two of two: 45.)
__host__ __device__ constexpr int stages(int mode, int Dp) { return mode == 1 && Dp <= 64 ? 4 : 2; }
constexpr int kAcc = 2;           // TMEM accumulators of 128 columns
// Filter warps: one per TMEM lane quarter in the sample pass (MODE 0), so that a
// row has one list, and two, of 64 columns each, in the other; then the loader's
// and the MMA issuer's warp.
constexpr int filter_warps(int mode) { return mode == 0 ? 4 : 8; }
constexpr int scan_threads(int mode) { return 32 * (filter_warps(mode) + 2); }

struct ScanArgs {
    KnnRows q, c;           // query rows; candidate rows (the sample or the rows themselves)
    int Dp, r;              // r: entries of a sample list
    float inv_s2, kappa, eps_abs;
    float *tau;             // [n] written by the sample pass, read by the other
    const uint32_t *qlist, *qcount;  // the query tiles to scan and how many; NULL: all
    const uint32_t *flag;   // with qlist: the tiles' flags, those with kLeft not scanned
    uint32_t *buf;          // [n][2][cap] candidates (ordered positions)
    uint32_t *cnt;          // [n][2] candidates found (more than cap: the first cap are in buf)
    int cap;
    unsigned *err;
    u64 *stats;
};

// MODE 1: the visits decided before the first tile, 32 a word (2 KB; all visits
// up to n = 2.1M).  The loader alone took 1.4 us for each 32 visits, of which it
// keeps about four, while its two stages ran dry: with all warps deciding first,
// the second pass takes 45 ms instead of 56 at n = 1M, D = 128.
constexpr int kKeepWords = 512;

// A row with up to kHopeless times the candidates that it has room for gets a
// narrower threshold; beyond, its distances tie or lie within the rounding of its
// tile's rows, and the tile is left to the one-pass search.  (Whole numbers: 200,000
// rows of 0 .. 3 in 8 dimensions, P in 34 ms, 57 with all tiles left over and 46
// by the one-pass search alone; 10 one-hot attributes of 5 values 58, 95 and 85.
// Where nothing helps the passes are lost: 128 dimensions, 300 off the origin, 428
// against 426; ending the hopeless scans early saved 2 and cost 1 % of every scan.)
constexpr uint32_t kHopeless = 4u;
constexpr uint32_t kAgain = 1u, kLeft = 2u;  // tile flags

// The i-th candidate tile a CTA visits: outward from its own neighbourhood.
__device__ __forceinline__ int64_t tile_at(int64_t own, int64_t i, int64_t T) {
    const int64_t off = (i & 1) ? (i + 1) / 2 : -(i / 2);
    return ((own + off) % T + T) % T;
}

// Shared memory: A tile, the stages of candidate tiles and of kHG floats, then for
// the sample pass the lists (128 rows x rs floats, rs odd).  At k = 90 two CTAs
// fit on an SM in both passes.
__host__ __device__ inline size_t scan_smem(int mode, int Dp, int r) {
    size_t b = (size_t)(1 + stages(mode, Dp)) * kTcRows * Dp * 2 +
               (size_t)stages(mode, Dp) * kHG * 4 + 1024;
    if (mode == 0) b += (size_t)kTcRows * (r | 1) * 4;
    return b;
}

// v[j] of 32 registers by a tree of selections.
__device__ __forceinline__ float pick32(const uint32_t (&v)[32], int j) {
    uint32_t t[16];
#pragma unroll
    for (int q = 0; q < 16; q++) t[q] = (j & 1) ? v[2 * q + 1] : v[2 * q];
#pragma unroll
    for (int q = 0; q < 8; q++) t[q] = (j & 2) ? t[2 * q + 1] : t[2 * q];
#pragma unroll
    for (int q = 0; q < 4; q++) t[q] = (j & 4) ? t[2 * q + 1] : t[2 * q];
#pragma unroll
    for (int q = 0; q < 2; q++) t[q] = (j & 8) ? t[2 * q + 1] : t[2 * q];
    return __uint_as_float((j & 16) ? t[1] : t[0]);
}

// MODE 0: the sample pass; MODE 1: the candidates.  One CTA per 128 query rows,
// warp roles as in the one-pass search: a loader that skips tiles beyond the
// rows' thresholds (triangle inequality on centroids and radii) and streams
// the others into shared memory by bulk copies, an MMA issuer, and the filter
// warps, one (MODE 0) or two (MODE 1) per quarter of the rows.  A value costs a packed half FMA
// and add and one funnel shift that collects the sign bits of e_j - t, e_j =
// (1-eps)|c~_j|^2 - 2 q~.c~_j, with the chunk's largest kappa |q~||c~| in t.
template <int MODE, int kStages>
__global__ void __launch_bounds__(scan_threads(MODE), 2) k_knn_scan(const ScanArgs a) {
    constexpr int kFilterWarps = filter_warps(MODE), kThreads = scan_threads(MODE);
    constexpr int kLoadWarp = kFilterWarps, kMmaWarp = kFilterWarps + 1;
    constexpr int kChunks = 16 / kFilterWarps;  // 32-column chunks of a tile per warp
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t bar_a, bar_sf[kStages], bar_se[kStages], bar_tf[kAcc], bar_te[kAcc],
        bar_hf[kStages], bar_he[kStages];
    __shared__ uint32_t tslot;
    __shared__ volatile int s_abort;
    __shared__ volatile float s_taumax[kFilterWarps];
    __shared__ volatile int s_tile[8];
    __shared__ float s_cq[128];
    __shared__ uint32_t s_keep[MODE == 1 ? kKeepWords : 1];
    uint8_t *smem = smem_raw + ((1024u - (tc::smem_u32(smem_raw) & 1023u)) & 1023u);
    const int64_t n = a.q.n, T = a.c.T;
    const uint32_t tile_bytes = (uint32_t)kTcRows * a.Dp * 2;
    uint8_t *sA = smem;
    uint8_t *sB = smem + tile_bytes;
    float *hbuf = reinterpret_cast<float *>(sB + (size_t)kStages * tile_bytes);
    const int rs = a.r | 1;
    float *lists = hbuf + kStages * kHG;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (MODE == 1 && a.qlist && blockIdx.x >= *a.qcount) return;
    const int64_t qt = MODE == 1 && a.qlist ? a.qlist[blockIdx.x] : blockIdx.x, q0 = qt * kTcRows;
    if (MODE == 1 && a.qlist && (a.flag[qt] & kLeft)) return;
    const int64_t own = MODE == 0 ? min(T - 1, qt / kScanStride) : qt;

    if (MODE == 0)
        for (int e = tid; e < kTcRows * rs; e += kThreads) lists[e] = INFINITY;
    if (warp == kMmaWarp) tc::tmem_alloc(&tslot, kAcc * kTcCols);
    if (tid == 0) {
        tc::mbar_init(&bar_a, 1);
        for (int s = 0; s < kStages; s++) {
            tc::mbar_init(&bar_sf[s], 1);
            tc::mbar_init(&bar_se[s], 1);
            tc::mbar_init(&bar_hf[s], 1);
            tc::mbar_init(&bar_he[s], kFilterWarps);
        }
        for (int b = 0; b < kAcc; b++) {
            tc::mbar_init(&bar_tf[b], 1);
            tc::mbar_init(&bar_te[b], kFilterWarps);
        }
        s_abort = 0;
        for (int w = 0; w < kFilterWarps; w++) s_taumax[w] = INFINITY;
    }
    for (int d = tid; d < a.Dp; d += kThreads) s_cq[d] = a.q.cent[qt * a.Dp + d];
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tbase = tslot;
    const float rq = a.q.rad[qt];
    // The lane's tile of the visits i0 .. i0 + 31, and which of the 32 a row's
    // neighbours can be in: its centroid is no farther than the radii and the
    // largest threshold.
    const auto keep32 = [&](int64_t i0, float taum, int64_t &tl) {
        const int64_t il = i0 + lane;
        const bool in = il < T;
        tl = in ? tile_at(own, il, T) : 0;
        float dd = 0.f;
        if (in) {
            const float4 *ct = reinterpret_cast<const float4 *>(a.c.cent + tl * a.Dp);
            for (int d4 = 0; d4 < a.Dp / 4; d4++) {
                const float4 c = __ldg(ct + d4);
                const float e0 = s_cq[4 * d4] - c.x, e1 = s_cq[4 * d4 + 1] - c.y;
                const float e2 = s_cq[4 * d4 + 2] - c.z, e3 = s_cq[4 * d4 + 3] - c.w;
                dd = fmaf(e0, e0, fmaf(e1, e1, fmaf(e2, e2, fmaf(e3, e3, dd))));
            }
        }
        const float lbd = sqrtf(dd) * 0.9999f - rq - (in ? a.c.rad[tl] : 0.f);
        const bool skip = in && il > 0 && lbd > 0.f && lbd * lbd > taum * 1.0001f;
        return __ballot_sync(0xffffffffu, in && !skip);
    };
    float taum = INFINITY;
    if (MODE == 1) {
        taum = 0.f;
        for (int r = lane; r < kTcRows; r += 32)
            if (q0 + r < n) taum = fmaxf(taum, a.tau[q0 + r]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) taum = fmaxf(taum, __shfl_xor_sync(0xffffffffu, taum, o));
        // the thresholds being known, all warps decide about the first
        // 32 kKeepWords visits
        for (int w = warp; w < kKeepWords && (int64_t)w * 32 < T; w += kThreads / 32) {
            int64_t tl;
            const unsigned keep = keep32((int64_t)w * 32, taum, tl);
            if (lane == 0) s_keep[w] = keep;
        }
        __syncthreads();
    }

    if (warp == kLoadWarp) {
        // ---- loader.  The kept tiles form a sequence j = 0, 1, ... that the
        // other warps follow through s_tile; the entry after the last is -1
        // (its barriers completed without data).
        if (lane == 0) {
            tc::mbar_expect_tx(&bar_a, tile_bytes);
            tc::bulk_g2s(sA, a.q.img + qt * tile_bytes, tile_bytes, &bar_a);
        }
        int64_t j = 0, n_sf = 0, n_hf = 0;
        u64 n_skip = 0u;
        bool fail = false, ended = false;
        for (int64_t i0 = 0; i0 <= T && !fail; i0 += 32) {
            if (__shfl_sync(0xffffffffu, s_abort, 0)) break;
            if (MODE == 0) {
                taum = 0.f;
#pragma unroll
                for (int w = 0; w < kFilterWarps; w++) taum = fmaxf(taum, s_taumax[w]);
            }
            int64_t tl;
            unsigned keep;
            if (MODE == 1 && i0 < 32 * kKeepWords) {
                tl = i0 + lane < T ? tile_at(own, i0 + lane, T) : 0;
                keep = i0 < T ? s_keep[i0 >> 5] : 0u;
            } else {
                keep = keep32(i0, taum, tl);
            }
            n_skip += (u64)(min((int64_t)32, T - i0) - __popc(keep));
            const bool last_block = i0 + 32 > T;
            while (keep || last_block) {
                const bool end = keep == 0u;  // (only in the last block)
                int64_t t = -1;
                if (!end) {
                    const int src = __ffs(keep) - 1;
                    keep &= keep - 1u;
                    t = __shfl_sync(0xffffffffu, tl, src);
                }
                const int s = (int)(j % kStages);
                bool ok = j < kStages ||
                          tc::mbar_wait_sleep(&bar_se[s], (uint32_t)((j / kStages - 1) & 1), kTcPolls,
                                              kTcSleepNs);
                ok = __all_sync(0xffffffffu, ok);
                if (ok) {
                    if (lane == 0) {
                        s_tile[j & 7] = (int)t;
                        if (end) {
                            tc::mbar_arrive(&bar_sf[s]);
                        } else {
                            tc::mbar_expect_tx(&bar_sf[s], tile_bytes);
                            tc::bulk_g2s(sB + (size_t)s * tile_bytes, a.c.img + t * tile_bytes,
                                         tile_bytes, &bar_sf[s]);
                        }
                    }
                    if (!end) n_sf++;
                    __syncwarp();
                    ok = j < kStages ||
                         tc::mbar_wait_sleep(&bar_he[s], (uint32_t)((j / kStages - 1) & 1), kTcPolls,
                                             kTcSleepNs);
                    ok = __all_sync(0xffffffffu, ok);
                    if (ok) {
                        if (lane == 0) {
                            if (end) {
                                tc::mbar_arrive(&bar_hf[s]);
                            } else {
                                tc::mbar_expect_tx(&bar_hf[s], kHG * 4);
                                tc::bulk_g2s(hbuf + s * kHG, a.c.HG + t * kHG, kHG * 4, &bar_hf[s]);
                            }
                        }
                        if (!end) n_hf++;
                    }
                }
                if (!ok) {
                    fail = true;
                    if (lane == 0) {
                        s_abort = 1;
                        atomicOr(a.err, (unsigned)PXSNE_DEVERR_TIMEOUT);
                    }
                }
                __syncwarp();
                ended = end && !fail;
                if (fail || end) break;
                j++;
            }
        }
        if (lane == 0) {
            // (the second scan's tiles were counted by the first)
            if (MODE == 1 && !a.qlist) atomicAdd(&a.stats[2], n_skip);
            atomicAdd(&a.stats[3], (u64)n_sf);
            if (MODE == 1 && a.qlist) atomicAdd(&a.stats[4], 1ull);
            // copies still in flight complete before the CTA exits (those of the
            // last kept tiles; after the end mark the copies into the slots it
            // reused are known complete)
            const int64_t ws = ended ? kStages - 1 : kStages;
            tc::mbar_wait(&bar_a, 0u, kTcPolls);
            for (int64_t q = (n_sf > ws ? n_sf - ws : 0); q < n_sf; q++)
                tc::mbar_wait(&bar_sf[q % kStages], (uint32_t)((q / kStages) & 1), kTcPolls);
            for (int64_t q = (n_hf > ws ? n_hf - ws : 0); q < n_hf; q++)
                tc::mbar_wait(&bar_hf[q % kStages], (uint32_t)((q / kStages) & 1), kTcPolls);
        }
    } else if (warp == kMmaWarp) {
        // ---- MMA issuer
        if (lane == 0) {
            const uint32_t idesc = tc::idesc_f16(kTcRows, kTcCols, 0);
            const uint32_t a0 = tc::smem_u32(sA);
            bool ok = tc::mbar_wait(&bar_a, 0u, kTcPolls);
            int64_t i = 0;
            bool ended = false;
            for (; ok && i <= T && !s_abort; i++) {
                const int s = (int)(i % kStages), b = (int)(i % kAcc);
                ok = tc::mbar_wait_sleep(&bar_sf[s], (uint32_t)((i / kStages) & 1), kTcPolls,
                                         kTcSleepNs);
                if (ok && i >= kAcc)
                    ok = tc::mbar_wait_sleep(&bar_te[b], (uint32_t)((i / kAcc - 1) & 1), kTcPolls,
                                             kTcSleepNs);
                if (!ok) break;
                tc::fence_after();
                if (s_tile[i & 7] < 0) {
                    tc::mbar_arrive(&bar_tf[b]);
                    ended = true;
                    break;
                }
                const uint32_t b0 = tc::smem_u32(sB + (size_t)s * tile_bytes);
                for (int kk = 0; kk < a.Dp / 16; kk++) {
                    const uint32_t off =
                        (uint32_t)(kk >> 2) * (kTcRows * 128) + (uint32_t)(kk & 3) * 32;
                    tc::mma_f16(tbase + (uint32_t)(b * kTcCols), tc::sdesc_sw128(a0 + off),
                                tc::sdesc_sw128(b0 + off), idesc, kk > 0 ? 1u : 0u);
                }
                tc::commit(&bar_se[s]);
                tc::commit(&bar_tf[b]);
            }
            if (!ok) {
                s_abort = 1;
                atomicOr(a.err, (unsigned)PXSNE_DEVERR_TIMEOUT);
            }
            // MMAs still in flight finish before TMEM is freed
            const int64_t wa = ended ? kAcc - 1 : kAcc;
            for (int64_t j = (i > wa ? i - wa : 0); j < i; j++)
                tc::mbar_wait(&bar_tf[j % kAcc], (uint32_t)((j / kAcc) & 1), kTcPolls);
        }
    } else {
        // ---- filter: warp `quarter` (and quarter + 4) owns query rows q0 + 32
        // quarter + lane, taking its kChunks chunks of a tile's columns
        const int quarter = warp & 3, half = warp >> 2;
        const int64_t qi = q0 + 32 * quarter + lane;
        const bool qvalid = qi < n;
        const float qn2 = qvalid ? a.q.nrm[qi] : 0.f;
        const float onem = 1.0f - a.eps_abs;
        const float2 cneg = make_float2(-2.0f * a.inv_s2, -2.0f * a.inv_s2);
        const float Bq = a.kappa * sqrtf(qn2);
        // MODE 1: sqrt(tau) + |q~ - q|; a chunk's threshold adds its rows'
        // largest rounding error
        const float sqE = MODE == 1 && qvalid ? sqrtf(a.tau[qi]) + a.q.rerr[qi] : 0.f;
        uint32_t *mine = MODE == 1 ? a.buf + ((size_t)(qvalid ? qi : 0) * 2 + half) * a.cap : nullptr;
        uint32_t found = 0u;
        // MODE 0: max-heap of the row's r smallest e_j
        float *heap = lists + (size_t)(32 * quarter + lane) * rs;
        float root = INFINITY;
        // the row's own column among the candidates, if it is one
        const int64_t self = MODE == 1 ? qi
                             : (qi >= kScanPhase && (qi - kScanPhase) % kScanStride == 0)
                                 ? (qi - kScanPhase) / kScanStride
                                 : -1;
        for (int64_t i = 0; i <= T; i++) {
            const int b = (int)(i % kAcc), hs = (int)(i % kStages);
            const uint32_t par = (uint32_t)((i / kAcc) & 1), hpar = (uint32_t)((i / kStages) & 1);
            const bool got =
                __all_sync(0xffffffffu, tc::mbar_wait_sleep(&bar_tf[b], par, kTcPolls, kTcSleepNs) &&
                                            tc::mbar_wait_sleep(&bar_hf[hs], hpar, kTcPolls, kTcSleepNs) &&
                                            !s_abort);
            if (!got) {
                if (lane == 0 && !s_abort) atomicOr(a.err, (unsigned)PXSNE_DEVERR_TIMEOUT);
                s_abort = 1;
                break;
            }
            tc::fence_after();
            const int tt = s_tile[i & 7];
            if (tt < 0) break;
            const int64_t c0 = (int64_t)tt * kTcCols;
            const float *hb = hbuf + hs * kHG;
#pragma unroll
            for (int cc = 0; cc < kChunks; cc++) {
                const int ci = kChunks * half + cc, cb = 32 * ci;
                uint32_t raw[32];
                tc::tmem_ld32_async(
                    tbase + ((uint32_t)(32 * quarter) << 16) + (uint32_t)(b * kTcCols + cb), raw);
                tc::tmem_wait_ld();
                if (cc == kChunks - 1) {  // the accumulator is free
                    tc::fence_before();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive(&bar_te[b]);
                }
                float t;
                if (MODE == 1) {
                    // e_j <= (sqrt(tau) + E_q + max E_c)^2 - (1-eps)|q~|^2 + kappa |q~| max |c~|,
                    // the square raised by 2^-16 for the roundings of tau, the
                    // exact distances and t itself; never infinite, so that
                    // padding (e = +inf) does not pass
                    const float tE = sqE + hb[2 * kTcCols + 8 + ci];
                    t = fmaf(tE * tE, 1.52587890625e-05f, tE * tE) - onem * qn2 +
                        Bq * hb[2 * kTcCols + 4 + ci];
                    t = qvalid ? fminf(t, 3.402823466e38f) : -3.402823466e38f;
                } else {
                    t = qvalid ? fminf(root, 3.402823466e38f) : -3.402823466e38f;
                }
                const float2 nt = make_float2(-t, -t);
                uint32_t sm = 0u;  // bit 31 - j: column j passes
#pragma unroll
                for (int j4 = 0; j4 < 8; j4++) {
                    const float4 h4 = *reinterpret_cast<const float4 *>(hb + cb + 4 * j4);
                    const float2 e0 = __ffma2_rn(make_float2(__uint_as_float(raw[4 * j4]),
                                                             __uint_as_float(raw[4 * j4 + 1])),
                                                 cneg, make_float2(h4.x, h4.y));
                    const float2 e1 = __ffma2_rn(make_float2(__uint_as_float(raw[4 * j4 + 2]),
                                                             __uint_as_float(raw[4 * j4 + 3])),
                                                 cneg, make_float2(h4.z, h4.w));
                    const float2 f0 = __fadd2_rn(e0, nt), f1 = __fadd2_rn(e1, nt);
                    sm = __funnelshift_l(__float_as_uint(f0.x), sm, 1);
                    sm = __funnelshift_l(__float_as_uint(f0.y), sm, 1);
                    sm = __funnelshift_l(__float_as_uint(f1.x), sm, 1);
                    sm = __funnelshift_l(__float_as_uint(f1.y), sm, 1);
                    if (MODE == 0) {
                        raw[4 * j4] = __float_as_uint(e0.x);
                        raw[4 * j4 + 1] = __float_as_uint(e0.y);
                        raw[4 * j4 + 2] = __float_as_uint(e1.x);
                        raw[4 * j4 + 3] = __float_as_uint(e1.y);
                    }
                }
                const int64_t js = self - (c0 + cb);
                if (js >= 0 && js < 32) sm &= ~(0x80000000u >> (int)js);
                if (MODE == 1) {
                    while (sm) {
                        const int j = __clz(sm);
                        sm ^= 0x80000000u >> j;
                        if (found < (uint32_t)a.cap) mine[found] = (uint32_t)(c0 + cb + j);
                        found++;
                    }
                } else {
                    while (sm) {
                        const int j = __clz(sm);
                        sm ^= 0x80000000u >> j;
                        const float e = pick32(raw, j);
                        if (!(e < root)) continue;
                        int p = 0;
                        for (;;) {
                            int c = 2 * p + 1;
                            if (c >= a.r) break;
                            float vc = heap[c];
                            if (c + 1 < a.r) {
                                const float vr = heap[c + 1];
                                if (vr > vc) {
                                    vc = vr;
                                    c++;
                                }
                            }
                            if (!(vc > e)) break;
                            heap[p] = vc;
                            p = c;
                        }
                        heap[p] = e;
                        root = heap[0];
                    }
                    __syncwarp();
                }
            }
            __syncwarp();
            if (lane == 0) tc::mbar_arrive(&bar_he[hs]);
            if (MODE == 0) {
                float tm = qvalid ? root + qn2 : -INFINITY;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) tm = fmaxf(tm, __shfl_xor_sync(0xffffffffu, tm, o));
                if (lane == 0) s_taumax[warp] = tm;
            }
        }
        if (MODE == 1 && qvalid) a.cnt[qi * 2 + half] = found;
        if (MODE == 0 && qvalid) a.tau[qi] = fmaxf(root + qn2, 0.f);
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (warp == kMmaWarp) tc::tmem_dealloc(tbase, kAcc * kTcCols);
}

// ---- exact distances and the k nearest
// One warp per row, 32 candidates at a time: their FP32 rows come into shared
// memory by one bulk copy per candidate (an odd number of 16-byte units apart,
// so that the lanes' 16-byte reads do not conflict),
// then every lane sums its candidate's squared differences in index order.
// (Lanes reading their candidate's row from global memory touch 32 lines per
// load; at n = 1M the 113 GB of rows come at 6.8 TB/s, and staging half rows, with
// twice the warps per SM, changed nothing.)  The candidates within tau go to a key buffer (distance, then row
// index); it is sorted by a bitonic network in registers, 8 or 16 keys per lane.
constexpr int kPickWarps = 2;
constexpr int kPickKeys = 512;  // most candidates within tau

template <int V>
__device__ __forceinline__ void sort_buffer(u64 *keys, int cnt, int lane) {
    u64 key[V];
#pragma unroll
    for (int v = 0; v < V; v++) key[v] = v * 32 + lane < cnt ? keys[v * 32 + lane] : ~0ull;
    sort_keys<V>(key, lane);
    __syncwarp();
#pragma unroll
    for (int v = 0; v < V; v++) keys[lane * V + v] = key[v];
    __syncwarp();
}

struct PickArgs {
    int64_t n;
    int ld, k, cap;
    float enough;  // k and 3.75 deviations
    const float *X;
    float *tau;                      // a row that falls short gets a wider one, a row
                                     // with too many a narrower one
    const uint32_t *qlist, *qcount;  // the query tiles to take and how many; NULL: all
    const uint32_t *buf, *cnt, *order;
    int32_t *out_idx;
    float *out_d2;
    // per query tile, kAgain: in retry (a second scan with its rows' new
    // thresholds), kLeft: in failed (the one-pass search)
    uint32_t *flag, *retry, *nretry, *failed, *nfailed;
    unsigned *err;
    u64 *stats;
};

// Floats from one staged row to the next: an odd number of 16-byte units.
__host__ __device__ inline int pick_pitch(int ld) { return ((ld >> 2) | 1) << 2; }

__host__ __device__ inline size_t pick_smem(int ld) {
    // per warp: keys, the query row, 32 candidate rows
    return (size_t)kPickWarps * ((size_t)33 * pick_pitch(ld) * 4 + kPickKeys * 8);
}

__global__ void __launch_bounds__(kPickWarps * 32) k_knn_pick(const PickArgs a) {
    extern __shared__ __align__(16) uint8_t pick_raw[];
    __shared__ uint64_t s_bar[kPickWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ls = pick_pitch(a.ld);
    uint8_t *base = pick_raw + (size_t)warp * (pick_smem(a.ld) / kPickWarps);
    u64 *keys = reinterpret_cast<u64 *>(base);
    float *qrow = reinterpret_cast<float *>(keys + kPickKeys);
    float *rows = qrow + ls;
    const uint32_t bytes = (uint32_t)a.ld * 4u;
    uint64_t *bar = &s_bar[warp];
    if (lane == 0) tc::mbar_init(bar, 1);
    __syncthreads();
    uint32_t phase = 0u;
    u64 n_exact = 0u, n_kept = 0u;
    bool ok = true;
    const int64_t rows_all = a.qlist ? (int64_t)*a.qcount * kTcRows : a.n;
    for (int64_t q = blockIdx.x * (int64_t)kPickWarps + warp; ok && q < rows_all;
         q += (int64_t)gridDim.x * kPickWarps) {
        const int64_t row = a.qlist ? (int64_t)a.qlist[q / kTcRows] * kTcRows + q % kTcRows : q;
        if (row >= a.n) continue;
        const uint32_t fl = __ldcg(&a.flag[row / kTcRows]);
        const uint32_t c0 = a.cnt[2 * row], c1 = a.cnt[2 * row + 1];
        const float tau = a.tau[row];
        // a tile that another of its rows has left to the one-pass search
        if (__any_sync(0xffffffffu, fl & kLeft)) continue;
        const uint32_t *b0 = a.buf + (size_t)row * 2 * a.cap, *b1 = b0 + a.cap;
        // the candidates that are in the buffers, and whether that is all of them
        const uint32_t m0 = min(c0, (uint32_t)a.cap), tot = m0 + min(c1, (uint32_t)a.cap);
        const bool all = c0 <= (uint32_t)a.cap && c1 <= (uint32_t)a.cap;
        bool good = c0 <= kHopeless * (uint32_t)a.cap && c1 <= kHopeless * (uint32_t)a.cap;
        uint32_t kept = 0u;
        if (good)
            for (int d = lane; d < (a.ld >> 2); d += 32)
                reinterpret_cast<float4 *>(qrow)[d] =
                    __ldg(reinterpret_cast<const float4 *>(a.X + row * a.ld) + d);
        for (uint32_t e0 = 0u; good && e0 < tot; e0 += 32u) {
            const uint32_t e = e0 + lane, m = min(32u, tot - e0);
            uint32_t cand = e < tot ? (e < m0 ? b0[e] : b1[e - m0]) : 0u;
            // (a padding column passes the filter only where its terms are NaN)
            const bool real = e < tot && cand < (uint32_t)a.n;
            if (!real) cand = 0u;
            __syncwarp();
            tc::fence_proxy_async();
            if (lane == 0) tc::mbar_expect_tx(bar, m * bytes);
            __syncwarp();
            if (e < tot) tc::bulk_g2s(rows + lane * ls, a.X + (int64_t)cand * a.ld, bytes, bar);
            ok = __all_sync(0xffffffffu, tc::mbar_wait(bar, phase & 1u, kTcPolls));
            phase++;
            if (!ok) break;
            float s = 0.f;
            const float4 *pc = reinterpret_cast<const float4 *>(rows + lane * ls);
            const float4 *pq = reinterpret_cast<const float4 *>(qrow);
#pragma unroll 8
            for (int d = 0; d < (a.ld >> 2); d++) {
                const float4 u = pq[d], v = pc[d];
                float t = u.x - v.x;
                s = fmaf(t, t, s);
                t = u.y - v.y;
                s = fmaf(t, t, s);
                t = u.z - v.z;
                s = fmaf(t, t, s);
                t = u.w - v.w;
                s = fmaf(t, t, s);
            }
            const bool in = real && s <= tau;
            const unsigned im = __ballot_sync(0xffffffffu, in);
            const uint32_t at = kept + __popc(im & ((1u << lane) - 1u));
            if (in && at < (uint32_t)kPickKeys)
                keys[at] = ((u64)__float_as_uint(s) << 32) | __ldg(a.order + cand);
            kept += __popc(im);
        }
        good = good && ok;
        __syncwarp();
        const uint32_t have = min(kept, (uint32_t)kPickKeys);
        if (good) {
            n_exact += tot;
            if (have <= 256u) sort_buffer<8>(keys, (int)have, lane);
            else sort_buffer<16>(keys, (int)have, lane);
        }
        if (!good || !all || kept != have || kept < (uint32_t)a.k) {
            // A threshold that should do.  Too many candidates: the k-th nearest of
            // those that were sorted bounds the k-th nearest; where they are a part,
            // so in all likelihood does the one that as large a part of `enough`
            // reach.  Too few: half of them lie within keys[kept / 2], so the same
            // factor again should about double them.
            float next = -1.f;
            if (good && (kept != have || !all)) {
                const float of = all ? (float)kept : (float)(c0 + c1) * (float)kept / (float)tot;
                const int at = min(a.k - 1, (int)(a.enough * (float)have / of));
                if ((uint32_t)at < have) {
                    const float v = __uint_as_float((uint32_t)(keys[at] >> 32));
                    if (v < tau) next = v;
                }
            } else if (good && a.retry && kept >= 8u) {
                const float half = __uint_as_float((uint32_t)(keys[kept >> 1] >> 32));
                const float wider = half > 0.f ? tau * (tau / half) : 0.f;
                if (wider > tau && wider < 3.402823466e38f) next = wider;
            }
            const uint32_t t = (uint32_t)(row / kTcRows);
            if (next >= 0.f && all && kept != have) {
                // all its candidates are at hand: the same row again
                if (lane == 0) a.tau[row] = next;
                q -= (int64_t)gridDim.x * kPickWarps;
            } else if (lane == 0) {
                if (next >= 0.f && a.retry) {
                    a.tau[row] = next;
                    if (!(atomicOr(&a.flag[t], kAgain) & kAgain)) a.retry[atomicAdd(a.nretry, 1u)] = t;
                } else if (!(atomicOr(&a.flag[t], kLeft) & kLeft)) {
                    a.failed[atomicAdd(a.nfailed, 1u)] = t;
                    atomicAdd(&a.stats[5], 1ull);
                }
                if (!ok) atomicOr(a.err, (unsigned)PXSNE_DEVERR_TIMEOUT);
            }
            __syncwarp();
            continue;
        }
        n_kept += kept;
        const int64_t orow = a.order[row];
        for (int e = lane; e < a.k; e += 32) {
            const u64 v = keys[e];
            a.out_idx[orow * a.k + e] = (int32_t)(uint32_t)v;
            a.out_d2[orow * a.k + e] = __uint_as_float((uint32_t)(v >> 32));
        }
        __syncwarp();
    }
    if (!ok) tc::mbar_wait(bar, (phase - 1u) & 1u, kTcPolls);  // copies in flight land first
    if (lane == 0) {
        atomicAdd(&a.stats[0], n_exact);
        atomicAdd(&a.stats[1], n_kept);
    }
}

// Entries of a sample list: of the k nearest, k / kScanStride are in the sample
// on average; 3.75 standard deviations and one more leave a chance of at most
// 2e-4 per row that the threshold comes out below the k-th distance, less than
// that where the locality order spreads the sample evenly (the tile is then scanned
// again: 0.65 % of them at n = 1M, 0.9 % at 10M; four and a half deviations would
// spare that but bring 12 % more candidates to every row).
int sample_rank(int k) {
    const double m = (double)k / kScanStride;
    return (int)std::ceil(m + 3.75 * std::sqrt(m * (1.0 - 1.0 / kScanStride)) + 1.0);
}

// Room per half of a row's candidates: about 8 r rows reach the threshold, half
// of them in each half of the tiles' columns; the filter's band lets through up
// to about half as many again, and small sets vary more.
int half_cap(int r) { return (4 * r * 5 / 2 + 64 + 31) / 32 * 32; }

}  // namespace

// The sample must hold a few lists' worth of rows; the sort holds kPickKeys.
bool knn_scan_takes(int64_t n, int k, int Dp, int smem_max) {
    const int r = sample_rank(k);
    return Dp <= 128 && scan_sample_rows(n) >= 4 * r && kScanStride * r * 3 / 2 <= kPickKeys &&
           scan_smem(0, Dp, r) <= (size_t)smem_max && pick_smem(Dp) <= (size_t)smem_max;
}

cudaError_t launch_knn_scan(const pxsne_ctx *c, const KnnScan &a, int sms, uint32_t *failed, uint32_t *nfailed,
                            cudaStream_t st) {
    const int64_t n = a.q.n, T = a.q.T;
    const int r = sample_rank(a.k), cap = half_cap(r);
    cudaError_t e;
    float *tau = nullptr;
    uint32_t *buf = nullptr, *cnt = nullptr, *flag = nullptr;
    if ((e = palloc(c, &tau, (size_t)n * 4, st))) return e;
    if ((e = palloc(c, &buf, (size_t)n * 2 * cap * 4, st))) return e;
    if ((e = palloc(c, &cnt, (size_t)n * 2 * 4, st))) return e;
    // flags and the retry list of the tiles, and its length
    if ((e = palloc(c, &flag, (size_t)(2 * T + 1) * 4, st))) return e;
    uint32_t *retry = flag + T, *nretry = flag + 2 * T;
    if ((e = cudaMemsetAsync(flag, 0, (size_t)(2 * T + 1) * 4, st))) return e;
    if ((e = cudaMemsetAsync(nfailed, 0, 4, st))) return e;
    // (a scan that gives up leaves its rows without candidates)
    if ((e = cudaMemsetAsync(tau, 0, (size_t)n * 4, st))) return e;
    if ((e = cudaMemsetAsync(cnt, 0, (size_t)n * 2 * 4, st))) return e;
    ScanArgs s{a.q, a.s, a.Dp, r, a.inv_s2, a.kappa, a.eps_abs, tau, nullptr, nullptr, flag, buf, cnt, cap,
               a.err, a.stats};
    const int sm0 = (int)scan_smem(0, a.Dp, r), sm1 = (int)scan_smem(1, a.Dp, r);
    const auto scan1 = stages(1, a.Dp) == 4 ? k_knn_scan<1, 4> : k_knn_scan<1, 2>;
    const int smp = (int)pick_smem(a.ld);
    if ((e = allow_smem(k_knn_scan<0, 2>))) return e;
    if ((e = allow_smem(scan1))) return e;
    if ((e = allow_smem(k_knn_pick))) return e;
    int per = 1;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_knn_pick, kPickWarps * 32, smp)))
        return e;
    const int64_t need = (n + kPickWarps - 1) / kPickWarps;
    const unsigned pgrid =
        (unsigned)std::min<int64_t>(need, (int64_t)std::max(1, per) * std::max(1, sms));
    k_knn_scan<0, 2><<<(unsigned)T, scan_threads(0), sm0, st>>>(s);
    if ((e = cudaGetLastError())) return e;
    s.c = a.q;
    scan1<<<(unsigned)T, scan_threads(1), sm1, st>>>(s);
    if ((e = cudaGetLastError())) return e;
    PickArgs p{n, a.ld, a.k, cap, (float)a.k + 3.75f * std::sqrt((float)a.k) + 1.f, a.q.X, tau, nullptr, nullptr, buf, cnt, a.order, a.out_idx, a.out_d2,
               flag, retry, nretry, failed, nfailed, a.err, a.stats};
    k_knn_pick<<<pgrid, kPickWarps * 32, smp, st>>>(p);
    if ((e = cudaGetLastError())) return e;
    // the tiles with a row that fell short or had too many, once more (their number is on the
    // device: CTAs past it return at once)
    s.qlist = p.qlist = retry;
    s.qcount = p.qcount = nretry;
    p.retry = nullptr;
    scan1<<<(unsigned)T, scan_threads(1), sm1, st>>>(s);
    if ((e = cudaGetLastError())) return e;
    k_knn_pick<<<pgrid, kPickWarps * 32, smp, st>>>(p);
    if ((e = cudaGetLastError())) return e;
    pfree(c, tau, st);
    pfree(c, buf, st);
    pfree(c, cnt, st);
    return pfree(c, flag, st);
}

}  // namespace pxsne
