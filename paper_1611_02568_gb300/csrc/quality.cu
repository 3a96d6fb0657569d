// Neighbourhood precision (Eq. nei_prec): (1 / (k n)) sum_i |N_D^k(i) ∩ N_d^k(i)|,
// with N_D^k(i) the first k high-dimensional neighbours of point i and
// N_d^k(i) its k nearest neighbours in the 2-D embedding.
//
// k_nbr_precision  one warp per point (in tree order): exact 2-D k nearest
//                  neighbours by a ring search over the cells of one level of the
//                  current tree (the points of a cell are contiguous in the
//                  counting-sort permutation); squared distances in FP64 with
//                  explicit round-to-nearest operations, ties to the lower index
#include <algorithm>

#include "common.cuh"

namespace pxsne {

constexpr int kPrecMaxK = 32;
constexpr int kPrecWarps = 8;

__device__ __forceinline__ double d2_fp64(uint2 a, uint2 b, double s0, double s1) {
    const double dx = __dmul_rn(s0, (double)((int64_t)a.x - (int64_t)b.x));
    const double dy = __dmul_rn(s1, (double)((int64_t)a.y - (int64_t)b.y));
    return __dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy));
}

// The state of the Hilbert curve two levels below a cell of state s, for each of
// the 16 pairs of Morton digits, two bits each.
constexpr uint32_t hil_next2(uint32_t s) {
    uint32_t w = 0u;
    for (uint32_t q = 0u; q < 16u; q++) {
        const uint32_t t = hil_child(s, hil_pos(s, q >> 2));
        w |= hil_child(t, hil_pos(t, q & 3u)) << (2u * q);
    }
    return w;
}

// The search runs on level l0 of the tree (2^l0 cells per axis, about one point
// per cell of a full screen: on the pixels themselves a sparse screen costs
// hundreds of empty ones per point), or on the first finer one whose cell around
// the point is not crowded.  The lanes take up to 32 cells of a ring,
// then up to 32 of their points at a time, one distance per lane; lane a keeps
// the a-th nearest so far, and a better point enters by one shift across the
// warp.  Distances are compared by their bits (non-negative doubles order like
// integers; FP64 issues at a small fraction of the integer rate).  n = 100,000,
// k = 10 on 2048^2: 4.1 ms with one thread per point over the pixels and its
// list in local memory, 0.26 so.
__global__ void __launch_bounds__(kPrecWarps * 32)
    k_nbr_precision(int n, int L, int l0, int K1, int k, const uint2 *__restrict__ z,
                    const uint32_t *__restrict__ perm, const float *__restrict__ recn,
                    const uint32_t *__restrict__ leaf_start,
                    const uint32_t *__restrict__ blk_off, const int32_t *__restrict__ knn_hd,
                    int kh, const DevScalars *__restrict__ sc, int32_t *__restrict__ hits,
                    unsigned long long *total) {
    __shared__ unsigned s_hits[kPrecWarps];
    __shared__ uint32_t s_next[4];
    if (threadIdx.x == 0) {
        constexpr uint32_t k0 = hil_next2(0u), k1 = hil_next2(1u), k2 = hil_next2(2u),
                           k3 = hil_next2(3u);
        s_next[0] = k0;
        s_next[1] = k1;
        s_next[2] = k2;
        s_next[3] = k3;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int t = blockIdx.x * kPrecWarps + warp;
    unsigned h = 0u;
    if (t < n) {
        const uint32_t i = perm[t];
        const uint2 zi = z[i];
        const uint32_t mi = morton2(zi.x >> (32 - L), zi.y >> (32 - L));
        int l = l0;
        while (l < L && recn[rec_offset(l) + (mi >> (2 * (L - l)))] > 64.f) l++;
        const float *cell_n = recn + rec_offset(l);
        const int F = 32 - l, R = 1 << l, up = 2 * (L - l);
        const int px = (int)(zi.x >> F), py = (int)(zi.y >> F);
        const bool hil = hil_order(L);
        const double s0 = sc->s[0], s1 = sc->s[1];
        // smallest cell side in y-units
        const double w = ldexp(s0 < s1 ? s0 : s1, F);
        u64 bd = ~0ull;  // lane a < k: the a-th nearest (distance bits, index)
        int32_t bj = 0x7fffffff;
        u64 kd = ~0ull;  // the k-th
        int32_t kj = 0x7fffffff;
        for (int rho = 0; rho <= R; rho++) {
            // every cell at Chebyshev distance >= rho holds points at distance
            // >= (rho - 1) w; stop when the k-th distance is strictly below that
            if (rho >= 2 && kd != ~0ull) {
                const double b = (double)(rho - 1) * w;
                if (__longlong_as_double((long long)kd) < b * b * (1.0 - 1e-12)) break;
            }
            const int side = 2 * rho, cells = rho == 0 ? 1 : 4 * side;
            for (int q0 = 0; q0 < cells; q0 += 32) {
                // this lane's cell: the ring's four sides of 2 rho cells each
                const int q = q0 + lane;
                uint32_t cnt = 0u, start = 0u;
                if (q < cells) {
                    const int sd = rho == 0 ? 0 : q / side, o = rho == 0 ? 0 : q % side;
                    const int x = px + (sd == 0 ? o - rho : sd == 1 ? rho : sd == 2 ? rho - o : -rho);
                    const int y = py + (sd == 0 ? -rho : sd == 1 ? o - rho : sd == 2 ? rho : rho - o);
                    if (x >= 0 && y >= 0 && x < R && y < R) {
                        const uint32_t m = morton2((uint32_t)x, (uint32_t)y);
                        cnt = (uint32_t)cell_n[m];  // (exact float)
                        if (cnt != 0u) {
                            uint32_t first = m << up;
                            // along the curve the first leaf of a cell is its first
                            // or, where the state's bit 1 is set, its last one
                            if (hil) {
                                uint32_t s = 0u;
                                int b = 2 * l;
                                if (l & 1) {
                                    b -= 2;
                                    s = hil_child(0u, hil_pos(0u, m >> b));
                                }
                                while (b > 0) {
                                    b -= 4;
                                    s = (s_next[s] >> (2u * ((m >> b) & 15u))) & 3u;
                                }
                                if (s & 2u) first += (1u << up) - 1u;
                            }
                            start = blk_off[first >> (2 * K1)] + leaf_start[first];
                        }
                    }
                }
                uint32_t inc = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += v;
                }
                const uint32_t tot = __shfl_sync(0xffffffffu, inc, 31);
                for (uint32_t e0 = 0u; e0 < tot; e0 += 32u) {
                    const uint32_t e = e0 + lane;
                    // the cell that holds the e-th point: the first whose
                    // inclusive count exceeds e
                    int c = 0;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) {
                        const uint32_t v = __shfl_sync(0xffffffffu, inc, c + o - 1);
                        if (v <= e) c += o;
                    }
                    c = min(c, 31);
                    const uint32_t cs = __shfl_sync(0xffffffffu, start, c);
                    const uint32_t ce = __shfl_sync(0xffffffffu, inc - cnt, c);
                    u64 dd = ~0ull;
                    int32_t j = 0x7fffffff;
                    if (e < tot) {
                        j = (int32_t)perm[cs + (e - ce)];
                        if ((uint32_t)j != i)
                            dd = (u64)__double_as_longlong(d2_fp64(zi, z[j], s0, s1));
                    }
                    unsigned m = __ballot_sync(0xffffffffu, dd < kd || (dd == kd && dd != ~0ull && j < kj));
                    while (m) {
                        const int src = __ffs(m) - 1;
                        m &= m - 1u;
                        const u64 nd = __shfl_sync(0xffffffffu, dd, src);
                        const int32_t nj = __shfl_sync(0xffffffffu, j, src);
                        if (!(nd < kd || (nd == kd && nj < kj))) continue;  // (the same for all)
                        const bool after = bd > nd || (bd == nd && bj > nj);
                        const u64 pd = __shfl_up_sync(0xffffffffu, bd, 1);
                        const int32_t pj = __shfl_up_sync(0xffffffffu, bj, 1);
                        const unsigned am = __ballot_sync(0xffffffffu, after);
                        const int at = __ffs(am) - 1;  // its place: the first that follows it
                        if (after) {
                            bd = lane == at ? nd : pd;
                            bj = lane == at ? nj : pj;
                        }
                        kd = __shfl_sync(0xffffffffu, bd, k - 1);
                        kj = __shfl_sync(0xffffffffu, bj, k - 1);
                    }
                }
            }
        }
        const int32_t hd = lane < k ? knn_hd[(int64_t)i * kh + lane] : -1;
        for (int a = 0; a < k; a++) {
            const int32_t j = __shfl_sync(0xffffffffu, bj, a);
            h += __any_sync(0xffffffffu, hd == j) ? 1u : 0u;
        }
        if (lane == 0) hits[i] = (int32_t)h;
    }
    if (lane == 0) s_hits[warp] = h;
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long s = 0ull;
        for (int q = 0; q < kPrecWarps; q++) s += s_hits[q];
        if (s) atomicAdd(total, s);
    }
}

cudaError_t launch_nbr_precision(pxsne_ctx *c, int k, const int32_t *knn_hd, int kh,
                                 int32_t *hits, unsigned long long *total) {
    const int n = (int)c->n;
    const int K1 = c->L < kPyrK ? c->L : kPyrK;
    int l = 1;
    while (l < c->L && (int64_t(1) << (2 * l)) < (int64_t)n) l++;
    k_nbr_precision<<<(n + kPrecWarps - 1) / kPrecWarps, kPrecWarps * 32, 0, c->stream>>>(
        n, c->L, l, K1, k, c->z, c->perm, c->recn, c->leaf_start, c->blk_off, knn_hd,
        kh, c->sc, hits, total);
    return cudaGetLastError();
}

}  // namespace pxsne
