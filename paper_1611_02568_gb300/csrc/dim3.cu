// The 3-D embedding (dim = 3): PixelSNE on a voxel grid, the extension the
// paper's introduction names beside the 2-D screen.  Each point's position is
// u32 fixed point on three axes (voxel = z >> (32 - L), 2^L voxels per axis),
// the pixel quadtree becomes a voxel octree (eight children per cell, Morton
// bits x, y, z from the least significant), and every other step is the 2-D
// method with a third coordinate:
//
//   k3_minmax, k3_map   Eq. z1/z2 per axis (FP64), the state's start
//   k3_update           Eq. grad and the gains/momentum step per coordinate
//   k3_snap             the exact-integer rescale of Sec. 4.2 per axis, the
//                       voxel snap and the leaf histogram (counts, exact sums)
//   k3_level, k3_top, k3_perm  the octree's upper levels with their cells'
//                       records; the counting sort of the points by voxel
//   k3_traverse         Barnes-Hut (Eq. bh_criteria) on the octree, one point
//                       per lane, 32 points of consecutive voxels per warp, the
//                       siblings as packed FP32 pairs; k3_traverse_pt the same
//                       for small sets, one warp per point
//   k3_attract          Eq. grad's first term over P, one warp per row
//   k3_kl, k3_centre_y  Eq. cost_func; the embedding's output
//
// The kernels follow the 2-D ones' arithmetic: exact offsets from the split
// centre of mass, FP32 forces, FP64 Z and KL.
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace pxsne {

namespace {

constexpr double kR3 = 4294967296.0;  // 2^32 ulps per axis
constexpr int kT3Warps = 4;           // warps per traversal CTA
constexpr int kT3Stack = 72;          // entries per warp; depth <= 7 L + 1 <= 64

__host__ __device__ inline int64_t off3(int l) { return ((int64_t(1) << (3 * l)) - 1) / 7; }

// Every third bit from bit 0 (10 of them), and back.
__device__ __forceinline__ uint32_t spread3(uint32_t x) {
    x &= 0x3ffu;
    x = (x | (x << 16)) & 0x030000ffu;
    x = (x | (x << 8)) & 0x0300f00fu;
    x = (x | (x << 4)) & 0x030c30c3u;
    return (x | (x << 2)) & 0x09249249u;
}
__device__ __forceinline__ uint32_t gather3(uint32_t x) {
    x &= 0x09249249u;
    x = (x | (x >> 2)) & 0x030c30c3u;
    x = (x | (x >> 4)) & 0x0300f00fu;
    x = (x | (x >> 8)) & 0x030000ffu;
    return (x | (x >> 16)) & 0x3ffu;
}

// Morton key of voxel (px, py, pz): bit b of x at 3b, of y at 3b + 1, of z at 3b + 2.
__device__ __forceinline__ uint32_t morton3(uint32_t px, uint32_t py, uint32_t pz) {
    return spread3(px) | (spread3(py) << 1) | (spread3(pz) << 2);
}

// Coordinate `axis` (0, 1, 2) of a cell from its Morton index.
__device__ __forceinline__ uint32_t demorton3(uint32_t m, int axis) { return gather3(m >> axis); }

__device__ __forceinline__ float rcp3(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Ordered u32 key of a float (for the integer min/max atomics), and back.
__device__ __forceinline__ uint32_t key3(float f) {
    const uint32_t b = __float_as_uint(f);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float unkey3(uint32_t k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// Per-iteration scalars of the 3-D state from s (one thread).
__device__ void derive3(DevScalars *sc, float theta, int L) {
    for (int d = 0; d < 3; d++) {
        sc->inv_s3[d] = 1.0 / sc->s3[d];
        sc->sf3[d] = (float)sc->s3[d];
    }
    const double th2 = (double)theta * (double)theta;
    const double ss = sc->s3[0] * sc->s3[0] + sc->s3[1] * sc->s3[1] + sc->s3[2] * sc->s3[2];
    for (int l = 0; l <= kMaxL + 1; l++) {
        if (l > L) {
            sc->T3[l] = INFINITY;
            continue;
        }
        // the cell diagonal squared, W^2 (s0^2 + s1^2 + s2^2), W = 2^(32-l) ulps;
        // Eq. bh_criteria accepts when r_c^2 < theta^2 d^2
        const double rc2 = ldexp(1.0, 64 - 2 * l) * ss;
        sc->T3[l] = th2 > 0.0 ? (float)(rc2 / th2) : INFINITY;
    }
}

__device__ void reset_mm3(DevScalars *sc, int par) {
    for (int d = 0; d < 3; d++) {
        sc->mm3[par][d] = 0x7fffffffffffffffll;
        sc->mm3[par][3 + d] = (i64)0x8000000000000000ull;
    }
}

__global__ void k3_set_scalars(DevScalars *sc, double s0, double s1, double s2, int t, float theta,
                               int L) {
    sc->s3[0] = s0;
    sc->s3[1] = s1;
    sc->s3[2] = s2;
    sc->t = t;
    sc->Z = 0.0;
    derive3(sc, theta, L);
    reset_mm3(sc, 0);
    reset_mm3(sc, 1);
}

// ---- the start (Eq. z1/z2 per axis)
__global__ void k3_minmax(int n, const float *__restrict__ Y, uint32_t *mm, DevScalars *sc) {
    uint32_t lo[3] = {0xffffffffu, 0xffffffffu, 0xffffffffu}, hi[3] = {0u, 0u, 0u};
    bool bad = false;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        for (int d = 0; d < 3; d++) {
            const float y = Y[3 * (int64_t)i + d];
            bad |= !isfinite(y);
            const uint32_t k = key3(y);
            lo[d] = min(lo[d], k);
            hi[d] = max(hi[d], k);
        }
    for (int d = 0; d < 3; d++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo[d] = min(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
            hi[d] = max(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
        }
    }
    if ((threadIdx.x & 31) == 0)
        for (int d = 0; d < 3; d++) {
            atomicMin(&mm[d], lo[d]);
            atomicMax(&mm[3 + d], hi[d]);
        }
    if (bad) atomicOr(&sc->err, (unsigned)PXSNE_DEVERR_NONFINITE);
}

__global__ void k3_map(int n, int L, float theta, const float *__restrict__ Y,
                       const uint32_t *__restrict__ mm, uint4 *__restrict__ z,
                       float4 *__restrict__ u, float4 *__restrict__ gains, DevScalars *sc) {
    double mn[3], rg[3];
    for (int d = 0; d < 3; d++) {
        mn[d] = (double)unkey3(mm[d]);
        rg[d] = (double)unkey3(mm[3 + d]) - mn[d];
    }
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) {
        for (int d = 0; d < 3; d++) sc->s3[d] = rg[d] > 0.0 ? rg[d] / kR3 : 1.0 / kR3;
        derive3(sc, theta, L);
        sc->t = 0;
        sc->Z = 0.0;
        reset_mm3(sc, 0);
        reset_mm3(sc, 1);
    }
    if (i >= n) return;
    uint32_t q3[3] = {0u, 0u, 0u};
    for (int d = 0; d < 3; d++) {
        if (!(rg[d] > 0.0)) continue;
        const double q = floor(((double)Y[3 * (int64_t)i + d] - mn[d]) * kR3 / rg[d]);
        q3[d] = q >= kR3 - 1.0 ? 0xffffffffu : (uint32_t)q;
    }
    z[i] = make_uint4(q3[0], q3[1], q3[2], 0u);
    u[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    gains[i] = make_float4(1.f, 1.f, 1.f, 0.f);
}

// ---- the gradient step per coordinate, and the extremes of zhat per axis
__global__ void __launch_bounds__(256)
    k3_update(int n, UpdateParams p, const uint4 *__restrict__ z, const float4 *__restrict__ Frep,
              const float4 *__restrict__ Fattr, float4 *__restrict__ u, float4 *__restrict__ gains,
              long long *__restrict__ zhat, DevScalars *sc) {
    __shared__ i64 s_mm[6][8];
    const int t = sc->t;
    const float alpha = t < p.exag_iters ? p.exag : 1.0f;
    const float mu = t < p.mom_switch ? p.mom0 : p.mom1;
    // 1 / Z once per CTA (an FP64 division)
    __shared__ float s_invZ;
    if (threadIdx.x == 0) {
        const double Z = sc->Z;
        s_invZ = Z > 0.0 ? (float)(1.0 / Z) : 0.0f;
    }
    __syncthreads();
    const float invZ = s_invZ;
    const double is0 = sc->inv_s3[0], is1 = sc->inv_s3[1], is2 = sc->inv_s3[2];
    i64 lo[3], hi[3];
    for (int d = 0; d < 3; d++) {
        lo[d] = 0x7fffffffffffffffll;
        hi[d] = (i64)0x8000000000000000ull;
    }
    unsigned err = 0u;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const float4 fr = Frep[i], fa = Fattr[i];
        float4 uu = u[i], gg = gains[i];
        const uint4 zz = z[i];
        i64 zh[3];
        zh[0] = step1(fa.x, fr.x, alpha, invZ, mu, p, uu.x, gg.x, zz.x, is0, err);
        zh[1] = step1(fa.y, fr.y, alpha, invZ, mu, p, uu.y, gg.y, zz.y, is1, err);
        zh[2] = step1(fa.z, fr.z, alpha, invZ, mu, p, uu.z, gg.z, zz.z, is2, err);
        u[i] = uu;
        gains[i] = gg;
        for (int d = 0; d < 3; d++) {
            zhat[3 * (int64_t)i + d] = zh[d];
            lo[d] = min(lo[d], zh[d]);
            hi[d] = max(hi[d], zh[d]);
        }
    }
    for (int d = 0; d < 3; d++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lo[d] = min(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], o));
            hi[d] = max(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], o));
        }
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0)
        for (int d = 0; d < 3; d++) {
            s_mm[d][w] = lo[d];
            s_mm[3 + d][w] = hi[d];
        }
    if (err) atomicOr(&sc->err, err);
    __syncthreads();
    if (threadIdx.x < 6) {
        const int k = threadIdx.x;
        const int nw = blockDim.x >> 5;
        i64 v = s_mm[k][0];
        for (int q = 1; q < nw; q++) v = k < 3 ? min(v, s_mm[k][q]) : max(v, s_mm[k][q]);
        long long *dst = reinterpret_cast<long long *>(&sc->mm3[t & 1][k]);
        if (k < 3) atomicMin(dst, (long long)v);
        else atomicMax(dst, (long long)v);
    }
}

// ---- the rescale (Sec. 4.2, exact integers, R = 2^32 per axis), the voxel
// snap and the leaf histogram; the rank of each point inside its voxel is the
// count before it (the order inside a voxel enters no result)
__global__ void k3_snap(int n, int L, int rescale, float theta, const long long *__restrict__ zhat,
                        uint4 *__restrict__ z, uint32_t *__restrict__ rank,
                        uint32_t *__restrict__ cnt, u64 *__restrict__ sx, u64 *__restrict__ sy,
                        u64 *__restrict__ sz, DevScalars *sc) {
    const int F = 32 - L;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t zv[3];
    if (rescale) {
        const int par = sc->t & 1;
        i64 mn[3];
        u64 g[3];
        double q[3];
        __shared__ double s_q[3];
        for (int d = 0; d < 3; d++) {
            mn[d] = sc->mm3[par][d];
            g[d] = (u64)(sc->mm3[par][3 + d] - mn[d]) + 1ull;
        }
        // one FP64 division per axis and CTA (the same for every point)
        if (threadIdx.x < 3) s_q[threadIdx.x] = kR3 / (double)g[threadIdx.x];
        __syncthreads();
        for (int d = 0; d < 3; d++) q[d] = s_q[d];
        if (i == 0) {
            // Eq. beta_scaling carried as s_d <- (s_d * gamma_d) / 2^32
            for (int d = 0; d < 3; d++) sc->s3[d] = (sc->s3[d] * (double)g[d]) / kR3;
            derive3(sc, theta, L);
            reset_mm3(sc, par ^ 1);
        }
        if (i >= n) return;
        for (int d = 0; d < 3; d++)
            zv[d] = rescale_exact((u64)(zhat[3 * (int64_t)i + d] - mn[d]), g[d], q[d],
                                  u64(1) << 32);
        z[i] = make_uint4(zv[0], zv[1], zv[2], 0u);
    } else {
        if (i >= n) return;
        const uint4 v = z[i];
        zv[0] = v.x;
        zv[1] = v.y;
        zv[2] = v.z;
    }
    const uint32_t m = morton3(zv[0] >> F, zv[1] >> F, zv[2] >> F);
    rank[i] = atomicAdd(&cnt[m], 1u);
    atomicAdd(&sx[m], (u64)zv[0]);
    atomicAdd(&sy[m], (u64)zv[1]);
    atomicAdd(&sz[m], (u64)zv[2]);
}

// The records.  The eight siblings of a node share a group of 56 floats, as
// in 2-D a structure of arrays: the negated halves -c_hi_x [8], -c_lo_x [8], and
// the same for y and z, of their centres of mass (record_axis), then their
// counts [8].  The group of the children (level l + 1) of cell m of level l is
// group off3(l) + m, so that child c of group G has its own children in group
// 8 G + 1 + c.  Only groups with a point are written; an empty sibling's centre
// weighs nothing.
constexpr int kGroup3 = 56;  // floats per sibling group, 14 float4s

__device__ __forceinline__ void put_record3(float *rec, int l, int64_t c, uint32_t N, u64 X, u64 Y,
                                            u64 Zs) {
    float *g = rec + (off3(l - 1) + (c >> 3)) * kGroup3 + (c & 7);
    float h[3] = {0.f, 0.f, 0.f}, e[3] = {0.f, 0.f, 0.f};
    if (N != 0u) {
        const int sh = 32 - l;
        record_axis(N, X, demorton3((uint32_t)c, 0) << sh, sh, h[0], e[0]);
        record_axis(N, Y, demorton3((uint32_t)c, 1) << sh, sh, h[1], e[1]);
        record_axis(N, Zs, demorton3((uint32_t)c, 2) << sh, sh, h[2], e[2]);
    }
#pragma unroll
    for (int d = 0; d < 3; d++) {
        g[16 * d] = -h[d];
        g[16 * d + 8] = -e[d];
    }
    g[48] = (float)N;
}

// The sum over the eight threads of a sibling group, for all of them.
__device__ __forceinline__ void sum8(unsigned mask, uint32_t &N, u64 &X, u64 &Y, u64 &Zs) {
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) {
        N += __shfl_xor_sync(mask, N, o);
        X += __shfl_xor_sync(mask, X, o);
        Y += __shfl_xor_sync(mask, Y, o);
        Zs += __shfl_xor_sync(mask, Zs, o);
    }
}

// One level of the octree from the one below: a thread per sibling group of
// level h.  Writes the group's records, the count and sums of its parent, and
// the children's starts among the group's points: a point's place in the
// counting sort is the sum of its cells' starts over the levels, so no scan of
// the voxels is needed.  clear: the cells are the leaves, and an occupied one
// goes back to zero once read (the next histogram starts from zeros without a
// memset of every leaf).  A group without a point costs its 32 bytes of counts
// and a zero for its parent: what bounds the kernel on a sparse grid is how many
// bytes of counts are in flight, hence the whole group per thread.  n = 200,000
// on 256^3, all levels: 0.10 ms; a thread per cell 0.39, three levels per CTA of
// 512 cells 0.33, and with every cell's sums read and records written and a scan
// of the voxel counts 0.44.
__global__ void __launch_bounds__(256)
    k3_level(int h, int clear, uint32_t *cnt, u64 *sx, u64 *sy, u64 *sz, float4 *__restrict__ rec,
             uint32_t *__restrict__ pref) {
    const int64_t grp = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (grp >= (int64_t(1) << (3 * (h - 1)))) return;
    const int64_t up = off3(h - 1) + grp, at = off3(h) + 8 * grp;
    uint32_t N[8];
    uint32_t gN = 0u;
    // (off3(h) is odd: the counts of a group are not 16-byte aligned, the
    // threads of a warp still read one run of bytes)
#pragma unroll
    for (int c = 0; c < 8; c++) {
        N[c] = cnt[at + c];
        gN += N[c];
    }
    cnt[up] = gN;
    if (gN == 0u) return;
    uint32_t run = 0u;
#pragma unroll
    for (int c = 0; c < 8; c++) {
        if (N[c] != 0u) {
            pref[at + c] = run;
            if (clear) cnt[at + c] = 0u;
        }
        run += N[c];
    }
    float4 *g = rec + (off3(h - 1) + grp) * (kGroup3 / 4);
    g[12] = make_float4((float)N[0], (float)N[1], (float)N[2], (float)N[3]);
    g[13] = make_float4((float)N[4], (float)N[5], (float)N[6], (float)N[7]);
    const int sh = 32 - h;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        u64 *s = d == 0 ? sx : d == 1 ? sy : sz;
        u64 S[8], sum = 0ull;
#pragma unroll
        for (int c = 0; c < 8; c++) S[c] = N[c] != 0u ? s[at + c] : 0ull;
        // the group's corner, and whether child c lies on its far side
        const uint32_t base = gather3((uint32_t)(grp >> d)) << (sh + 1);
        float hi[8], lo[8];
#pragma unroll
        for (int c = 0; c < 8; c++) {
            hi[c] = lo[c] = 0.f;
            if (N[c] != 0u) {
                record_axis(N[c], S[c], base + (((uint32_t)c >> d) & 1u) * (1u << sh), sh, hi[c], lo[c]);
                if (clear) s[at + c] = 0ull;
            }
            sum += S[c];
        }
        s[up] = sum;
        g[4 * d] = make_float4(-hi[0], -hi[1], -hi[2], -hi[3]);
        g[4 * d + 1] = make_float4(-hi[4], -hi[5], -hi[6], -hi[7]);
        g[4 * d + 2] = make_float4(-lo[0], -lo[1], -lo[2], -lo[3]);
        g[4 * d + 3] = make_float4(-lo[4], -lo[5], -lo[6], -lo[7]);
    }
}

// The top K levels in one CTA: a thread per cell of level K, whose starts among
// all points it writes.
template <int K>
__global__ void __launch_bounds__(1 << (3 * K))
    k3_top(int clear, uint32_t *cnt, u64 *sx, u64 *sy, u64 *sz, float *__restrict__ rec,
           uint32_t *__restrict__ pref) {
    constexpr int NT = 1 << (3 * K);
    constexpr unsigned MASK = NT >= 32 ? 0xffffffffu : (1u << (NT & 31)) - 1u;
    __shared__ uint32_t s_w[NT >= 32 ? NT / 32 : 1];
    __shared__ uint32_t s_n[NT / 8];
    __shared__ u64 s_s[3][NT / 8];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t at = off3(K) + tid;
    uint32_t N = cnt[at];
    u64 X = 0ull, Y = 0ull, Zs = 0ull;
    if (N != 0u) {
        X = sx[at];
        Y = sy[at];
        Zs = sz[at];
        if (clear) {
            cnt[at] = 0u;
            sx[at] = 0ull;
            sy[at] = 0ull;
            sz[at] = 0ull;
        }
    }
    uint32_t inc = N;
#pragma unroll
    for (int o = 1; o < (NT >= 32 ? 32 : NT); o <<= 1) {
        const uint32_t t = __shfl_up_sync(MASK, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31 || tid == NT - 1) s_w[warp] = inc;
    __syncthreads();
    uint32_t before = 0u;
    for (int w = 0; w < warp; w++) before += s_w[w];
    pref[at] = before + inc - N;
#pragma unroll
    for (int k = 0; k < K; k++) {
        // level K - k: 8^(K - k) threads hold its cells
        const int cells = NT >> (3 * k);
        const bool in = tid < cells;
        uint32_t gN = N;
        u64 gX = X, gY = Y, gZ = Zs;
        // (whole warps, or the CTA's only one: the shuffles need them all)
        if (tid < ((cells + 31) & ~31)) {
            sum8(MASK, gN, gX, gY, gZ);
            if (in && gN != 0u) put_record3(rec, K - k, tid, N, X, Y, Zs);
        }
        if (in && (tid & 7) == 0) {
            s_n[tid >> 3] = gN;
            s_s[0][tid >> 3] = gX;
            s_s[1][tid >> 3] = gY;
            s_s[2][tid >> 3] = gZ;
        }
        __syncthreads();
        const bool up = tid < (cells >> 3);
        N = up ? s_n[tid] : 0u;
        X = up ? s_s[0][tid] : 0ull;
        Y = up ? s_s[1][tid] : 0ull;
        Zs = up ? s_s[2][tid] : 0ull;
        if (up) cnt[off3(K - k - 1) + tid] = N;
        __syncthreads();
    }
}

// the counting sort by voxel: perm[start of the voxel + rank] = i; the
// iteration counter advances here for an iteration
__global__ void k3_perm(int n, int L, const uint4 *__restrict__ z, const uint32_t *__restrict__ rank,
                        const uint32_t *__restrict__ pref, uint32_t *__restrict__ perm,
                        DevScalars *sc, int bump_t) {
    const int F = 32 - L;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (bump_t && i == 0) sc->t += 1;
    if (i >= n) return;
    const uint4 v = z[i];
    const uint32_t m = morton3(v.x >> F, v.y >> F, v.z >> F);
    uint32_t pos = rank[i], a = m;
    int l = L;
    for (; l > 3; l--, a >>= 3) pos += pref[off3(l) + a];
    pos += pref[off3(l) + a];  // the top level's starts are among all points
    if (pos < (uint32_t)n) perm[pos] = (uint32_t)i;
    else atomicOr(&sc->err, (unsigned)PXSNE_DEVERR_STACK);
}

// ---- Barnes-Hut on the octree.  A warp takes 32 points consecutive in voxel
// order, one per lane, and walks the octree depth-first; each stack entry is a
// node with the mask of the lanes whose point opens it, so every point sees
// exactly the cells its own depth-first search would, in the tree's order.
// As in 2-D the siblings enter the arithmetic as packed pairs straight from their
// group's arrays, children at the voxel level are always accepted (bounded
// depth) except a point's own voxel, used without the point itself, and above
// it Eq. bh_criteria decides, the cell holding a point is opened, and a cell
// of one point, whose centre is that point exactly, is accepted by all others.
// 200,000 points on 256^3 (late state): 2.2 ms, 3.5 with one scalar child after
// the other and single points opened down to their voxels.
struct Point3 {
    float2 h[3], l[3];
};
__device__ __forceinline__ float2 b3(float v) { return make_float2(v, v); }
__device__ __forceinline__ Point3 point3(uint4 z) {
    const uint32_t v[3] = {z.x, z.y, z.z};
    Point3 p;
#pragma unroll
    for (int d = 0; d < 3; d++) {
        p.h[d] = b3((float)(v[d] & 0xffff0000u));
        p.l[d] = b3((float)(v[d] & 0xffffu));
    }
    return p;
}
__device__ __forceinline__ float2 half2of(float4 v, int p) {
    return p ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
}

// The force sums of a point, even and odd siblings apart.
struct Sum3 {
    float2 f[3], z;
};

// Pair p (0, 1) of one half (four siblings, r = its six arrays' float4s): the
// offsets in ulps from the pair's centres.
__device__ __forceinline__ void offset3(const float4 (&r)[6], int p, const Point3 &pt,
                                        float2 (&dx)[3]) {
#pragma unroll
    for (int d = 0; d < 3; d++)
        dx[d] = __fadd2_rn(__fadd2_rn(pt.h[d], half2of(r[2 * d], p)),
                           __fadd2_rn(pt.l[d], half2of(r[2 * d + 1], p)));
}

// y-units and the squared distances.
__device__ __forceinline__ float2 dist3(float2 (&dx)[3], const float2 (&s)[3]) {
#pragma unroll
    for (int d = 0; d < 3; d++) dx[d] = __fmul2_rn(dx[d], s[d]);
    return __ffma2_rn(dx[0], dx[0], __ffma2_rn(dx[1], dx[1], __fmul2_rn(dx[2], dx[2])));
}

__device__ __forceinline__ void add3(Sum3 &a, float2 N, float2 d2, const float2 (&dx)[3]) {
    const float2 w = __fadd2_rn(b3(1.0f), d2);
    const float2 q = make_float2(rcp3(w.x), rcp3(w.y));
    const float2 Nq = __fmul2_rn(N, q);
    a.z = __fadd2_rn(a.z, Nq);
    const float2 Nq2 = __fmul2_rn(Nq, q);
#pragma unroll
    for (int d = 0; d < 3; d++) a.f[d] = __ffma2_rn(Nq2, dx[d], a.f[d]);
}

// Takes the point itself out of its own voxel (slot of the pair's two): one
// fewer, the centre of mass of the others.
__device__ __forceinline__ void take_out3(int slot, float2 &N, float2 (&dx)[3]) {
    const float Nc = slot ? N.y : N.x, r = Nc - 1.0f;
    const float k = r > 0.0f ? Nc / r : 1.0f;
    if (slot) {
        N.y = r;
        for (int d = 0; d < 3; d++) dx[d].y *= k;
    } else {
        N.x = r;
        for (int d = 0; d < 3; d++) dx[d].x *= k;
    }
}

// Cells of one point are accepted by all others by the same rule as in 2-D
// (single_base, common.cuh).
template <bool OWN>
__device__ __forceinline__ float base3(const DevScalars *sc) {
    return single_base(OWN || underflows(sc->sf3[0]) || underflows(sc->sf3[1]) ||
                       underflows(sc->sf3[2]));
}
// What a point (its voxel's Morton index mi) has to take out of its sum.
template <bool OWN>
__device__ __forceinline__ float own_single3(float base, const float4 *__restrict__ rec, int L,
                                             uint32_t mi) {
    if (OWN || base == -kManyT || L < 2) return 0.f;
    const float *g = reinterpret_cast<const float *>(rec) + (off3(L - 2) + (mi >> 6)) * kGroup3;
    return g[48 + ((mi >> 3) & 7u)] == 1.f ? 1.f : 0.f;
}

struct __align__(8) T3Entry {
    uint32_t node, mask;  // (children's level << 28) | their group; lanes that open it
};

template <bool OWN>
__global__ void __launch_bounds__(kT3Warps * 32, 4)
    k3_traverse(int n, int L, const uint4 *__restrict__ z, const uint32_t *__restrict__ perm,
                const float4 *__restrict__ rec, DevScalars *sc, float4 *__restrict__ Frep,
                float *__restrict__ Zi) {
    __shared__ T3Entry s_stk[kT3Warps][kT3Stack];
    __shared__ float2 s_T[kMaxL + 2];  // a level's threshold on d^2, and single_base
    if (threadIdx.x < kMaxL + 2) s_T[threadIdx.x] = make_float2(sc->T3[threadIdx.x], base3<OWN>(sc));
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int idx = (blockIdx.x * kT3Warps + w) * 32 + lane;
    const bool valid = idx < n;
    const unsigned act = __ballot_sync(0xffffffffu, valid);
    if (act == 0u) return;
    const int F = 32 - L;
    const uint32_t i = valid ? perm[idx] : 0u;
    const uint4 zi = z[i];
    const uint32_t mi = morton3(zi.x >> F, zi.y >> F, zi.z >> F);
    const uint32_t own_grp = (uint32_t)off3(L - 1) + (mi >> 3);
    const Point3 pt = point3(zi);
    const float2 s[3] = {b3(sc->sf3[0]), b3(sc->sf3[1]), b3(sc->sf3[2])};
    Sum3 a{{b3(0.f), b3(0.f), b3(0.f)}, b3(0.f)};
    T3Entry *stk = s_stk[w];
    if (lane == 0) stk[0] = T3Entry{1u << 28, act};  // the root's children: level 1, group 0
    int sp = 1;
    __syncwarp();
    bool overflow = false;
    while (sp > 0) {
        sp--;
        T3Entry top = stk[sp];
        __syncwarp();
        top.node = __shfl_sync(0xffffffffu, top.node, 0);
        top.mask = __shfl_sync(0xffffffffu, top.mask, 0);
        const uint32_t grp = top.node & 0x0fffffffu;
        const int lc = (int)(top.node >> 28);
        const bool me = (top.mask >> lane) & 1u;
        const float4 *g = rec + (size_t)grp * (kGroup3 / 4);
        // the counts and the first half's records are requested together (both
        // halves' took registers: 6.7 against 6.2 ms for four iterations)
        const float4 nv[2] = {__ldg(g + 12), __ldg(g + 13)};
        float4 rr[2][6];
#pragma unroll
        for (int q = 0; q < 6; q++) rr[0][q] = __ldg(g + 2 * q);
        if (lc == L) {
            const bool own = me && own_grp == grp;
            const bool any_own = __any_sync(0xffffffffu, own);
#pragma unroll
            for (int hf = 0; hf < 2; hf++) {
                if (nv[hf].x + nv[hf].y + nv[hf].z + nv[hf].w == 0.f) continue;
                if (hf == 1)
                    for (int q = 0; q < 6; q++) rr[1][q] = __ldg(g + 2 * q + 1);
                const float4(&r)[6] = rr[hf];
#pragma unroll
                for (int p = 0; p < 2; p++) {
                    float2 N = half2of(nv[hf], p);
                    if (N.x + N.y == 0.f) continue;
                    float2 dx[3];
                    offset3(r, p, pt, dx);
                    if (any_own && own && (int)((mi & 7u) >> 1) == 2 * hf + p)
                        take_out3((int)(mi & 1u), N, dx);
                    const float2 d2 = dist3(dx, s);
                    add3(a, make_float2(me ? N.x : 0.f, me ? N.y : 0.f), d2, dx);
                }
            }
        } else {
            const float2 Tb = s_T[lc];
            const float Tl = Tb.x, base = OWN ? single_base(true) : Tb.y;
            const uint32_t mine = OWN ? mi >> (3 * (L - lc)) : 0u;
            const uint32_t first = OWN ? 8u * (grp - (uint32_t)off3(lc - 1)) : 0u;
            if (sp + 8 > kT3Stack) {
                overflow = true;
                break;
            }
            // lanes 0 .. 7 keep the acceptances of their child
            unsigned taken = 0u;
#pragma unroll
            for (int hf = 0; hf < 2; hf++) {
                if (nv[hf].x + nv[hf].y + nv[hf].z + nv[hf].w == 0.f) continue;
                if (hf == 1)
                    for (int q = 0; q < 6; q++) rr[1][q] = __ldg(g + 2 * q + 1);
                const float4(&r)[6] = rr[hf];
#pragma unroll
                for (int p = 0; p < 2; p++) {
                    const int c = 4 * hf + 2 * p;
                    const float2 N = half2of(nv[hf], p);
                    if (N.x + N.y == 0.f) continue;
                    float2 dx[3];
                    offset3(r, p, pt, dx);
                    const float2 d2 = dist3(dx, s);
                    const float2 tb = __ffma2_rn(N, b3(kManyT), b3(base));
                    const bool a0 = me && d2.x > fminf(tb.x, Tl) && (!OWN || mine != first + c);
                    const bool a1 = me && d2.y > fminf(tb.y, Tl) && (!OWN || mine != first + c + 1);
                    add3(a, make_float2(a0 ? N.x : 0.f, a1 ? N.y : 0.f), d2, dx);
                    const unsigned b0 = __ballot_sync(0xffffffffu, a0);
                    const unsigned b1 = __ballot_sync(0xffffffffu, a1);
                    if (lane == c) taken = b0;
                    if (lane == c + 1) taken = b1;
                }
            }
            // they push their child if it holds several points and some lane opens it
            const float nn = lane < 8 ? __ldg(reinterpret_cast<const float *>(g + 12) + lane) : 0.f;
            const unsigned o = top.mask & ~taken;
            const bool push = nn > 1.f && o != 0u;
            const unsigned pm = __ballot_sync(0xffffffffu, push);
            if (push)
                stk[sp + __popc(pm & ((1u << lane) - 1u))] =
                    T3Entry{((uint32_t)(lc + 1) << 28) | (8u * grp + 1u + (uint32_t)lane), o};
            sp += __popc(pm);
        }
        __syncwarp();
    }
    if (valid) {
        Frep[i] = make_float4(a.f[0].x + a.f[0].y, a.f[1].x + a.f[1].y, a.f[2].x + a.f[2].y, 0.f);
        Zi[i] = a.z.x + a.z.y - own_single3<OWN>(s_T[0].y, rec, L, mi);
    }
    if (overflow && lane == 0) atomicOr(&sc->err, (unsigned)PXSNE_DEVERR_STACK);
}

// One warp per point, up to 32 of its open nodes at a time (the 2-D kernel's
// scheme, forces.cu): for sets too small to fill the chip with warps of 32
// points.  A step adds at most 256 nodes of the next level, so a node of level
// l waits at most 256 l places above kPt3Deep + 224.
constexpr int kPt3Warps = 4;
constexpr int kPt3Ring = 4096;
constexpr int kPt3Deep = kPt3Ring - 256 * kMaxL3 - 256;
static_assert(kPt3Deep >= 256, "ring of the point traversal");
constexpr size_t kPt3Smem = (size_t)kPt3Warps * kPt3Ring * 4;
template <bool OWN>
__global__ void __launch_bounds__(kPt3Warps * 32)
    k3_traverse_pt(int n, int L, const uint4 *__restrict__ z, const uint32_t *__restrict__ perm,
                   const float4 *__restrict__ rec, const DevScalars *__restrict__ sc,
                   float4 *__restrict__ Frep, float *__restrict__ Zi) {
    extern __shared__ uint32_t s_ring[];
    __shared__ float s_T[kMaxL + 2];
    if (threadIdx.x < kMaxL + 2) s_T[threadIdx.x] = sc->T3[threadIdx.x];
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int idx = blockIdx.x * kPt3Warps + w;
    if (idx >= n) return;  // whole warps; no block barrier follows
    uint32_t *ring = s_ring + w * kPt3Ring;
    const int F = 32 - L;
    const uint32_t i = perm[idx];
    const uint4 zi = z[i];
    const uint32_t mi = morton3(zi.x >> F, zi.y >> F, zi.z >> F);
    const uint32_t own_grp = (uint32_t)off3(L - 1) + (mi >> 3);
    const Point3 pt = point3(zi);
    const float2 s[3] = {b3(sc->sf3[0]), b3(sc->sf3[1]), b3(sc->sf3[2])};
    const float base = base3<OWN>(sc);
    Sum3 a{{b3(0.f), b3(0.f), b3(0.f)}, b3(0.f)};
    const unsigned before = (1u << lane) - 1u;
    if (lane == 0) ring[0] = 1u << 28;
    uint32_t head = 0u, size = 1u;
    __syncwarp();
    while (size > 0u) {
        const uint32_t k = min(size, 32u);
        const uint32_t at = size <= (uint32_t)kPt3Deep ? head : head + size - k;
        if (size <= (uint32_t)kPt3Deep) head += k;
        size -= k;
        const bool act = (uint32_t)lane < k;
        const uint32_t node = act ? ring[(at + lane) & (kPt3Ring - 1)] : 1u << 28;
        __syncwarp();
        const uint32_t grp = node & 0x0fffffffu;
        const int lc = (int)(node >> 28);
        const bool leaf = lc == L;
        const float4 *g = rec + (size_t)grp * (kGroup3 / 4);
        const float Tl = s_T[lc];
        const bool own = act && leaf && own_grp == grp;
        const uint32_t mine = OWN ? mi >> (3 * (L - lc)) : 0u;
        const uint32_t first = OWN ? 8u * (grp - (uint32_t)off3(lc - 1)) : 0u;
        unsigned open = 0u;  // this lane's children to open
#pragma unroll
        for (int hf = 0; hf < 2; hf++) {
            const float4 nv = act ? __ldg(g + 12 + hf) : make_float4(0.f, 0.f, 0.f, 0.f);
            if (nv.x + nv.y + nv.z + nv.w == 0.f) continue;
            float4 r[6];
#pragma unroll
            for (int q = 0; q < 6; q++) r[q] = __ldg(g + 2 * q + hf);
#pragma unroll
            for (int p = 0; p < 2; p++) {
                const int c = 4 * hf + 2 * p;
                const float2 N0 = half2of(nv, p);
                float2 N = N0, dx[3];
                offset3(r, p, pt, dx);
                if (own && (int)((mi & 7u) >> 1) == 2 * hf + p) take_out3((int)(mi & 1u), N, dx);
                const float2 d2 = dist3(dx, s);
                const float2 tb = __ffma2_rn(N0, b3(kManyT), b3(base));
                const float T0 = leaf ? -1.0f : fminf(tb.x, Tl), T1 = leaf ? -1.0f : fminf(tb.y, Tl);
                const bool a0 = d2.x > T0 && (!OWN || leaf || mine != first + c);
                const bool a1 = d2.y > T1 && (!OWN || leaf || mine != first + c + 1);
                add3(a, make_float2(a0 ? N.x : 0.f, a1 ? N.y : 0.f), d2, dx);
                // (a voxel is never opened, whatever a non-finite distance says)
                open |= (!a0 && !leaf && N0.x > 1.f ? 1u : 0u) << c;
                open |= (!a1 && !leaf && N0.y > 1.f ? 2u : 0u) << c;
            }
        }
        __syncwarp();
        const uint32_t child = ((uint32_t)(lc + 1) << 28) | (8u * grp + 1u);
        uint32_t end = head + size;
#pragma unroll
        for (int c = 0; c < 8; c++) {
            const bool o = (open >> c) & 1u;
            const unsigned b = __ballot_sync(0xffffffffu, o);
            if (o) ring[(end + __popc(b & before)) & (kPt3Ring - 1)] = child + (uint32_t)c;
            end += __popc(b);
        }
        size = end - head;
        __syncwarp();
    }
    float v[4] = {a.f[0].x + a.f[0].y, a.f[1].x + a.f[1].y, a.f[2].x + a.f[2].y, a.z.x + a.z.y};
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int d = 0; d < 4; d++) v[d] += __shfl_xor_sync(0xffffffffu, v[d], o);
    if (lane == 0) {
        Frep[i] = make_float4(v[0], v[1], v[2], 0.f);
        Zi[i] = v[3] - own_single3<OWN>(base, rec, L, mi);
    }
}

// ---- Eq. grad's first term, one warp per row of P (rows padded with zero
// entries that point at the row itself); z_i - z_j exact in float from the
// 16-bit halves, one rounding
__global__ void __launch_bounds__(256)
    k3_attract(int n, const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
               const float *__restrict__ val, const uint4 *__restrict__ z,
               const DevScalars *__restrict__ sc, float4 *__restrict__ Fattr) {
    const int lane = threadIdx.x & 31;
    const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (row >= n) return;
    const float s0 = sc->sf3[0], s1 = sc->sf3[1], s2 = sc->sf3[2];
    const uint4 zi = z[row];
    const float xh = (float)(zi.x & 0xffff0000u), xl = (float)(zi.x & 0xffffu);
    const float yh = (float)(zi.y & 0xffff0000u), yl = (float)(zi.y & 0xffffu);
    const float zh = (float)(zi.z & 0xffff0000u), zl = (float)(zi.z & 0xffffu);
    float fx = 0.f, fy = 0.f, fz = 0.f;
    for (int64_t e = rp[row] + lane; e < rp[row + 1]; e += 32) {
        const int32_t j = __ldcs(col + e);
        const float p = __ldcs(val + e);
        const uint4 zj = z[j];
        const float dx =
            ((xh - (float)(zj.x & 0xffff0000u)) + (xl - (float)(zj.x & 0xffffu))) * s0;
        const float dy =
            ((yh - (float)(zj.y & 0xffff0000u)) + (yl - (float)(zj.y & 0xffffu))) * s1;
        const float dz =
            ((zh - (float)(zj.z & 0xffff0000u)) + (zl - (float)(zj.z & 0xffffu))) * s2;
        const float wgt = __fdividef(1.0f, 1.0f + fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
        const float pw = p * wgt;
        fx = fmaf(pw, dx, fx);
        fy = fmaf(pw, dy, fy);
        fz = fmaf(pw, dz, fz);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        fx += __shfl_xor_sync(0xffffffffu, fx, o);
        fy += __shfl_xor_sync(0xffffffffu, fy, o);
        fz += __shfl_xor_sync(0xffffffffu, fz, o);
    }
    if (lane == 0) Fattr[row] = make_float4(fx, fy, fz, 0.f);
}

// ---- Eq. cost_func: sum p (ln p + ln(1 + d^2)) + (sum p) ln Z, FP32 terms
// accumulated in FP64 in a fixed order, the last block adding the partials
__device__ double block_sum3(double v, double *s_red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) s_red[warp] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int k = 0; k < (int)(blockDim.x >> 5); k++) t += s_red[k];
    __syncthreads();
    return t;
}

__global__ void __launch_bounds__(256)
    k3_kl(int n, const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
          const float *__restrict__ val, const uint4 *__restrict__ z, DevScalars *sc,
          double *__restrict__ part, double *out) {
    __shared__ double s_red[8];
    __shared__ bool s_last;
    const int lane = threadIdx.x & 31;
    const int warps_total = gridDim.x * (blockDim.x >> 5);
    const float s0 = sc->sf3[0], s1 = sc->sf3[1], s2 = sc->sf3[2];
    double acc = 0.0, psum = 0.0;
    for (int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); row < n;
         row += warps_total) {
        const uint4 zi = z[row];
        for (int64_t e = rp[row] + lane; e < rp[row + 1]; e += 32) {
            const float p = val[e];
            if (!(p > 0.f)) continue;
            const uint4 zj = z[col[e]];
            const float dx = (float)((int64_t)zi.x - (int64_t)zj.x) * s0;
            const float dy = (float)((int64_t)zi.y - (int64_t)zj.y) * s1;
            const float dz = (float)((int64_t)zi.z - (int64_t)zj.z) * s2;
            acc += (double)(p * (logf(p) + log1pf(fmaf(dx, dx, fmaf(dy, dy, dz * dz)))));
            psum += (double)p;
        }
    }
    const double a = block_sum3(acc, s_red);
    const double ps = block_sum3(psum, s_red);
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = a;
        part[2 * blockIdx.x + 1] = ps;
        __threadfence();
        const unsigned tk = atomicAdd(&sc->ticket2, 1u);
        s_last = (tk == gridDim.x - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (threadIdx.x == 0) {
        double A = 0.0, S = 0.0;
        volatile double *vp = part;
        for (int k = 0; k < (int)gridDim.x; k++) {
            A += vp[2 * k];
            S += vp[2 * k + 1];
        }
        *out = A + S * log(sc->Z);
        sc->ticket2 = 0u;
    }
}

// ---- output: y = s z minus the per-axis mean (FP64 sums), voxels z >> F
__global__ void k3_sum_y(int n, const uint4 *__restrict__ z, const DevScalars *sc, double *sums) {
    double a[3] = {0.0, 0.0, 0.0};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const uint4 v = z[i];
        a[0] += (double)v.x * sc->s3[0];
        a[1] += (double)v.y * sc->s3[1];
        a[2] += (double)v.z * sc->s3[2];
    }
    for (int d = 0; d < 3; d++) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a[d] += __shfl_xor_sync(0xffffffffu, a[d], o);
        if ((threadIdx.x & 31) == 0) atomicAdd(&sums[d], a[d]);
    }
}

__global__ void k3_write_y(int n, int L, const uint4 *__restrict__ z, const DevScalars *sc,
                           const double *sums, float *Y, int32_t *pix) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint4 v = z[i];
    const uint32_t zz[3] = {v.x, v.y, v.z};
    for (int d = 0; d < 3; d++) {
        if (Y) Y[3 * (int64_t)i + d] = (float)((double)zz[d] * sc->s3[d] - sums[d] / (double)n);
        if (pix) pix[3 * (int64_t)i + d] = (int32_t)(zz[d] >> (32 - L));
    }
}

// The leaf histogram of the current state, for inspection (the iteration's
// own is cleared by the first reduction once read).
__global__ void k3_leaf_hist(int n, int L, const uint4 *__restrict__ z, uint32_t *cnt, u64 *sx,
                             u64 *sy, u64 *sz) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int F = 32 - L;
    const uint4 v = z[i];
    const uint32_t m = morton3(v.x >> F, v.y >> F, v.z >> F);
    atomicAdd(&cnt[m], 1u);
    atomicAdd(&sx[m], (u64)v.x);
    atomicAdd(&sy[m], (u64)v.y);
    atomicAdd(&sz[m], (u64)v.z);
}

__global__ void k3_morton(int n, int L, const uint4 *__restrict__ z, uint32_t *__restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint4 v = z[i];
    out[i] = morton3(v.x >> (32 - L), v.y >> (32 - L), v.z >> (32 - L));
}

__global__ void k3_fill(int n, float4 *p, float4 v) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = v;
}

}  // namespace

cudaError_t launch_fill3(pxsne_ctx *c, float4 *p, float x, float y, float z) {
    const int n = (int)c->n;
    k3_fill<<<(n + 255) / 256, 256, 0, c->stream>>>(n, p, make_float4(x, y, z, 0.f));
    return cudaGetLastError();
}

int64_t cells3(int L) { return off3(L + 1); }
int64_t level_offset3(int l) { return off3(l); }

cudaError_t launch_leaf_hist3(pxsne_ctx *c, uint32_t *cnt, u64 *sums) {
    const int n = (int)c->n;
    const size_t leaves = size_t(1) << (3 * c->L);
    cudaError_t e;
    if ((e = cudaMemsetAsync(cnt, 0, leaves * 4, c->stream))) return e;
    if ((e = cudaMemsetAsync(sums, 0, 3 * leaves * 8, c->stream))) return e;
    k3_leaf_hist<<<(n + 255) / 256, 256, 0, c->stream>>>(n, c->L, c->z3, cnt, sums, sums + leaves,
                                                         sums + 2 * leaves);
    return cudaGetLastError();
}

cudaError_t launch_morton3(pxsne_ctx *c, uint32_t *out) {
    const int n = (int)c->n;
    k3_morton<<<(n + 255) / 256, 256, 0, c->stream>>>(n, c->L, c->z3, out);
    return cudaGetLastError();
}

template <class T>
static cudaError_t alloc_n(T **p, size_t count) {
    if (*p) {
        cudaFree(*p);
        *p = nullptr;
    }
    return cudaMalloc(reinterpret_cast<void **>(p), (count ? count : 1) * sizeof(T));
}

template <class T>
static void free_p(T *&p) {
    if (p) cudaFree(p);
    p = nullptr;
}

cudaError_t alloc3(pxsne_ctx *c) {
    const size_t n = (size_t)c->n;
    const int64_t cells = cells3(c->L);
    cudaError_t e;
    if ((e = alloc_n(&c->z3, n))) return e;
    if ((e = alloc_n(&c->zhat3, 3 * n))) return e;
    if ((e = alloc_n(&c->u3, n))) return e;
    if ((e = alloc_n(&c->gains3, n))) return e;
    if ((e = alloc_n(&c->Frep3, n))) return e;
    if ((e = alloc_n(&c->Fattr3, n))) return e;
    if ((e = alloc_n(&c->cnt3, (size_t)cells))) return e;
    if ((e = alloc_n(&c->sum3, 3 * (size_t)cells))) return e;
    // groups of siblings: one per cell above the leaves
    const size_t groups = (size_t)off3(c->L);
    if ((e = alloc_n(&c->rec3, groups * (kGroup3 / 4)))) return e;
    if ((e = alloc_n(&c->pref3, (size_t)cells))) return e;
    // the leaf histogram starts from zeros; the first reduction clears what it read
    if ((e = cudaMemsetAsync(c->cnt3, 0, (size_t)cells * sizeof(uint32_t), c->stream))) return e;
    if ((e = cudaMemsetAsync(c->sum3, 0, 3 * (size_t)cells * sizeof(u64), c->stream))) return e;
    c->dev_bytes += (int64_t)n * (16 + 24 + 16 * 4) + cells * (4 + 24) +
                    (int64_t)groups * kGroup3 * 4 + cells * 4;
    return cudaSuccess;
}

void free3(pxsne_ctx *c) {
    free_p(c->z3);
    free_p(c->zhat3);
    free_p(c->u3);
    free_p(c->gains3);
    free_p(c->Frep3);
    free_p(c->Fattr3);
    free_p(c->cnt3);
    free_p(c->sum3);
    free_p(c->rec3);
    free_p(c->pref3);
}

cudaError_t launch_set_scalars3(pxsne_ctx *c, const double *s, int t) {
    k3_set_scalars<<<1, 1, 0, c->stream>>>(c->sc, s[0], s[1], s[2], t, c->p.theta, c->L);
    return cudaGetLastError();
}

cudaError_t launch_init3(pxsne_ctx *c, const float *Y0dev, double *scratch) {
    cudaStream_t st = c->stream;
    const int n = (int)c->n;
    uint32_t *mm = reinterpret_cast<uint32_t *>(scratch);
    const uint32_t init[6] = {0xffffffffu, 0xffffffffu, 0xffffffffu, 0u, 0u, 0u};
    cudaError_t e;
    if ((e = cudaMemcpyAsync(mm, init, sizeof(init), cudaMemcpyHostToDevice, st))) return e;
    const int blocks = std::min((n + 255) / 256, 1184);
    k3_minmax<<<blocks > 0 ? blocks : 1, 256, 0, st>>>(n, Y0dev, mm, c->sc);
    k3_map<<<(n + 255) / 256, 256, 0, st>>>(n, c->L, c->p.theta, Y0dev, mm, c->z3, c->u3,
                                             c->gains3, c->sc);
    return cudaGetLastError();
}

// the tree of the current state (rescale: zhat -> z first, an iteration)
static cudaError_t tree3(pxsne_ctx *c, bool rescale) {
    cudaStream_t st = c->stream;
    const int L = c->L, n = (int)c->n;
    const int64_t cells = cells3(L);
    const int64_t lo = off3(L);
    uint32_t *cnt = c->cnt3;
    u64 *sx = c->sum3, *sy = c->sum3 + cells, *sz = c->sum3 + 2 * cells;
    cudaError_t e;
    // the leaves are zero here (set at allocation, cleared by the first
    // reduction after each histogram)
    k3_snap<<<(n + 255) / 256, 256, 0, st>>>(n, L, rescale ? 1 : 0, c->p.theta, c->zhat3, c->z3,
                                              c->rank, cnt + lo, sx + lo, sy + lo, sz + lo, c->sc);
    if ((e = cudaGetLastError())) return e;
    // the octree from the bottom, and the voxel order
    float *rec = reinterpret_cast<float *>(c->rec3);
    for (int h = L; h > 3; h--) {
        const int64_t m = int64_t(1) << (3 * (h - 1));
        k3_level<<<(unsigned)((m + 255) / 256), 256, 0, st>>>(h, h == L ? 1 : 0, cnt, sx, sy, sz,
                                                              c->rec3, c->pref3);
        if ((e = cudaGetLastError())) return e;
    }
    const int clear = L <= 3 ? 1 : 0;
    if (L >= 3) k3_top<3><<<1, 512, 0, st>>>(clear, cnt, sx, sy, sz, rec, c->pref3);
    else if (L == 2) k3_top<2><<<1, 64, 0, st>>>(clear, cnt, sx, sy, sz, rec, c->pref3);
    else k3_top<1><<<1, 8, 0, st>>>(clear, cnt, sx, sy, sz, rec, c->pref3);
    if ((e = cudaGetLastError())) return e;
    k3_perm<<<(n + 255) / 256, 256, 0, st>>>(n, L, c->z3, c->rank, c->pref3, c->perm, c->sc,
                                              rescale ? 1 : 0);
    return cudaGetLastError();
}

// Sets below kTrav3PointTo points take a warp per point: an iteration at n =
// 2,000 on 64^3 takes 56 against 134 us, at 20,000 on 128^3 307 against 447, at
// 40,000 on 256^3 812 against 678.
constexpr int64_t kTrav3PointTo = 24576;

static cudaError_t traverse3(pxsne_ctx *c) {
    cudaStream_t st = c->stream;
    const int n = (int)c->n;
    // the own-cell test is redundant below theta = 1 (with a margin for the
    // rounding of d^2)
    const bool own = c->p.theta >= 0.999f;
    if (c->n < kTrav3PointTo) {
        cudaError_t e = cudaFuncSetAttribute(own ? k3_traverse_pt<true> : k3_traverse_pt<false>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)kPt3Smem);
        if (e) return e;
        const unsigned blocks = (unsigned)((n + kPt3Warps - 1) / kPt3Warps);
        auto k = own ? k3_traverse_pt<true> : k3_traverse_pt<false>;
        k<<<blocks, kPt3Warps * 32, kPt3Smem, st>>>(n, c->L, c->z3, c->perm, c->rec3, c->sc,
                                                    c->Frep3, c->Zi);
    } else {
        const int per_block = kT3Warps * 32;
        auto k = own ? k3_traverse<true> : k3_traverse<false>;
        k<<<(n + per_block - 1) / per_block, per_block, 0, st>>>(n, c->L, c->z3, c->perm, c->rec3,
                                                                 c->sc, c->Frep3, c->Zi);
    }
    return cudaGetLastError();
}

static cudaError_t attract3(pxsne_ctx *c, cudaStream_t st) {
    const int n = (int)c->n;
    k3_attract<<<(unsigned)(((int64_t)n * 32 + 255) / 256), 256, 0, st>>>(
        n, c->rp, c->col, c->val, c->z3, c->sc, c->Fattr3);
    return cudaGetLastError();
}

cudaError_t launch_prime3(pxsne_ctx *c, bool rescale) {
    cudaError_t e = tree3(c, rescale);
    if (e) return e;
    if ((e = traverse3(c))) return e;
    if ((e = attract3(c, c->stream))) return e;
    return launch_zsum(c);
}

// One iteration; the attraction, which needs only the rescaled positions and
// P, runs on the side stream beside the traversal, as in 2-D.
cudaError_t launch_iteration3(pxsne_ctx *c) {
    UpdateParams p;
    p.eta = c->p.eta;
    p.exag = c->p.exaggeration;
    p.mom0 = c->p.momentum0;
    p.mom1 = c->p.momentum1;
    p.min_gain = c->p.min_gain;
    p.exag_iters = c->p.exag_iters;
    p.mom_switch = c->p.momentum_switch;
    const int n = (int)c->n;
    const int blocks = std::max(1, std::min((n + 255) / 256, 4 * std::max(c->sms, 1)));
    k3_update<<<blocks, 256, 0, c->stream>>>(n, p, c->z3, c->Frep3, c->Fattr3, c->u3, c->gains3,
                                              c->zhat3, c->sc);
    cudaError_t e = cudaGetLastError();
    if (e) return e;
    if (!c->side) return launch_prime3(c, true);
    if ((e = tree3(c, true))) return e;
    if ((e = cudaEventRecord(c->ev_fork, c->stream))) return e;
    if ((e = traverse3(c))) return e;
    if ((e = launch_zsum(c))) return e;
    if ((e = cudaStreamWaitEvent(c->side, c->ev_fork, 0))) return e;
    if ((e = attract3(c, c->side))) return e;
    if ((e = cudaEventRecord(c->ev_join, c->side))) return e;
    return cudaStreamWaitEvent(c->stream, c->ev_join, 0);
}

cudaError_t launch_kl3(pxsne_ctx *c, double *out_dev) {
    k3_kl<<<c->klblocks, 256, 0, c->stream>>>((int)c->n, c->rp, c->col, c->val, c->z3, c->sc,
                                              c->klpart, out_dev);
    return cudaGetLastError();
}

cudaError_t launch_centre_y3(pxsne_ctx *c, float *Ydev, int32_t *pixdev, double *scratch) {
    cudaStream_t st = c->stream;
    const int n = (int)c->n;
    cudaError_t e;
    if ((e = cudaMemsetAsync(scratch, 0, 3 * sizeof(double), st))) return e;
    k3_sum_y<<<std::min((n + 255) / 256, 1184), 256, 0, st>>>(n, c->z3, c->sc, scratch);
    k3_write_y<<<(n + 255) / 256, 256, 0, st>>>(n, c->L, c->z3, c->sc, scratch, Ydev, pixdev);
    return cudaGetLastError();
}

}  // namespace pxsne
