// Forces of the PixelSNE gradient (Eq. grad) on the pixel-aligned tree.
//
//   k_bh_traverse  repulsion by Barnes-Hut (Sec. 3.3, Eq. bh_criteria) on the
//                  dense pyramid, one warp per 32 points in tree order (64
//                  for large sets with geometric centres or on a crowded
//                  screen), the siblings as packed FP32 pairs; each point
//                  keeps its own accept/open decisions (lane masks per stack
//                  entry), so it sees exactly the cells its own depth-first
//                  search would
//   k_bh_traverse_pt  the same for small sets, one warp per point
//   k_attract      attraction over the CSR of P, one warp per row
//   k_zsum         Z = sum_i Z_i in FP64, fixed summation order
//   k_kl           Eq. cost_func, sums in three floats and FP64
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace pxsne {

// One warp = 32 PPL points consecutive in tree order, PPL (1 or 2) per lane.
// Each stack
// entry is a node whose four children are to be tested, with the mask of the
// lanes whose point opened it, so every point sees exactly the cells its own
// depth-first search would.  The four children are taken as two packed FP32
// pairs of siblings: the records keep each sibling group as a structure of
// arrays (common.cuh), so that a pair's coordinates are two adjacent words of
// a 16-byte load and enter the packed operations as they are, while a point's
// own coordinates are broadcast into packed registers once per 32 points.
// (Each component is rounded to nearest exactly as the scalar operation.)  The
// per-node step is branch-free within a level: every lane computes its point's
// offsets, distances and kernel values, and the accept/open decisions only
// gate the accumulation and the push.  Empty children add zero.  Children at
// the leaf level are always accepted (bounded depth, Sec. 4.1) except for a
// point's own pixel, which is used without the point itself; children above
// it follow Eq. bh_criteria, and the cell holding a point's own pixel is
// opened.  A point accumulates its cells in the fixed depth-first order of the
// tree (even and odd siblings in two sums, added at the end), so its result
// does not depend on the warp it shares.
// The kernel is bound by its issue slots: about 110 instructions per node of 32
// points, of which the packed arithmetic and reciprocals are about 35.  The
// siblings' pairs replaced pairs of a lane's two points, whose cell data had to
// be broadcast into packed registers for every child (59 instructions per child
// of 64 points): together with accepting single points early, 20 iterations at
// n = 1M went from 31.1 to 27.7 ms and five at 70,000 from 1.37 to 0.88 ms (beside
// the attraction; 64 points per warp and pairs of siblings: 28.8 and 1.18 ms).
// CENTRE = 0: centre of mass; 1: geometric cell centre.  COUNT = 1 also
// counts tested and accepted (point, cell) pairs.
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    return __ffma2_rn(a, b, c);
}
__device__ __forceinline__ float2 bc2(float v) { return make_float2(v, v); }
// The kernel value 1 / (1 + d^2) (argument >= 1): the hardware's approximate
// reciprocal (PTX rcp.approx, relative error within 2^-23), one instruction.
__device__ __forceinline__ float rcp1(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// COUNT: one (node, non-empty child) step's tested and accepted points, added
// to the CTA's counters of the child's level by lane 0.
__device__ __forceinline__ void count_level(u64 *lv, bool me, bool acc, bool step, int lane) {
    const unsigned t = __popc(__ballot_sync(0xffffffffu, me));
    const unsigned a = __popc(__ballot_sync(0xffffffffu, acc));
    if (lane == 0) {
        atomicAdd(&lv[0], (u64)t);
        atomicAdd(&lv[1], (u64)a);
        if (step) atomicAdd(&lv[2], 1ull);
    }
}

// A coordinate's two 16-bit halves as floats, each offset by a power of two
// that leaves the half's bits as the mantissa: hi_bits(v) = 2^39 + (v >> 16)
// 2^16 (ulp 2^16 at 2^39) and lo_bits(v) = 2^23 + (v & 0xffff) (ulp 1 at
// 2^23), both exact and built by bit operations instead of integer-to-float
// conversions.  The difference of two such values cancels the offset
// exactly, so (hi_bits(a) - hi_bits(b)) + (lo_bits(a) - lo_bits(b)) is the
// exact difference of the halves with one final rounding, as when the halves
// are converted and subtracted directly.
__device__ __forceinline__ float hi_bits(uint32_t v) {
    return __uint_as_float(0x53000000u | (v >> 16));
}
__device__ __forceinline__ float lo_bits(uint32_t v) {
    return __uint_as_float(0x4B000000u | (v & 0xffffu));
}

// Eq. grad, first term: Fattr_i = sum_j p_ij w_ij (y_i - y_j), one warp per
// row (row lengths vary with the in-degree of the kNN graph; a warp per row
// keeps long rows from stalling short ones).  It runs over the relabelled copy
// of P (rows and columns in the tree order of a recent state), so a row's
// gathered positions zp[j] lie close together in memory, and writes each row's
// force back under the point's own index.  Each lane keeps four entries in
// flight; P is streamed with evict-first loads so that the positions stay in
// L2.  z_i - z_j is formed exactly in float from the 16-bit halves of the
// fixed-point coordinates (both differences are exact; one final rounding).
// Entry order within a row is that of P, so the sums equal those over P.
struct AttractArgs {
    const int64_t *rp;
    const int32_t *col;
    const float *val;
    const uint2 *z;         // positions under the relabelled labels
    const uint32_t *aperm;  // relabelled row -> point
    float2 *Fattr;
};

__device__ __forceinline__ void attract_row(int row, int lane, const AttractArgs &a, float sf0,
                                            float sf1) {
    constexpr int U = 4;
    const int64_t *__restrict__ rp = a.rp;
    const int32_t *__restrict__ col = a.col;
    const float *__restrict__ val = a.val;
    const uint2 *__restrict__ z = a.z;
    const uint2 zi = z[row];
    // the row's halves offset by the same constants as hi_bits / lo_bits
    const float xh = hi_bits(zi.x), xl = lo_bits(zi.x);
    const float yh = hi_bits(zi.y), yl = lo_bits(zi.y);
    const int64_t e0 = rp[row], e1 = rp[row + 1];
    float fx = 0.f, fy = 0.f;
    // software pipeline: the next batch of P is requested while the current
    // batch's positions are being gathered
    int32_t jn[U];
    float pn[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
        const int64_t q = e0 + lane + 32 * u;
        jn[u] = q < e1 ? __ldcs(col + q) : row;
        pn[u] = q < e1 ? __ldcs(val + q) : 0.f;
    }
    for (int64_t e = e0 + lane; e < e1; e += 32 * U) {
        int32_t j[U];
        float p[U];
        uint2 zj[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            j[u] = jn[u];
            p[u] = pn[u];
            zj[u] = z[j[u]];
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t q = e + 32 * (U + u);
            jn[u] = q < e1 ? __ldcs(col + q) : row;
            pn[u] = q < e1 ? __ldcs(val + q) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const float dx = ((xh - hi_bits(zj[u].x)) + (xl - lo_bits(zj[u].x))) * sf0;
            const float dy = ((yh - hi_bits(zj[u].y)) + (yl - lo_bits(zj[u].y))) * sf1;
            const float w = __fdividef(1.0f, 1.0f + fmaf(dx, dx, dy * dy));
            const float pw = p[u] * w;
            fx = fmaf(pw, dx, fx);
            fy = fmaf(pw, dy, fy);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        fx += __shfl_xor_sync(0xffffffffu, fx, o);
        fy += __shfl_xor_sync(0xffffffffu, fy, o);
    }
    if (lane == 0) a.Fattr[a.aperm[row]] = make_float2(fx, fy);
}

// A point as the traversal holds it: each coordinate's two 16-bit halves
// (both exact in float, see rec in common.cuh) broadcast into packed pairs.
struct TravPoint {
    float2 hx, lx, hy, ly;
};
__device__ __forceinline__ TravPoint trav_point(uint2 z) {
    return TravPoint{bc2((float)(z.x & 0xffff0000u)), bc2((float)(z.x & 0xffffu)),
                     bc2((float)(z.y & 0xffff0000u)), bc2((float)(z.y & 0xffffu))};
}

// The four children of one node as two packed pairs (children 0, 1 and 2, 3).
// CENTRE = 0: the group's records (negated centres of mass), loaded.
// CENTRE = 1: the geometric centres from the node's corner (exact floats) and
// width 2^(33 - lc): child ch's centre is a quarter or three quarters across
// on each axis, so the two pairs share their x offsets.
template <int CENTRE>
struct Siblings {
    float4 hx, lx, hy, ly;  // CENTRE = 1: hx.xy the pair's x, hy.xy the two rows' y
    __device__ __forceinline__ void load(const float4 *__restrict__ rec, int at, int lc,
                                         uint32_t m) {
        if (CENTRE == 0) {
            hx = __ldg(rec + at);
            lx = __ldg(rec + at + 1);
            hy = __ldg(rec + at + 2);
            ly = __ldg(rec + at + 3);
        } else {
            const float wp = __int_as_float((127 + 33 - lc) << 23);
            const float px = (float)gather_bits16(m) * wp, py = (float)gather_bits16(m >> 1) * wp;
            hx = make_float4(-fmaf(wp, 0.25f, px), -fmaf(wp, 0.75f, px), 0.f, 0.f);
            hy = make_float4(-fmaf(wp, 0.25f, py), -fmaf(wp, 0.75f, py), 0.f, 0.f);
        }
    }
    // Offsets z - c (one rounding) of the point from pair p's two centres.
    __device__ __forceinline__ void offset(int p, const TravPoint &z, float2 &dx, float2 &dy) const {
        if (CENTRE == 0) {
            const float2 cx = p ? make_float2(hx.z, hx.w) : make_float2(hx.x, hx.y);
            const float2 ex = p ? make_float2(lx.z, lx.w) : make_float2(lx.x, lx.y);
            const float2 cy = p ? make_float2(hy.z, hy.w) : make_float2(hy.x, hy.y);
            const float2 ey = p ? make_float2(ly.z, ly.w) : make_float2(ly.x, ly.y);
            dx = add2(add2(z.hx, cx), add2(z.lx, ex));
            dy = add2(add2(z.hy, cy), add2(z.ly, ey));
        } else {
            dx = add2(add2(z.hx, make_float2(hx.x, hx.y)), z.lx);
            dy = add2(add2(z.hy, bc2(p ? hy.y : hy.x)), z.ly);
        }
    }
};

// A stack entry: the record offset of a node's sibling group of children
// (rec_offset(lc) + 4 m, lc their level, m the node's Morton index; a multiple
// of 4) in the low 28 bits as a count of groups, lc above, and for each of a
// lane's PPL points the mask of the lanes whose point opens the node.
template <int PPL>
struct TravEntry;
template <>
struct __align__(8) TravEntry<1> {
    uint32_t node, m[1];
};
template <>
struct __align__(16) TravEntry<2> {
    uint32_t node, m[2], pad;
};

// The threshold's term for cells of one point (single_base; geometric centres: no
// such rule).  It is read with the level's threshold where it is no constant: a
// register for it across the walk, or a load of its own, cost 1.6 % of an iteration
// at n = 70,000.
template <int CENTRE, bool OWN>
__device__ __forceinline__ constexpr bool trav_const() {
    return CENTRE != 0 || OWN;
}
template <int CENTRE, bool OWN>
__device__ __forceinline__ float trav_base(const DevScalars *sc) {
    if (CENTRE != 0) return 0.f;
    return single_base(OWN || underflows(sc->sf[0]) || underflows(sc->sf[1]));
}

// What a point (its pixel's Morton index mi) has to take out of its sum: 1 where
// every point accepts cells of one point (single_base) and it is alone in a cell
// above the pixels.
template <int CENTRE, bool OWN>
__device__ __forceinline__ float own_single(float base, const float *__restrict__ recn, int L,
                                            uint32_t mi) {
    if (CENTRE != 0 || OWN || base == -kManyT || L < 2) return 0.f;
    return recn[rec_offset(L - 1) + (mi >> 2)] == 1.f ? 1.f : 0.f;
}

template <int CENTRE, int COUNT, bool OWN, int PPL>
__global__ void __launch_bounds__(kTravWarps * 32, 16)
    k_bh_traverse(int n, int L, const uint2 *__restrict__ z, const uint32_t *__restrict__ perm,
                  const float4 *__restrict__ rec, const float *__restrict__ recn,
                  DevScalars *sc, float2 *__restrict__ Frep, float *__restrict__ Zi) {
    __shared__ TravEntry<PPL> s_stk[kTravWarps][kTravStack];
    __shared__ float2 s_T[kMaxL + 2];  // a level's threshold on d^2, and single_base
    const int stk_lim = sc->stack_limit > 0 ? min(max(sc->stack_limit, 4), kTravStack) : kTravStack;
    // COUNT: (tested, accepted, warp steps) by level of the child
    __shared__ u64 s_lv[COUNT ? kMaxL + 2 : 1][3];
    if (threadIdx.x < kMaxL + 2) {
        s_T[threadIdx.x] = make_float2(sc->T[threadIdx.x], trav_base<CENTRE, OWN>(sc));
        if (COUNT) s_lv[threadIdx.x][0] = s_lv[threadIdx.x][1] = s_lv[threadIdx.x][2] = 0ull;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int F = 32 - L;
    const float2 sf0 = bc2(sc->sf[0]), sf1 = bc2(sc->sf[1]);
    const unsigned before = (1u << lane) - 1u;
    uint32_t n_acc = 0u, n_tst = 0u, n_stp = 0u, n_nod = 0u;
    TravEntry<PPL> *stk = s_stk[w];
    // Each warp takes the next 32 PPL points of the tree order until none are
    // left: a warp whose points are cheap moves on instead of idling until
    // the slowest warp of its CTA is done.
    for (;;) {
        unsigned chunk = 0u;
        if (lane == 0) chunk = atomicAdd(&sc->trav_next, 1u);
        chunk = __shfl_sync(0xffffffffu, chunk, 0);
        if ((int64_t)chunk * (32 * PPL) >= n) break;
        unsigned act[PPL];
        uint32_t i[PPL], mi[PPL];
        TravPoint pt[PPL];
        float2 fx[PPL], fy[PPL], zs[PPL];
#pragma unroll
        for (int a = 0; a < PPL; a++) {
            const int idx = (int)chunk * (32 * PPL) + 32 * a + lane;
            act[a] = __ballot_sync(0xffffffffu, idx < n);
            i[a] = idx < n ? perm[idx] : 0u;
            const uint2 zi = z[i[a]];
            mi[a] = morton2(zi.x >> F, zi.y >> F);
            pt[a] = trav_point(zi);
            fx[a] = fy[a] = zs[a] = bc2(0.f);
        }

        // The root contains every point: start with its four children (level
        // 1, group 1 of the records).
        if (lane == 0) {
            TravEntry<PPL> e;
            e.node = (1u << 28) | 1u;
#pragma unroll
            for (int a = 0; a < PPL; a++) e.m[a] = act[a];
            stk[0] = e;
        }
        int sp = 1;
        __syncwarp();
        bool overflow = false;
        while (sp > 0) {
            sp--;
            TravEntry<PPL> top = stk[sp];
            __syncwarp();
            // the entry is the same for every lane: taken from lane 0, so that
            // the node, its level and addresses are known to be warp-uniform
            top.node = __shfl_sync(0xffffffffu, top.node, 0);
            bool me[PPL];
#pragma unroll
            for (int a = 0; a < PPL; a++) {
                top.m[a] = __shfl_sync(0xffffffffu, top.m[a], 0);
                me[a] = (top.m[a] >> lane) & 1u;
            }
            const uint32_t grp = top.node & 0x0fffffffu;
            const int lc = (int)(top.node >> 28);  // level of the children
            // the counts and the four children's records are requested
            // together (one latency per node)
            const float4 nv = __ldg(reinterpret_cast<const float4 *>(recn) + grp);
            Siblings<CENTRE> sib;
            // the node's Morton index, from rec_offset(lc) = (4^lc + 8) / 3
            const uint32_t m = (CENTRE == 1 || OWN || COUNT) ? grp - (uint32_t)(rec_offset(lc) >> 2) : 0u;
            sib.load(rec, (int)(4u * grp), lc, m);
            if (COUNT) {
                n_nod++;
                n_stp += (nv.x != 0.f) + (nv.y != 0.f) + (nv.z != 0.f) + (nv.w != 0.f);
            }
            if (lc == L) {
                const uint32_t g0 = (uint32_t)(rec_offset(L) >> 2);
                bool own[PPL], any = false;
#pragma unroll
                for (int a = 0; a < PPL; a++) {
                    own[a] = me[a] && (mi[a] >> 2) + g0 == grp;
                    any |= own[a];
                }
                const bool any_own = __any_sync(0xffffffffu, any);
#pragma unroll
                for (int p = 0; p < 2; p++) {
                    const float2 N0 = p ? make_float2(nv.z, nv.w) : make_float2(nv.x, nv.y);
                    if (N0.x + N0.y == 0.f) continue;
#pragma unroll
                    for (int a = 0; a < PPL; a++) {
                        float2 N = N0, dx, dy;
                        sib.offset(p, pt[a], dx, dy);
                        if (any_own) {  // a point's own pixel: take the point out
                            const bool o0 = own[a] && (mi[a] & 3u) == 2u * p;
                            const bool o1 = own[a] && (mi[a] & 3u) == 2u * p + 1u;
                            if (o0) {
                                const float r = N.x - 1.0f;
                                if (CENTRE == 0 && r > 0.0f) {
                                    const float k = N.x / r;
                                    dx.x *= k;
                                    dy.x *= k;
                                }
                                N.x = r;
                            }
                            if (o1) {
                                const float r = N.y - 1.0f;
                                if (CENTRE == 0 && r > 0.0f) {
                                    const float k = N.y / r;
                                    dx.y *= k;
                                    dy.y *= k;
                                }
                                N.y = r;
                            }
                        }
                        dx = mul2(dx, sf0);
                        dy = mul2(dy, sf1);
                        const float2 d2 = fma2(dx, dx, mul2(dy, dy));
                        if (COUNT) {
                            const bool a0 = me[a] && N.x > 0.f, a1 = me[a] && N.y > 0.f;
                            if (N0.x != 0.f) {
                                n_tst += me[a];
                                n_acc += a0;
                                count_level(s_lv[lc], me[a], a0, a == 0, lane);
                            }
                            if (N0.y != 0.f) {
                                n_tst += me[a];
                                n_acc += a1;
                                count_level(s_lv[lc], me[a], a1, a == 0, lane);
                            }
                        }
                        const float2 w1 = add2(bc2(1.0f), d2);
                        const float2 q = make_float2(rcp1(w1.x), rcp1(w1.y));
                        const float2 Nq =
                            mul2(make_float2(me[a] ? N.x : 0.0f, me[a] ? N.y : 0.0f), q);
                        zs[a] = add2(zs[a], Nq);
                        const float2 Nq2 = mul2(Nq, q);
                        fx[a] = fma2(Nq2, dx, fx[a]);
                        fy[a] = fma2(Nq2, dy, fy[a]);
                    }
                }
            } else {
                // Eq. bh_criteria's threshold on d^2.  The centre of a cell that
                // holds one point is that point exactly, so opening it down to
                // its pixel would end in the same term: it is accepted at once
                // by every point but the one in it (single_base).  Empty cells
                // add nothing.
                const float2 Tb = s_T[lc];
                const float Tl = Tb.x, base = trav_const<CENTRE, OWN>() ? trav_base<CENTRE, OWN>(sc) : Tb.y;
                constexpr float few = CENTRE == 0 ? 1.0f : 0.0f;
                // room for the (at most four) entries this node may push
                if (sp + 4 > stk_lim) {
                    overflow = true;
                    break;
                }
                unsigned acc[PPL][4];
#pragma unroll
                for (int p = 0; p < 2; p++) {
                    const float2 N = p ? make_float2(nv.z, nv.w) : make_float2(nv.x, nv.y);
                    const float2 tb = fma2(N, bc2(kManyT), bc2(base));
                    const float T0 = fminf(tb.x, Tl), T1 = fminf(tb.y, Tl);
#pragma unroll
                    for (int a = 0; a < PPL; a++) {
                        // a point's own cell: opened by the criterion itself when
                        // theta < 1 (the point and the centre of mass lie in the
                        // cell, so d <= r_c < r_c / theta); tested explicitly
                        // otherwise
                        const uint32_t mine = OWN || COUNT ? mi[a] >> (2 * (L - lc)) : 0u;
                        float2 dx, dy;
                        sib.offset(p, pt[a], dx, dy);
                        dx = mul2(dx, sf0);
                        dy = mul2(dy, sf1);
                        const float2 d2 = fma2(dx, dx, mul2(dy, dy));
                        const bool a0 = me[a] && d2.x > T0 && (!OWN || mine != 4u * m + 2u * p);
                        const bool a1 = me[a] && d2.y > T1 && (!OWN || mine != 4u * m + 2u * p + 1u);
                        if (COUNT) {  // (its own cell is no interaction)
                            const bool c0 = a0 && mine != 4u * m + 2u * p;
                            const bool c1 = a1 && mine != 4u * m + 2u * p + 1u;
                            if (N.x != 0.f) {
                                n_tst += me[a];
                                n_acc += c0;
                                count_level(s_lv[lc], me[a], c0, a == 0, lane);
                            }
                            if (N.y != 0.f) {
                                n_tst += me[a];
                                n_acc += c1;
                                count_level(s_lv[lc], me[a], c1, a == 0, lane);
                            }
                        }
                        const float2 w1 = add2(bc2(1.0f), d2);
                        const float2 q = make_float2(rcp1(w1.x), rcp1(w1.y));
                        const float2 Nq = mul2(make_float2(a0 ? N.x : 0.0f, a1 ? N.y : 0.0f), q);
                        zs[a] = add2(zs[a], Nq);
                        const float2 Nq2 = mul2(Nq, q);
                        fx[a] = fma2(Nq2, dx, fx[a]);
                        fy[a] = fma2(Nq2, dy, fy[a]);
                        acc[a][2 * p] = __ballot_sync(0xffffffffu, a0);
                        acc[a][2 * p + 1] = __ballot_sync(0xffffffffu, a1);
                    }
                }
                // lanes 0..3 push the children that some point opens
                const float na = (lane & 1) ? nv.y : nv.x, nc = (lane & 1) ? nv.w : nv.z;
                const float nn = (lane & 2) ? nc : na;
                TravEntry<PPL> e;
                unsigned some = 0u;
#pragma unroll
                for (int a = 0; a < PPL; a++) {
                    const unsigned oa = (lane & 1) ? acc[a][1] : acc[a][0];
                    const unsigned oc = (lane & 1) ? acc[a][3] : acc[a][2];
                    e.m[a] = top.m[a] & ~((lane & 2) ? oc : oa);
                    some |= e.m[a];
                }
                // the group of child c's children (rec_offset(l + 1) = 4
                // rec_offset(l) - 8): 4 grp - 2 + c, one level down
                e.node = ((uint32_t)(lc + 1) << 28) | (4u * grp - 2u + (uint32_t)lane);
                const bool push = lane < 4 && some != 0u && nn > few;
                const unsigned pm = __ballot_sync(0xffffffffu, push);
                if (push) stk[sp + __popc(pm & before)] = e;
                sp += __popc(pm);
            }
            __syncwarp();
        }
#pragma unroll
        for (int a = 0; a < PPL; a++)
            if ((act[a] >> lane) & 1u) {
                Frep[i[a]] = make_float2(fx[a].x + fx[a].y, fy[a].x + fy[a].y);
                Zi[i[a]] = zs[a].x + zs[a].y - own_single<CENTRE, OWN>(s_T[0].y, recn, L, mi[a]);
            }
        if (overflow && lane == 0) atomicOr(&sc->err, (unsigned)PXSNE_DEVERR_STACK);
        __syncwarp();
    }
    // every warp has taken its last chunk: the last one out resets the counter
    // for the next launch
    if (lane == 0 && atomicAdd(&sc->trav_done, 1u) == gridDim.x * kTravWarps - 1u) {
        sc->trav_next = 0u;
        sc->trav_done = 0u;
    }
    if (COUNT) {
        __syncthreads();
        if (threadIdx.x < (L + 1) * 3) {
            const int l = threadIdx.x / 3, q = threadIdx.x % 3;
            if (s_lv[l][q]) atomicAdd(&sc->lvl[l][q], s_lv[l][q]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            n_acc += __shfl_xor_sync(0xffffffffu, n_acc, o);
            n_tst += __shfl_xor_sync(0xffffffffu, n_tst, o);
        }
        if (lane == 0) {
            atomicAdd(&sc->n_accept, (u64)n_acc);
            atomicAdd(&sc->n_test, (u64)n_tst);
            atomicAdd(&sc->n_steps, (u64)n_stp);
            atomicAdd(&sc->n_nodes, (u64)n_nod);
        }
    }
}

// The traversal of small sets, one warp per point: with a few thousand points
// the kernel above has a few dozen warps on the whole chip, each walking its
// tree one node after another, and the time is that chain's latency.  Here the
// lanes take up to 32 of the point's open nodes at a time (all four children
// of a node as two packed pairs), so that the chain is about one step per
// level: 5 us instead of 55 at n = 2000 (20 iterations 0.93 ms when it came, 2.05
// with the kernel above; 0.72 with the smaller steps since).  The open nodes wait in a ring in shared memory, taken oldest first
// (breadth first); above kPtDeep waiting nodes the newest are taken first,
// which bounds the ring: such a step takes the 32 newest, of level l or deeper,
// and puts at most 128 of level l + 1 or deeper in their place, so that a
// node of level l waits at most 128 l places above kPtDeep + 96.  What a lane
// sums, and in which order, depends on the point's own walk only.
constexpr int kPtWarps = 4;
constexpr int kPtRing = 2048;
constexpr int kPtDeep = kPtRing - 128 * kMaxL - 128;
static_assert(kPtDeep >= 128, "ring of the point traversal");
template <int CENTRE, int COUNT, bool OWN>
__global__ void __launch_bounds__(kPtWarps * 32)
    k_bh_traverse_pt(int n, int L, const uint2 *__restrict__ z, const uint32_t *__restrict__ perm,
                     const float4 *__restrict__ rec, const float *__restrict__ recn,
                     DevScalars *sc, float2 *__restrict__ Frep, float *__restrict__ Zi) {
    __shared__ uint32_t s_ring[kPtWarps][kPtRing];
    __shared__ float s_T[kMaxL + 2];
    if (threadIdx.x < kMaxL + 2) s_T[threadIdx.x] = sc->T[threadIdx.x];
    __syncthreads();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int idx = blockIdx.x * kPtWarps + w;
    if (idx >= n) return;  // whole warps; no block barrier follows
    uint32_t *ring = s_ring[w];
    const int F = 32 - L;
    const float2 sf0 = bc2(sc->sf[0]), sf1 = bc2(sc->sf[1]);
    const float base = trav_base<CENTRE, OWN>(sc);
    const unsigned before = (1u << lane) - 1u;
    const uint32_t g0 = (uint32_t)(rec_offset(L) >> 2);
    const uint32_t i = perm[idx];
    const uint2 zi = z[i];
    const uint32_t mi = morton2(zi.x >> F, zi.y >> F);
    const TravPoint pt = trav_point(zi);
    float2 fx = bc2(0.f), fy = bc2(0.f), zs = bc2(0.f);
    uint32_t n_acc = 0u, n_tst = 0u, n_stp = 0u, n_nod = 0u;
    if (lane == 0) ring[0] = (1u << 28) | 1u;
    uint32_t head = 0u, size = 1u;
    __syncwarp();
    while (size > 0u) {
        const uint32_t k = min(size, 32u);
        const uint32_t at = size <= (uint32_t)kPtDeep ? head : head + size - k;
        if (size <= (uint32_t)kPtDeep) head += k;
        size -= k;
        const bool act = (uint32_t)lane < k;
        const uint32_t node = act ? ring[(at + lane) & (kPtRing - 1)] : (1u << 28) | 1u;
        __syncwarp();
        const uint32_t grp = node & 0x0fffffffu;
        const int lc = (int)(node >> 28);
        const bool leaf = lc == L;
        float4 nv = __ldg(reinterpret_cast<const float4 *>(recn) + grp);
        if (!act) nv = make_float4(0.f, 0.f, 0.f, 0.f);
        Siblings<CENTRE> sib;
        const uint32_t m = (CENTRE == 1 || OWN || COUNT) ? grp - (uint32_t)(rec_offset(lc) >> 2) : 0u;
        sib.load(rec, (int)(4u * grp), lc, m);
        const float Tl = s_T[lc];
        constexpr float few = CENTRE == 0 ? 1.0f : 0.0f;
        const bool own = leaf && act && (mi >> 2) + g0 == grp;
        const uint32_t mine = OWN || COUNT ? mi >> (2 * (L - lc)) : 0u;
        bool open[4];
        if (COUNT && act) n_nod++;
#pragma unroll
        for (int p = 0; p < 2; p++) {
            const float2 N0 = p ? make_float2(nv.z, nv.w) : make_float2(nv.x, nv.y);
            float2 N = N0, dx, dy;
            sib.offset(p, pt, dx, dy);
            if (own) {  // the point's own pixel: take the point out
                const bool second = mi & 1u;
                if (((mi >> 1) & 1u) == (uint32_t)p) {
                    const float Nc = second ? N.y : N.x, r = Nc - 1.0f;
                    const float kk = (CENTRE == 0 && r > 0.0f) ? Nc / r : 1.0f;
                    if (second) {
                        N.y = r;
                        dx.y *= kk;
                        dy.y *= kk;
                    } else {
                        N.x = r;
                        dx.x *= kk;
                        dy.x *= kk;
                    }
                }
            }
            dx = mul2(dx, sf0);
            dy = mul2(dy, sf1);
            const float2 d2 = fma2(dx, dx, mul2(dy, dy));
            // thresholds as above; a pixel is always accepted
            const float2 tb = fma2(N0, bc2(kManyT), bc2(base));
            const float T0 = leaf ? -1.0f : fminf(tb.x, Tl), T1 = leaf ? -1.0f : fminf(tb.y, Tl);
            const bool a0 = d2.x > T0 && (!OWN || leaf || mine != 4u * m + 2u * p);
            const bool a1 = d2.y > T1 && (!OWN || leaf || mine != 4u * m + 2u * p + 1u);
            if (COUNT) {
                const bool f0 = N0.x != 0.f, f1 = N0.y != 0.f;
                const uint32_t ts = (f0 ? 1u : 0u) + (f1 ? 1u : 0u);
                // (its own cell above the pixels is no interaction)
                const bool c0 = a0 && (leaf || mine != 4u * m + 2u * p);
                const bool c1 = a1 && (leaf || mine != 4u * m + 2u * p + 1u);
                const uint32_t ac = (f0 && c0 && N.x > 0.f ? 1u : 0u) + (f1 && c1 && N.y > 0.f ? 1u : 0u);
                // a warp step: the lanes that test their nodes' same child at
                // once, those of each level counted apart
                const unsigned m0 = __match_any_sync(0xffffffffu, f0 ? lc : -1);
                const unsigned m1 = __match_any_sync(0xffffffffu, f1 ? lc : -1);
                const uint32_t st = (f0 && lane == __ffs(m0) - 1 ? 1u : 0u) +
                                    (f1 && lane == __ffs(m1) - 1 ? 1u : 0u);
                n_tst += ts;
                n_acc += ac;
                n_stp += st;
                if (ts) atomicAdd(&sc->lvl[lc][0], (u64)ts);
                if (ac) atomicAdd(&sc->lvl[lc][1], (u64)ac);
                if (st) atomicAdd(&sc->lvl[lc][2], (u64)st);
            }
            const float2 w1 = add2(bc2(1.0f), d2);
            const float2 q = make_float2(rcp1(w1.x), rcp1(w1.y));
            const float2 Nq = mul2(make_float2(a0 ? N.x : 0.0f, a1 ? N.y : 0.0f), q);
            zs = add2(zs, Nq);
            const float2 Nq2 = mul2(Nq, q);
            fx = fma2(Nq2, dx, fx);
            fy = fma2(Nq2, dy, fy);
            // (a pixel is never opened, whatever a non-finite distance says)
            open[2 * p] = !a0 && !leaf && N0.x > few;
            open[2 * p + 1] = !a1 && !leaf && N0.y > few;
        }
        const uint32_t child = ((uint32_t)(lc + 1) << 28) | (4u * grp - 2u);
        uint32_t end = head + size;
#pragma unroll
        for (int c = 0; c < 4; c++) {
            const unsigned b = __ballot_sync(0xffffffffu, open[c]);
            if (open[c]) ring[(end + __popc(b & before)) & (kPtRing - 1)] = child + (uint32_t)c;
            end += __popc(b);
        }
        size = end - head;
        __syncwarp();
    }
    float vx = fx.x + fx.y, vy = fy.x + fy.y, vz = zs.x + zs.y;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        vx += __shfl_xor_sync(0xffffffffu, vx, o);
        vy += __shfl_xor_sync(0xffffffffu, vy, o);
        vz += __shfl_xor_sync(0xffffffffu, vz, o);
    }
    if (lane == 0) {
        Frep[i] = make_float2(vx, vy);
        Zi[i] = vz - own_single<CENTRE, OWN>(base, recn, L, mi);
    }
    if (COUNT) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            n_acc += __shfl_xor_sync(0xffffffffu, n_acc, o);
            n_tst += __shfl_xor_sync(0xffffffffu, n_tst, o);
            n_stp += __shfl_xor_sync(0xffffffffu, n_stp, o);
            n_nod += __shfl_xor_sync(0xffffffffu, n_nod, o);
        }
        if (lane == 0) {
            atomicAdd(&sc->n_accept, (u64)n_acc);
            atomicAdd(&sc->n_test, (u64)n_tst);
            atomicAdd(&sc->n_steps, (u64)n_stp);
            atomicAdd(&sc->n_nodes, (u64)n_nod);
        }
    }
}

// The attraction as its own kernel: one warp per row, the warps of a small
// persistent grid taking the rows `rows` at a time until none are left, so
// that it runs beside the traversal on the SMs' spare registers.
constexpr int kAttRows = 4;
// Below this many rows a warp takes one at a time: the whole grid then has less
// than six rows a warp, and at n = 2000, where fours left three SMs of four
// without any, the launch is the length of one warp's share.  (20 iterations of
// 2000 points with this, the last CTA's pyramid and the scalars' lanes: 0.91 to
// 0.69 ms.)  From here on fours save three quarters of the counter's atomics.
constexpr int kAttRowsFrom = 65536;
__global__ void __launch_bounds__(256)
    k_attract(int n, int rows, AttractArgs a, DevScalars *sc) {
    const int lane = threadIdx.x & 31;
    const float sf0 = sc->sf[0], sf1 = sc->sf[1];
    for (;;) {
        unsigned chunk = 0u;
        if (lane == 0) chunk = atomicAdd(&sc->att_next, 1u);
        chunk = __shfl_sync(0xffffffffu, chunk, 0);
        if ((int64_t)chunk * rows >= n) break;
        const int r0 = (int)chunk * rows, r1 = min(n, r0 + rows);
        for (int row = r0; row < r1; row++) attract_row(row, lane, a, sf0, sf1);
    }
    if (lane == 0 && atomicAdd(&sc->att_done, 1u) == gridDim.x * (blockDim.x >> 5) - 1u) {
        sc->att_next = 0u;
        sc->att_done = 0u;
    }
}

// Relabelling: new label r is the point perm[r] (tree order of the last
// tree).  Maps, padded row lengths under the new labels, and the positions.
__global__ void k_relabel_maps(int n, const uint32_t *__restrict__ perm,
                               const int64_t *__restrict__ rp, const uint2 *__restrict__ z,
                               uint32_t *__restrict__ aperm, uint32_t *__restrict__ ainv,
                               uint32_t *__restrict__ len2, uint2 *__restrict__ zp) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const uint32_t i = perm[r];
    aperm[r] = i;
    ainv[i] = (uint32_t)r;
    len2[r] = (uint32_t)(rp[i + 1] - rp[i]);
    zp[r] = z[i];
}

// Row r of the relabelled P is row aperm[r] of P with every column j replaced
// by ainv[j], entries in the same order; one warp per row, 16-byte quads (rows
// are padded to multiples of four on both sides).
__global__ void __launch_bounds__(256)
    k_relabel_rows(int n, const uint32_t *__restrict__ aperm, const uint32_t *__restrict__ ainv,
                   const int64_t *__restrict__ rp, const int4 *__restrict__ col4,
                   const float4 *__restrict__ val4, const int64_t *__restrict__ rp2,
                   int4 *__restrict__ col2, float4 *__restrict__ val2) {
    const int lane = threadIdx.x & 31;
    const int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (r >= n) return;
    const uint32_t i = aperm[r];
    const int64_t q0 = rp[i] >> 2, q1 = rp[i + 1] >> 2, d0 = rp2[r] >> 2;
    for (int64_t q = q0 + lane; q < q1; q += 32) {
        const int4 c = __ldcs(col4 + q);
        const float4 v = __ldcs(val4 + q);
        col2[d0 + (q - q0)] = make_int4((int)ainv[c.x], (int)ainv[c.y], (int)ainv[c.z],
                                        (int)ainv[c.w]);
        val2[d0 + (q - q0)] = v;
    }
}

// Deterministic FP64 block sum (fixed tree order) of blockDim.x values.
__device__ double block_sum_f64(double v, double *s_red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) s_red[warp] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0) {
        const int nw = blockDim.x >> 5;
        for (int k = 0; k < nw; k++) t += s_red[k];
    }
    __syncthreads();
    return t;
}

// Z = sum_i Z_i: each block sums a fixed contiguous chunk, the last block to
// finish adds the partials in index order.
__global__ void __launch_bounds__(512)
    k_zsum(int n, const float *__restrict__ Zi, double *__restrict__ part, DevScalars *sc) {
    __shared__ double s_red[16];
    __shared__ bool s_last;
    const int chunk = (n + gridDim.x - 1) / gridDim.x;
    const int a = blockIdx.x * chunk, b = min(n, a + chunk);
    double v = 0.0;
    for (int k = a + threadIdx.x; k < b; k += blockDim.x) v += (double)Zi[k];
    const double t = block_sum_f64(v, s_red);
    if (gridDim.x == 1) {
        if (threadIdx.x == 0) sc->Z = t;
        return;
    }
    if (threadIdx.x == 0) {
        part[blockIdx.x] = t;
        __threadfence();
        const unsigned tk = atomicAdd(&sc->ticket, 1u);
        s_last = (tk == gridDim.x - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double w = 0.0;
    for (int k = threadIdx.x; k < (int)gridDim.x; k += blockDim.x)
        w += reinterpret_cast<volatile double *>(part)[k];
    const double Z = block_sum_f64(w, s_red);
    if (threadIdx.x == 0) {
        sc->Z = Z;
        sc->ticket = 0u;
    }
}

static AttractArgs attract_args(const pxsne_ctx *c) {
    return AttractArgs{c->rp2, c->col2, c->val2, c->zp, c->aperm, c->Fattr};
}

static bool crowded(const pxsne_ctx *c) {
    return trav_crowded(c->n, c->L, c->p.screen_x, c->p.screen_y);
}

// One wave of a few CTAs per SM (kTravCtasPerSm), fewer when the points fill
// fewer.
template <int CENTRE, int COUNT, bool OWN, int PPL>
static void traverse_as(pxsne_ctx *c, cudaStream_t st) {
    const int n = (int)c->n;
    const int per_block = kTravWarps * 32 * PPL;
    const int ctas = CENTRE == 0 && crowded(c) ? kTravCrowdedCtasPerSm : kTravCtasPerSm;
    const int blocks = std::min((n + per_block - 1) / per_block, ctas * std::max(c->sms, 1));
    k_bh_traverse<CENTRE, COUNT, OWN, PPL><<<blocks, kTravWarps * 32, 0, st>>>(
        n, c->L, c->z, c->perm, c->rec, c->recn, c->sc, c->Frep, c->Zi);
}

template <int CENTRE, int COUNT, bool OWN>
static void traverse_n(pxsne_ctx *c, cudaStream_t st) {
    // (the stack test hook is the other kernels')
    if (c->n < kTravPointTo && c->stack_limit == 0) {
        const int n = (int)c->n;
        k_bh_traverse_pt<CENTRE, COUNT, OWN><<<(n + kPtWarps - 1) / kPtWarps, kPtWarps * 32, 0, st>>>(
            n, c->L, c->z, c->perm, c->rec, c->recn, c->sc, c->Frep, c->Zi);
    } else if (CENTRE == 0 ? crowded(c) && c->n >= kTravCrowdedPair
                           : c->n >= kTravPairFrom) {
        traverse_as<CENTRE, COUNT, OWN, 2>(c, st);
    } else {
        traverse_as<CENTRE, COUNT, OWN, 1>(c, st);
    }
}

static cudaError_t traverse(pxsne_ctx *c, cudaStream_t st, bool count) {
    // the own-cell test is redundant below theta = 1 (with a margin for the
    // rounding of d^2)
    const bool own = c->p.theta >= 0.999f;
    if (c->p.centre_mode == 0) {
        if (count) own ? traverse_n<0, 1, true>(c, st) : traverse_n<0, 1, false>(c, st);
        else own ? traverse_n<0, 0, true>(c, st) : traverse_n<0, 0, false>(c, st);
    } else {
        if (count) own ? traverse_n<1, 1, true>(c, st) : traverse_n<1, 1, false>(c, st);
        else own ? traverse_n<1, 0, true>(c, st) : traverse_n<1, 0, false>(c, st);
    }
    return cudaGetLastError();
}

cudaError_t launch_attract(pxsne_ctx *c, cudaStream_t st) {
    const int n = (int)c->n;
    const int rows = n < kAttRowsFrom ? 1 : kAttRows;
    // (few rows: fewer and larger CTAs; the same up to 32,000 rows, 158.0 against
    // 158.8 us an iteration at 60,000)
    const int warps = rows == 1 ? 8 : kAttWarps;
    const int need = (int)((int64_t(n) + warps * rows - 1) / (warps * rows));
    const int blocks = std::min(need, kAttCtasPerSm * kAttWarps / warps * std::max(c->sms, 1));
    k_attract<<<blocks, warps * 32, 0, st>>>(n, rows, attract_args(c), c->sc);
    return cudaGetLastError();
}

static cudaError_t zsum(pxsne_ctx *c, cudaStream_t st) {
    k_zsum<<<c->zblocks, 512, 0, st>>>((int)c->n, c->Zi, c->zpart, c->sc);
    return cudaGetLastError();
}

cudaError_t launch_zsum(pxsne_ctx *c) { return zsum(c, c->stream); }

cudaError_t launch_relabel(pxsne_ctx *c, cudaStream_t st) {
    const int n = (int)c->n;
    k_relabel_maps<<<(n + 255) / 256, 256, 0, st>>>(n, c->perm, c->rp, c->z, c->aperm, c->ainv,
                                                     c->rl2, c->zp);
    cudaError_t e = cudaGetLastError();
    if (e) return e;
    if ((e = scan_u32_to_i64(c, c->rl2, n, c->rp2, st))) return e;
    const unsigned blocks = (unsigned)(((int64_t)n * 32 + 255) / 256);
    k_relabel_rows<<<blocks, 256, 0, st>>>(n, c->aperm, c->ainv, c->rp,
                                           reinterpret_cast<const int4 *>(c->col),
                                           reinterpret_cast<const float4 *>(c->val), c->rp2,
                                           reinterpret_cast<int4 *>(c->col2),
                                           reinterpret_cast<float4 *>(c->val2));
    return cudaGetLastError();
}

// The traversal of the current tree again, with the work counters (the
// tree's snap kernel reset them); Frep and Zi are rewritten with the same
// values.
cudaError_t launch_count_traversal(pxsne_ctx *c) { return traverse(c, c->stream, true); }

__global__ void k_accumulate_counters(DevScalars *sc) {
    sc->tot[0] += sc->n_accept;
    sc->tot[1] += sc->n_test;
    sc->tot[2] += sc->n_steps;
    sc->tot[3] += sc->n_nodes;
}

cudaError_t launch_accumulate_counters(pxsne_ctx *c) {
    k_accumulate_counters<<<1, 1, 0, c->stream>>>(c->sc);
    return cudaGetLastError();
}

cudaError_t launch_traverse_zsum(pxsne_ctx *c) {
    cudaError_t e = traverse(c, c->stream, false);
    if (e) return e;
    return zsum(c, c->stream);
}

// Sequential forces (traversal, attraction, Z) with optional timing marks.
cudaError_t launch_forces(pxsne_ctx *c, cudaEvent_t *marks) {
    cudaStream_t st = c->stream;
    cudaError_t e;
    if (marks && (e = cudaEventRecord(marks[KG_TRAVERSE], st))) return e;
    // the initial state's traversal keeps the work counters (the level
    // counters restart with it); a timed one is the kernel of the iteration
    // itself
    if (!marks && (e = cudaMemsetAsync(c->sc->lvl, 0, sizeof(c->sc->lvl), st))) return e;
    if ((e = traverse(c, st, marks == nullptr))) return e;
    if (marks && (e = cudaEventRecord(marks[KG_ATTRACT], st))) return e;
    if ((e = launch_attract(c, st))) return e;
    if (marks && (e = cudaEventRecord(marks[KG_ZSUM], st))) return e;
    if ((e = zsum(c, st))) return e;
    if (marks && (e = cudaEventRecord(marks[KG_COUNT], st))) return e;
    return cudaSuccess;
}

// A sum of FP32 terms carried as three floats: the rounding error of every
// addition to one word is found exactly (Knuth's two-sum) and added to the next, and
// only the last one rounds.  After N terms the error is at most N^3 2^-74 of their
// absolute sum, which is less than that of N FP64 additions (N 2^-53) up to 1,400
// terms; with roundings of either sign it is about N^1.5 2^-72 against N^0.5 2^-54.
struct FloatSum {
    float h, m, l;
    static __device__ __forceinline__ float two_sum(float &a, float x) {
        const float s = __fadd_rn(a, x), b = __fsub_rn(s, a);
        const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, b)), __fsub_rn(x, b));
        a = s;
        return e;
    }
    __device__ __forceinline__ void add(float x) { l = __fadd_rn(l, two_sum(m, two_sum(h, x))); }
    __device__ __forceinline__ double sum() const { return (double)h + ((double)m + (double)l); }
};

// Eq. cost_func: C = sum_ij p_ij ln(p_ij Z / w_ij)
//                  = sum p (ln p - ln w) + (sum p) ln Z,
// one warp per row, fixed order: a lane's FP32 terms (700 of them at n = 1M) in three
// floats, FP64 across lanes and blocks.  FP64 additions and conversions issue at a
// small fraction of the FP32 rate: 100,000 points, 13.5M entries, the whole call
// 278 us; 284 with two floats, whose error of 2^-37 on a row of 200,000 entries is
// more than FP64's, 296 with two floats and FP64 after every row (288 with the
// three); the kernel alone took 400 with two FP64 additions per entry.
__global__ void __launch_bounds__(256)
    k_kl(int n, const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
         const float *__restrict__ val, const uint2 *__restrict__ z, DevScalars *sc,
         double *__restrict__ part, double *out) {
    __shared__ double s_red[8];
    __shared__ bool s_last;
    const int lane = threadIdx.x & 31;
    const int warps_total = gridDim.x * (blockDim.x >> 5);
    const float sf0 = sc->sf[0], sf1 = sc->sf[1];
    FloatSum ka{0.f, 0.f, 0.f}, kp{0.f, 0.f, 0.f};
    for (int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); row < n;
         row += warps_total) {
        const uint2 zi = z[row];
        const float xh = hi_bits(zi.x), xl = lo_bits(zi.x);
        const float yh = hi_bits(zi.y), yl = lo_bits(zi.y);
        const int64_t e1 = rp[row + 1];
        for (int64_t e = rp[row] + lane; e < e1; e += 32) {
            const float p = __ldcs(val + e);
            const uint2 zj = z[__ldcs(col + e)];
            if (!(p > 0.f)) continue;
            const float dx = ((xh - hi_bits(zj.x)) + (xl - lo_bits(zj.x))) * sf0;
            const float dy = ((yh - hi_bits(zj.y)) + (yl - lo_bits(zj.y))) * sf1;
            ka.add(p * (logf(p) + log1pf(fmaf(dx, dx, dy * dy))));
            kp.add(p);
        }
    }
    const double acc = ka.sum(), psum = kp.sum();
    const double a = block_sum_f64(acc, s_red);
    const double ps = block_sum_f64(psum, s_red);
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
    double A = 0.0, S = 0.0;
    volatile double *vp = part;
    for (int k = threadIdx.x; k < (int)gridDim.x; k += blockDim.x) {
        A += vp[2 * k];
        S += vp[2 * k + 1];
    }
    A = block_sum_f64(A, s_red);
    S = block_sum_f64(S, s_red);
    if (threadIdx.x == 0) {
        *out = A + S * log(sc->Z);
        sc->ticket2 = 0u;
    }
}

cudaError_t launch_kl(pxsne_ctx *c, double *out_dev) {
    const int blocks = std::max(1, std::min(c->klblocks, ((int)c->n + 7) / 8));
    k_kl<<<blocks, 256, 0, c->stream>>>((int)c->n, c->rp, c->col, c->val, c->z, c->sc, c->klpart,
                                        out_dev);
    return cudaGetLastError();
}

}  // namespace pxsne
