// PCA to d_out dimensions, the standard pre-processing the paper applies to all
// datasets before P is built (Sec. 5.1.1).
//
//   k_colsum_f64   column sums (FP64 accumulation), k_mean the FP32 means
//   k_cov          covariance (X - mu)^T (X - mu) / (n - 1): 128 x 128 output
//                  tiles per CTA over a slice of rows in FP32, slices added in
//                  FP64
//   k_sym_mul, k_gram, k_chol_inv, k_apply   block subspace iteration in FP64:
//                  Y = C Q, Q = Y R^-1 with R^T R = Y^T Y
//   k_project      (X - mu) V for the leading eigenvectors V
// The eigenvectors come from block subspace iteration with a Rayleigh-Ritz
// step in FP64 (cyclic Jacobi on the small projected matrix, on the host).
#include <algorithm>
#include <cmath>
#include <random>
#include <vector>

#include "common.cuh"

namespace pxsne {
namespace {

__global__ void k_colsum_f64(int64_t n, int D, const float *__restrict__ X, double *sum) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= D) return;
    double s = 0.0;
    for (int64_t r = blockIdx.y; r < n; r += gridDim.y) s += X[r * D + c];
    atomicAdd(&sum[c], s);
}

// mean[c] = sum[c] / n, and the covariance of the upper triangle divided by
// n - 1 and mirrored.
__global__ void k_mean(int64_t n, int D, const double *__restrict__ sum, float *__restrict__ mean) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < D) mean[c] = (float)(sum[c] / (double)n);
}
__global__ void k_mirror(int64_t n, int D, double *cov) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= (int64_t)D * D) return;
    const int a = (int)(i / D), b = (int)(i % D);
    if (b < a) return;
    const double v = cov[i] / (double)(n - 1);
    cov[i] = v;
    cov[(int64_t)b * D + a] = v;
}

// Covariance sums.  A CTA of 256 threads takes a 128 x 128 tile of the upper
// triangle over a slice of rows; a thread sums 8 x 8 entries (rows and columns
// 4 apart in halves, so that its operands are four 16-byte shared loads per
// row of X), each over the slice's rows in order.  70,000 x 784: 3.1 ms, with
// 64 x 64 tiles of scalar loads and the mean's FP64 quotient formed for every
// element 13.4.
constexpr int kCT = 128;   // covariance tile
constexpr int kCR = 16;    // rows per shared-memory stage
constexpr int kCRows = 4096;  // rows per slice (grid z)

__global__ void __launch_bounds__(256, 2)
    k_cov(int64_t n, int D, const float *__restrict__ X, const float *__restrict__ mean,
          double *cov) {
    __shared__ __align__(16) float sa[kCR][kCT], sb[kCR][kCT];
    const int a0 = blockIdx.x * kCT, b0 = blockIdx.y * kCT;
    if (b0 < a0) return;  // lower triangle mirrored at the end
    const int64_t r0 = (int64_t)blockIdx.z * kCRows;
    const int64_t r1 = r0 + kCRows < n ? r0 + kCRows : n;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    const int cc = tid & 127, rh = tid >> 7;  // staging: a column, every other row
    const float ma = a0 + cc < D ? mean[a0 + cc] : 0.f, mb = b0 + cc < D ? mean[b0 + cc] : 0.f;
    float acc[8][8] = {};
    for (int64_t rb = r0; rb < r1; rb += kCR) {
#pragma unroll
        for (int q = 0; q < kCR / 2; q++) {
            const int rr = 2 * q + rh;
            const int64_t r = rb + rr;
            float va = 0.f, vb = 0.f;
            if (r < r1) {
                if (a0 + cc < D) va = X[r * D + a0 + cc] - ma;
                if (b0 + cc < D) vb = X[r * D + b0 + cc] - mb;
            }
            sa[rr][cc] = va;
            sb[rr][cc] = vb;
        }
        __syncthreads();
#pragma unroll 4
        for (int rr = 0; rr < kCR; rr++) {
            float xa[8], xb[8];
#pragma unroll
            for (int h = 0; h < 2; h++) {
                const float4 u = *reinterpret_cast<const float4 *>(&sa[rr][64 * h + 4 * ty]);
                const float4 v = *reinterpret_cast<const float4 *>(&sb[rr][64 * h + 4 * tx]);
                xa[4 * h] = u.x; xa[4 * h + 1] = u.y; xa[4 * h + 2] = u.z; xa[4 * h + 3] = u.w;
                xb[4 * h] = v.x; xb[4 * h + 1] = v.y; xb[4 * h + 2] = v.z; xb[4 * h + 3] = v.w;
            }
#pragma unroll
            for (int u = 0; u < 8; u++)
#pragma unroll
                for (int v = 0; v < 8; v++) acc[u][v] = fmaf(xa[u], xb[v], acc[u][v]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < 8; u++)
#pragma unroll
        for (int v = 0; v < 8; v++) {
            const int a = a0 + 64 * (u >> 2) + 4 * ty + (u & 3);
            const int b = b0 + 64 * (v >> 2) + 4 * tx + (v & 3);
            if (a < D && b < D && b >= a) atomicAdd(&cov[(int64_t)a * D + b], (double)acc[u][v]);
        }
}

// out = (X - mean) V: 64 rows x 64 components per CTA, a thread 4 x 4 of them,
// each summed over the dimensions in order.  70,000 x 784 -> 50: 0.34 ms; one
// thread per output, dividing for the mean at every term, took 43.
constexpr int kPD = 32;  // dimensions per stage
__global__ void __launch_bounds__(256)
    k_project(int64_t n, int D, int dout, const float *__restrict__ X,
              const float *__restrict__ mean, const float *__restrict__ V,
              float *__restrict__ out) {
    __shared__ float sx[64][kPD + 1];
    __shared__ __align__(16) float sv[kPD][64];
    const int64_t r0 = (int64_t)blockIdx.x * 64;
    const int c0 = blockIdx.y * 64;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    float acc[4][4] = {};
    for (int d0 = 0; d0 < D; d0 += kPD) {
        for (int q = tid; q < 64 * kPD; q += 256) {
            const int rr = q / kPD, dd = q % kPD;
            sx[rr][dd] = (r0 + rr < n && d0 + dd < D) ? X[(r0 + rr) * D + d0 + dd] - mean[d0 + dd] : 0.f;
        }
        for (int q = tid; q < 64 * kPD; q += 256) {
            const int dd = q / 64, c = q % 64;
            sv[dd][c] = (d0 + dd < D && c0 + c < dout) ? V[(int64_t)(d0 + dd) * dout + c0 + c] : 0.f;
        }
        __syncthreads();
        const int m = D - d0 < kPD ? D - d0 : kPD;
        for (int dd = 0; dd < m; dd++) {
            const float4 v = *reinterpret_cast<const float4 *>(&sv[dd][4 * tx]);
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const float x = sx[4 * ty + u][dd];
                acc[u][0] = fmaf(x, v.x, acc[u][0]);
                acc[u][1] = fmaf(x, v.y, acc[u][1]);
                acc[u][2] = fmaf(x, v.z, acc[u][2]);
                acc[u][3] = fmaf(x, v.w, acc[u][3]);
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int u = 0; u < 4; u++)
#pragma unroll
        for (int v = 0; v < 4; v++) {
            const int64_t r = r0 + 4 * ty + u;
            const int c = c0 + 4 * tx + v;
            if (r < n && c < dout) out[r * dout + c] = acc[u][v];
        }
}

// ---- the subspace iteration's steps, all FP64 (D x b blocks, row-major).
// FP64 issues at about two FMAs a cycle and SM here, so the iteration is bound
// by Y = C Q (D^2 b FMAs); what matters is that every SM has its share.

// Y = A Q, A [rows x m], Q [m x b]: a thread per output, `per` rows of A per
// CTA, staged 32 columns at a time (A by rows, Q shared by the CTA's rows).
constexpr int kMulK = 32;
__global__ void k_mul(int rows, int m, int b, int per, const double *__restrict__ A,
                      const double *__restrict__ Q, double *__restrict__ Y) {
    extern __shared__ double s_mul[];
    double *sA = s_mul, *sQ = s_mul + per * kMulK;
    const int r0 = blockIdx.x * per;
    const int c0 = blockIdx.y * 32;
    const int c = threadIdx.x & 31, r = threadIdx.x >> 5;  // blockDim = 32 per
    double acc = 0.0;
    for (int k0 = 0; k0 < m; k0 += kMulK) {
        sA[r * kMulK + c] = (r0 + r < rows && k0 + c < m) ? A[(int64_t)(r0 + r) * m + k0 + c] : 0.0;
        for (int q = threadIdx.x; q < kMulK * 32; q += blockDim.x) {
            const int kk = q >> 5, cc = q & 31;
            sQ[q] = (k0 + kk < m && c0 + cc < b) ? Q[(int64_t)(k0 + kk) * b + c0 + cc] : 0.0;
        }
        __syncthreads();
#pragma unroll 8
        for (int kk = 0; kk < kMulK; kk++) acc = fma(sA[r * kMulK + kk], sQ[kk * 32 + c], acc);
        __syncthreads();
    }
    if (r0 + r < rows && c0 + c < b) Y[(int64_t)(r0 + r) * b + c0 + c] = acc;
}

// G[i][j] = sum over rows of A[.][i] B[.][j] (b x b), a warp per entry.
__global__ void k_gram(int D, int b, const double *__restrict__ A, const double *__restrict__ B,
                       double *__restrict__ G) {
    const int e = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (e >= b * b) return;
    const int i = e / b, j = e % b;
    double s = 0.0;
    for (int a = lane; a < D; a += 32) s = fma(A[(int64_t)a * b + i], B[(int64_t)a * b + j], s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) G[e] = s;
}

// One CTA: Cholesky G = R^T R (R upper triangular) and W = R^-1 in shared
// memory.  A pivot that has lost all but a few digits against its column's
// norm sets *bad (the block is close to rank-deficient) and W is not used.
constexpr int kCholMax = 112;  // b x b doubles of shared memory twice
__global__ void __launch_bounds__(512)
    k_chol_inv(int b, const double *__restrict__ G, double *__restrict__ W, int *bad) {
    extern __shared__ double s_ch[];
    double *R = s_ch, *I = s_ch + b * b;
    __shared__ int s_bad;
    __shared__ double s_f[kCholMax];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = blockDim.x >> 5;
    for (int q = tid; q < b * b; q += blockDim.x) {
        R[q] = G[q];
        I[q] = (q / b == q % b) ? 1.0 : 0.0;
    }
    if (tid == 0) s_bad = 0;
    __syncthreads();
    // eliminating row k of [G | 1] from the rows below leaves D R' | L^-1 in
    // place (of R' the upper triangle, its mirror being the same numbers), with
    // R = D^-1/2 of the rows and W = R^-1 = (D^-1/2 L^-1)^T.  One SM issues a
    // warp's FP64 operation in 16 cycles, so the step is bound by their number:
    // the rows' factors are formed once (not by every lane), the reciprocal by
    // one lane, and a row's two parts are one run of lanes.
    for (int k = 0; k < b; k++) {
        if (warp == 0) {
            double inv = 0.0;
            if (lane == 0) {
                inv = 1.0 / R[k * b + k];
                if (!(R[k * b + k] > 1e-12 * G[k * b + k])) s_bad = 1;
            }
            inv = __shfl_sync(0xffffffffu, inv, 0);
            for (int i = k + 1 + lane; i < b; i += 32) s_f[i] = R[k * b + i] * inv;
        }
        __syncthreads();
        for (int i = k + 1 + warp; i < b; i += warps) {
            const double f = s_f[i];
            const int nr = b - i, len = nr + k + 1;  // columns i .. of R', 0 .. k of L^-1
            for (int c = lane; c < len; c += 32) {
                double *row = c < nr ? R + i * b + i + c : I + i * b + c - nr;
                const double *piv = c < nr ? R + k * b + i + c : I + k * b + c - nr;
                *row -= f * *piv;
            }
        }
        __syncthreads();
    }
    for (int q = tid; q < b * b; q += blockDim.x) {
        const int i = q / b, j = q % b;  // W[j][i] = L^-1[i][j] / sqrt(D_i)
        W[j * b + i] = j <= i ? I[q] / sqrt(R[i * b + i]) : 0.0;
    }
    if (tid == 0 && s_bad) *bad = 1;
}

// Symmetric eigendecomposition of a small b x b matrix (cyclic Jacobi, FP64):
// on return A's diagonal holds the eigenvalues and U (row-major) the
// eigenvectors as columns.
void jacobi_eig(int b, std::vector<double> &A, std::vector<double> &U) {
    U.assign((size_t)b * b, 0.0);
    for (int i = 0; i < b; i++) U[(size_t)i * b + i] = 1.0;
    for (int sweep = 0; sweep < 60; sweep++) {
        double off = 0.0, tot = 0.0;
        for (int i = 0; i < b; i++)
            for (int j = 0; j < b; j++) {
                const double v = A[(size_t)i * b + j] * A[(size_t)i * b + j];
                tot += v;
                if (i != j) off += v;
            }
        if (off <= 1e-30 * tot || off == 0.0) break;
        for (int p = 0; p < b; p++)
            for (int q = p + 1; q < b; q++) {
                const double apq = A[(size_t)p * b + q];
                if (std::fabs(apq) < 1e-300) continue;
                const double app = A[(size_t)p * b + p], aqq = A[(size_t)q * b + q];
                // rotation angle zeroing A[p][q]: tan(2 phi) = 2 apq / (aqq - app)
                const double tau = (aqq - app) / (2.0 * apq);
                const double t = (tau >= 0 ? 1.0 : -1.0) / (std::fabs(tau) + std::sqrt(1.0 + tau * tau));
                const double c = 1.0 / std::sqrt(1.0 + t * t), s = t * c;
                for (int k = 0; k < b; k++) {  // columns p, q
                    const double akp = A[(size_t)k * b + p], akq = A[(size_t)k * b + q];
                    A[(size_t)k * b + p] = c * akp - s * akq;
                    A[(size_t)k * b + q] = s * akp + c * akq;
                }
                for (int k = 0; k < b; k++) {  // rows p, q
                    const double apk = A[(size_t)p * b + k], aqk = A[(size_t)q * b + k];
                    A[(size_t)p * b + k] = c * apk - s * aqk;
                    A[(size_t)q * b + k] = s * apk + c * aqk;
                }
                for (int k = 0; k < b; k++) {
                    const double ukp = U[(size_t)k * b + p], ukq = U[(size_t)k * b + q];
                    U[(size_t)k * b + p] = c * ukp - s * ukq;
                    U[(size_t)k * b + q] = s * ukp + c * ukq;
                }
            }
    }
}

// Modified Gram-Schmidt on the b columns of Q (D x b, row-major).
void orthonormalize(int D, int b, std::vector<double> &Q) {
    for (int j = 0; j < b; j++) {
        for (int i = 0; i < j; i++) {
            double d = 0.0;
            for (int a = 0; a < D; a++) d += Q[(size_t)a * b + i] * Q[(size_t)a * b + j];
            for (int a = 0; a < D; a++) Q[(size_t)a * b + j] -= d * Q[(size_t)a * b + i];
        }
        double nn = 0.0;
        for (int a = 0; a < D; a++) nn += Q[(size_t)a * b + j] * Q[(size_t)a * b + j];
        nn = std::sqrt(nn);
        for (int a = 0; a < D; a++) Q[(size_t)a * b + j] = nn > 0 ? Q[(size_t)a * b + j] / nn : 0.0;
    }
}

// The iteration on the host: Q (the random start) becomes the orthonormal
// block, T = Q^T C Q.
void subspace_host(int D, int b, int iters, const std::vector<double> &C, std::vector<double> &Q,
                   std::vector<double> &T) {
    std::vector<double> Y((size_t)D * b);
    auto mul = [&](const std::vector<double> &q, std::vector<double> &y) {
        std::fill(y.begin(), y.end(), 0.0);
        for (int a = 0; a < D; a++)
            for (int c = 0; c < D; c++) {
                const double cac = C[(size_t)a * D + c];
                const double *qc = &q[(size_t)c * b];
                double *ya = &y[(size_t)a * b];
                for (int j = 0; j < b; j++) ya[j] += cac * qc[j];
            }
    };
    orthonormalize(D, b, Q);
    for (int it = 0; it < iters; it++) {
        mul(Q, Y);
        Q.swap(Y);
        orthonormalize(D, b, Q);
    }
    mul(Q, Y);
    for (int i = 0; i < b; i++)
        for (int j = 0; j < b; j++) {
            double s = 0.0;
            for (int a = 0; a < D; a++) s += Q[(size_t)a * b + i] * Y[(size_t)a * b + j];
            T[(size_t)i * b + j] = s;
        }
}

// The same on the device.  The block's QR factorisation is unique up to signs
// (positive diagonal here and there), so Cholesky of its Gram matrix gives the
// columns that Gram-Schmidt does, up to rounding; the last one is done twice,
// which leaves the columns orthonormal to FP64 rounding.  False: a
// factorisation broke down or an error (Q is then the start still).  It does
// so first where the spectrum spans six decades and more: the first product's
// columns are all alike there, while later ones have turned to directions of
// their own.  So the flag is read after the first product (standard deviations
// falling as 0.85^i, 5,000 x 200: 42.2 ms; 48.7 with the flag read at the end).
template <class Check>
bool subspace_device(int D, int b, int iters, const double *dC, double *dwork,
                     std::vector<double> &Q, std::vector<double> &T, cudaStream_t st, Check &&ck) {
    double *dQ = dwork, *dY = dQ + (size_t)D * b, *dG = dY + (size_t)D * b, *dW = dG + (size_t)b * b;
    int *bad = reinterpret_cast<int *>(dW + (size_t)b * b);
    const size_t ch_smem = (size_t)2 * b * b * 8;
    // rows of Y per CTA: about one CTA per SM and 32 columns
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int cb = (b + 31) / 32;
    int per = (D * cb + std::max(sms, 1) - 1) / std::max(sms, 1);
    per = std::min(32, std::max(1, per));
    const size_t mul_smem = (size_t)(per * kMulK + kMulK * 32) * 8;
    bool ok = ck(allow_smem(k_chol_inv));
    ok = ok && ck(cudaMemsetAsync(bad, 0, sizeof(int), st));
    ok = ok && ck(cudaMemcpyAsync(dQ, Q.data(), (size_t)D * b * 8, cudaMemcpyHostToDevice, st));
    if (!ok) return false;
    const unsigned gram_blocks = (unsigned)((b * b + 7) / 8);
    auto mul = [&](const double *A, int m, const double *q, double *y) {
        const dim3 g((unsigned)((D + per - 1) / per), (unsigned)cb);
        k_mul<<<g, 32 * per, mul_smem, st>>>(D, m, b, per, A, q, y);
    };
    // y <- y R^-1, through the other block
    auto orthonormal = [&](double *&y, double *&other) {
        k_gram<<<gram_blocks, 256, 0, st>>>(D, b, y, y, dG);
        k_chol_inv<<<1, 512, ch_smem, st>>>(b, dG, dW, bad);
        mul(y, b, dW, other);
        std::swap(y, other);
    };
    int hbad = 0;
    orthonormal(dQ, dY);
    for (int it = 0; it < iters; it++) {
        mul(dC, D, dQ, dY);
        std::swap(dQ, dY);
        orthonormal(dQ, dY);
        if (it == 0) {
            ok = ck(cudaGetLastError());
            ok = ok && ck(cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, st));
            ok = ok && ck(cudaStreamSynchronize(st));
            if (!ok || hbad) return false;
        }
    }
    orthonormal(dQ, dY);
    mul(dC, D, dQ, dY);
    k_gram<<<gram_blocks, 256, 0, st>>>(D, b, dQ, dY, dG);
    ok = ck(cudaGetLastError());
    ok = ok && ck(cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, st));
    ok = ok && ck(cudaStreamSynchronize(st));
    if (!ok || hbad) return false;
    ok = ck(cudaMemcpyAsync(Q.data(), dQ, (size_t)D * b * 8, cudaMemcpyDeviceToHost, st));
    ok = ok && ck(cudaMemcpyAsync(T.data(), dG, (size_t)b * b * 8, cudaMemcpyDeviceToHost, st));
    return ok && ck(cudaStreamSynchronize(st));
}

}  // namespace
}  // namespace pxsne

using namespace pxsne;

extern "C" int pxsne_pca(const float *X, int64_t n, int32_t D, int32_t dout, float *Xout,
                         float *components, float *eigenvalues, int on_device, uint64_t seed) {
    if (!X || !Xout || n < 2 || D < 1 || dout < 1 || dout > D) return PXSNE_E_ARG;
    cudaStream_t st = nullptr;
    if (cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking)) return PXSNE_E_CUDA;
    int rc = PXSNE_OK;
    auto ck = [&](cudaError_t e) {
        if (e != cudaSuccess && rc == PXSNE_OK) {
            cudaGetLastError();
            rc = e == cudaErrorMemoryAllocation ? PXSNE_E_OOM : PXSNE_E_CUDA;
        }
        return rc == PXSNE_OK;
    };
    float *dX = nullptr, *dO = nullptr, *dV = nullptr, *dmean = nullptr;
    double *dsum = nullptr, *dcov = nullptr, *dwork = nullptr;
    const float *Xs = X;
    if (!on_device) {
        ck(cudaMallocAsync(&dX, (size_t)n * D * 4, st));
        if (rc == PXSNE_OK) ck(cudaMemcpyAsync(dX, X, (size_t)n * D * 4, cudaMemcpyHostToDevice, st));
        Xs = dX;
    }
    const int b = std::min<int>(D, dout + 16);
    ck(cudaMallocAsync(&dsum, (size_t)D * 8, st));
    ck(cudaMallocAsync(&dmean, (size_t)D * 4, st));
    ck(cudaMallocAsync(&dcov, (size_t)D * D * 8, st));
    // Q, Y (D x b), G, W (b x b), the flag
    ck(cudaMallocAsync(&dwork, (size_t)(2 * (int64_t)D * b + 2 * (int64_t)b * b + 1) * 8, st));
    if (rc == PXSNE_OK) {
        ck(cudaMemsetAsync(dsum, 0, (size_t)D * 8, st));
        ck(cudaMemsetAsync(dcov, 0, (size_t)D * D * 8, st));
        const dim3 gs((D + 127) / 128, 256);
        k_colsum_f64<<<gs, 128, 0, st>>>(n, D, Xs, dsum);
        k_mean<<<(D + 127) / 128, 128, 0, st>>>(n, D, dsum, dmean);
        const dim3 gc((D + kCT - 1) / kCT, (D + kCT - 1) / kCT, (unsigned)((n + kCRows - 1) / kCRows));
        k_cov<<<gc, 256, 0, st>>>(n, D, Xs, dmean, dcov);
        k_mirror<<<(unsigned)(((int64_t)D * D + 255) / 256), 256, 0, st>>>(n, D, dcov);
        ck(cudaGetLastError());
    }
    std::vector<double> lam(dout);
    std::vector<float> Vf((size_t)D * dout);
    if (rc == PXSNE_OK) {
        // block subspace iteration on C, then Rayleigh-Ritz
        std::vector<double> Q((size_t)D * b), T((size_t)b * b), U;
        std::mt19937_64 rng(seed);
        std::normal_distribution<double> nd(0.0, 1.0);
        for (auto &q : Q) q = nd(rng);
        const int iters = (b == D) ? 1 : 40;
        bool done = false;
        if (b <= kCholMax) done = subspace_device(D, b, iters, dcov, dwork, Q, T, st, ck);
        if (!done && rc == PXSNE_OK) {
            // a block near rank-deficiency (fewer rows or directions than
            // columns), or too wide for the factorisation's shared memory
            std::vector<double> C((size_t)D * D);
            ck(cudaMemcpyAsync(C.data(), dcov, (size_t)D * D * 8, cudaMemcpyDeviceToHost, st));
            ck(cudaStreamSynchronize(st));
            if (rc == PXSNE_OK) subspace_host(D, b, iters, C, Q, T);
        }
        if (rc == PXSNE_OK) {
        for (int i = 0; i < b; i++)
            for (int j = i + 1; j < b; j++) {
                const double v = 0.5 * (T[(size_t)i * b + j] + T[(size_t)j * b + i]);
                T[(size_t)i * b + j] = T[(size_t)j * b + i] = v;
            }
        jacobi_eig(b, T, U);
        std::vector<int> order(b);
        for (int i = 0; i < b; i++) order[i] = i;
        std::sort(order.begin(), order.end(),
                  [&](int x, int y) { return T[(size_t)x * b + x] > T[(size_t)y * b + y]; });
        // V = Q U of the leading columns, signs fixed so that each column's
        // largest |component| is positive
        std::vector<double> Us((size_t)b * dout), V((size_t)D * dout, 0.0);
        for (int j = 0; j < b; j++)
            for (int c = 0; c < dout; c++) Us[(size_t)j * dout + c] = U[(size_t)j * b + order[c]];
        for (int a = 0; a < D; a++)
            for (int j = 0; j < b; j++) {
                const double q = Q[(size_t)a * b + j];
                for (int c = 0; c < dout; c++) V[(size_t)a * dout + c] += q * Us[(size_t)j * dout + c];
            }
        for (int c = 0; c < dout; c++) {
            lam[c] = T[(size_t)order[c] * b + order[c]];
            double best = 0.0;
            int ba = 0;
            for (int a = 0; a < D; a++)
                if (std::fabs(V[(size_t)a * dout + c]) > best) {
                    best = std::fabs(V[(size_t)a * dout + c]);
                    ba = a;
                }
            const double sg = V[(size_t)ba * dout + c] < 0 ? -1.0 : 1.0;
            for (int a = 0; a < D; a++)
                Vf[(size_t)a * dout + c] = (float)(sg * V[(size_t)a * dout + c]);
        }
        if (components) std::copy(Vf.begin(), Vf.end(), components);
        if (eigenvalues)
            for (int c = 0; c < dout; c++) eigenvalues[c] = (float)lam[c];
        ck(cudaMallocAsync(&dV, (size_t)D * dout * 4, st));
        float *out = Xout;
        if (!on_device) ck(cudaMallocAsync(&dO, (size_t)n * dout * 4, st)), out = dO;
        if (rc == PXSNE_OK) {
            ck(cudaMemcpyAsync(dV, Vf.data(), (size_t)D * dout * 4, cudaMemcpyHostToDevice, st));
            const dim3 gp((unsigned)((n + 63) / 64), (unsigned)((dout + 63) / 64));
            k_project<<<gp, 256, 0, st>>>(n, D, dout, Xs, dmean, dV, out);
            ck(cudaGetLastError());
            if (!on_device)
                ck(cudaMemcpyAsync(Xout, dO, (size_t)n * dout * 4, cudaMemcpyDeviceToHost, st));
            ck(cudaStreamSynchronize(st));
        }
        }
    }
    if (dX) cudaFreeAsync(dX, st);
    if (dO) cudaFreeAsync(dO, st);
    if (dV) cudaFreeAsync(dV, st);
    if (dsum) cudaFreeAsync(dsum, st);
    if (dcov) cudaFreeAsync(dcov, st);
    if (dmean) cudaFreeAsync(dmean, st);
    if (dwork) cudaFreeAsync(dwork, st);
    cudaStreamSynchronize(st);
    cudaStreamDestroy(st);
    return rc;
}
