// Gradient of an eigenvalue loss with respect to the stored CSR values
// (differentiation of the FEAST result; the guide has no counterpart).
// For a simple eigenpair of A x = lambda B x with x^T B x = 1,
// d lambda / d a_ij = x_i x_j and d lambda / d b_ij = -lambda x_i x_j
// (first-order perturbation of a single stored entry).  For the loss
// L = sum_k g_k lambda_k the entry-wise gradient over a CSR pattern is
//   grad[p] = sum_k w_k x_k[i_p] x_k[j_p],  w_k = g_k (for A) or -g_k lambda_k (for B),
// a sampled dense-dense product (SDDMM) over the pattern.
#include <algorithm>

#include "feast_internal.cuh"

namespace feast {

// Xr is row-major n x m (eigenvectors in columns).  Weights: w_k = g_k, or
// w_k = -g_k lambda_k when lam is given (entries of B).  half: the pattern is
// one triangle of a symmetric matrix, so a stored off-diagonal value stands
// for both (i, j) and (j, i) and its derivative is twice the entry-wise one.
// Eight lanes per row i, four rows per warp; a lane holds columns l, l + 8, ...
// of w o x_i in registers (up to kGradReg of them, in shared memory to 256) and
// its share of an entry's sum, which three shuffles complete; four entries are
// in flight.  Bound: FP64 issue, then L2 (each row of X is read once per entry
// of its column).  A warp per row spent its time on five FP64 shuffle-and-add
// steps per entry (48^3, 71 vectors: 453 us, this form 190; the sums alone need
// 54 M FP64 FMA, about 95 us).
static constexpr int kGradLanes = 8;
static constexpr int kGradReg = 16;

template <bool SMEM>
__global__ void __launch_bounds__(256) eig_grad(int n, const int* __restrict__ ia, const int* __restrict__ ja, int m,
                                                const double* __restrict__ Xr, const double* __restrict__ gw,
                                                const double* __restrict__ lam, int half, double* __restrict__ grad)
{
    extern __shared__ double u_sm[];
    const int l = threadIdx.x & (kGradLanes - 1), grp = threadIdx.x / kGradLanes;
    const unsigned mask = 0xffu << (threadIdx.x & 24);
    double* us = u_sm + (size_t)grp * m;
    const int rows = gridDim.x * (blockDim.x / kGradLanes);
    for (int i = blockIdx.x * (blockDim.x / kGradLanes) + grp; i < n; i += rows) {
        const double* xi = Xr + (size_t)i * m;
        double u[kGradReg];
        if (SMEM) {
            __syncwarp(mask);
            for (int k = l; k < m; k += kGradLanes) us[k] = (lam ? -gw[k] * lam[k] : gw[k]) * __ldg(xi + k);
            __syncwarp(mask);
        } else {
#pragma unroll
            for (int q = 0; q < kGradReg; ++q) {
                const int k = l + q * kGradLanes;
                u[q] = k < m ? (lam ? -gw[k] * lam[k] : gw[k]) * __ldg(xi + k) : 0.0;
            }
        }
        const int p0 = ia[i], p1 = ia[i + 1];
        for (int p = p0; p < p1; p += 4) {
            int j[4];
            double s[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                j[e] = ja[min(p + e, p1 - 1)];
                s[e] = 0.0;
            }
            if (SMEM) {
                for (int k = l; k < m; k += kGradLanes) {
                    const double uk = us[k];
#pragma unroll
                    for (int e = 0; e < 4; ++e) s[e] = fma(uk, __ldg(Xr + (size_t)j[e] * m + k), s[e]);
                }
            } else {
#pragma unroll
                for (int q = 0; q < kGradReg; ++q) {
                    const int k = l + q * kGradLanes;
                    if (q * kGradLanes < m) {  // uniform
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (k < m && p + e < p1) s[e] = fma(u[q], __ldg(Xr + (size_t)j[e] * m + k), s[e]);
                    }
                }
            }
            // lanes 0, 2, 4, 6 end with the sums of entries 0..3: halve the values kept per step
            const bool hi4 = l & 4, hi2 = l & 2;
            double a0 = hi4 ? s[2] : s[0], a1 = hi4 ? s[3] : s[1];
            a0 += __shfl_xor_sync(mask, hi4 ? s[0] : s[2], 4);
            a1 += __shfl_xor_sync(mask, hi4 ? s[1] : s[3], 4);
            double b = hi2 ? a1 : a0;
            b += __shfl_xor_sync(mask, hi2 ? a0 : a1, 2);
            b += __shfl_xor_sync(mask, b, 1);
            const int e = l >> 1;
            if (!(l & 1) && p + e < p1) grad[p + e] = (half && ja[p + e] != i) ? 2.0 * b : b;
        }
    }
}

// The same for more columns than that: sixteen lanes per row, w o x_i in shared
// memory, two entries in flight, the columns in chunks (an entry's sums added up
// in grad), so that enough warps fit beside the weights and the rows of X that
// they read stay in L1.
static constexpr int kPairLanes = 16;

__global__ void __launch_bounds__(256) eig_grad_pairs(int n, const int* __restrict__ ia, const int* __restrict__ ja, int m,
                                                      int chunk, const double* __restrict__ Xr, const double* __restrict__ gw,
                                                      const double* __restrict__ lam, int half, double* __restrict__ grad)
{
    extern __shared__ double u_sm[];
    const int l = threadIdx.x & (kPairLanes - 1), grp = threadIdx.x / kPairLanes;
    const unsigned mask = 0xffffu << (threadIdx.x & 16);
    double* us = u_sm + (size_t)grp * chunk;
    const int rows = gridDim.x * (blockDim.x / kPairLanes);
    for (int i = blockIdx.x * (blockDim.x / kPairLanes) + grp; i < n; i += rows) {
        const int p0 = ia[i], p1 = ia[i + 1];
        for (int c0 = 0; c0 < m; c0 += chunk) {
            const int mc = min(chunk, m - c0);
            const double* X = Xr + c0;
            __syncwarp(mask);
            for (int k = l; k < mc; k += kPairLanes)
                us[k] = (lam ? -gw[c0 + k] * lam[c0 + k] : gw[c0 + k]) * __ldg(X + (size_t)i * m + k);
            __syncwarp(mask);
            for (int p = p0; p < p1; p += 2) {
                const int j0 = ja[p], j1 = ja[min(p + 1, p1 - 1)];
                double s0 = 0.0, s1 = 0.0;
#pragma unroll 4
                for (int k = l; k < mc; k += kPairLanes) {
                    const double uk = us[k];
                    s0 = fma(uk, __ldg(X + (size_t)j0 * m + k), s0);
                    s1 = fma(uk, __ldg(X + (size_t)j1 * m + k), s1);
                }
                // lanes 0 and 8 end with the sums of the two entries
                const bool hi = l & 8;
                double b = (hi ? s1 : s0) + __shfl_xor_sync(mask, hi ? s0 : s1, 8);
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) b += __shfl_xor_sync(mask, b, o);
                const int q = p + (l >> 3);
                if (!(l & 7) && q < p1) {
                    if (half && ja[q] != i) b *= 2.0;
                    grad[q] = c0 > 0 ? grad[q] + b : b;
                }
            }
        }
    }
}

// The same with a warp per row and an entry at a time; with QUADS rows of eight
// entries and more take four.  For few rows, and for columns so many that an
// entry's five steps weigh little beside its terms.
template <bool QUADS>
__global__ void __launch_bounds__(256) eig_grad_warp(int n, const int* __restrict__ ia, const int* __restrict__ ja, int m,
                                                     const double* __restrict__ Xr, const double* __restrict__ gw,
                                                     const double* __restrict__ lam, int half, double* __restrict__ grad)
{
    extern __shared__ double u_sm[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    double* u = u_sm + (size_t)wib * m;
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int i = warp; i < n; i += nwarps) {
        for (int k = lane; k < m; k += 32) {
            const double w = lam ? -gw[k] * lam[k] : gw[k];
            u[k] = w * Xr[(size_t)i * m + k];
        }
        __syncwarp();
        int p = ia[i];
        if constexpr (QUADS) {
            const int p1 = ia[i + 1];
            if (p1 - p >= 8)
                for (; p + 4 <= p1; p += 4) {
                    const double* x[4];
                    double s[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        x[e] = Xr + (size_t)ja[p + e] * m;
                        s[e] = 0.0;
                    }
#pragma unroll 4
                    for (int k = lane; k < m; k += 32) {
                        const double uk = u[k];
#pragma unroll
                        for (int e = 0; e < 4; ++e) s[e] = fma(uk, __ldg(x[e] + k), s[e]);
                    }
                    // lanes 0, 8, 16, 24 end with the sums of the four entries
                    const bool hi = lane & 16, hj = lane & 8;
                    double a0 = hi ? s[2] : s[0], a1 = hi ? s[3] : s[1];
                    a0 += __shfl_xor_sync(0xffffffffu, hi ? s[0] : s[2], 16);
                    a1 += __shfl_xor_sync(0xffffffffu, hi ? s[1] : s[3], 16);
                    double b = (hj ? a1 : a0) + __shfl_xor_sync(0xffffffffu, hj ? a0 : a1, 8);
#pragma unroll
                    for (int o = 4; o > 0; o >>= 1) b += __shfl_xor_sync(0xffffffffu, b, o);
                    const int q = p + (lane >> 3);
                    if (!(lane & 7)) grad[q] = (half && ja[q] != i) ? 2.0 * b : b;
                }
        }
        for (; p < ia[i + 1]; ++p) {
            const int j = ja[p];
            double s = 0.0;
            for (int k = lane; k < m; k += 32) s = fma(u[k], __ldg(Xr + (size_t)j * m + k), s);
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) grad[p] = (half && j != i) ? 2.0 * s : s;
        }
        __syncwarp();
    }
}

// Which form (us at 40^3 7-point / 300 x 300 5-point / 24^3 27-point):
//   columns       128          256          384          640             1000
//   8 lanes   183 262 149  325 437 210  465 655 333   943 1284 532   2336 2878 998
//   pairs     212 233 163  355 394 257  492 561 353   842  950 523   1249 1400 809
//   a warp    299 310 251  415 434 339  530 557 427   782  836 592   1610 1674 1037
// Eight lanes up to 256 columns (their weights are 64 KB a CTA there), pairs to
// 512 and above 896, a warp between.  With fewer than 16 rows per SM eight lanes a
// row leave the chip idle: from 64 columns a warp per row with quads (8^3
// 27-point, 128 columns 55 -> 30 us, 512 columns 124 -> 67), above 512 columns
// also with fewer than 32 rows per SM (16^3 7-point, 1,500 columns 228 -> 128).
cudaError_t launch_eig_grad(int n, const int* ia, const int* ja, int m, const double* Xr, const double* gw,
                            double* grad, cudaStream_t s, const double* lam, int half)
{
    if (n <= 0) return cudaSuccess;
    if (m <= 0 || m > 2048) return cudaErrorInvalidValue;
    const bool few = n < 16 * num_sms() ? m >= 64 : n < 32 * num_sms() && m > 512;
    const bool warp = few || (m > 512 && m <= 896);
    const bool regs = m <= kGradLanes * kGradReg, pairs = m > 256;
    const int chunk = std::min(m, pairs ? 512 : 256);
    const int per = warp ? 8 : pairs ? 256 / kPairLanes : 256 / kGradLanes;  // rows per CTA
    const size_t smem = warp ? (size_t)per * m * sizeof(double) : regs ? 0 : (size_t)per * chunk * sizeof(double);
    const int blocks = (int)std::min<long long>(((long long)n + per - 1) / per, (long long)num_sms() * 16);
    auto launch = [&](auto kern, auto... args) {
        if (smem > 48 * 1024) {
            const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
        kern<<<blocks, 256, smem, s>>>(n, ia, ja, m, args..., Xr, gw, lam, half, grad);
        count_launches(1);
        return cudaGetLastError();
    };
    if (few) return launch(eig_grad_warp<true>);
    if (warp) return launch(eig_grad_warp<false>);
    if (pairs) return launch(eig_grad_pairs, chunk);
    return regs ? launch(eig_grad<false>) : launch(eig_grad<true>);
}

}  // namespace feast
