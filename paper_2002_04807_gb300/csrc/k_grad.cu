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
// of w o x_i in registers (up to kGradReg of them, in shared memory beyond) and
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

cudaError_t launch_eig_grad(int n, const int* ia, const int* ja, int m, const double* Xr, const double* gw,
                            double* grad, cudaStream_t s, const double* lam, int half)
{
    if (n <= 0) return cudaSuccess;
    if (m <= 0 || m > 2048) return cudaErrorInvalidValue;
    const bool regs = m <= kGradLanes * kGradReg;
    // rows per CTA: 32, fewer where their weights would not fit in shared memory
    int threads = 256;
    while (!regs && threads > 32 && (size_t)(threads / kGradLanes) * m * sizeof(double) > 64 * 1024) threads /= 2;
    const size_t smem = regs ? 0 : (size_t)(threads / kGradLanes) * m * sizeof(double);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(eig_grad<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const int per = threads / kGradLanes;
    const long long blocks = std::min<long long>(((long long)n + per - 1) / per, (long long)num_sms() * 16);
    if (regs) eig_grad<false><<<(int)blocks, threads, 0, s>>>(n, ia, ja, m, Xr, gw, lam, half, grad);
    else eig_grad<true><<<(int)blocks, threads, smem, s>>>(n, ia, ja, m, Xr, gw, lam, half, grad);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace feast
