// One-CTA Cholesky factorization and triangular inverse used by the reduced
// generalized eigenproblem A_Q v = lambda B_Q v of the Rayleigh-Ritz step
// (FEAST v4.0 guide, Sec. 1.1; the guide's dense reduced solvers are the
// LAPACK sygv family, whose first step is B = L L^T).
//
// With B~ = L L^T and X = L^{-1}, S = D X^T satisfies S^T B_Q S = I for the
// diagonal scaling D, so the generalized problem turns into the standard one
// S^T A_Q S w = lambda w.  When the filtered subspace is nearly B-orthogonal
// (every loop after the first few), B~ is close to I, L is close to I and
// S^T A_Q S stays close to diagonal, so the Jacobi sweeps that follow converge
// in a few sweeps.
#pragma once

namespace feast {

static constexpr double kCholCondMax = 1e8;  // accepted bound on ||L^{-1}||_F^2

// Position of X[k][c] (c < k) in the m x m array: the strict upper triangle,
// rows and columns reversed, so that the columns c of one k are contiguous.
__device__ __forceinline__ size_t chol_inv_at(int m, int k, int c) { return (size_t)(m - 1 - k) * m + (m - 1 - c); }

// All threads of the CTA call this.  M: m x m row-major holding the symmetric
// positive definite B~ (lower triangle read).  On return true: lower triangle
// of M (with the diagonal) = L, xd[i] = 1 / L_ii, strict upper triangle of M =
// the strict lower triangle of X (at chol_inv_at).  Returns false when a pivot
// is not positive or ||X||_F^2 > kCholCondMax; M is then partially
// overwritten.  cj: m doubles of scratch; red: blockDim.x doubles of shared
// scratch.
// Bound: one SM's FP64 pipe, which a warp instruction holds for 16 cycles
// however few of its lanes work.  So one thread takes the pivot's root and
// reciprocal (all warps doing so took most of the 1.66 ms at m = 150), the
// columns are scaled by the reciprocal, and the inverse is formed row by row
// with a thread per column and the sum cut into G parts, without shuffles.
__device__ inline bool cta_chol_inv(int m, double* M, double* xd, double* cj, double* red)
{
    const int tid = threadIdx.x, nt = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    for (int j = 0; j < m; ++j) {
        if (tid == 0) {
            const double d = M[(size_t)j * m + j];
            const double l = d > 0.0 ? sqrt(d) : 0.0;
            M[(size_t)j * m + j] = l;
            xd[j] = red[0] = l > 0.0 ? 1.0 / l : 0.0;
        }
        __syncthreads();
        const double r = red[0];
        if (!(r > 0.0)) return false;  // same value in every thread: uniform exit
        for (int i = j + 1 + tid; i < m; i += nt) {
            const double v = M[(size_t)i * m + j] * r;
            M[(size_t)i * m + j] = v;
            cj[i] = v;
        }
        __syncthreads();
        for (int i = j + 1 + warp; i < m; i += nw) {
            const double ci = cj[i];
            for (int k = j + 1 + lane; k <= i; k += 32) M[(size_t)i * m + k] -= ci * cj[k];
        }
        __syncthreads();
    }
    // X[i][c] = -(1/L_ii) (L[i][c] / L_cc + sum_{c<k<i} L[i][k] X[k][c])
    const int mc = (m + 31) / 32 * 32, G = nt / mc;
    const int c = tid % mc, g = tid / mc;
    double nrm = 0.0;
    for (int i = tid; i < m; i += nt) nrm = fma(xd[i], xd[i], nrm);
    for (int i = 1; i < m; ++i) {
        const double* Li = M + (size_t)i * m;
        if (G >= 1) {
            double s = 0.0;
            if (g < G && c < i)
                for (int k = c + 1 + g; k < i; k += G) s = fma(Li[k], M[chol_inv_at(m, k, c)], s);
            red[tid] = s;
            __syncthreads();
            if (tid < i) {  // g = 0, c = tid
                for (int q = 1; q < G; ++q) s += red[q * mc + c];
                const double x = -xd[i] * fma(Li[c], xd[c], s);
                M[chol_inv_at(m, i, c)] = x;
                nrm = fma(x, x, nrm);
            }
        } else {
            for (int cc = tid; cc < i; cc += nt) {
                double s = Li[cc] * xd[cc];
                for (int k = cc + 1; k < i; ++k) s = fma(Li[k], M[chol_inv_at(m, k, cc)], s);
                const double x = -xd[i] * s;
                M[chol_inv_at(m, i, cc)] = x;
                nrm = fma(x, x, nrm);
            }
        }
        __syncthreads();
    }
    for (int o = 16; o > 0; o >>= 1) nrm += __shfl_xor_sync(0xffffffffu, nrm, o);
    __syncthreads();
    if (lane == 0) red[warp] = nrm;
    __syncthreads();
    double tot = 0.0;
    for (int w = 0; w < nw; ++w) tot += red[w];
    __syncthreads();
    return tot <= kCholCondMax;
}

}  // namespace feast
