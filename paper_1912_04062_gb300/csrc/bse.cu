// bse.cu -- device kernels of the Bethe-Salpeter driver around the skew
// solver (Sec. 3: the structure-preserving method for a definite
// H_BS = [[A, B], [-conj(B), -conj(A)]], A Hermitian, B complex symmetric):
//   1. M = J H = [[Re(A+B), Im(A-B)], [-Im(A+B), Re(A-B)]] (Eq. SymmetricM),
//      real symmetric, positive definite when H_BS is definite;
//   2. M = L L^T (Cholesky, lower);
//   3. the skew-symmetric eigenproblem of K = L^T J L, J = [[0, I], [-I, 0]];
//   4. the eigenvectors back: x = L^-T z solves H x = -i lambda x, and
//      psi = Q x with the unitary Q = [[I, -iI], [I, iI]] / sqrt(2) of
//      Theorem 1 is the eigenvector of H_BS for lambda > 0; psi is scaled to
//      psi^H S psi = 1, S = diag(I, -I) (for orthonormal z it is 1/lambda).
// Steps 2 and 4 are blocked by 64: the diagonal blocks and the panels'
// triangular solves are kernels of their own, the trailing updates FP64
// products (lower tiles for the Cholesky, full for the back substitution).
#include <cmath>

#include "common.cuh"
#include "internal.h"

namespace sk {
namespace {

constexpr int CB = 64;

__global__ void bse_build_m_kernel(int h, const double* __restrict__ Ar, const double* __restrict__ Ai, int lda,
                                   const double* __restrict__ Br, const double* __restrict__ Bi, int ldb,
                                   double* __restrict__ M, int ldm) {
    const long long N = 2LL * h, total = N * N;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(e % N), j = (int)(e / N);
        const int bi = i >= h, bj = j >= h, ii = i - bi * h, jj = j - bj * h;
        const double ar = Ar[ii + (size_t)jj * lda], ai = Ai[ii + (size_t)jj * lda];
        const double br = Br[ii + (size_t)jj * ldb], bm = Bi[ii + (size_t)jj * ldb];
        double v;
        if (!bi && !bj) v = ar + br;          // Re(A + B)
        else if (!bi && bj) v = ai - bm;      // Im(A - B)
        else if (bi && !bj) v = -(ai + bm);   // -Im(A + B)
        else v = ar - br;                     // Re(A - B)
        M[i + (size_t)j * ldm] = v;
    }
}

// Unblocked Cholesky of the kb x kb diagonal block (lower, in place), right
// looking; a pivot that is not positive and finite records
// SKEW_ERR_NOT_DEFINITE and stops the factorisation of the block.  A serial
// chain of a square root, a quotient (about 600 clocks each) and an update per
// column: two barriers a column, the roots beside the block so that every
// thread can test the pivot itself, and the update on thread columns without
// an integer division.
__global__ void __launch_bounds__(256) chol_diag_kernel(int kb, double* __restrict__ D, int ld, int* status) {
    __shared__ double S[CB][CB + 1], root[CB];
    const int t = threadIdx.x, q = t & (CB - 1);
    for (int e = t; e < CB * CB; e += 256) {
        const int i = e % CB, j = e / CB;
        S[i][j] = (i < kb && i >= j) ? D[i + (size_t)j * ld] : 0.0;
    }
    __syncthreads();
    int done = kb;
    for (int j = 0; j < kb; j++) {
        const double d = S[j][j];
        if (!(d > 0.0) || !isfinite(d)) {
            if (t == 0) sk_set_error(status, SKEW_ERR_NOT_DEFINITE);
            done = j;
            break;  // every thread reads the same pivot
        }
        if (t < CB && t >= j) {
            const double r = sqrt(d);
            if (t == j) root[j] = r;
            else S[t][j] /= r;
        }
        __syncthreads();
        if (q > j) {
            const double w = S[q][j];
#pragma unroll 4
            for (int i = j + 1 + (t >> 6); i < kb; i += 4)
                if (q <= i) S[i][q] = fma(-S[i][j], w, S[i][q]);
        }
        __syncthreads();
    }
    for (int e = t; e < CB * CB; e += 256) {
        const int i = e % CB, j = e / CB;
        if (i < kb && i >= j) D[i + (size_t)j * ld] = (i == j && j < done) ? root[j] : S[i][j];
    }
}

// The two triangular solves with a diagonal block, a warp to each right-hand
// side (8 to a CTA): lane l holds entries l and l + 32, each step's solution is
// broadcast by a shuffle and taken off the rest.  64 steps of a short chain,
// bound by it and by the FP64 pipe of the SMs that have a CTA.  The form with a
// right-hand side per thread had 64 quotients of 600 clocks in a chain on the
// few SMs that its CTAs of 128 filled: 139 us a panel and 173 us a block of the
// back substitution at 2h = 1200 (now 29 and 28), whatever their width.  The
// driver at h = 600: 29.0 -> 24.7 ms.
constexpr int TR = 8;

// L (lower, kb x kb at ld) and the reciprocals of its diagonal; zero and one
// beyond kb, so that the steps there change nothing.
__device__ inline void load_diag_block(int t, int kb, const double* __restrict__ L, int ld, double (*Ls)[CB + 1],
                                       double* inv) {
    for (int e = t; e < CB * CB; e += 256) {
        const int i = e % CB, j = e / CB;
        Ls[i][j] = (i < kb && i >= j) ? L[i + (size_t)j * ld] : (i == j ? 1.0 : 0.0);
    }
    __syncthreads();
    if (t < CB) inv[t] = 1.0 / Ls[t][t];
    __syncthreads();
}

// s / d from y = 1 / d, corrected once (the largest relative error over 2.3e8
// random arguments was 0.999 2^-53, as that of the division)
__device__ __forceinline__ double quot_corrected(double s, double d, double y) {
    const double x = s * y;
    return fma(fma(-x, d, s), y, x);
}

// Panel below a factored diagonal block: P <- P L11^-T (row r: x L11^T = p by
// forward substitution), and NP = -P for the trailing update's second factor.
__global__ void __launch_bounds__(256) chol_panel_kernel(int m, int kb, const double* __restrict__ L11, int ld,
                                                         double* __restrict__ P, double* __restrict__ NP, int ldn) {
    __shared__ double Ls[CB][CB + 1], inv[CB], X[TR][CB + 1];
    const int t = threadIdx.x, w = t >> 5, lane = t & 31, r0 = blockIdx.x * TR;
    for (int e = t; e < TR * CB; e += 256) {
        const int r = e % TR, j = e / TR;
        X[r][j] = (r0 + r < m && j < kb) ? P[r0 + r + (size_t)j * ld] : 0.0;
    }
    load_diag_block(t, kb, L11, ld, Ls, inv);
    double a = X[w][lane], b = X[w][lane + 32];
    for (int j = 0; j < 32; j++) {
        const double x = quot_corrected(__shfl_sync(~0u, a, j), Ls[j][j], inv[j]);
        if (lane == j) a = x;
        if (lane > j) a = fma(-x, Ls[lane][j], a);
        b = fma(-x, Ls[lane + 32][j], b);
    }
    for (int j = 0; j < 32; j++) {
        const double x = quot_corrected(__shfl_sync(~0u, b, j), Ls[j + 32][j + 32], inv[j + 32]);
        if (lane == j) b = x;
        if (lane > j) b = fma(-x, Ls[lane + 32][j + 32], b);
    }
    X[w][lane] = a;
    X[w][lane + 32] = b;
    __syncthreads();
    for (int e = t; e < TR * CB; e += 256) {
        const int r = e % TR, j = e / TR;
        if (r0 + r < m && j < kb) {
            P[r0 + r + (size_t)j * ld] = X[r][j];
            NP[r0 + r + (size_t)j * ldn] = -X[r][j];
        }
    }
}

// K = L^T J L on 32-tiles I >= J of its lower triangle, mirrored with the sign
// changed (K is skew).  Bound by the FP64 pipe, so the work is what counts:
// (J L)[k, j] is L[k + h, j] for k < h and -L[k - h, j] below, and with L lower
// a tile's k runs over [i0, h) and [max(i0, h + j0), N) only, 5/6 h^3 FMAs
// of the 8 h^3 of a full product.  Small tiles because the longest one, the
// first, is then a quarter as long as a 64-tile; rows in ascending order start
// the long ones first.  N = 1200: 0.59 ms against 3.6 for the full product on
// 64-tiles; the driver at h = 600 24.7 -> 21.6 ms, outputs equal to 5e-17.
constexpr int KT = 32;

__global__ void __launch_bounds__(256) bse_k_kernel(int h, const double* __restrict__ L, int ld,
                                                    double* __restrict__ K, int ldk) {
    __shared__ double As[KT][KT + 1], Bs[KT][KT + 1];
    const int N = 2 * h, t = threadIdx.x, tx = t & 15, ty = t >> 4;
    // invert blockIdx = I (I + 1) / 2 + J
    const long long b = blockIdx.x;
    int I = (int)((sqrt(8.0 * (double)b + 1.0) - 1.0) * 0.5);
    while ((long long)(I + 1) * (I + 2) / 2 <= b) I++;
    while ((long long)I * (I + 1) / 2 > b) I--;
    const int i0 = I * KT, j0 = (int)(b - (long long)I * (I + 1) / 2) * KT;
    double acc[2][2] = {};
    for (int half = 0; half < 2; half++) {
        const int kbeg = half ? max(i0, h + j0) : i0, kend = half ? N : h;
        for (int k0 = kbeg; k0 < kend; k0 += KT) {
            for (int e = t; e < KT * KT; e += 256) {
                const int k = k0 + e % KT, c = e / KT, i = i0 + c, j = j0 + c, r = half ? k - h : k + h;
                As[e % KT][c] = (k < kend && i <= k) ? L[k + (size_t)i * ld] : 0.0;
                const double v = (k < kend && j <= r) ? L[r + (size_t)j * ld] : 0.0;
                Bs[e % KT][c] = half ? -v : v;
            }
            __syncthreads();
#pragma unroll 8
            for (int k = 0; k < KT; k++) {
                const double a0 = As[k][tx], a1 = As[k][tx + 16], b0 = Bs[k][ty], b1 = Bs[k][ty + 16];
                acc[0][0] = fma(a0, b0, acc[0][0]);
                acc[0][1] = fma(a0, b1, acc[0][1]);
                acc[1][0] = fma(a1, b0, acc[1][0]);
                acc[1][1] = fma(a1, b1, acc[1][1]);
            }
            __syncthreads();
        }
    }
    for (int r = 0; r < 2; r++)
        for (int c = 0; c < 2; c++) {
            const int i = i0 + tx + 16 * r, j = j0 + ty + 16 * c;
            if (i >= N || i < j) continue;
            K[i + (size_t)j * ldk] = i == j ? 0.0 : acc[r][c];
            if (i > j) K[j + (size_t)i * ldk] = -acc[r][c];
        }
}

// Back substitution with one diagonal block: X_I <- L_II^-T X_I, a warp per
// right-hand side column (L_II^T x = z: x_j = (z_j - sum_{l > j} L_lj x_l) / L_jj).
__global__ void __launch_bounds__(256) trsm_lt_diag_kernel(int kb, const double* __restrict__ Lii, int ld,
                                                           double* __restrict__ X, int ldx, int ncols) {
    __shared__ double Ls[CB][CB + 1], inv[CB];
    const int t = threadIdx.x, lane = t & 31;
    load_diag_block(t, kb, Lii, ld, Ls, inv);
    const int c = blockIdx.x * TR + (t >> 5);
    if (c >= ncols) return;
    double* x0 = X + (size_t)c * ldx;
    double a = (lane < kb) ? x0[lane] : 0.0, b = (lane + 32 < kb) ? x0[lane + 32] : 0.0;
    for (int j = 31; j >= 0; j--) {
        const double x = quot_corrected(__shfl_sync(~0u, b, j), Ls[j + 32][j + 32], inv[j + 32]);
        if (lane == j) b = x;
        if (lane < j) b = fma(-x, Ls[j + 32][lane + 32], b);
        a = fma(-x, Ls[j + 32][lane], a);
    }
    for (int j = 31; j >= 0; j--) {
        const double x = quot_corrected(__shfl_sync(~0u, a, j), Ls[j][j], inv[j]);
        if (lane == j) a = x;
        if (lane < j) a = fma(-x, Ls[j][lane], a);
    }
    if (lane < kb) x0[lane] = a;
    if (lane + 32 < kb) x0[lane + 32] = b;
}

// psi = Q x sqrt(lambda), x = Xr + i Xi (2h x nev), Q = [[I, -iI], [I, iI]] / sqrt(2)
__global__ void bse_psi_kernel(int h, int nev, const double* __restrict__ Xr, const double* __restrict__ Xi, int ldx,
                               const double* __restrict__ lambda, double* __restrict__ Pr, double* __restrict__ Pi,
                               int ldp) {
    const long long total = (long long)h * nev;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(e % h), k = (int)(e / h);
        const double s = sqrt(fmax(lambda[k], 0.0)) * 0.70710678118654752440;
        const size_t c = (size_t)k * ldx, o = (size_t)k * ldp;
        const double rt = Xr[c + i], rb = Xr[c + i + h], it = Xi[c + i], ib = Xi[c + i + h];
        Pr[o + i] = s * (rt + ib);
        Pi[o + i] = s * (it - rb);
        Pr[o + i + h] = s * (rt - ib);
        Pi[o + i + h] = s * (it + rb);
    }
}

inline int grid_of(long long total) {
    long long g = (total + 255) / 256;
    return (int)(g > 16384 ? 16384 : (g < 1 ? 1 : g));
}

}  // namespace

cudaError_t bse_build_m(cudaStream_t st, int h, const double* Ar, const double* Ai, int lda, const double* Br,
                        const double* Bi, int ldb, double* M, int ldm) {
    bse_build_m_kernel<<<grid_of(4LL * h * h), 256, 0, st>>>(h, Ar, Ai, lda, Br, Bi, ldb, M, ldm);
    count_launch();
    return cudaGetLastError();
}

// M (N x N, ld) <- its lower Cholesky factor; NP: scratch of N x 64.
cudaError_t cholesky_lower(cudaStream_t st, int N, double* M, int ld, double* NP, int* status) {
    for (int k0 = 0; k0 < N; k0 += CB) {
        const int kb = (N - k0 < CB) ? N - k0 : CB;
        double* D = M + k0 + (size_t)k0 * ld;
        chol_diag_kernel<<<1, 256, 0, st>>>(kb, D, ld, status);
        count_launch();
        const int m = N - k0 - kb;
        if (m <= 0) break;
        double* P = D + kb;
        chol_panel_kernel<<<(m + TR - 1) / TR, 256, 0, st>>>(m, kb, D, ld, P, NP, m);
        count_launch();
        // A22 += P (-P)^T on the lower 64-tiles
        if (const cudaError_t e = gemm_lower_tiles(st, m, kb, P, ld, NP, m, D + kb + (size_t)kb * ld, ld, false))
            return e;
    }
    return cudaGetLastError();
}

cudaError_t bse_k(cudaStream_t st, int h, const double* L, int ld, double* K, int ldk) {
    const long long T = (2LL * h + KT - 1) / KT;
    bse_k_kernel<<<(unsigned)(T * (T + 1) / 2), 256, 0, st>>>(h, L, ld, K, ldk);
    count_launch();
    return cudaGetLastError();
}

// X (N x ncols, ld ldx) <- L^-T X for the lower factor L, by blocks of 64 from
// the bottom: X_I <- L_II^-T X_I, then X_{0:I} -= L_{I, 0:I}^T X_I.
cudaError_t trsm_lower_t(cudaStream_t st, int N, const double* L, int ld, double* X, int ldx, int ncols) {
    if (N <= 0 || ncols <= 0) return cudaSuccess;
    const int nb = (N + CB - 1) / CB;
    for (int b = nb - 1; b >= 0; b--) {
        const int i0 = b * CB, kb = (N - i0 < CB) ? N - i0 : CB;
        trsm_lt_diag_kernel<<<(ncols + TR - 1) / TR, 256, 0, st>>>(kb, L + i0 + (size_t)i0 * ld, ld, X + i0, ldx,
                                                                    ncols);
        count_launch();
        if (i0 > 0) {
            // X[0:i0, :] -= (L[i0:i0+kb, 0:i0])^T X[i0:i0+kb, :]
            if (const cudaError_t e = gemm(st, true, false, i0, ncols, kb, -1.0, L + i0, ld, X + i0, ldx, 1.0, X, ldx))
                return e;
        }
    }
    return cudaGetLastError();
}

cudaError_t bse_psi(cudaStream_t st, int h, int nev, const double* Xr, const double* Xi, int ldx,
                    const double* lambda, double* Pr, double* Pi, int ldp) {
    bse_psi_kernel<<<grid_of((long long)h * nev), 256, 0, st>>>(h, nev, Xr, Xi, ldx, lambda, Pr, Pi, ldp);
    count_launch();
    return cudaGetLastError();
}

}  // namespace sk
