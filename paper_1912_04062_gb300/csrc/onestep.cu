// onestep.cu -- one-step Householder tridiagonalisation of a skew-symmetric
// matrix (the direct form of Sec. 2.3.1: A -> T without the band in between)
// over the whole GPU, and the FP64 back-transformation by its reflectors.
//
// Why one step: the FP64 pipe of this part does 1.68 FMA per clock and SM
// (measured), so even a matrix-vector product is bound by the arithmetic and
// not by memory (one element read per 3 FMAs needs 2.8 TB/s over 152 SMs).
// The two-step route's advantage, products instead of matrix-vector work, is
// therefore worth nothing in FP64, while its bulge chase (a chain of 2 n
// dependent tasks) and its second back-transformation (another 4 n^2 nev flops)
// remain.  Per column c the kernel needs ONE exchange between the CTAs:
//
//   every CTA owns the rows i = g (mod G) of the full skew matrix (shared
//   memory, the rest in L2/HBM) and keeps the current reflector u and
//   p = A u whole in shared memory;
//   1. gather (q_j, a_j), j > c: q = A x of the previous reflector's
//      unscaled column x and a = column c before its rank-2 update.  With
//      u = x - beta e_0:  A u = q - beta a, so the product could be formed
//      before beta was known and the norm, sqrt and division are off the
//      critical path;
//   2. every CTA forms p, the updated column x = a + sigma (u p_c - p u_c) and, later,
//      its norm redundantly (same order everywhere: same bits);
//   3. one pass over the own rows applies A += u w^T - w u^T (Eqs. 2-6 with
//      u1 = -u2) and multiplies the result by x; the sums and the next column's
//      elements are published.
//
#include <algorithm>
#include <cfloat>

#include "common.cuh"
#include "internal.h"
#include "onestep_dev.cuh"

namespace sk {

using namespace onestep;

namespace {

constexpr int OT = 256;     // threads of the reduction kernel
constexpr int OMAXR = 64;   // rows of one CTA at most (n <= 64 G)
// Dynamic shared memory at most: of 227 KB, the static arrays take about 5.3 KB.
// The kernels' limits are set to constants, so that calls of several threads
// cannot take them from one another.
constexpr int OS_SMEM = 221 * 1024, WY_SMEM = 226 * 1024;

struct OsArgs {
    int n;
    double* F;     // full skew matrix by rows, F[i * n + j]; rows that are not in shared memory are updated here
    double* V;     // reflectors by columns (ld n), zeroed by the caller: v[k + 1] = 1
    double* tau;   // n entries
    double* alpha; // T[k, k + 1]
    double2* qa;   // 2 n: (q, a), double-buffered
    unsigned* ctr; // arrivals, zeroed by onestep_full
    const unsigned long long* amax;  // max |A| (os_scale)
    int* status;
    unsigned cap;
    int srows;     // own rows kept in shared memory (the last ones: they live longest)
};

__global__ void __launch_bounds__(OT, 1) onestep_kernel(OsArgs o) {
    extern __shared__ __align__(16) double os_sm[];
    __shared__ double s_part[OMAXR][OCW];
    __shared__ double2 s_coef[OMAXR];  // sigma u_i, -sigma p_i of the own rows
    __shared__ double s_red[4];
    __shared__ double s_sc[4];  // beta, sigma, 1 / u_0, u_0
    __shared__ int s_ok;
    const int n = o.n, G = gridDim.x, g = blockIdx.x;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int ldn = n | 1;
    double* u = os_sm;           // u of the pending update (indices k ..)
    double* p = u + ldn;         // A u of it
    double* x = p + ldn;         // the column being eliminated
    double* rows = x + ldn;
    const int Rt = (n - 1 - g) / G + 1;              // own rows: g, g + G, ...
    const int rs0 = Rt > o.srows ? Rt - o.srows : 0; // the first one in shared memory
    const int ilast = g + (Rt - 1) * G;
    const double scale = os_scale(*o.amax);
    for (int r = rs0; r < Rt; r++)
        for (int j = t; j < n; j += OT) rows[(size_t)(r - rs0) * ldn + j] = scale * o.F[(size_t)(g + r * G) * n + j];
    if (scale != 1.0)  // row 0 is read by all below, and never again
        for (int r = g == 0 ? 1 : 0; r < rs0; r++)
            for (int j = t; j < n; j += OT) o.F[(size_t)(g + r * G) * n + j] *= scale;
    unsigned target = 0;
    double beta = 0.0, sigma = 0.0;
    for (int k = 0; k + 1 < n; k++) {
        if (ilast < k + 1) return;  // no rows left: the others do not count on this CTA any more
        // ---- 1. gather; p of the previous reflector, the updated column x
        const double2* qa = o.qa + (size_t)(k & 1) * n;
        if (k == 0) {
            // column 0 of A, nothing pending: element (j, 0) = -element (0, j)
            for (int j = t; j < n; j += OT) {
                x[j] = -scale * o.F[j];
                u[j] = 0.0;
                p[j] = 0.0;
            }
        } else {
            // two elements are under way while element k is waited for
            const int j0 = k + 1 + t, j1 = j0 + OT;
            double2 e0 = make_double2(0.0, 0.0), e1 = e0;
            if (j0 < n) e0 = __ldcg(qa + j0);
            if (j1 < n) e1 = __ldcg(qa + j1);
            const double2 qk = __ldcg(qa + k);
            const double uk = -sigma * u[k], pk = sigma * fma(-beta, qk.y, qk.x);
            if (j0 < n) {
                const double pj = fma(-beta, e0.y, e0.x);
                p[j0] = pj;
                x[j0] = fma(u[j0], pk, fma(pj, uk, e0.y));
            }
            if (j1 < n) {
                const double pj = fma(-beta, e1.y, e1.x);
                p[j1] = pj;
                x[j1] = fma(u[j1], pk, fma(pj, uk, e1.y));
            }
#pragma unroll 4
            for (int j = j1 + OT; j < n; j += OT) {
                const double2 e = __ldcg(qa + j);
                const double pj = fma(-beta, e.y, e.x);
                p[j] = pj;
                x[j] = fma(u[j], pk, fma(pj, uk, e.y));
            }
        }
        __syncthreads();
        if (k == n - 2) {
            // T[n-1, n-2] = x_{n-1}; this CTA owns the last row
            if (t == 0) o.alpha[k] = -x[n - 1];
            break;
        }
        // ---- 2. update the own rows i > k and multiply by x
        const int rf = (k + 1 > g) ? (k + 1 - g + G - 1) / G : 0;  // first own row below k
        const int R = Rt - rf;
        const int rg = max(rs0, rf) - rf;  // rows of global memory
        for (int r = t; r < R; r += OT)
            s_coef[r] = make_double2(sigma * u[g + (rf + r) * G], -sigma * p[g + (rf + r) * G]);
        __syncthreads();
        const int nss = R - rg >= 16 ? 1 : R - rg >= 8 ? 2 : R - rg >= 4 ? 4 : 8, nsg = rg >= 16 ? 4 : 8;
        os_pass<8>(nsg, nss, R, rg, o.F + (size_t)(g + rf * G) * n, rows + (size_t)(rf + rg - rs0) * ldn, n, ldn, g + rf * G, G,
                   k, s_coef, u, p, x, warp, lane, s_part);
        __syncthreads();
        if (warp == 0) {
            // ---- 3. publish the products and the next column, arrive, wait
            double2* out = o.qa + (size_t)((k + 1) & 1) * n;
            for (int r = lane; r < R; r += 32) {
                const int i = g + (rf + r) * G;
                const double* row = r >= rg ? rows + (size_t)(rf + r - rs0) * ldn : o.F + (size_t)i * n;
                __stcg(out + i, make_double2(os_row_sum(s_part[r], r < rg ? nsg : nss), row[k + 1]));
            }
            __syncwarp();
            target += (unsigned)min(G, n - 1 - k);
            if (lane == 0) {
                int ok = 1;
                if (G > 1) {
                    sk_atom_add_release(o.ctr, 1u);
                    unsigned polls = 0;
                    while (sk_ld_acquire(o.ctr) < target) {
                        ++polls;
                        if (polls > o.cap || ((polls & 255u) == 0 && *(volatile int*)o.status != 0)) {
                            ok = 0;
                            break;
                        }
                        if (polls > 256) __nanosleep(64);
                    }
                    if (!ok) sk_set_error(o.status, SKEW_ERR_DEVICE_TIMEOUT);
                }
                s_ok = ok;
            }
        } else if (warp >= 4) {
            // ---- meanwhile: the norm of x below its first element, beta and
            // sigma (H = I - sigma u u^T, sigma = 2 / |u|^2 = -1 / (beta u_0))
            double nr = 0.0;
            for (int j = k + 2 + (t - 128); j < n; j += 128) nr = fma(x[j], x[j], nr);
            nr = sk_warp_sum(nr);
            if (lane == 0) s_red[warp - 4] = nr;
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (warp == 4 && lane == 0) {
                const double s2 = (s_red[0] + s_red[1]) + (s_red[2] + s_red[3]);
                const double x0 = x[k + 1];
                double b = x0, sg = 0.0, inv = 0.0;
                if (os_tail(s2)) {
                    const double rr = sqrt(fma(x0, x0, s2));
                    b = (x0 >= 0.0) ? -rr : rr;
                    sg = -1.0 / (b * (x0 - b));
                    inv = -sg * b;
                }
                s_sc[0] = b;
                s_sc[1] = sg;
                s_sc[2] = inv;
                s_sc[3] = x0 - b;
            }
        }
        __syncthreads();
        if (!s_ok) return;
        beta = s_sc[0];
        sigma = s_sc[1];
        // ---- the reflector out, scaled to a unit leading element
        {
            const double inv = s_sc[2], u0 = s_sc[3];
            for (int r = t; r < R; r += OT) {
                const int i = g + (rf + r) * G;
                o.V[(size_t)k * n + i] = (i == k + 1) ? 1.0 : x[i] * inv;
            }
            if (ilast == n - 1 && t == 0) {
                o.tau[k] = sigma * u0 * u0;
                o.alpha[k] = -beta;
            }
            if (t == 0) x[k + 1] = u0;  // x_0 itself is not read above
            double* sw = u;
            u = x;
            x = sw;
        }
        __syncthreads();
    }
    // the CTA of the last row has written every entry
    const double s = os_scale(__ldcg(o.amax));
    if (s != 1.0) {
        __syncthreads();
        for (int j = t; j < n - 1; j += OT) o.alpha[j] /= s;
    }
}

// Full skew matrix by rows from the strict lower triangle of A (column-major):
// F[i * n + j] = A(i, j) below the diagonal, -A(j, i) above.  32 x 32 tiles
// through shared memory, both sides coalesced.  amax: max |A| (os_scale).
__global__ void __launch_bounds__(256)
os_full_kernel(int n, const double* __restrict__ A, int lda, double* __restrict__ F, unsigned long long* amax, int check,
               int* status) {
    __shared__ double tile[32][33];
    const int bi = blockIdx.x * 32, bj = blockIdx.y * 32;
    if (bi < bj) return;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    bool bad = false;
    unsigned long long m = 0;
    for (int jj = ty; jj < 32; jj += 8) {
        const int i = bi + tx, j = bj + jj;
        double v = 0.0;
        if (i < n && j < n && i > j) {
            v = A[(size_t)j * lda + i];
            if (check && !isfinite(v)) bad = true;
            const unsigned long long b = os_abs_bits(v);
            m = b > m ? b : m;
        }
        tile[jj][tx] = v;
        // F(j, i) = -A(i, j); the diagonal and the part above it of a diagonal tile come below
        if (i < n && j < n && i > j) F[(size_t)j * n + i] = -v;
        if (i < n && i == j) F[(size_t)j * n + i] = 0.0;
    }
    __syncthreads();
    for (int ii = ty; ii < 32; ii += 8) {
        const int i = bi + ii, j = bj + tx;
        if (i < n && j < n && i > j) F[(size_t)i * n + j] = tile[tx][ii];
    }
    m = os_warp_max(m);
    if (tx == 0 && m > *(volatile unsigned long long*)amax) atomicMax(amax, m);
    if (bad) sk_set_error(status, SKEW_ERR_NONFINITE);
}

__global__ void __launch_bounds__(160)
os_gram_kernel(int n, const double* __restrict__ V, int ldv, double* __restrict__ part) {
    const int p = blockIdx.x, s = blockIdx.y, P = gridDim.x;
    const int lo = p * PB + 1 + s * GR;
    if (lo >= n) return;
    os_gram_body(V + (size_t)p * PB * ldv, ldv, lo, min(n, lo + GR), part + ((size_t)s * P + p) * PB * PB);
}

__global__ void __launch_bounds__(256)
os_gram_sum_kernel(int n, const double* __restrict__ part, const double* __restrict__ tau, double* __restrict__ Gt,
                   int scaled) {
    const int p = blockIdx.x, P = gridDim.x;
    const int m = n - (p * PB + 1), S = (m + GR - 1) / GR;
    os_gram_sum_body(part + (size_t)p * PB * PB, (size_t)P * PB * PB, S, tau + p * PB, Gt + (size_t)p * PB * PB, scaled,
                     blockIdx.y * 256 + threadIdx.x, gridDim.y * 256);
}

template <int E>
__global__ void __launch_bounds__(WT, 1)
os_wy_kernel(int n, int nev, const double* __restrict__ V, const double* __restrict__ Gt,
             const double* __restrict__ tau, const double* __restrict__ Qi, double* __restrict__ Zre,
             double* __restrict__ Zim, int ldz) {
    extern __shared__ __align__(16) double wy_sm[];
    os_wy_body<E>(n, nev, blockIdx.x * E, V, Gt, tau, Qi, Zre, Zim, ldz, wy_sm);
}

template <int E>
cudaError_t wy_launch(cudaStream_t st, int n, int nev, const double* V, const double* Gt, const double* tau,
                      const double* Qi, double* Zre, double* Zim, int ldz) {
    const size_t dyn = wy_smem(n, E);
    if (const cudaError_t e = cudaFuncSetAttribute(os_wy_kernel<E>, cudaFuncAttributeMaxDynamicSharedMemorySize, WY_SMEM))
        return e;
    os_wy_kernel<E><<<(nev + E - 1) / E, WT, dyn, st>>>(n, nev, V, Gt, tau, Qi, Zre, Zim, ldz);
    count_launch();
    return cudaGetLastError();
}

int os_srows(int n, int G) {
    const int rmax = (n + G - 1) / G;
    const size_t vec = 3 * sizeof(double) * (size_t)(n | 1), row = sizeof(double) * (size_t)(n | 1);
    const size_t cap = OS_SMEM;
    const int fit = vec + row > cap ? 0 : (int)((cap - vec) / row);
    return std::min(rmax, fit);
}

}  // namespace

size_t onestep_ws(int n) {
    Carve cv(nullptr, ~size_t(0));
    cv.take<double2>(2 * (size_t)(n > 0 ? n : 1));
    cv.take<unsigned>(16);
    return cv.off + 256;
}

int onestep_vcols(int n) { return n > 2 ? (n - 2 + 63) / 64 * 64 : 64; }

namespace {
// [0] arrivals, [2..3] max |A|
unsigned* carve_os(Carve& cv, int n, double2** qa) {
    *qa = cv.take<double2>(2 * (size_t)n);
    return cv.take<unsigned>(16);
}
}  // namespace

int onestep_full(cudaStream_t st, int n, const double* A, int lda, double* F, int check, void* ws, size_t ws_bytes,
                 int* status) {
    Carve cv(ws, ws_bytes);
    double2* qa;
    unsigned* ctr = carve_os(cv, n, &qa);
    if (!cv.ok) return SKEW_ERR_WORKSPACE;
    if (const cudaError_t e = cudaMemsetAsync(ctr, 0, 16 * sizeof(unsigned), st)) return cuda_fail(e);
    const int nb = (n + 31) / 32;
    os_full_kernel<<<dim3(nb, nb), 256, 0, st>>>(n, A, lda, F, reinterpret_cast<unsigned long long*>(ctr + 2), check,
                                                 status);
    count_launch();
    return cuda_ok(cudaGetLastError());
}

int onestep_reduce(cudaStream_t st, int n, double* F, double* V, double* tau, double* alpha, void* ws,
                   size_t ws_bytes, int* d_status, unsigned spin_cap) {
    if (n < 2) return 0;
    Carve cv(ws, ws_bytes);
    OsArgs o{};
    o.ctr = carve_os(cv, n, &o.qa);
    if (!cv.ok) return SKEW_ERR_WORKSPACE;
    o.amax = reinterpret_cast<const unsigned long long*>(o.ctr + 2);
    const size_t vc = (size_t)onestep_vcols(n);
    if (const cudaError_t e = cudaMemsetAsync(V, 0, sizeof(double) * vc * n, st)) return cuda_fail(e);
    if (const cudaError_t e = cudaMemsetAsync(tau, 0, sizeof(double) * vc, st)) return cuda_fail(e);
    // two rows per CTA and more
    const int G = std::min(device_sms(), (n + 1) / 2);
    if (n > OMAXR * G) return SKEW_ERR_UNSUPPORTED;
    o.n = n;
    o.F = F;
    o.V = V;
    o.tau = tau;
    o.alpha = alpha;
    o.status = d_status;
    o.cap = spin_cap ? spin_cap : SK_SPIN_CAP;
    o.srows = os_srows(n, G);
    const size_t dyn = sizeof(double) * (size_t)(n | 1) * (3 + (size_t)o.srows);
    if (const cudaError_t e =
            cudaFuncSetAttribute(onestep_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, OS_SMEM))
        return cuda_fail(e);
    void* args[] = {&o};
    KtScope kt(st, KT_PANEL_QR);
    const cudaError_t e = cudaLaunchCooperativeKernel((void*)onestep_kernel, dim3(G), dim3(OT), args, dyn, st);
    count_launch();
    if (e == cudaErrorCooperativeLaunchTooLarge) return SKEW_ERR_LAUNCH;
    return cuda_ok(e);
}

// Eigenvectors of one wave in shared memory: every CTA one slab.
static int wy_e(int n, int nev) {
    const int sms = device_sms();
    const int e = (nev + sms - 1) / sms;
    return (e <= 6 && wy_smem(n, e) <= (size_t)WY_SMEM) ? e : 0;
}

bool onestep_wy_fits(int n, int nev) { return wy_e(n, nev) > 0; }

size_t onestep_back_ws(int n) {
    const size_t P = (size_t)(onestep_vcols(n) / PB), S = (size_t)((n + GR - 1) / GR);
    Carve cv(nullptr, ~size_t(0));
    cv.take<double>(P * S * PB * PB);
    cv.take<double>(P * PB * PB);
    return cv.off + 256;
}

namespace {
// V^T V of every panel (os_gram_sum_kernel's two forms)
cudaError_t os_gram(cudaStream_t st, int n, const double* V, const double* tau, double* part, double* G, int scaled) {
    const int P = (n - 2 + PB - 1) / PB, S = (n - 1 + GR - 1) / GR;
    os_gram_kernel<<<dim3(P, S), 160, 0, st>>>(n, V, n, part);
    os_gram_sum_kernel<<<dim3(P, 4), 256, 0, st>>>(n, part, tau, G, scaled);
    count_launch(2);
    return cudaGetLastError();
}
}  // namespace

int onestep_back(cudaStream_t st, int n, int nev, const double* V, const double* tau, const double* Qi, double* Zre,
                 double* Zim, int ldz, void* ws, size_t ws_bytes) {
    const int E = wy_e(n, nev);
    if (E <= 0) return SKEW_ERR_UNSUPPORTED;
    const size_t P = (size_t)(onestep_vcols(n) / PB), S = (size_t)((n + GR - 1) / GR);
    Carve cv(ws, ws_bytes);
    double* part = cv.take<double>(P * S * PB * PB);
    double* Gt = cv.take<double>(P * PB * PB);
    if (!cv.ok) return SKEW_ERR_WORKSPACE;
    KtScope kt(st, KT_GEMM_F64);
    if (n > 2) {
        if (const cudaError_t e = os_gram(st, n, V, tau, part, Gt, 1)) return cuda_fail(e);
    }
    cudaError_t e;
    switch (E) {
    case 1: e = wy_launch<1>(st, n, nev, V, Gt, tau, Qi, Zre, Zim, ldz); break;
    case 2: e = wy_launch<2>(st, n, nev, V, Gt, tau, Qi, Zre, Zim, ldz); break;
    case 3: e = wy_launch<3>(st, n, nev, V, Gt, tau, Qi, Zre, Zim, ldz); break;
    case 4: e = wy_launch<4>(st, n, nev, V, Gt, tau, Qi, Zre, Zim, ldz); break;
    case 5: e = wy_launch<5>(st, n, nev, V, Gt, tau, Qi, Zre, Zim, ldz); break;
    default: e = wy_launch<6>(st, n, nev, V, Gt, tau, Qi, Zre, Zim, ldz); break;
    }
    return cuda_ok(e);
}

int onestep_tfactors(cudaStream_t st, int n, const double* V, const double* tau, double* Tfac, void* ws,
                     size_t ws_bytes) {
    if (n < 3) return 0;
    const size_t P = (size_t)(onestep_vcols(n) / PB), S = (size_t)((n + GR - 1) / GR);
    Carve cv(ws, ws_bytes);
    double* part = cv.take<double>(P * S * PB * PB);
    double* G = cv.take<double>(P * PB * PB);
    if (!cv.ok) return SKEW_ERR_WORKSPACE;
    KtScope kt(st, KT_GEMM_F64);
    if (const cudaError_t e = os_gram(st, n, V, tau, part, G, 0)) return cuda_fail(e);
    return cuda_ok(tfactor_panels(st, (int)P, tau, G, Tfac));
}

}  // namespace sk
