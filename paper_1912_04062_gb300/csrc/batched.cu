// batched.cu -- many independent skew eigenproblems of small and medium order
// (the paper solves one matrix per run; this is the batched form of the
// one-step route for orders up to BATCH_MAX = 1024).
//
// The batch goes through the route stage by stage, each stage one launch over
// all matrices (work tables built once per plan), so every stage spreads over
// the whole GPU whatever the sizes are:
//   1. reduction (Householder, A <- A + v p^T - p v^T with p = tau A v, Eqs. 2-6
//      with u1 = -u2), the only stage with a chain per matrix.  Orders above
//      BATCH_ONE_CTA: one thread-block cluster a matrix (cluster_reduce_kernel),
//      its CTAs own interleaved rows and exchange one vector a column through
//      distributed shared memory; clusters take matrices from a work counter,
//      largest first.  Smaller ones: one CTA a matrix (bt_persistent_kernel:
//      ctas_per_sm CTAs per SM, orders up to smem_max_n in shared memory; the
//      tunables of skew_batched_config).
//   2. eigenvalues: FP32 brackets and FP64 multisection on the zero-diagonal
//      form (Sec. 3), a few lanes an eigenvalue;
//   3. vectors of S by twisted factorisations, clusters by Gram-Schmidt or
//      inverse iteration;
//   4. the D map (Algorithm 1 step 3) and the reflectors in 64-wide compact WY
//      panels (Eq. 7), a few vectors a CTA.
// One CTA a matrix for the whole route (before) left a batch waiting for its
// largest matrices: 96 matrices of order 32 .. 1024 took 1388 ms.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "internal.h"
#include "onestep_dev.cuh"
#include "tridiag_dev.cuh"

namespace sk {

using namespace onestep;

namespace {

constexpr int BT = 256;  // threads per CTA of the per-matrix kernels

constexpr int BL = 4;    // lanes an eigenvalue of the multisections
constexpr int BE = 4;    // eigenvectors a CTA of the back-transformation

struct BItem {
    int n, nev, lda, vectors;
    double* S;                   // working matrix (n x n) where it does not fit in shared memory
    const double* A;
    double *lambda, *Zre, *Zim;  // Z: n x nev, leading dimension n
    int* info;                   // caller's status word of this matrix (may be null)
    // per-matrix scratch
    double *V, *tau, *alpha, *Qi;  // V: n x onestep_vcols(n), tau as many
    double* as;                    // alpha scaled (tri_prep)
    double *a2e, *b2e;  // the bidiagonal of the zero-diagonal form, scaled and squared (ceil(n/2) each)
    float* a2s;         // alpha^2 / g^2
    double* lohi;       // brackets, then the flags of the vectors' residual tests
    tri::TriScalars* sc;
    tri::InvitBufs bf;
    int* fail;
    double *gpart, *G;  // Gram partials and matrices of the panels
};

// One unit of a stage's work: a matrix and a place in it.
struct BUnit {
    int item, at;
};

__device__ double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();  // red may still be read from a previous call
    if (l == 0) red[w] = v;
    __syncthreads();
    double s = 0.0;
    for (int k = 0; k < BT / 32; k++) s += red[k];
    return s;
}

__host__ __device__ inline int bt_vcols(int n) { return n > 2 ? (n - 2 + PB - 1) / PB * PB : PB; }

// Tridiagonalisation of one matrix by the whole CTA.  S: the working matrix
// (shared memory, ld n + 1, or the matrix's global copy, ld n); v, p: n
// doubles of shared memory; red: 32 doubles of shared memory.
__device__ void bt_reduce_body(const BItem& it, double* S, int ld, double* v, double* p, double* red) {
    const int n = it.n, t = threadIdx.x;
    // S(i, j) = A(i, j) below the diagonal, -A(j, i) above: only the strict
    // lower triangle of A is read
    for (int e = t; e < n * n; e += BT) {
        const int i = e % n, j = e / n;
        double x = 0.0;
        if (i > j) x = it.A[i + (size_t)j * it.lda];
        else if (i < j) x = -it.A[j + (size_t)i * it.lda];
        S[i + (size_t)j * ld] = x;
    }
    __syncthreads();
    for (int c = 0; c + 2 < n; c++) {
        double a = 0.0;
        for (int i = c + 2 + t; i < n; i += BT) a = fma(S[i + (size_t)c * ld], S[i + (size_t)c * ld], a);
        a = block_sum(a, red);
        const double x0 = S[(c + 1) + (size_t)c * ld];
        double tau, beta, sc;
        if (a == 0.0) {
            tau = 0.0;
            beta = x0;
            sc = 0.0;
        } else {
            const double rr = sqrt(x0 * x0 + a);
            beta = (x0 >= 0.0) ? -rr : rr;
            tau = (beta - x0) / beta;
            sc = 1.0 / (x0 - beta);
        }
        for (int i = t; i < n; i += BT) {
            const double vi = i <= c ? 0.0 : (i == c + 1) ? 1.0 : S[i + (size_t)c * ld] * sc;
            v[i] = vi;
            it.V[i + (size_t)c * n] = vi;
        }
        if (t == 0) {
            it.tau[c] = tau;
            it.alpha[c] = -beta;  // T[c, c+1] = -T[c+1, c]
        }
        __syncthreads();
        if (tau != 0.0) {
            // p = tau S22 v, S22 = S[c+1:, c+1:]
            for (int i = c + 1 + t; i < n; i += BT) {
                double s2 = 0.0;
                for (int j = c + 1; j < n; j++) s2 = fma(S[i + (size_t)j * ld], v[j], s2);
                p[i] = tau * s2;
            }
            __syncthreads();
            // S22 += v p^T - p v^T: each product is rounded on its own, so the
            // update of (j, i) is exactly minus that of (i, j); the strict lower
            // triangle is computed and its negation stored above (the diagonal
            // stays 0), which keeps S exactly skew with half the FP64 work of
            // updating the whole square, and the same values
            const int m = n - c - 1;
            for (int e = t; e < m * m; e += BT) {
                const int i = c + 1 + e % m, j = c + 1 + e / m;
                if (i > j) {
                    const double x =
                        S[i + (size_t)j * ld] + __dsub_rn(__dmul_rn(v[i], p[j]), __dmul_rn(p[i], v[j]));
                    S[i + (size_t)j * ld] = x;
                    S[j + (size_t)i * ld] = -x;
                }
            }
        }
        __syncthreads();
    }
    if (t == 0 && n >= 2) it.alpha[n - 2] = S[(n - 2) + (size_t)(n - 1) * ld];
    __syncthreads();
    // the columns that fill up the last panel
    const int vc = bt_vcols(n), c0 = n > 2 ? n - 2 : 0;
    for (int e = t; e < (vc - c0) * n; e += BT) it.V[(size_t)c0 * n + e] = 0.0;
    for (int c = c0 + t; c < vc; c += BT) it.tau[c] = 0.0;
    __syncthreads();
}

// Reduction of the small orders: CTAs take matrices from *next over order[]
// (largest first) until the list is exhausted.  MINB = CTAs per SM the
// registers are budgeted for.
template <int MINB>
__global__ void __launch_bounds__(BT, MINB)
bt_persistent_kernel(const BItem* __restrict__ items, const int* __restrict__ order, int count,
                     int* __restrict__ next, int smem_n) {
    extern __shared__ double bsm[];
    __shared__ int s_q;
    const int t = threadIdx.x;
    for (;;) {
        __syncthreads();  // the previous matrix is finished with shared memory and s_q
        if (t == 0) s_q = atomicAdd(next, 1);
        __syncthreads();
        const int q = s_q;
        if (q >= count) break;
        const BItem it = items[order[q]];
        const int n = it.n;
        if (n <= smem_n) {
            double* S = bsm;
            double* v = S + (size_t)n * (n + 1);
            bt_reduce_body(it, S, n + 1, v, v + n, v + 2 * n);
        } else {
            bt_reduce_body(it, it.S, n, bsm, bsm + n, bsm + 2 * n);
        }
    }
}

// ---- reduction of the larger orders: one cluster a matrix --------------------
// The column step of onestep_kernel (onestep.cu) with the cluster in place of
// the grid: the CTAs' (q, a) pairs go straight into every CTA's shared memory
// and one hardware cluster barrier a column orders them (about 300 clocks,
// against 3000 for an exchange through L2).  The norm of the column, its square
// root and division (2500 clocks) are then the longest chain at small orders,
// so four warps form them while eight apply the update.
constexpr int CT = 384;     // 8 warps of the pass, 4 of the norm
constexpr int CMAXR = 114;  // rows of one CTA at most (order 1024 in a cluster of 9)
constexpr int CSMEM = 210 * 1024;

SK_DEV uint32_t cl_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
SK_DEV uint32_t cl_size() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
SK_DEV void cl_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address of this CTA's shared p in CTA `rank` of the cluster.
SK_DEV uint32_t cl_map(const void* p, uint32_t rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}

// Shared memory of a CTA for order n in a cluster of G: u, p, x, the exchange
// buffers, then as many own rows as fit.
__host__ __device__ inline int cl_ld(int n) { return (n + 2) & ~1; }
__host__ __device__ inline int cl_rows(int n, int G) {
    const int rmax = (n + G - 1) / G, ld = cl_ld(n);
    const int fit = (CSMEM / 8 - 7 * ld) / ld;
    return fit < rmax ? fit : rmax;
}

// One matrix by the cluster.  S: its rows that do not fit in shared memory.
// check: values that are not finite are reported in *status.
SK_DEV void cluster_reduce_body(int n, const double* __restrict__ A, int lda, double* S, double* V, double* tau,
                                double* alpha, int check, int* status) {
    extern __shared__ __align__(16) double cl_sm[];
    __shared__ double s_part[CMAXR][OCW];
    __shared__ double2 s_coef[CMAXR];  // sigma u_i, -sigma p_i of the own rows
    __shared__ double s_red[4];
    __shared__ double s_sc[4];
    __shared__ unsigned long long s_amax[16];  // max |A| over each CTA's rows
    __shared__ unsigned long long s_wmax[CT / 32];
    const int G = (int)cl_size(), g = (int)cl_rank();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int ldn = cl_ld(n);
    double* u = cl_sm;
    double* p = u + ldn;
    double* x = p + ldn;
    double2* qa = reinterpret_cast<double2*>(x + ldn);  // 2 n, double-buffered
    double* rows = x + 5 * ldn;
    const int srows = cl_rows(n, G);
    const int Rt = g < n ? (n - 1 - g) / G + 1 : 0;  // own rows: none past a small order
    const int rs0 = Rt > srows ? Rt - srows : 0, ilast = g + (Rt - 1) * G;
    // own rows of the full skew matrix: -A(j, i) right of the diagonal
    // (contiguous), A(i, j) left of it
    unsigned long long am = 0;
    for (int r = 0; r < Rt; r++) {
        const int i = g + r * G;
        double* row = r >= rs0 ? rows + (size_t)(r - rs0) * ldn : S + (size_t)i * n;
        for (int j = t; j < n; j += CT) {
            const double v = j > i ? -A[(size_t)i * lda + j] : j < i ? A[(size_t)j * lda + i] : 0.0;
            if (check && !isfinite(v)) sk_set_error(status, SKEW_ERR_NONFINITE);
            row[j] = v;
            const unsigned long long b = os_abs_bits(v);
            am = b > am ? b : am;
        }
    }
    am = os_warp_max(am);
    if (lane == 0) s_wmax[warp] = am;
    __syncthreads();
    if (warp == 0) {
        am = os_warp_max(lane < CT / 32 ? s_wmax[lane] : 0ull);
        if (lane < G)
            asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(cl_map(s_amax + g, (uint32_t)lane)), "l"(am)
                         : "memory");
    }
    // zeros of V above the reflectors and in the columns that fill up the
    // last panel (the values come after the first barrier below)
    const int vc = bt_vcols(n);
    for (int c = g; c < vc; c += G) {
        const int hi = c < n - 2 ? c + 1 : n;
        for (int i = t; i < hi; i += CT) V[(size_t)c * n + i] = 0.0;
    }
    if (g == 0)
        for (int c = n - 2 + t; c < vc; c += CT) tau[c] = 0.0;
    cl_barrier();
    am = 0;
    for (int c = 0; c < G; c++) am = s_amax[c] > am ? s_amax[c] : am;
    const double scale = os_scale(am);
    if (scale != 1.0) {
        for (int r = 0; r < Rt; r++) {
            double* row = r >= rs0 ? rows + (size_t)(r - rs0) * ldn : S + (size_t)(g + r * G) * n;
            for (int j = t; j < n; j += CT) row[j] *= scale;
        }
    }
    double beta = 0.0, sigma = 0.0;
    for (int k = 0; k + 1 < n; k++) {
        const bool act = ilast > k;  // rows left
        const int rf = (k + 1 > g) ? (k + 1 - g + G - 1) / G : 0, R = Rt - rf;
        if (act) {
            const double2* in = qa + (size_t)(k & 1) * n;
            if (k == 0) {
                for (int j = t; j < n; j += CT) {
                    x[j] = j > 0 ? scale * A[j] : 0.0;
                    u[j] = 0.0;
                    p[j] = 0.0;
                }
            } else {
                const double2 qk = in[k];
                const double uk = -sigma * u[k], pk = sigma * fma(-beta, qk.y, qk.x);
                for (int j = k + 1 + t; j < n; j += CT) {
                    const double2 e = in[j];
                    const double pj = fma(-beta, e.y, e.x);
                    p[j] = pj;
                    x[j] = fma(u[j], pk, fma(pj, uk, e.y));
                }
            }
        }
        __syncthreads();
        if (k == n - 2) {
            if (act && t == 0) alpha[k] = -x[n - 1];
            break;
        }
        const int rg = max(rs0, rf) - rf;  // rows of global memory
        // a function of the order left alone: a matrix's result does not
        // depend on the size of the cluster
        const int m = n - k - 1, nseg = m >= 288 ? 1 : m >= 144 ? 2 : m >= 72 ? 4 : 8;
        if (act && warp < OCW) {
            for (int r = t; r < R; r += 256)
                s_coef[r] = make_double2(sigma * u[g + (rf + r) * G], -sigma * p[g + (rf + r) * G]);
            asm volatile("bar.sync 1, 256;" ::: "memory");
            os_pass<4>(nseg, nseg, R, rg, S + (size_t)(g + rf * G) * n, rows + (size_t)(rf + rg - rs0) * ldn, n, ldn,
                       g + rf * G, G, k, s_coef, u, p, x, warp, lane, s_part);
            asm volatile("bar.sync 1, 256;" ::: "memory");
            // publish (q_i, a_i) of the own rows to every CTA
            double2* out = qa + (size_t)((k + 1) & 1) * n;
            for (int r = t; r < R; r += 256) {
                const int i = g + (rf + r) * G;
                const double* row = r >= rg ? rows + (size_t)(rf + r - rs0) * ldn : S + (size_t)i * n;
                const double sum = os_row_sum(s_part[r], nseg);
                const double av = row[k + 1];
                for (int c = 0; c < G; c++)
                    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(cl_map(out + i, (uint32_t)c)),
                                 "d"(sum), "d"(av)
                                 : "memory");
            }
        } else if (act) {
            // the norm of x below its first element, beta and sigma
            double nr = 0.0;
            for (int j = k + 2 + (t - 256); j < n; j += 128) nr = fma(x[j], x[j], nr);
            nr = sk_warp_sum(nr);
            if (lane == 0) s_red[warp - OCW] = nr;
            asm volatile("bar.sync 2, 128;" ::: "memory");
            if (t == 256) {
                const double s2 = (s_red[0] + s_red[1]) + (s_red[2] + s_red[3]);
                const double x0 = x[k + 1];
                double b = x0, sg = 0.0, inv = 0.0;
                if (os_tail(s2)) {
                    const double rr = sqrt(fma(x0, x0, s2));
                    b = (x0 >= 0.0) ? -rr : rr;
                    // this chain is the longest of a column at small orders
                    const double den = b * (x0 - b);
                    sg = den > -1e270 && den < -1e-270 ? -tri::rcp_fast(den) : -1.0 / den;
                    inv = -sg * b;
                }
                s_sc[0] = b;
                s_sc[1] = sg;
                s_sc[2] = inv;
                s_sc[3] = x0 - b;
            }
        }
        cl_barrier();
        if (act) {
            beta = s_sc[0];
            sigma = s_sc[1];
            const double inv = s_sc[2], u0 = s_sc[3];
            for (int r = t; r < R; r += CT) {
                const int i = g + (rf + r) * G;
                V[(size_t)k * n + i] = (i == k + 1) ? 1.0 : x[i] * inv;
            }
            if (ilast == n - 1 && t == 0) {
                tau[k] = sigma * u0 * u0;
                alpha[k] = -beta;
            }
            if (t == 0) x[k + 1] = u0;  // x_0 itself is not read above
            double* sw = u;
            u = x;
            x = sw;
        }
        __syncthreads();
    }
    if (scale != 1.0 && ilast == n - 1) {  // this CTA has written every entry
        __syncthreads();
        for (int j = t; j < n - 1; j += CT) alpha[j] /= scale;
    }
}

__global__ void __launch_bounds__(CT, 1)
cluster_reduce_kernel(const BItem* __restrict__ items, const int* __restrict__ order, int count,
                      int* __restrict__ next) {
    __shared__ int s_q;
    for (;;) {
        cl_barrier();  // nobody writes into this CTA's shared memory any more
        if (cl_rank() == 0 && threadIdx.x == 0) {
            const int q = atomicAdd(next, 1);
            for (uint32_t c = 0; c < cl_size(); c++)
                asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(cl_map(&s_q, c)), "r"(q) : "memory");
        }
        cl_barrier();
        const int q = s_q;
        if (q >= count) return;
        const BItem it = items[order[q]];
        cluster_reduce_body(it.n, it.A, it.lda, it.S, it.V, it.tau, it.alpha, 0, nullptr);
    }
}

// One matrix, one cluster.
__global__ void __launch_bounds__(CT, 1)
cluster_reduce_one_kernel(int n, const double* __restrict__ A, int lda, double* V, double* tau, double* alpha,
                          int check, int* status) {
    cl_barrier();  // every CTA of the cluster has started
    cluster_reduce_body(n, A, lda, nullptr, V, tau, alpha, check, status);
    cl_barrier();  // no CTA leaves while another may still write to it
}

// ---- eigenvalues and vectors of every tridiagonal ----------------------------
// ||S||_1, the power-of-two scaling and the scaled forms (tri_prep_kernel's)
__global__ void __launch_bounds__(BT) bt_prep_kernel(const BItem* __restrict__ items, int* __restrict__ nclu) {
    const BItem it = items[blockIdx.x];
    const int n = it.n, t = threadIdx.x;
    __shared__ double red[BT / 32];
    double gm = 0.0, am = 0.0;
    for (int i = t; i < n; i += BT) {
        const double al = (i < n - 1) ? it.alpha[i] : 0.0, ap = (i > 0) ? it.alpha[i - 1] : 0.0;
        gm = fmax(gm, fabs(al) + fabs(ap));
        am = fmax(am, fabs(al));
    }
    for (int o = 16; o > 0; o >>= 1) {
        gm = fmax(gm, __shfl_xor_sync(0xffffffffu, gm, o));
        am = fmax(am, __shfl_xor_sync(0xffffffffu, am, o));
    }
    if ((t & 31) == 0) red[t >> 5] = gm;
    __syncthreads();
    double g = 0.0;
    for (int w = 0; w < BT / 32; w++) g = fmax(g, red[w]);
    __syncthreads();
    if ((t & 31) == 0) red[t >> 5] = am;
    __syncthreads();
    double a = 0.0;
    for (int w = 0; w < BT / 32; w++) a = fmax(a, red[w]);
    const double down = tri::pow2_down(g), ig = g > 0.0 ? 1.0 / g : 0.0;
    if (t == 0) {
        it.sc->g = g;
        it.sc->pivmin = DBL_MIN * fmax(1.0, a * a);
        it.sc->down = down;
        it.sc->up = 1.0 / down;
        *it.fail = 0x7fffffff;
        if (blockIdx.x == 0) *nclu = 0;
    }
    for (int i = t; i < n - 1; i += BT) {
        const double al = it.alpha[i], s = al * ig;
        it.as[i] = al * down;
        it.a2s[i] = (float)(s * s);
    }
    for (int i = t; i < (n + 1) / 2; i += BT) {
        const double x = (2 * i <= n - 2) ? it.alpha[2 * i] * down : 0.0;
        const double y = (2 * i + 1 <= n - 2) ? it.alpha[2 * i + 1] * down : 0.0;
        it.a2e[i] = x * x;
        it.b2e[i] = y * y;
    }
}

// One warp a unit: 32 / BL eigenvalues.  Four lanes an eigenvalue: a batch
// keeps the FP64 pipes busy, and fewer lanes spend fewer counts (15 steps of 4
// against 7 of 32).
__global__ void __launch_bounds__(64) bt_bisect_kernel(const BItem* __restrict__ items,
                                                       const BUnit* __restrict__ units, int count) {
    const int w = blockIdx.x * 2 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (w >= count) return;
    const BUnit b = units[w];
    const BItem it = items[b.item];
    const int k = b.at + lane / BL, q = lane % BL;
    if (k >= it.nev) return;  // whole lane groups leave together
    tri::bisect32_body<BL>(it.n, k, q, lane, it.a2s, it.lohi);
    __syncwarp(tri::lane_group<BL>(lane));
    tri::bisect_bd_body<BL>(it.n, k, q, lane, it.sc, it.lohi, it.lambda, it.a2e, it.b2e);
}

__device__ __forceinline__ double bt_ctol(int n) { return fmin(1e-3, 10.0 / ((double)n * sqrt((double)n))); }

__global__ void __launch_bounds__(32) bt_twist_kernel(const BItem* __restrict__ items,
                                                      const BUnit* __restrict__ units, int maxit) {
    const BUnit b = units[blockIdx.x];
    const BItem it = items[b.item];
    tri::twist_body(it.n, it.nev, b.at, threadIdx.x, it.as, it.alpha, it.lambda, it.sc, bt_ctol(it.n), maxit, 1, it.bf,
                    it.Qi, it.lohi, it.fail);
}

// Clusters of every matrix: (matrix, first eigenvalue, size).
__global__ void __launch_bounds__(128) bt_clu_list_kernel(const BItem* __restrict__ items, int3* __restrict__ list,
                                                          int* __restrict__ nclu) {
    const BItem it = items[blockIdx.x];
    if (!it.vectors) return;
    const double ctol = bt_ctol(it.n) * it.sc->g;
    for (int k = threadIdx.x; k + 1 < it.nev; k += 128) {
        if (!tri::starts_cluster(it.lambda, k, ctol) || tri::starts_cluster(it.lambda, k + 1, ctol)) continue;
        int k1 = k + 2;
        while (k1 < it.nev && !tri::starts_cluster(it.lambda, k1, ctol)) k1++;
        list[atomicAdd(nclu, 1)] = make_int3(blockIdx.x, k, k1 - k);
    }
}

__global__ void __launch_bounds__(tri::CLU_T) bt_clu_kernel(const BItem* __restrict__ items,
                                                            const int3* __restrict__ list,
                                                            const int* __restrict__ nclu, int maxit) {
    const int nc = *nclu;
    for (int b = blockIdx.x; b < nc; b += gridDim.x) {
        __syncthreads();  // the previous cluster is done with shared memory
        const BItem it = items[list[b].x];
        tri::clu_body(it.n, it.nev, list[b].y, list[b].z, it.alpha, it.lambda, it.sc->g, maxit, it.bf, it.Qi, it.lohi,
                      it.fail);
    }
}

// ---- back-transformation -------------------------------------------------------
__global__ void __launch_bounds__(160) bt_gram_kernel(const BItem* __restrict__ items,
                                                      const BUnit* __restrict__ units) {
    const BUnit b = units[blockIdx.x];
    const BItem it = items[b.item];
    const int p = b.at & 0xffff, s = b.at >> 16, P = bt_vcols(it.n) / PB;
    const int lo = p * PB + 1 + s * GR;
    os_gram_body(it.V + (size_t)p * PB * it.n, it.n, lo, min(it.n, lo + GR), it.gpart + ((size_t)s * P + p) * PB * PB);
}

__global__ void __launch_bounds__(256) bt_gram_sum_kernel(const BItem* __restrict__ items,
                                                          const BUnit* __restrict__ units) {
    const BUnit b = units[blockIdx.x];
    const BItem it = items[b.item];
    const int p = b.at, P = bt_vcols(it.n) / PB, m = it.n - (p * PB + 1);
    os_gram_sum_body(it.gpart + (size_t)p * PB * PB, (size_t)P * PB * PB, (m + GR - 1) / GR, it.tau + p * PB,
                     it.G + (size_t)p * PB * PB, 1, blockIdx.y * 256 + threadIdx.x, gridDim.y * 256);
}

__global__ void __launch_bounds__(WT, 1) bt_wy_kernel(const BItem* __restrict__ items,
                                                      const BUnit* __restrict__ units) {
    extern __shared__ __align__(16) double wy_sm[];
    const BUnit b = units[blockIdx.x];
    const BItem it = items[b.item];
    os_wy_body<BE>(it.n, it.nev, b.at, it.V, it.G, it.tau, it.Qi, it.Zre, it.Zim, it.n, wy_sm);
}

__global__ void bt_status_kernel(const BItem* __restrict__ items, int count) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= count) return;
    const BItem it = items[b];
    if (it.info) *it.info = (it.vectors && *it.fail < it.nev) ? SKEW_INFO_INVIT_BASE + *it.fail : 0;
}

// The stages' work tables of a batch (units largest matrix first).
struct BTables {
    std::vector<BUnit> bisect, twist, gram, gsum, wy;
    std::vector<int> order;  // larger orders first: order[0 .. nlarge) take clusters
    int nlarge = 0, nvec = 0;
    long long cap_clu = 0;
};

BTables batch_tables(int count, const BatchProblem* pr) {
    BTables t;
    t.order.resize((size_t)count);
    for (int b = 0; b < count; b++) t.order[(size_t)b] = b;
    // longest processing time first: largest order first
    std::stable_sort(t.order.begin(), t.order.end(), [&](int x, int y) { return pr[x].n > pr[y].n; });
    for (int b : t.order) {
        const int n = pr[b].n, nev = pr[b].nev, P = bt_vcols(n) / PB;
        if (n > BATCH_ONE_CTA) t.nlarge++;
        for (int k = 0; k < nev; k += 32 / BL) t.bisect.push_back({b, k});
        if (!pr[b].Zre) continue;
        t.nvec++;
        t.cap_clu += nev / 2;
        for (int k = 0; k < nev; k += 16) t.twist.push_back({b, k});
        for (int k = 0; k < nev; k += BE) t.wy.push_back({b, k});
        if (n > 2)
            for (int p = 0; p < P; p++) {
                t.gsum.push_back({b, p});
                for (int s = 0; p * PB + 1 + s * GR < n; s++) t.gram.push_back({b, p | s << 16});
            }
    }
    return t;
}

struct BCarve {
    std::vector<BItem> items;
    BItem* d_items;
    int* d_order;
    BUnit *d_bisect, *d_twist, *d_gram, *d_gsum, *d_wy;
    int3* d_clu;
    int* d_cnt;  // two work counters and the cluster count
};

// Places every buffer of a batch (base == nullptr: sizing only).
size_t carve_small(Carve& cv, int count, const BatchProblem* pr, const BTables& tb, BCarve* out) {
    std::vector<BItem> items((size_t)count);
    BCarve c{};
    c.d_items = cv.take<BItem>((size_t)(count > 0 ? count : 1));
    c.d_order = cv.take<int>((size_t)(count > 0 ? count : 1));
    c.d_bisect = cv.take<BUnit>(tb.bisect.size() + 1);
    c.d_twist = cv.take<BUnit>(tb.twist.size() + 1);
    c.d_gram = cv.take<BUnit>(tb.gram.size() + 1);
    c.d_gsum = cv.take<BUnit>(tb.gsum.size() + 1);
    c.d_wy = cv.take<BUnit>(tb.wy.size() + 1);
    c.d_clu = cv.take<int3>((size_t)tb.cap_clu + 1);
    c.d_cnt = cv.take<int>(4);
    for (int b = 0; b < count; b++) {
        const BatchProblem& q = pr[b];
        BItem& it = items[(size_t)b];
        const size_t n = (size_t)q.n, ne = (size_t)(q.nev > 0 ? q.nev : 1), vc = (size_t)bt_vcols(q.n);
        it.n = q.n;
        it.nev = q.nev;
        it.lda = q.lda;
        it.vectors = q.Zre != nullptr;
        it.A = q.A;
        it.lambda = q.lambda;
        it.Zre = q.Zre;
        it.Zim = q.Zim;
        it.info = q.info;
        // global working copy: for the small orders used whenever the launch
        // keeps this order out of shared memory (a launch parameter, 0..160)
        it.S = cv.take<double>(n * n);
        it.V = cv.take<double>(n * vc);
        it.tau = cv.take<double>(vc);
        it.alpha = cv.take<double>(n);
        it.as = cv.take<double>(n);
        it.a2e = cv.take<double>(n / 2 + 1);
        it.b2e = cv.take<double>(n / 2 + 1);
        it.a2s = cv.take<float>(n);
        it.lohi = cv.take<double>(2 * ne);
        it.sc = cv.take<tri::TriScalars>(1);
        it.fail = cv.take<int>(1);
        if (it.vectors) {
            it.Qi = cv.take<double>(n * ne);
            it.bf.u0 = cv.take<double>(n * ne);
            it.bf.u1 = cv.take<double>(n * ne);
            it.bf.u2 = cv.take<double>(n * ne);
            it.bf.ml = cv.take<double>(n * ne);
            it.bf.sw = cv.take<unsigned char>(n * ne);
            const size_t P = vc / PB, S = (n + GR - 1) / GR;
            it.gpart = cv.take<double>(P * S * PB * PB);
            it.G = cv.take<double>(P * PB * PB);
        }
    }
    if (out) {
        *out = c;
        out->items = std::move(items);
    }
    return cv.off;
}

size_t smem_reduce(int n) { return sizeof(double) * ((size_t)n * (n + 1) + 2 * (size_t)n + 32); }

}  // namespace

size_t batched_small_ws(int count, const BatchProblem* pr) {
    Carve cv(nullptr, ~size_t(0));
    carve_small(cv, count, pr, batch_tables(count, pr), nullptr);
    return cv.off + 256;
}

namespace {

// Largest order kept in shared memory for a given shared-memory budget per CTA.
int smem_n_for(size_t budget) {
    int n = 2;
    while (n < BATCH_ONE_CTA && smem_reduce(n + 1) <= budget) n++;
    return n;
}

template <int MINB>
int prepare_persistent(int smem_n, int nmax, int count, BatchLaunch* out) {
    const size_t dyn_global = sizeof(double) * (2 * (size_t)nmax + 32);
    const size_t dyn = smem_n >= 2 ? std::max(smem_reduce(smem_n), dyn_global) : dyn_global;
    auto kern = bt_persistent_kernel<MINB>;
    // a constant: plans of other thresholds, in other threads too, launch the
    // same kernel with what they need
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_reduce(BATCH_ONE_CTA)) !=
        cudaSuccess)
        return SKEW_ERR_LAUNCH;
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, BT, dyn) != cudaSuccess || occ < 1)
        return SKEW_ERR_LAUNCH;
    const int per_sm = occ < MINB ? occ : MINB;
    int grid = per_sm * device_sms();
    if (grid > count) grid = count;
    out->ctas = MINB;
    out->grid = grid;
    out->dyn = dyn;
    out->smem_n = smem_n;
    return 0;
}

}  // namespace

skew_batched_config& batched_default_config() {
    static skew_batched_config c{2, 112, {0, 0}};
    return c;
}

int batched_config_check(const skew_batched_config& c) {
    if (c.ctas_per_sm < 1 || c.ctas_per_sm > 4) return -1;
    if (c.smem_max_n < 0 || c.smem_max_n > BATCH_SMALL_MAX) return -2;
    return 0;
}

namespace {

// Time of the larger orders (largest first) on `fit` clusters of G CTAs, in
// clocks: each matrix goes to the cluster that is free first, and takes 3500
// clocks a column and n^3 FMAs at 1.45 per clock and SM (both measured).
double cluster_span(const std::vector<int>& ns, int G, int fit) {
    std::vector<double> heap((size_t)fit, 0.0);
    const auto later = [](double x, double y) { return x > y; };
    double end = 0.0;
    for (int n : ns) {
        std::pop_heap(heap.begin(), heap.end(), later);
        heap.back() += 3500.0 * n + (double)n * n * n / (1.45 * G);
        end = std::max(end, heap.back());
        std::push_heap(heap.begin(), heap.end(), later);
    }
    return end;
}

// Cluster size of the larger orders' reduction.  Large clusters finish one
// matrix sooner but leave SMs of a GPC unused (measured on 152 SMs: 7 clusters
// of 16, 13 of 10, 15 of 9, 36 of 4 fit), so a few matrices take 16 and a
// long batch 9 or 4: whichever ends first by cluster_span.
int pick_clusters(const std::vector<int>& ns, BatchPlanDev* out) {
    out->cl_size = out->cl_count = 0;
    if (ns.empty()) return 0;
    auto kern = cluster_reduce_kernel;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, CSMEM) != cudaSuccess)
        return SKEW_ERR_LAUNCH;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) cudaGetLastError();
    double best = 0.0;
    for (int G : {16, 12, 10, 9, 8, 6, 5, 4}) {
        if (ns[0] > CMAXR * G) continue;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(G * device_sms()));
        cfg.blockDim = dim3(CT);
        cfg.dynamicSmemBytes = CSMEM;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = (unsigned)G;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        int fit = 0;
        if (cudaOccupancyMaxActiveClusters(&fit, kern, &cfg) != cudaSuccess || fit < 1) {
            cudaGetLastError();
            continue;
        }
        const double t = cluster_span(ns, G, fit);
        if (out->cl_size == 0 || t < best) {
            best = t;
            out->cl_size = G;
            out->cl_count = std::min(fit, (int)ns.size());
        }
    }
    return out->cl_size > 0 ? 0 : SKEW_ERR_LAUNCH;
}

}  // namespace

int cluster_reduce(cudaStream_t st, int n, const double* A, int lda, double* V, double* tau, double* alpha, int check,
                   int* d_status) {
    if (n < 2 || n > CLUSTER_ONE_MAX) return SKEW_ERR_UNSUPPORTED;
    auto kern = cluster_reduce_one_kernel;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, CSMEM) != cudaSuccess)
        return SKEW_ERR_LAUNCH;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) cudaGetLastError();
    KtScope kt(st, KT_PANEL_QR);
    for (int G = 16; G >= 8; G /= 2) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)G);
        cfg.blockDim = dim3(CT);
        cfg.dynamicSmemBytes = CSMEM;
        cfg.stream = st;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = (unsigned)G;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, n, A, lda, V, tau, alpha, check, d_status);
        if (e == cudaSuccess) {
            count_launch();
            return 0;
        }
        cudaGetLastError();
        if (G == 8) return cuda_fail(e);
    }
    return SKEW_ERR_LAUNCH;
}

// Launch parameters for a configuration (sets the kernels' attributes; no
// stream work).
int batched_prepare(const BatchPlanDev& d, const skew_batched_config& cfg, BatchLaunch* out) {
    if (batched_config_check(cfg)) return SKEW_ERR_UNSUPPORTED;
    const int dyn_wy = (int)wy_smem(BATCH_MAX, BE);  // a constant: plans of several threads share the kernel
    if (cudaFuncSetAttribute(bt_wy_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn_wy) != cudaSuccess)
        return SKEW_ERR_LAUNCH;
    // the shared-memory threshold: no more than the per-SM budget allows, nor than
    // the orders that this kernel gets
    int dev = 0, smem_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    const size_t budget = (size_t)smem_sm / (size_t)cfg.ctas_per_sm - 2048;
    const int small = d.count - d.nlarge, cnt = small > 0 ? small : 1;
    const int nmax = std::min(d.nmax, BATCH_ONE_CTA);
    int smem_n = small > 0 ? std::min(cfg.smem_max_n, nmax) : 0;
    if (smem_n >= 2) smem_n = std::min(smem_n, smem_n_for(budget));
    switch (cfg.ctas_per_sm) {
    case 1: return prepare_persistent<1>(smem_n, nmax, cnt, out);
    case 2: return prepare_persistent<2>(smem_n, nmax, cnt, out);
    case 3: return prepare_persistent<3>(smem_n, nmax, cnt, out);
    default: return prepare_persistent<4>(smem_n, nmax, cnt, out);
    }
}

// Stream work only: clear the work counters, launch the stages (capturable).
int batched_exec(cudaStream_t st, const BatchPlanDev& d, const BatchLaunch& L, int maxit) {
    if (d.count <= 0) return 0;
    if (const cudaError_t e = cudaMemsetAsync(d.cnt, 0, 2 * sizeof(int), st)) return cuda_fail(e);
    const BItem* items = static_cast<const BItem*>(d.items);
    auto units = [](const void* p) { return static_cast<const BUnit*>(p); };
    int* nclu = d.cnt + 2;
    if (d.nlarge > 0) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)(d.cl_size * d.cl_count));
        cfg.blockDim = dim3(CT);
        cfg.dynamicSmemBytes = CSMEM;
        cfg.stream = st;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = (unsigned)d.cl_size;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        if (const cudaError_t e = cudaLaunchKernelEx(&cfg, cluster_reduce_kernel, items, d.order, d.nlarge, d.cnt))
            return cuda_fail(e);
        count_launch();
    }
    if (const int small = d.count - d.nlarge; small > 0) {
        const int* order = d.order + d.nlarge;
        int* next = d.cnt + 1;
        switch (L.ctas) {
        case 1: bt_persistent_kernel<1><<<L.grid, BT, L.dyn, st>>>(items, order, small, next, L.smem_n); break;
        case 2: bt_persistent_kernel<2><<<L.grid, BT, L.dyn, st>>>(items, order, small, next, L.smem_n); break;
        case 3: bt_persistent_kernel<3><<<L.grid, BT, L.dyn, st>>>(items, order, small, next, L.smem_n); break;
        default: bt_persistent_kernel<4><<<L.grid, BT, L.dyn, st>>>(items, order, small, next, L.smem_n);
        }
        count_launch();
    }
    bt_prep_kernel<<<d.count, BT, 0, st>>>(items, nclu);
    bt_bisect_kernel<<<(d.nbisect + 1) / 2, 64, 0, st>>>(items, units(d.bisect), d.nbisect);
    count_launch(2);
    if (d.ntwist > 0) {
        bt_twist_kernel<<<d.ntwist, 32, 0, st>>>(items, units(d.twist), maxit);
        bt_clu_list_kernel<<<d.count, 128, 0, st>>>(items, static_cast<int3*>(d.clu), nclu);
        bt_clu_kernel<<<2 * device_sms(), tri::CLU_T, 0, st>>>(items, static_cast<const int3*>(d.clu), nclu, maxit);
        count_launch(3);
        if (d.ngram > 0) {
            bt_gram_kernel<<<d.ngram, 160, 0, st>>>(items, units(d.gram));
            bt_gram_sum_kernel<<<dim3(d.ngsum, 4), 256, 0, st>>>(items, units(d.gsum));
            count_launch(2);
        }
        bt_wy_kernel<<<d.nwy, WT, wy_smem(d.nmax, BE), st>>>(items, units(d.wy));
        count_launch();
    }
    bt_status_kernel<<<(d.count + 127) / 128, 128, 0, st>>>(items, d.count);
    count_launch();
    return cuda_ok(cudaGetLastError());
}

int batched_launch(cudaStream_t st, const BatchPlanDev& d, const skew_batched_config& cfg, int maxit) {
    if (d.count <= 0) return 0;
    BatchLaunch L{};
    if (const int rc = batched_prepare(d, cfg, &L)) return rc;
    return batched_exec(st, d, L, maxit);
}

// Places the item and work tables in the workspace and uploads them
// (synchronously with respect to the host buffers: pageable copies).
int batched_upload(cudaStream_t st, int count, const BatchProblem* pr, void* ws, size_t ws_bytes, BatchPlanDev* out) {
    if (count <= 0) return 0;
    for (int b = 0; b < count; b++)
        if (pr[b].n < 2 || pr[b].n > BATCH_MAX) return SKEW_ERR_UNSUPPORTED;
    const BTables tb = batch_tables(count, pr);
    Carve cv(ws, ws_bytes);
    BCarve bc{};
    carve_small(cv, count, pr, tb, &bc);
    if (!cv.ok) return SKEW_ERR_WORKSPACE;
    cudaError_t e = cudaSuccess;
    auto up = [&](void* dst, const void* src, size_t bytes) {
        if (e == cudaSuccess && bytes > 0) e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, st);
    };
    up(bc.d_items, bc.items.data(), sizeof(BItem) * bc.items.size());
    up(bc.d_order, tb.order.data(), sizeof(int) * tb.order.size());
    up(bc.d_bisect, tb.bisect.data(), sizeof(BUnit) * tb.bisect.size());
    up(bc.d_twist, tb.twist.data(), sizeof(BUnit) * tb.twist.size());
    up(bc.d_gram, tb.gram.data(), sizeof(BUnit) * tb.gram.size());
    up(bc.d_gsum, tb.gsum.data(), sizeof(BUnit) * tb.gsum.size());
    up(bc.d_wy, tb.wy.data(), sizeof(BUnit) * tb.wy.size());
    if (e != cudaSuccess) return cuda_fail(e);
    *out = BatchPlanDev{};
    out->items = bc.d_items;
    out->order = bc.d_order;
    out->bisect = bc.d_bisect;
    out->twist = bc.d_twist;
    out->gram = bc.d_gram;
    out->gsum = bc.d_gsum;
    out->wy = bc.d_wy;
    out->clu = bc.d_clu;
    out->cnt = bc.d_cnt;
    out->nbisect = (int)tb.bisect.size();
    out->ntwist = (int)tb.twist.size();
    out->ngram = (int)tb.gram.size();
    out->ngsum = (int)tb.gsum.size();
    out->nwy = (int)tb.wy.size();
    out->count = count;
    out->nlarge = tb.nlarge;
    out->nmax = 2;
    for (int b = 0; b < count; b++) out->nmax = pr[b].n > out->nmax ? pr[b].n : out->nmax;
    std::vector<int> ns;
    for (int i = 0; i < tb.nlarge; i++) ns.push_back(pr[tb.order[(size_t)i]].n);
    return pick_clusters(ns, out);
}

int batched_small(cudaStream_t st, int count, const BatchProblem* pr, void* ws, size_t ws_bytes, int maxit) {
    if (count <= 0) return 0;
    BatchPlanDev d{};
    if (const int rc = batched_upload(st, count, pr, ws, ws_bytes, &d)) return rc;
    return batched_launch(st, d, batched_default_config(), maxit);
}

}  // namespace sk
