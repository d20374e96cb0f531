// tridiag.cu -- eigenpairs of the symmetric tridiagonal S = tridiag(alpha, 0,
// alpha) obtained from the skew tridiagonal T by Lemma 1 (Eq. 1:
// -i D^H T D = S, D = diag(i^r)), and the D back transformation of
// Algorithm 1 step 3.
//
// Sec. 3 (the solver BSEPACK adapted from ScaLAPACK): bisection + inverse
// iteration, each in the form that suits a slow FP64 pipe.
//   * Eigenvalues: Sturm counts for the nev largest on [-g, g], g = ||S||_1.
//     FP64 runs at 1/64 of the FP32 rate and the recurrence is a division
//     chain, so FP32 counts of S / g bracket each eigenvalue to 8 eps32 first
//     (four lanes multisect).  Where the vectors are not refined, FP64 counts
//     on the zero-diagonal form check the bracket, widened by 64 eps32, and
//     finish it with 2 to 32 lanes an eigenvalue, as many as fill the FP64
//     pipes (32 lanes: a factor 33 a count, 7 counts instead of 30); where they
//     are, double-float counts (FP32 pairs) narrow it to 2^-42.  Each floating-point Sturm count is
//     exact for a matrix perturbed by a few units of its roundoff (Kahan),
//     hence the widening before each check.
//   * Vectors: the twisted factorisation of S - lambda I (stationary and
//     progressive transforms met at the row of the smallest |gamma|: Fernando;
//     Parlett and Dhillon), FP64, two lanes a vector, and where no refinement
//     follows one more solve with it (one shot alone: orthogonality 3.2 n eps
//     at n = 1001, with the solve 0.3): two passes each way instead of two or
//     three pivoted LU solves.  Vectors closer than ctol are a cluster: gaps above 1e-9 g
//     leave them independent and one modified Gram-Schmidt pass orthogonalises
//     them; tighter ones iterate in lockstep (pivoted LU solves from a
//     counter-based (splitmix64) start vector, each member's on its own
//     thread, the cluster's CTA orthogonalising between them; before a
//     refinement in double-float, eps = 2^-44).
//     The largest-modulus entry of each vector is made positive.
//     Before a refinement, vectors of eigenvalues near 0 get halves (even and
//     odd rows) of equal norm (tridiag_dev.cuh, PAIR_TOL).
//   With both the FP64 solve takes 1.2, 3.9 and 12.8 ms at n = 500, 1501
//   and 4096 (nev = n / 2), against 5.9, 17.6 and 48 ms for two-lane bisection
//   from a double-float bracket and pivoted inverse iteration alone.
// Vectors are kept interleaved, Q[i * nev + k], so consecutive threads
// (consecutive k) touch consecutive addresses in every sweep over i.
#include <algorithm>
#include <cfloat>
#include <cmath>

#include "common.cuh"
#include "internal.h"
#include "tridiag_dev.cuh"

namespace sk {
namespace {

using namespace tri;

#ifndef BISECT_LANES
#define BISECT_LANES 2
#endif


__global__ void tri_prep_kernel(int n, const double* __restrict__ alpha, double* __restrict__ a2,
                                float* __restrict__ a2s, float* __restrict__ a2l, float* __restrict__ alh,
                                float* __restrict__ all_, TriScalars* sc, double* __restrict__ a2e,
                                double* __restrict__ b2e, int full, int* __restrict__ fail) {
    if (threadIdx.x == 0) *fail = 0x7fffffff;
    __shared__ double red[32];
    double gmax = 0.0, amax = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        double al = (i < n - 1) ? alpha[i] : 0.0;
        double ap = (i > 0) ? alpha[i - 1] : 0.0;
        if (i < n - 1 && full) a2[i] = al * al;
        gmax = fmax(gmax, fabs(al) + fabs(ap));
        amax = fmax(amax, al * al);
    }
    // block max (reuse the sum helper pattern with fmax)
    for (int o = 16; o > 0; o >>= 1) {
        gmax = fmax(gmax, __shfl_xor_sync(0xffffffffu, gmax, o));
        amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ double red2[32];
    if (lane == 0) { red[warp] = gmax; red2[warp] = amax; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double g = 0.0, a = 0.0;
        for (int w = 0; w < (int)(blockDim.x + 31) / 32; w++) { g = fmax(g, red[w]); a = fmax(a, red2[w]); }
        sc->g = g;
        sc->pivmin = DBL_MIN * fmax(1.0, a);
        sc->down = pow2_down(g);
        sc->up = 1.0 / sc->down;
        red[0] = g;
        red[1] = sc->down;
    }
    __syncthreads();
    // alpha^2 / g^2 as an FP32 pair (a2s + a2l) for the bracketing passes
    // (entries below FLT_MIN become 0: a perturbation far below their
    // tolerances)
    const double g = red[0], ig2 = (g > 0.0) ? 1.0 / (g * g) : 0.0, down = red[1];
    // alpha scaled by a power of two (exact), and the bidiagonal of the
    // zero-diagonal form from it: a_i = alpha_{2i}, b_i = alpha_{2i+1}, squared
    for (int i = threadIdx.x; i < n - 1 && !full; i += blockDim.x) a2[i] = alpha[i] * down;
    for (int i = threadIdx.x; i < (n + 1) / 2; i += blockDim.x) {
        const double a = (2 * i <= n - 2) ? alpha[2 * i] * down : 0.0;
        const double b = (2 * i + 1 <= n - 2) ? alpha[2 * i + 1] * down : 0.0;
        a2e[i] = a * a;
        b2e[i] = b * b;
    }
    for (int i = threadIdx.x; i < n - 1; i += blockDim.x) {
        const double v = alpha[i] * alpha[i] * ig2;
        const float h = (float)v;
        a2s[i] = h;
        a2l[i] = (float)(v - (double)h);
        const float ah = (float)alpha[i];  // alpha itself as a pair (double-float inverse iteration)
        alh[i] = ah;
        all_[i] = (float)(alpha[i] - (double)ah);
    }
}

// as[i] = alpha[i] scaled (tri_prep_kernel's array when it held alpha^2 so far)
__global__ void tri_scale_kernel(int n, const double* __restrict__ alpha, const TriScalars* sc,
                                 double* __restrict__ as) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n - 1; i += gridDim.x * blockDim.x)
        as[i] = alpha[i] * sc->down;
}

constexpr float PIV_DF = 7.888609052210118e-31f;  // 2^-100: pivots of S / g raised to this

// Double-float Sturm count of S / g at x (the recurrence of sturm()).
__device__ __forceinline__ int sturm_df(int n, const float* __restrict__ a2s, const float* __restrict__ a2l, Df x) {
    int cnt = 0;
    Df d = {-x.h, -x.l};
    if (fabsf(d.h) < PIV_DF) d = {-PIV_DF, 0.f};
    cnt += (d.h < 0.f);
    for (int i = 1; i < n; i++) {
        const Df t = df_add(x, df_div({a2s[i - 1], a2l[i - 1]}, d));
        d = {-t.h, -t.l};
        if (fabsf(d.h) < PIV_DF) d = {-PIV_DF, 0.f};
        cnt += (d.h < 0.f);
    }
    return cnt;
}

template <int L>
__global__ void bisect32_kernel(int n, int nev, const float* __restrict__ a2s, double* __restrict__ lohi) {
    const int gt = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = gt / L;
    if (k < nev) bisect32_body<L>(n, k, gt % L, threadIdx.x & 31, a2s, lohi);
}

// Second pass: L lanes multisect the FP32 bracket (widened by FP32_SLACK
// eps32, checked with double-float counts and widened eightfold until the
// check holds) with double-float counts down to DF_WIDTH.  Writes the
// bracket (units of g) back and, in lambda, its midpoint times g.
constexpr double DF_WIDTH = 1.0 / 4398046511104.0;  // 2^-42
template <int L>
__global__ void bisect_df_kernel(int n, int nev, const float* __restrict__ a2s, const float* __restrict__ a2l,
                                 const TriScalars* sc, double* __restrict__ lohi, double* __restrict__ lambda) {
    const int gt = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = gt / L, q = gt % L, lane = threadIdx.x & 31;
    if (k >= nev) return;
    const unsigned gmask = lane_group<L>(lane);
    const int j = n - 1 - k;
    const double g = sc->g;
    if (n == 1 || g == 0.0) {
        if (q == 0) lambda[k] = 0.0;
        return;
    }
    const double glo = -1.0 - 1e-6, ghi = 1.0 + 1e-6;
    double lo = glo, hi = ghi;
    double slack = FP32_SLACK * FLT_EPSILON;
    for (int tries = 0; tries < 8; tries++) {
        const double a = fmax(glo, lohi[2 * k] - slack), b = fmin(ghi, lohi[2 * k + 1] + slack);
        bool mine = true;
        if (q == 0) mine = (a == glo) || sturm_df(n, a2s, a2l, df_of(a)) <= j;
        if (q == 1) mine = (b == ghi) || sturm_df(n, a2s, a2l, df_of(b)) > j;
        if ((__ballot_sync(gmask, !mine) & gmask) == 0u) {
            lo = a;
            hi = b;
            break;
        }
        slack *= 8.0;
    }
    for (int it = 0; it < 64; it++) {
        const double w = hi - lo;
        if (w <= DF_WIDTH) break;
        const double step = w * (1.0 / (L + 1));
        const double x = lo + (double)(q + 1) * step;
        const bool le = (x > lo && x < hi) ? (sturm_df(n, a2s, a2l, df_of(x)) <= j) : (x <= lo);
        const int nle = __popc(__ballot_sync(gmask, le) & gmask);
        const double nlo = (nle > 0) ? lo + (double)nle * step : lo;
        const double nhi = (nle < L) ? lo + (double)(nle + 1) * step : hi;
        if (!(nlo > lo || nhi < hi)) break;
        lo = nlo;
        hi = (nhi < hi) ? nhi : hi;
    }
    if (q == 0) {
        lohi[2 * k] = lo;
        lohi[2 * k + 1] = hi;
        lambda[k] = (lo + 0.5 * (hi - lo)) * g;
    }
}

constexpr double DF_SLACK = 1.0 / 68719476736.0;  // 2^-36: widening of a double-float bracket (units of g)

// FP64 multisection with L lanes per wanted eigenvalue: each lane counts at
// one of L equally spaced interior points, the interval shrinks to
// 1 / (L + 1) per step, down to 2 eps max(|lo|, |hi|).  The start is the
// double-float bracket (units of g) widened by DF_SLACK g once its ends pass
// the FP64 counts count(lo) <= j < count(hi); a bracket that fails is widened
// eightfold, up to the whole Gershgorin interval.
template <int L>
__global__ void bisect_kernel(int n, int nev, const double* __restrict__ a2, const TriScalars* sc,
                              const double* __restrict__ lohi, double* __restrict__ lambda) {
    const int gt = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = gt / L, q = gt % L, lane = threadIdx.x & 31;
    if (k >= nev) return;  // whole lane groups leave together (blockDim is a multiple of L)
    const unsigned gmask = lane_group<L>(lane);
    const double g = sc->g, pivmin = sc->pivmin;
    const int j = n - 1 - k;  // ascending index of the wanted eigenvalue
    // count(x) <= j: the wanted eigenvalue is >= x
    auto below = [&](double x) -> bool { return sturm(n, a2, pivmin, x) <= j; };
    if (n == 1 || g == 0.0) {
        if (q == 0) lambda[k] = 0.0;
        return;
    }
    const double glo = -g - 2.0 * DBL_EPSILON * g - pivmin, ghi = g + 2.0 * DBL_EPSILON * g + pivmin;
    double lo = glo, hi = ghi;
    double slack = DF_SLACK * g;
    for (int tries = 0; tries < 8; tries++) {
        const double a = fmax(glo, lohi[2 * k] * g - slack), b = fmin(ghi, lohi[2 * k + 1] * g + slack);
        // lane 0 checks the lower end, lane 1 the upper one
        bool mine = true;
        if (q == 0) mine = (a == glo) || below(a);
        if (q == 1) mine = (b == ghi) || !below(b);
        if ((__ballot_sync(gmask, !mine) & gmask) == 0u) {
            lo = a;
            hi = b;
            break;
        }
        slack *= 8.0;
    }
    for (int it = 0; it < 4000; it++) {
        const double w = hi - lo;
        const double tol = 2.0 * DBL_EPSILON * fmax(fabs(lo), fabs(hi)) + DBL_MIN;
        if (w <= tol) break;
        const double step = w / (double)(L + 1);
        const double x = lo + (double)(q + 1) * step;
        const bool le = (x > lo && x < hi) ? below(x) : (x <= lo);
        // counts grow with x: the lanes with lambda_j >= x_q are a prefix
        const int nle = __popc(__ballot_sync(gmask, le) & gmask);
        const double nlo = (nle > 0) ? lo + (double)nle * step : lo;
        const double nhi = (nle < L) ? lo + (double)(nle + 1) * step : hi;
        if (!(nlo > lo || nhi < hi)) break;  // no representable progress
        lo = nlo;
        hi = (nhi < hi) ? nhi : hi;
    }
    if (q == 0) lambda[k] = lo + 0.5 * (hi - lo);
}

template <int L>
__global__ void __launch_bounds__(64) bisect_bd_kernel(int n, int nev, const TriScalars* sc,
                                                       const double* __restrict__ lohi, double* __restrict__ lambda,
                                                       const double* __restrict__ a2e,
                                                       const double* __restrict__ b2e) {
    const int gt = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = gt / L;
    if (k < nev) bisect_bd_body<L>(n, k, gt % L, threadIdx.x & 31, sc, lohi, lambda, a2e, b2e);
}

// null: a single eigenvalue at NULL_TOL g or below counts as a cluster of one.
__global__ void clu_list_kernel(int nev, const double* __restrict__ lambda, const TriScalars* sc, double ctol_rel,
                                int null, int2* __restrict__ list, int* __restrict__ count) {
    __shared__ int c;
    if (threadIdx.x == 0) c = 0;
    __syncthreads();
    const double ctol = ctol_rel * sc->g;
    for (int k = threadIdx.x; k < nev; k += blockDim.x) {
        if (!starts_cluster(lambda, k, ctol)) continue;
        if (k + 1 == nev || starts_cluster(lambda, k + 1, ctol)) {
            if (null && lambda[k] <= NULL_TOL * sc->g) list[atomicAdd(&c, 1)] = make_int2(k, 1);
            continue;
        }
        int k1 = k + 2;
        while (k1 < nev && !starts_cluster(lambda, k1, ctol)) k1++;
        const int at = atomicAdd(&c, 1);  // clusters are independent: their order does not matter
        list[at] = make_int2(k, k1 - k);
    }
    __syncthreads();
    if (threadIdx.x == 0) *count = c;
}

__global__ void __launch_bounds__(CLU_T)
invit_clu_kernel(int n, int nev, const double* __restrict__ alpha, const double* __restrict__ lambda,
                 const TriScalars* sc, int maxit, InvitBufs bf, double* Q, const int2* __restrict__ list,
                 const int* __restrict__ count, double* __restrict__ need, int* __restrict__ fail) {
    const int nc = *count;
    for (int b = blockIdx.x; b < nc; b += gridDim.x) {
        __syncthreads();  // the previous cluster is done with shared memory
        clu_body(n, nev, list[b].x, list[b].y, alpha, lambda, sc->g, maxit, bf, Q, need, fail);
    }
}

// CTA-wide double-float sum (fixed order: deterministic).
__device__ __forceinline__ Df df_block_sum(Df v, float* rh, float* rl) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v = df_add(v, Df{__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)});
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) {
        rh[warp] = v.h;
        rl[warp] = v.l;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        Df s = {rh[0], rl[0]};
        for (int w = 1; w < nw; w++) s = df_add(s, Df{rh[w], rl[w]});
        rh[0] = s.h;
        rl[0] = s.l;
    }
    __syncthreads();
    const Df r = {rh[0], rl[0]};
    __syncthreads();
    return r;
}

// The lockstep cluster iteration in double-float (the vectors refined
// afterwards); the members are converted to FP64 when the cluster is done.
__global__ void __launch_bounds__(CLU_T)
invit_clu_df_kernel(int n, int nev, const float* __restrict__ alh, const float* __restrict__ all_,
                    const double* __restrict__ lambda, const TriScalars* sc, int maxit, InvitBufs bf,
                    double* Q, const int2* __restrict__ list, const int* __restrict__ count,
                    const double* __restrict__ need, int* __restrict__ fail) {
    __shared__ float rh[32], rl[32];
    __shared__ double red[32];
    __shared__ int redi[32];
    __shared__ int s_ff, s_bad;
    const int nc = *count;
    const double g = sc->g;
    const size_t ld = (size_t)nev;
    const double eps = 1.0 / 17592186044416.0;  // 2^-44
    const float ptol = (float)(eps * g);
    const float grow = (float)(1.0 / (100.0 * sqrt((double)n) * eps * g));
    const InvitDf v = invit_df_view(bf, Q);
    Df* Qd = v.Qd;
    const int t = threadIdx.x, T = blockDim.x;
    for (int b = blockIdx.x; b < nc; b += gridDim.x) {
        const int2 cl = list[b];
        const int k0 = cl.x, m = cl.y;
        if (n == 1 || g == 0.0) {
            for (int e = t; e < m * n; e += T) {
                const int j = e / n, i = e % n;
                Q[i * ld + k0 + j] = (i == k0 + j) ? 1.0 : 0.0;
            }
            continue;
        }
        if (!clu_tight(lambda, need, g, k0, m)) {
            clu_mgs(n, ld, Q, k0, m, red, redi);
            continue;
        }
        const bool pairs = lambda[k0 + m - 1] <= PAIR_TOL * g;  // halves by themselves
        // the cluster's iterations one after another; st (clu_next_state) is
        // the same in every thread
        int st = 0;
        for (int it = 0; it < maxit && st != 2; it++) {
            for (int j = t; j < m; j += T) {
                const int k = k0 + j;
                if (it == 0) {
                    const bool null = lambda[k] <= NULL_TOL * g;
                    invit_lu_df(n, alh, all_, null ? 0.0 : lambda[k], ptol, null ? ptol : 0.f, v, ld, k);
                    invit_start_df(n, Qd, ld, k);
                }
                invit_solve_df(n, v, ld, k);
            }
            if (t == 0) {
                s_ff = m;
                s_bad = 0;
            }
            __syncthreads();
            for (int j = 0; j < m; j++) {
                Df* qj = Qd + k0 + j;
                if (pairs) {
                    // |even|^2 and |odd|^2 of the vector (T is even: a thread's rows
                    // are of one half)
                    auto halves = [&]() -> double2 {
                        double s = 0.0;
                        for (int i = t; i < n; i += T) {
                            const double y = df_to_double(qj[i * ld]);
                            s = fma(y, y, s);
                        }
                        const double e = sk_block_sum((t & 1) ? 0.0 : s, red);
                        return make_double2(e, sk_block_sum((t & 1) ? s : 0.0, red));
                    };
                    const double2 before = halves();
                    // twice: with one shift the members can start nearly parallel
                    for (int h = 0; h < 2 * j; h++) {
                        const Df* qp = Qd + k0 + (h < j ? h : h - j);
                        Df d = {0.f, 0.f};
                        for (int i = t; i < n; i += T) d = df_add(d, df_mul(qp[i * ld], qj[i * ld]));
                        const Df de = df_block_sum((t & 1) ? Df{0.f, 0.f} : d, rh, rl);
                        const Df dd = df_block_sum((t & 1) ? d : Df{0.f, 0.f}, rh, rl);
                        const Df md = (t & 1) ? Df{-2.f * dd.h, -2.f * dd.l} : Df{-2.f * de.h, -2.f * de.l};
                        for (int i = t; i < n; i += T) qj[i * ld] = df_add(qj[i * ld], df_mul(md, qp[i * ld]));
                        __syncthreads();
                    }
                    const double2 s = halves();
                    if (!(s.x > 0.0) || !(s.y > 0.0) || !isfinite(s.x + s.y)) {
                        if (t == 0) {
                            s_bad = 1;
                            s_ff = min(s_ff, j);
                        }
                    } else {
                        const Df f = df_of(1.0 / sqrt(2.0 * ((t & 1) ? s.y : s.x)));
                        for (int i = t; i < n; i += T) qj[i * ld] = df_mul(qj[i * ld], f);
                        // nor may a half be the rounding of what the passes took off
                        if (t == 0 && (!(sqrt(s.x + s.y) >= (double)grow) || s.x < 1e-20 * before.x || s.y < 1e-20 * before.y))
                            s_ff = min(s_ff, j);
                    }
                    __syncthreads();
                    continue;
                }
                for (int p = 0; p < j; p++) {
                    const Df* qp = Qd + k0 + p;
                    Df d = {0.f, 0.f};
                    for (int i = t; i < n; i += T) d = df_add(d, df_mul(qp[i * ld], qj[i * ld]));
                    const Df md = df_neg(df_block_sum(d, rh, rl));
                    for (int i = t; i < n; i += T) qj[i * ld] = df_add(qj[i * ld], df_mul(md, qp[i * ld]));
                    __syncthreads();
                }
                float s = 0.f;
                for (int i = t; i < n; i += T) {
                    const float y = qj[i * ld].h;
                    s = fmaf(y, y, s);
                }
                const float nrm = sqrtf(sk_block_sum(s, rh));
                if (!(nrm > 0.f) || !isfinite(nrm)) {
                    if (t == 0) {
                        s_bad = 1;
                        s_ff = min(s_ff, j);
                    }
                } else {
                    const Df sc1 = {1.0f / nrm, 0.f};
                    for (int i = t; i < n; i += T) qj[i * ld] = df_mul(qj[i * ld], sc1);
                    if (t == 0 && !(nrm >= grow)) s_ff = min(s_ff, j);
                }
                __syncthreads();
            }
            bool fin, failed;
            const int nst = clu_next_state(st, s_ff, m, s_bad, it, maxit, fin, failed);
            if (failed && t == 0) atomicMin(fail, k0 + s_ff);
            if (fin) {
                for (int j = 0; j < m; j++) {
                    Df* qj = Qd + k0 + j;
                    const int imax = block_argmax(n, [&](int i) { return (double)fabsf(qj[i * ld].h); }, red, redi);
                    const bool neg = qj[imax * ld].h < 0.f;  // read by all before any flip
                    __syncthreads();
                    for (int i = t; i < n; i += T) {
                        const Df y = qj[i * ld];
                        Q[i * ld + k0 + j] = df_to_double(neg ? df_neg(y) : y);
                    }
                    __syncthreads();
                }
            }
            st = fin ? 2 : nst;
            __syncthreads();
        }
    }
}

__global__ void __launch_bounds__(32)
twist_kernel(int n, int nev, const double* __restrict__ as, const double* __restrict__ alpha,
             const double* __restrict__ lambda, const TriScalars* sc, double ctol_rel, int maxit, int polish,
             InvitBufs bf, double* Q, double* __restrict__ need, int* __restrict__ fail) {
    twist_body(n, nev, blockIdx.x * 16, threadIdx.x, as, alpha, lambda, sc, ctol_rel, maxit, polish, bf, Q, need,
               fail);
}

__global__ void invit_status_kernel(const int* fail, int nev, int* status) {
    if (threadIdx.x == 0 && *fail < nev) sk_set_error(status, SKEW_INFO_INVIT_BASE + *fail);
}

// Qi (n x nev interleaved: Qi[i * nev + k]) -> X (n x nev, ld ldz) [+ Y]:
// with dmap, entry i of column k is i^i * q: i mod 4 = 0 -> X = q, 1 -> Y = q,
// 2 -> X = -q, 3 -> Y = -q (Algorithm 1 step 3).
__global__ void transpose_dmap_kernel(int n, int nev, const double* __restrict__ Qi, double* __restrict__ X,
                                      double* __restrict__ Y, int ldz, int dmap) {
    __shared__ double tile[32][33];
    const int i0 = blockIdx.x * 32, k0 = blockIdx.y * 32;
    const int tx = threadIdx.x, ty = threadIdx.y;  // 32 x 8
    for (int r = ty; r < 32; r += 8) {
        int i = i0 + r, k = k0 + tx;
        tile[r][tx] = (i < n && k < nev) ? Qi[(size_t)i * nev + k] : 0.0;
    }
    __syncthreads();
    for (int c = ty; c < 32; c += 8) {
        int k = k0 + c, i = i0 + tx;
        if (i < n && k < nev) {
            double q = tile[tx][c];
            size_t at = (size_t)k * ldz + i;
            if (!dmap) {
                X[at] = q;
            } else {
                int m4 = i & 3;
                X[at] = (m4 == 0) ? q : (m4 == 2 ? -q : 0.0);
                Y[at] = (m4 == 1) ? q : (m4 == 3 ? -q : 0.0);
            }
        }
    }
}

__global__ void dmap_colmajor_kernel(int n, int k, const double* __restrict__ Q, int ldq, double* __restrict__ X,
                                     double* __restrict__ Y, int ldz) {
    size_t total = (size_t)n * k;
    for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
         e += (size_t)gridDim.x * blockDim.x) {
        int i = (int)(e % n), j = (int)(e / n);
        double q = Q[(size_t)j * ldq + i];
        int m4 = i & 3;
        X[(size_t)j * ldz + i] = (m4 == 0) ? q : (m4 == 2 ? -q : 0.0);
        Y[(size_t)j * ldz + i] = (m4 == 1) ? q : (m4 == 3 ? -q : 0.0);
    }
}

struct TriWs {
    double* a2;  // alpha^2 for the full-length counts, then alpha scaled by a power of two to g in [1, 2)
    double *a2e, *b2e;  // alpha_{2i}^2, alpha_{2i+1}^2 (zero-diagonal form, ceil(n/2) each)
    float *a2s, *a2l;  // alpha^2 / g^2 as an FP32 pair (bracketing passes)
    float *alh, *all_;  // alpha as an FP32 pair (double-float inverse iteration)
    double* lohi;   // FP32 brackets, 2 per wanted eigenvalue
    TriScalars* sc;
    int* fail;
    InvitBufs bf;
    int2* clist;  // clusters of two or more: (first index, size)
    int* ccount;
};

TriWs carve_tri(Carve& cv, int n, int nev) {
    TriWs w{};
    size_t nn = (size_t)(n > 0 ? n : 1), ne = (size_t)(nev > 0 ? nev : 1);
    w.a2 = cv.take<double>(nn);
    w.a2e = cv.take<double>(nn / 2 + 1);
    w.b2e = cv.take<double>(nn / 2 + 1);
    w.a2s = cv.take<float>(nn);
    w.a2l = cv.take<float>(nn);
    w.alh = cv.take<float>(nn);
    w.all_ = cv.take<float>(nn);
    w.lohi = cv.take<double>(2 * ne);
    w.sc = cv.take<TriScalars>(1);
    w.fail = cv.take<int>(1);
    w.bf.u0 = cv.take<double>(nn * ne);
    w.bf.u1 = cv.take<double>(nn * ne);
    w.bf.u2 = cv.take<double>(nn * ne);
    w.bf.ml = cv.take<double>(nn * ne);
    w.bf.sw = cv.take<unsigned char>(nn * ne);
    w.clist = cv.take<int2>(ne / 2 + 1);
    w.ccount = cv.take<int>(1);
    return w;
}

}  // namespace

size_t tridiag_ws(int n, int nev) {
    Carve cv(nullptr, ~size_t(0));
    carve_tri(cv, n, nev);
    return cv.off + 256;
}

int tridiag_eig(cudaStream_t st, int n, const double* alpha, int nev, double* lambda, double* Qi, void* ws,
                size_t ws_bytes, int* d_status, int maxit, bool fp64, bool bidiag) {
    if (n <= 0 || nev <= 0) return 0;
    Carve cv(ws, ws_bytes);
    TriWs w = carve_tri(cv, n, nev);
    if (!cv.ok) return SKEW_ERR_WORKSPACE;
    // full-length counts where the zero-diagonal form is not wanted
    const int full = fp64 && !(bidiag && 2 * nev <= n);
    tri_prep_kernel<<<1, 1024, 0, st>>>(n, alpha, w.a2, w.a2s, w.a2l, w.alh, w.all_, w.sc, w.a2e, w.b2e,
                                        full, w.fail);
    count_launch();
    const int sms = device_sms();
    {
        KtScope kt(st, KT_BISECT);
        // FP32 chains are bound by latency: 32 lanes an eigenvalue up to about
        // eight warps a scheduler, four beyond that
        const bool wide = nev <= sms * 32;
        if (wide)
            bisect32_kernel<32><<<(32 * nev + 127) / 128, 128, 0, st>>>(n, nev, w.a2s, w.lohi);
        else
            bisect32_kernel<4><<<(4 * nev + 127) / 128, 128, 0, st>>>(n, nev, w.a2s, w.lohi);
        count_launch();
        if (fp64 && !full) {
            // FP64 finish on the zero-diagonal form (half-length counts)
            int L = 32;
            while (L > 2 && (long long)nev * L > 32LL * 4 * sms) L >>= 1;
            const int grid = (int)(((long long)L * nev + 63) / 64);
            switch (L) {
            case 32: bisect_bd_kernel<32><<<grid, 64, 0, st>>>(n, nev, w.sc, w.lohi, lambda, w.a2e, w.b2e); break;
            case 16: bisect_bd_kernel<16><<<grid, 64, 0, st>>>(n, nev, w.sc, w.lohi, lambda, w.a2e, w.b2e); break;
            case 8: bisect_bd_kernel<8><<<grid, 64, 0, st>>>(n, nev, w.sc, w.lohi, lambda, w.a2e, w.b2e); break;
            case 4: bisect_bd_kernel<4><<<grid, 64, 0, st>>>(n, nev, w.sc, w.lohi, lambda, w.a2e, w.b2e); break;
            default: bisect_bd_kernel<2><<<grid, 64, 0, st>>>(n, nev, w.sc, w.lohi, lambda, w.a2e, w.b2e);
            }
            count_launch();
        } else {
            if (wide)
                bisect_df_kernel<32><<<(32 * nev + 127) / 128, 128, 0, st>>>(n, nev, w.a2s, w.a2l, w.sc, w.lohi,
                                                                             lambda);
            else
                bisect_df_kernel<4><<<(4 * nev + 127) / 128, 128, 0, st>>>(n, nev, w.a2s, w.a2l, w.sc, w.lohi,
                                                                           lambda);
            count_launch();
            if (fp64) {
                bisect_kernel<BISECT_LANES><<<(BISECT_LANES * nev + 63) / 64, 64, 0, st>>>(n, nev, w.a2, w.sc, w.lohi,
                                                                                            lambda);
                count_launch();
            }
        }
    }
    if (Qi) {
        // cluster tolerance relative to ||S||_1: 1e-3 for small n (the usual
        // inverse-iteration choice), shrinking like n^-1.5 so that clusters stay
        // small for dense spectra while eps*||S||/gap stays below n*eps.
        double ctol = fmin(1e-3, 10.0 / ((double)n * sqrt((double)n)));
        {
            KtScope kt(st, KT_INVIT);
            // singletons by twisted factorisations; clusters in lockstep, one CTA each
            if (full) {
                tri_scale_kernel<<<(n + 255) / 256, 256, 0, st>>>(n, alpha, w.sc, w.a2);
                count_launch();
            }
            twist_kernel<<<(nev + 15) / 16, 32, 0, st>>>(n, nev, w.a2, alpha, lambda, w.sc, ctol, maxit, fp64 ? 1 : 0,
                                                         w.bf, Qi, w.lohi, w.fail);
            clu_list_kernel<<<1, 1024, 0, st>>>(nev, lambda, w.sc, ctol, fp64 ? 0 : 1, w.clist, w.ccount);
            count_launch(2);
            const int cgrid = std::max(1, std::min(nev / 2, 2 * sms));
            if (fp64)
                invit_clu_kernel<<<cgrid, CLU_T, 0, st>>>(n, nev, alpha, lambda, w.sc, maxit, w.bf, Qi, w.clist,
                                                          w.ccount, w.lohi, w.fail);
            else
                invit_clu_df_kernel<<<cgrid, CLU_T, 0, st>>>(n, nev, w.alh, w.all_, lambda, w.sc, maxit, w.bf, Qi,
                                                             w.clist, w.ccount, w.lohi, w.fail);
            count_launch();
        }
        invit_status_kernel<<<1, 32, 0, st>>>(w.fail, nev, d_status);
        count_launch();
    }
    return cudaGetLastError() == cudaSuccess ? 0 : SKEW_ERR_CUDA;
}

cudaError_t interleaved_to_colmajor(cudaStream_t st, int n, int nev, const double* Qi, double* X, double* Y,
                                    int ldz, bool dmap) {
    if (n <= 0 || nev <= 0) return cudaSuccess;
    dim3 grid((n + 31) / 32, (nev + 31) / 32), block(32, 8);
    transpose_dmap_kernel<<<grid, block, 0, st>>>(n, nev, Qi, X, Y, ldz, dmap ? 1 : 0);
    count_launch();
    return cudaGetLastError();
}

cudaError_t dmap_colmajor(cudaStream_t st, int n, int k, const double* Q, int ldq, double* X, double* Y, int ldz) {
    if (n <= 0 || k <= 0) return cudaSuccess;
    size_t total = (size_t)n * k;
    int grid = (int)((total + 255) / 256 > 8192 ? 8192 : (total + 255) / 256);
    dmap_colmajor_kernel<<<grid, 256, 0, st>>>(n, k, Q, ldq, X, Y, ldz);
    count_launch();
    return cudaGetLastError();
}

}  // namespace sk
