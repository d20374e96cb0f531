// tridiag_dev.cuh -- device routines of the tridiagonal eigensolver (Sec. 3:
// bisection + inverse iteration on S = tridiag(alpha, 0, alpha)), shared by
// the single-matrix kernels and the batched ones.
#pragma once
#include <cfloat>
#include <cmath>

#include "common.cuh"

namespace sk {
namespace tri {

struct TriScalars {
    double g;       // ||S||_1
    double pivmin;  // DBL_MIN * max(1, max alpha^2)
    double down, up;  // powers of two: g down in [1, 2) (1 when g == 0), up = 1 / down
};

// 1 / d for 2^-1000 < |d| < 2^1000, to rounding (the largest relative error over
// 2.3e8 random arguments was 0.995 2^-53, as that of the division): the hardware's
// FP32 reciprocal of the significand (2^-23), its exponent set with integer
// operations, and one third-order Newton step y (1 + e + e^2), e = 1 - d y.
// Three FP64 instructions; the FP64 pipe issues one per 64 clocks and scheduler
// here, and the division takes nine (640 clocks with its addition, measured).
__device__ __forceinline__ double rcp_fast(double d) {
    const int hi = __double2hiint(d), lo = __double2loint(d);
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;"
        : "=f"(r)
        : "f"(__int_as_float(0x3f800000 | ((hi & 0xfffff) << 3) | (int)((unsigned)lo >> 29))));
    const int rb = __float_as_int(r);
    const int ex = (rb >> 23) - 127 + 1023 - (((hi >> 20) & 0x7ff) - 1023);
    const double y = __hiloint2double((hi & (int)0x80000000) | (ex << 20) | ((rb & 0x7fffff) >> 3), rb << 29);
    double e = fma(-d, y, 1.0);
    e = fma(e, e, e);
    return fma(y, e, y);
}

// Power of two that brings g > 0 into [1, 2).
__device__ __forceinline__ double pow2_down(double g) {
    int e;
    frexp(g, &e);  // g = f 2^e, f in [1/2, 1)
    return (g > 0.0 && isfinite(g)) ? ldexp(1.0, 1 - e) : 1.0;
}

__device__ __forceinline__ int sturm(int n, const double* __restrict__ a2, double pivmin, double x) {
    int cnt = 0;
    double d = -x;
    if (fabs(d) < pivmin) d = -pivmin;
    cnt += (d < 0.0);
    for (int i = 1; i < n; i++) {
        d = -x - a2[i - 1] / d;
        if (fabs(d) < pivmin) d = -pivmin;
        cnt += (d < 0.0);
    }
    return cnt;
}

// Zero-diagonal form (Sec. 2.2, remark after Algorithm 1): with the unknowns
// shuffled even first, S = [[0, B], [B^T, 0]], B lower bidiagonal with
// diagonal a_i = alpha_{2i} and subdiagonal b_i = alpha_{2i+1}; the
// eigenvalues >= 0 of S are the square roots of those of B B^T (order
// m = ceil(n/2)).  Number of eigenvalues of B B^T below t from the stationary
// qd transform of its L D L^T form (D_i = a_i^2, l_i = b_i / a_i):
// D+_i = a_i^2 + s_i, s_{i+1} = b_i^2 s_i / D+_i - t, s_0 = -t (one division per
// step over m steps, against n steps of the full Sturm count).
// The matrix is scaled to g in [1, 2) (entries a2e, b2e <= 4); with the quick
// reciprocal six FP64 instructions a step.  A quotient off by a
// unit of the last place is, like any rounding of the recurrence, a relative
// perturbation of a_i and b_i.  Pivots below 2^-900 are raised to it.
__device__ __forceinline__ int bd_count_scaled(int m, const double* __restrict__ a2e, const double* __restrict__ b2e,
                                               double t) {
    constexpr double PIV = 1.1830521861667747e-271;  // 2^-900
    int cnt = 0;
    double sv = -t;
#pragma unroll 4
    for (int i = 0; i < m; i++) {
        double d = a2e[i] + sv;
        const int e = (__double2hiint(d) >> 20) & 0x7ff;
        if (e <= 123) d = -PIV;  // |d| < 2^-899
        cnt += __double2hiint(d) < 0;
        sv = fma(b2e[i] * sv, rcp_fast(d), -t);
    }
    return cnt;
}

__device__ __forceinline__ double splitmix_uniform(unsigned long long seed, unsigned long long i) {
    // splitmix64 (Steele, Lea, Flood 2014) of seed * golden + i -> uniform(-1, 1)
    unsigned long long z = seed * 0x9E3779B97F4A7C15ULL + i + 0x632BE59BD9B4E019ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    z ^= z >> 31;
    return (double)(z >> 11) * (1.0 / 9007199254740992.0) * 2.0 - 1.0;
}

// ---- double-float (FP32 pair) arithmetic: Dekker, "A floating-point
// technique for extending the available precision" (1971); Knuth's two_sum.
// About 46 bits, at FP32-pipe latency.
struct Df {
    float h, l;
};
__device__ __forceinline__ Df df_of(double x) {
    const float h = (float)x;
    return {h, (float)(x - (double)h)};
}
__device__ __forceinline__ Df df_fast_two_sum(float a, float b) {
    const float s = a + b;
    return {s, b - (s - a)};
}
// (a + b) with an error below a few 2^-46 (|a| + |b|): as a perturbation of
// the shift and of the quotient separately, which a Sturm count tolerates
__device__ __forceinline__ Df df_add(Df a, Df b) {
    const float s = a.h + b.h;
    const float bb = s - a.h;
    const float e = (a.h - (s - bb)) + (b.h - bb);
    return df_fast_two_sum(s, e + (a.l + b.l));
}
// a / b: quotient of the leading parts, corrected by the exact remainder
__device__ __forceinline__ Df df_div(Df a, Df b) {
    const float q1 = __fdividef(a.h, b.h);
    const float p1 = q1 * b.h;
    const float p2 = fmaf(q1, b.h, -p1);
    const float r = (((a.h - p1) - p2) + a.l) - q1 * b.l;
    return df_fast_two_sum(q1, __fdividef(r, b.h));
}

__device__ __forceinline__ Df df_mul(Df a, Df b) {
    const float p = a.h * b.h;
    const float e = fmaf(a.h, b.h, -p) + (a.h * b.l + a.l * b.h);
    return df_fast_two_sum(p, e);
}
__device__ __forceinline__ Df df_neg(Df a) { return {-a.h, -a.l}; }
__device__ __forceinline__ double df_to_double(Df a) { return (double)a.h + (double)a.l; }

struct InvitBufs {
    double *u0, *u1, *u2, *ml;
    unsigned char* sw;
};

// ---- inverse iteration, one vector (column k of the interleaved buffers) ----
// LU with partial pivoting of S - lam I (U rows u0, u1, u2; multipliers ml;
// interchanges sw); pivots below ptol are raised to ptol, couplings below drop
// count as zero.
__device__ __forceinline__ void invit_lu(int n, const double* __restrict__ alpha, double lam, double ptol,
                                         const InvitBufs& bf, size_t ld, int k, double drop = 0.0) {
    auto edge = [&](int i) { return fabs(alpha[i]) < drop ? 0.0 : alpha[i]; };
    double a0 = -lam, a1 = edge(0);
    for (int i = 0; i < n - 1; i++) {
        const double l = edge(i), dn = -lam;
        const double un = (i + 1 < n - 1) ? edge(i + 1) : 0.0;
        const size_t at = i * ld + k;
        if (fabs(a0) >= fabs(l)) {
            double piv = a0;
            if (fabs(piv) < ptol) piv = (piv < 0.0) ? -ptol : ptol;
            double m = l / piv;
            bf.u0[at] = piv; bf.u1[at] = a1; bf.u2[at] = 0.0; bf.sw[at] = 0; bf.ml[at] = m;
            a0 = dn - m * a1;
            a1 = un;
        } else {
            double m = a0 / l;
            bf.u0[at] = l; bf.u1[at] = dn; bf.u2[at] = un; bf.sw[at] = 1; bf.ml[at] = m;
            double na0 = a1 - m * dn;
            a1 = -m * un;
            a0 = na0;
        }
    }
    if (fabs(a0) < ptol) a0 = (a0 < 0.0) ? -ptol : ptol;
    const size_t at = (size_t)(n - 1) * ld + k;
    bf.u0[at] = a0; bf.u1[at] = 0.0; bf.u2[at] = 0.0;
}

// The sweeps below are sequential in i and each thread owns column k: loads
// run IB elements ahead of the dependent arithmetic (a store to element i
// never precedes the load of element i), so the chain waits on global memory
// once per IB elements instead of once per element.
constexpr int INV_IB = 8;

// Counter-based start vector (splitmix64 of (k + 1, i)), normalised.
__device__ __forceinline__ void invit_start(int n, double* __restrict__ Q, size_t ld, int k) {
    double nrm = 0.0;
    for (int i = 0; i < n; i++) {
        double x = splitmix_uniform((unsigned long long)k + 1ULL, (unsigned long long)i);
        Q[i * ld + k] = x;
        nrm = fma(x, x, nrm);
    }
    nrm = 1.0 / sqrt(nrm);
    for (int i = 0; i < n; i++) Q[i * ld + k] *= nrm;
}

// One solve with the stored LU, in place on column k.
__device__ __forceinline__ void invit_solve(int n, const InvitBufs& bf, double* __restrict__ Q, size_t ld, int k) {
    // forward: interchanges and multipliers
    double prev = Q[k];
    for (int i0 = 0; i0 < n - 1; i0 += INV_IB) {
        double nx[INV_IB], ml[INV_IB];
        unsigned char sw[INV_IB];
#pragma unroll
        for (int u = 0; u < INV_IB; u++)
            if (i0 + u < n - 1) {
                const size_t at = (size_t)(i0 + u) * ld + k;
                nx[u] = Q[at + ld];
                ml[u] = bf.ml[at];
                sw[u] = bf.sw[at];
            }
#pragma unroll
        for (int u = 0; u < INV_IB; u++)
            if (i0 + u < n - 1) {
                double next = nx[u];
                if (sw[u]) { double tmp = prev; prev = next; next = tmp; }
                Q[(size_t)(i0 + u) * ld + k] = prev;
                prev = next - ml[u] * prev;
            }
    }
    Q[(size_t)(n - 1) * ld + k] = prev;
    // back substitution
    double y2 = 0.0, y1 = prev / bf.u0[(size_t)(n - 1) * ld + k];
    Q[(size_t)(n - 1) * ld + k] = y1;
    for (int i0 = n - 2; i0 >= 0; i0 -= INV_IB) {
        double q[INV_IB], u0[INV_IB], u1[INV_IB], u2[INV_IB];
#pragma unroll
        for (int u = 0; u < INV_IB; u++)
            if (i0 - u >= 0) {
                const size_t at = (size_t)(i0 - u) * ld + k;
                q[u] = Q[at];
                u0[u] = bf.u0[at];
                u1[u] = bf.u1[at];
                u2[u] = bf.u2[at];
            }
#pragma unroll
        for (int u = 0; u < INV_IB; u++)
            if (i0 - u >= 0) {
                double y = (q[u] - u1[u] * y1 - u2[u] * y2) / u0[u];
                Q[(size_t)(i0 - u) * ld + k] = y;
                y2 = y1;
                y1 = y;
            }
    }
}

// Largest-modulus entry of column k made positive (lowest index on ties).
__device__ __forceinline__ void invit_sign(int n, double* __restrict__ Q, size_t ld, int k) {
    int imax = 0;
    double vmax = fabs(Q[k]);
    for (int i = 1; i < n; i++) {
        double a = fabs(Q[i * ld + k]);
        if (a > vmax) { vmax = a; imax = i; }
    }
    if (Q[imax * ld + k] < 0.0)
        for (int i = 0; i < n; i++) Q[i * ld + k] = -Q[i * ld + k];
}

// Cluster membership: eigenvalue k continues the cluster of k - 1 unless
// lambda[k-1] - lambda[k] > ctol.
__device__ __forceinline__ bool starts_cluster(const double* __restrict__ lambda, int k, double ctol) {
    return k == 0 || lambda[k - 1] - lambda[k] > ctol;
}

// Inverse iteration for the cluster led by eigenvalue k0 (nothing unless k0
// starts a cluster): vectors into Q[i * nev + k], LU rows in bf (same layout).
// One thread handles the whole cluster, orthogonalising each new vector
// against the cluster's earlier vectors after every solve.  singles_only:
// clusters of two or more are left to the lockstep cluster kernel.
__device__ __forceinline__ void invit_cluster(int n, int nev, const double* __restrict__ alpha,
                                              const double* __restrict__ lambda, double g, double ctol_rel,
                                              int maxit, const InvitBufs& bf, double* __restrict__ Q,
                                              int* __restrict__ fail, int k0, bool singles_only = false) {
    const double ctol = ctol_rel * g;
    if (!starts_cluster(lambda, k0, ctol)) return;  // not a cluster leader
    int k1 = k0 + 1;
    while (k1 < nev && !starts_cluster(lambda, k1, ctol)) k1++;
    if (singles_only && k1 - k0 > 1) return;
    const size_t ld = (size_t)nev;
    if (n == 1 || g == 0.0) {
        for (int k = k0; k < k1; k++)
            for (int i = 0; i < n; i++) Q[i * ld + k] = (i == k) ? 1.0 : 0.0;
        return;
    }
    const double eps = DBL_EPSILON;
    const double ptol = eps * g;
    const double grow = 1.0 / (100.0 * sqrt((double)n) * eps * g);
    for (int k = k0; k < k1; k++) {
        invit_lu(n, alpha, lambda[k], ptol, bf, ld, k);
        invit_start(n, Q, ld, k);
        bool conv = false, done = false;
        for (int it = 0; it < maxit && !done; it++) {
            invit_solve(n, bf, Q, ld, k);
            // orthogonalise against the earlier vectors of the cluster
            for (int p = k0; p < k; p++) {
                double d = 0.0;
                for (int i = 0; i < n; i++) d = fma(Q[i * ld + p], Q[i * ld + k], d);
                for (int i = 0; i < n; i++) Q[i * ld + k] = fma(-d, Q[i * ld + p], Q[i * ld + k]);
            }
            double nrm = 0.0;
            for (int i = 0; i < n; i++) { double y = Q[i * ld + k]; nrm = fma(y, y, nrm); }
            nrm = sqrt(nrm);
            if (!(nrm > 0.0) || !isfinite(nrm)) break;
            const double inv = 1.0 / nrm;
            for (int i = 0; i < n; i++) Q[i * ld + k] *= inv;
            if (conv) done = true;
            else if (nrm >= grow) conv = true;
        }
        if (!conv) atomicMin(fail, k);
        invit_sign(n, Q, ld, k);
    }
}

// ---- one eigenvector by a twisted factorisation ------------------------------
// (Fernando, "On computing an eigenvector of a tridiagonal matrix", 1997;
// Parlett and Dhillon 1997.)  With the pivots d+ of S - lambda I from the top
// (d+_i = -lambda - alpha_{i-1} l+_{i-1}, l+_i = alpha_i / d+_i) and d- from the
// bottom (l-_i = alpha_i / d-_{i+1}), gamma_i = -lambda - alpha_{i-1} l+_{i-1} -
// alpha_i l-_i; at r = argmin |gamma_i| the vector z_r = 1, z_i = -l+_i z_{i+1}
// above, z_{i+1} = -l-_i z_i below has residual |gamma_r| / |z| (no pivoting, no
// start vector), and lambda + gamma_r / |z|^2 is its Rayleigh quotient.  Two
// lanes a vector: lane half 0 runs downwards, half 1 upwards, the same
// instructions on mirrored rows; sixteen vectors a warp.  as: alpha scaled to
// g in [1, 2).
constexpr int TW_IB = 8;

// Reciprocal pivots Y (of row i) and ratios L (of edge i, i + 1) at shift lam,
// this lane's direction.
__device__ __forceinline__ void twist_factor(int n, const double* __restrict__ as, double lam, int half, double* Y,
                                             double* L, size_t ld, int k, bool live) {
    constexpr double PIV = 4.909093465297727e-91;  // 2^-300
    double d = -lam;
    for (int s0 = 0; s0 < n; s0 += TW_IB) {
        double al[TW_IB];
#pragma unroll
        for (int u = 0; u < TW_IB; u++) {
            const int s = s0 + u;
            al[u] = (s < n - 1) ? as[half ? n - 2 - s : s] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < TW_IB; u++) {
            const int s = s0 + u;
            if (s < n) {
                if (((__double2hiint(d) >> 20) & 0x7ff) <= 723) d = -PIV;  // |d| < 2^-299
                const double y = rcp_fast(d), l = al[u] * y;
                if (live) {
                    Y[(size_t)(half ? n - 1 - s : s) * ld + k] = y;
                    if (s < n - 1) L[(size_t)(half ? n - 2 - s : s) * ld + k] = l;
                }
                d = fma(-al[u], l, -lam);
            }
        }
    }
}

// argmin |gamma_i| over the rows (the lower on ties) and gamma there.
__device__ __forceinline__ int twist_index(int n, const double* __restrict__ as, double lam, int half,
                                           const double* Lp, const double* Lm, size_t ld, int k, double* gam) {
    const int h = (n + 1) / 2, lo = half ? h : 0, hi = half ? n : h;
    long long best = 0x7fffffffffffffffLL;
    double bg = 0.0;
    int br = lo;
    for (int i0 = 0; i0 < h; i0 += TW_IB) {
        double a[TW_IB], b[TW_IB], al[TW_IB + 1];
#pragma unroll
        for (int u = 0; u < TW_IB; u++) {
            const int i = min(lo + i0 + u, n - 1);
            a[u] = i > 0 ? Lp[(size_t)(i - 1) * ld + k] : 0.0;
            b[u] = i < n - 1 ? Lm[(size_t)i * ld + k] : 0.0;
        }
#pragma unroll
        for (int u = 0; u <= TW_IB; u++) {
            const int e = min(lo + i0 + u, n - 1) - 1;
            al[u] = e >= 0 ? as[min(e, n - 2)] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < TW_IB; u++) {
            const double gm = fma(-al[u + 1], b[u], fma(-al[u], a[u], -lam));
            const long long m = __double_as_longlong(gm) & 0x7fffffffffffffffLL;
            if (lo + i0 + u < hi && m < best) {
                best = m;
                bg = gm;
                br = lo + i0 + u;
            }
        }
    }
    const long long ob = __shfl_xor_sync(0xffffffffu, best, 16);
    const double og = __shfl_xor_sync(0xffffffffu, bg, 16);
    const int orow = __shfl_xor_sync(0xffffffffu, br, 16);
    if (ob < best || (ob == best && orow < br)) {
        bg = og;
        br = orow;
    }
    *gam = bg;
    return br;
}

// One step of inverse iteration with the factorisation twisted at r: on entry
// Z holds b; afterwards gamma_r Y y of N y = b on this lane's side
// (the forward part).  Returns y_r (both lanes).
__device__ __forceinline__ double twist_forward(int n, int r, int half, double gam, const double* Y, const double* L,
                                                double* Z, size_t ld, int k, bool live) {
    double y = 0.0;
    for (int s0 = 0; s0 < n - 1; s0 += TW_IB) {
        double l[TW_IB], yi[TW_IB], zi[TW_IB];
#pragma unroll
        for (int u = 0; u < TW_IB; u++) {
            const int s = min(s0 + u, n - 2), row = half ? n - 1 - s : s;
            zi[u] = Z[(size_t)row * ld + k];
            yi[u] = Y[(size_t)row * ld + k];
            l[u] = s > 0 ? L[(size_t)(half ? n - 1 - s : s - 1) * ld + k] : 0.0;  // edge to the previous row
        }
#pragma unroll
        for (int u = 0; u < TW_IB; u++) {
            const int s = s0 + u, row = half ? n - 1 - s : s;
            const bool act = s < n - 1 && (half ? row > r : row < r);
            if (!__any_sync(0xffffffffu, act)) continue;
            const double yn = fma(-l[u], y, zi[u]);
            if (act) {
                y = yn;
                if (live) Z[(size_t)row * ld + k] = yn * (yi[u] * gam);
            }
        }
    }
    // this lane's share of y_r
    const double br = Z[(size_t)r * ld + k];
    const bool has = half ? r < n - 1 : r > 0;
    const double mine = has ? L[(size_t)(half ? r : r - 1) * ld + k] * y : 0.0;
    const double other = __shfl_xor_sync(0xffffffffu, mine, 16);
    return half ? (br - other) - mine : (br - mine) - other;
}

// Z outwards from the twist index r with z_r = zr: z_i = (add ? Z_i : 0) -
// l z_{previous}.  Returns |z|^2 and the sign of the entry of largest modulus
// (the lowest on ties).
__device__ __forceinline__ double twist_vector(int n, int r, double zr, bool add, int half, const double* L, double* Z,
                                               size_t ld, int k, bool live, bool* neg) {
    double z = zr, nrm = half ? 0.0 : zr * zr;
    long long best = half ? -1 : (__double_as_longlong(zr) & 0x7fffffffffffffffLL);
    int bi = r;
    bool bneg = zr < 0.0;
    if (live && !half) Z[(size_t)r * ld + k] = zr;
    for (int s0 = 0; s0 < n - 1; s0 += TW_IB) {
        double l[TW_IB], t[TW_IB];
#pragma unroll
        for (int u = 0; u < TW_IB; u++) {
            const int s = min(s0 + u, n - 2), e = half ? s : n - 2 - s;  // edge between rows e and e + 1
            l[u] = L[(size_t)e * ld + k];
            t[u] = add ? Z[(size_t)(half ? e + 1 : e) * ld + k] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < TW_IB; u++) {
            const int e = half ? s0 + u : n - 2 - (s0 + u);
            const bool act = s0 + u < n - 1 && (half ? e >= r : e < r);
            if (!__any_sync(0xffffffffu, act)) continue;
            const double zn = fma(-l[u], z, t[u]);
            const double sq = fma(zn, zn, nrm);
            if (act) {
                z = zn;
                nrm = sq;
                const int row = half ? e + 1 : e;
                if (live) Z[(size_t)row * ld + k] = z;
                const long long m = __double_as_longlong(z) & 0x7fffffffffffffffLL;
                if (m > best || (m == best && row < bi)) {
                    best = m;
                    bi = row;
                    bneg = __double_as_longlong(z) < 0;
                }
            }
        }
    }
    const long long ob = __shfl_xor_sync(0xffffffffu, best, 16);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, 16);
    const int on = __shfl_xor_sync(0xffffffffu, (int)bneg, 16);
    if (ob > best || (ob == best && oi < bi)) bneg = on != 0;
    *neg = bneg;
    // the same sum on both lanes of a pair
    const double other = __shfl_xor_sync(0xffffffffu, nrm, 16);
    return half ? other + nrm : nrm + other;
}

// Inverse iteration in double-float (about 2^-44 relative; Dekker's pair
// arithmetic runs at FP32 latency, the FP64 division chain here is about ten
// times longer): for a caller that refines the vectors afterwards.  The steps
// are those of the FP64 routines with the pivot floor and growth threshold
// taken at 2^-44; the LU rows and the vectors are kept as FP32 pairs in the
// same buffers, and the vectors are converted to FP64 at the end.  alpha as a
// pair: alh + all_.
struct InvitDf {
    Df *U0, *U1, *U2, *ML, *Qd;
    unsigned char* sw;
};
__device__ __forceinline__ InvitDf invit_df_view(const InvitBufs& bf, double* Q) {
    return {reinterpret_cast<Df*>(bf.u0), reinterpret_cast<Df*>(bf.u1), reinterpret_cast<Df*>(bf.u2),
            reinterpret_cast<Df*>(bf.ml), reinterpret_cast<Df*>(Q), bf.sw};
}

// drop: couplings below it count as zero (the blocks they leave each have a null
// vector of their own; couplings at rounding level would grow one past all others).
__device__ __forceinline__ void invit_lu_df(int n, const float* __restrict__ alh, const float* __restrict__ all_,
                                            double lam, float ptol, float drop, const InvitDf& v, size_t ld, int k) {
    const Df zero = {0.f, 0.f};
    const Df mlam = df_neg(df_of(lam));
    auto edge = [&](int i) { return fabsf(alh[i]) < drop ? zero : Df{alh[i], all_[i]}; };
    Df a0 = mlam, a1 = edge(0);
    for (int i = 0; i < n - 1; i++) {
        const Df l = edge(i);
        const Df un = (i + 1 < n - 1) ? edge(i + 1) : zero;
        const size_t at = i * ld + k;
        if (fabsf(a0.h) >= fabsf(l.h)) {
            Df piv = a0;
            if (fabsf(piv.h) < ptol) piv = {(piv.h < 0.f) ? -ptol : ptol, 0.f};
            const Df m = df_div(l, piv);
            v.U0[at] = piv; v.U1[at] = a1; v.U2[at] = zero; v.sw[at] = 0; v.ML[at] = m;
            a0 = df_add(mlam, df_neg(df_mul(m, a1)));
            a1 = un;
        } else {
            const Df m = df_div(a0, l);
            v.U0[at] = l; v.U1[at] = mlam; v.U2[at] = un; v.sw[at] = 1; v.ML[at] = m;
            const Df na0 = df_add(a1, df_neg(df_mul(m, mlam)));
            a1 = df_neg(df_mul(m, un));
            a0 = na0;
        }
    }
    if (fabsf(a0.h) < ptol) a0 = {(a0.h < 0.f) ? -ptol : ptol, 0.f};
    const size_t at = (size_t)(n - 1) * ld + k;
    v.U0[at] = a0; v.U1[at] = zero; v.U2[at] = zero;
}

__device__ __forceinline__ void invit_scale_df(int n, Df* __restrict__ Qd, size_t ld, int k, Df s) {
    for (int i0 = 0; i0 < n; i0 += INV_IB) {
        Df x[INV_IB];
#pragma unroll
        for (int u = 0; u < INV_IB; u++)
            if (i0 + u < n) x[u] = Qd[(size_t)(i0 + u) * ld + k];
#pragma unroll
        for (int u = 0; u < INV_IB; u++)
            if (i0 + u < n) Qd[(size_t)(i0 + u) * ld + k] = df_mul(x[u], s);
    }
}

// the FP64 routine's start vector, norm in FP32
__device__ __forceinline__ void invit_start_df(int n, Df* __restrict__ Qd, size_t ld, int k) {
    float nrm = 0.f;
    for (int i = 0; i < n; i++) {
        const Df x = df_of(splitmix_uniform((unsigned long long)k + 1ULL, (unsigned long long)i));
        Qd[i * ld + k] = x;
        nrm = fmaf(x.h, x.h, nrm);
    }
    invit_scale_df(n, Qd, ld, k, {1.0f / sqrtf(nrm), 0.f});
}

__device__ __forceinline__ void invit_solve_df(int n, const InvitDf& v, size_t ld, int k) {
    const Df zero = {0.f, 0.f};
    Df* Qd = v.Qd;
    // forward: interchanges and multipliers
    Df prev = Qd[k];
    for (int i0 = 0; i0 < n - 1; i0 += INV_IB) {
        Df nx[INV_IB], ml[INV_IB];
        unsigned char sw[INV_IB];
#pragma unroll
        for (int u = 0; u < INV_IB; u++)
            if (i0 + u < n - 1) {
                const size_t at = (size_t)(i0 + u) * ld + k;
                nx[u] = Qd[at + ld];
                ml[u] = v.ML[at];
                sw[u] = v.sw[at];
            }
#pragma unroll
        for (int u = 0; u < INV_IB; u++)
            if (i0 + u < n - 1) {
                Df next = nx[u];
                if (sw[u]) { const Df tmp = prev; prev = next; next = tmp; }
                Qd[(size_t)(i0 + u) * ld + k] = prev;
                prev = df_add(next, df_neg(df_mul(ml[u], prev)));
            }
    }
    // back substitution
    Df y2 = zero, y1 = df_div(prev, v.U0[(size_t)(n - 1) * ld + k]);
    Qd[(size_t)(n - 1) * ld + k] = y1;
    for (int i0 = n - 2; i0 >= 0; i0 -= INV_IB) {
        Df q[INV_IB], u0[INV_IB], u1[INV_IB], u2[INV_IB];
#pragma unroll
        for (int u = 0; u < INV_IB; u++)
            if (i0 - u >= 0) {
                const size_t at = (size_t)(i0 - u) * ld + k;
                q[u] = Qd[at];
                u0[u] = v.U0[at];
                u1[u] = v.U1[at];
                u2[u] = v.U2[at];
            }
#pragma unroll
        for (int u = 0; u < INV_IB; u++)
            if (i0 - u >= 0) {
                const Df r = df_add(q[u], df_neg(df_add(df_mul(u1[u], y1), df_mul(u2[u], y2))));
                const Df y = df_div(r, u0[u]);
                Qd[(size_t)(i0 - u) * ld + k] = y;
                y2 = y1;
                y1 = y;
            }
    }
}

// FP32 Sturm count of the scaled matrix S / g at x (|x| ~ 1): the recurrence
// of sturm() with pivots below FLT_MIN raised to FLT_MIN.
__device__ __forceinline__ int sturm32(int n, const float* __restrict__ a2s, float x) {
    int cnt = 0;
    float d = -x;
    if (fabsf(d) < FLT_MIN) d = -FLT_MIN;
    cnt += (d < 0.f);
    for (int i = 1; i < n; i++) {
        d = -x - __fdividef(a2s[i - 1], d);
        if (fabsf(d) < FLT_MIN) d = -FLT_MIN;
        cnt += (d < 0.f);
    }
    return cnt;
}

template <int L>
__device__ __forceinline__ unsigned lane_group(int lane) {
    return L == 32 ? 0xffffffffu : ((1u << (L & 31)) - 1u) << (lane & ~(L - 1));
}

// Bracketing pass in FP32 (64 times the FP64 rate on this part): L lanes
// per wanted eigenvalue multisect [-1, 1] for S / g down to 8 eps32.  A
// floating-point Sturm count is the exact count of a matrix whose entries are
// perturbed by a few units of roundoff (Kahan), so lambda_j lies within a few
// eps32 g of the FP32 bracket; the FP64 pass widens it by FP32_SLACK eps32 g
// and checks it with FP64 counts before trusting it.
template <int L>
__device__ __forceinline__ void bisect32_body(int n, int k, int q, int lane, const float* __restrict__ a2s,
                                              double* __restrict__ lohi) {
    const unsigned gmask = lane_group<L>(lane);
    const int j = n - 1 - k;
    float lo = -1.0f - 4.0f * FLT_EPSILON, hi = 1.0f + 4.0f * FLT_EPSILON;
    for (int it = 0; it < 64; it++) {
        const float w = hi - lo;
        if (w <= 8.0f * FLT_EPSILON) break;
        const float step = w * (1.0f / (L + 1));
        const float x = lo + (float)(q + 1) * step;
        const bool le = (x > lo && x < hi) ? (sturm32(n, a2s, x) <= j) : (x <= lo);
        const int nle = __popc(__ballot_sync(gmask, le) & gmask);
        const float nlo = (nle > 0) ? lo + (float)nle * step : lo;
        const float nhi = (nle < L) ? lo + (float)(nle + 1) * step : hi;
        if (!(nlo > lo || nhi < hi)) break;
        lo = nlo;
        hi = (nhi < hi) ? nhi : hi;
    }
    if (q == 0) {
        lohi[2 * k] = (double)lo;  // in units of g
        lohi[2 * k + 1] = (double)hi;
    }
}

constexpr double FP32_SLACK = 64.0;
// FP64 multisection on the zero-diagonal form (B B^T at x^2, m = ceil(n/2)
// steps; the wanted eigenvalues are >= 0, so the search stays in [0, g]),
// straight from the FP32 bracket.  The first step's points span the bracket
// widened by FP32_SLACK eps32 g; an eigenvalue outside them leaves the interval
// to the end of [0, g] on that side, so the bracket need not be trusted.
// Bound by the FP64 instructions of one chain (6 x 64 clocks a step when a
// scheduler has one warp), so L is the largest power of two that still gives
// every warp a scheduler of its own: 12 three-section steps from a
// double-float bracket took 3.3 ms at n = 500, nev = 250 with the passes
// before it.
template <int L>
__device__ __forceinline__ void bisect_bd_body(int n, int k, int q, int lane, const TriScalars* sc,
                                               const double* __restrict__ lohi, double* __restrict__ lambda,
                                               const double* __restrict__ a2e, const double* __restrict__ b2e) {
    const unsigned gmask = lane_group<L>(lane);
    const int m = (n + 1) / 2, j = m - 1 - k;
    if (n == 1 || sc->g == 0.0) {
        if (q == 0) lambda[k] = 0.0;
        return;
    }
    const double gs = sc->g * sc->down;  // in [1, 2)
    const double ghi = gs + 2.0 * DBL_EPSILON * gs;
    const double slack = FP32_SLACK * FLT_EPSILON * gs;
    double lo = 0.0, hi = ghi;
    // the first points: a, ..., b inclusive
    double a = fmax(0.0, lohi[2 * k] * gs - slack), step = (fmin(ghi, lohi[2 * k + 1] * gs + slack) - a) / (double)(L - 1);
    bool first = true;
    for (int it = 0; it < 4000; it++) {
        const double w = hi - lo;
        const double tol = 2.0 * DBL_EPSILON * hi + 1e-300;
        if (!(w > tol)) break;
        if (!first) {
            step = w / (double)(L + 1);
            a = lo + step;
        }
        const double x = a + (double)q * step;
        const bool le = (x > lo && x < hi) ? (bd_count_scaled(m, a2e, b2e, x * x) <= j) : (x <= lo);
        const int nle = __popc(__ballot_sync(gmask, le) & gmask);
        const double nlo = (nle > 0) ? fmax(lo, a + (double)(nle - 1) * step) : lo;
        const double nhi = (nle < L) ? fmin(hi, a + (double)nle * step) : hi;
        if (!first && !(nlo > lo || nhi < hi)) break;
        first = false;
        lo = nlo;
        hi = nhi;
    }
    if (q == 0) lambda[k] = (lo + 0.5 * (hi - lo)) * sc->up;
}

// ---- lockstep inverse iteration of clusters ---------------------------------
// A cluster (two or more eigenvalues closer than ctol) is iterated in lockstep
// rather than by one thread: in every iteration each member solves with its
// own LU on its own thread, then the cluster's CTA orthogonalises the members
// in index order (modified Gram-Schmidt, parallel over the rows), normalises
// them and applies the growth test to each; the cluster stops one iteration
// after all its members passed.  The vectors are an orthonormal basis of the
// same invariant subspace, and the critical path is one member's solves
// instead of the whole cluster's (16 x at the 1e-10 clusters of a clustered
// spectrum).  Singletons keep the one-thread path.
constexpr int CLU_T = 256;

// Clusters come in two kinds.  Where all neighbouring gaps exceed TIGHT g each
// member's own vector (twist_kernel) is accurate to about eps / TIGHT, and
// one modified Gram-Schmidt pass orthogonalises the members: the overlaps it
// removes are eps g / gap, which moves a residual by eps g only.  Tight
// clusters (or ones with a member that failed the residual test, need[2 k] !=
// 0) go through the lockstep iteration.
constexpr double TIGHT = 1e-9;

__device__ __forceinline__ bool clu_tight(const double* lambda, const double* need, double g, int k0, int m) {
    for (int j = 0; j < m; j++)
        if (need[2 * (k0 + j)] != 0.0 || (j + 1 < m && !(lambda[k0 + j] - lambda[k0 + j + 1] > TIGHT * g))) return true;
    return false;
}

// Row of the largest abs(x_i) (the lowest on ties), CTA-wide.
template <class F>
__device__ __forceinline__ int block_argmax(int n, F absval, double* rv, int* ri) {
    double best = -1.0;
    int bi = 0x7fffffff;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double a = absval(i);
        if (a > best) {
            best = a;
            bi = i;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) {
            best = ob;
            bi = oi;
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) {
        rv[warp] = best;
        ri[warp] = bi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < nw; w++)
            if (rv[w] > rv[0] || (rv[w] == rv[0] && ri[w] < ri[0])) {
                rv[0] = rv[w];
                ri[0] = ri[w];
            }
    }
    __syncthreads();
    const int r = ri[0];
    __syncthreads();
    return r < n ? r : 0;
}

// The Gram-Schmidt pass of a loose cluster: members in index order, each
// normalised, its largest-modulus entry positive.
__device__ __forceinline__ void clu_mgs(int n, size_t ld, double* Q, int k0, int m, double* red, int* redi) {
    const int t = threadIdx.x, T = blockDim.x;
    for (int j = 0; j < m; j++) {
        double* qj = Q + k0 + j;
        for (int p = 0; p < j; p++) {
            const double* qp = Q + k0 + p;
            double d = 0.0;
            for (int i = t; i < n; i += T) d = fma(qp[i * ld], qj[i * ld], d);
            d = sk_block_sum(d, red);
            for (int i = t; i < n; i += T) qj[i * ld] = fma(-d, qp[i * ld], qj[i * ld]);
            __syncthreads();
        }
        double s = 0.0;
        for (int i = t; i < n; i += T) s = fma(qj[i * ld], qj[i * ld], s);
        s = sk_block_sum(s, red);
        const int imax = block_argmax(n, [&](int i) { return fabs(qj[i * ld]); }, red, redi);
        const double f = (qj[imax * ld] < 0.0 ? -1.0 : 1.0) / sqrt(s);
        __syncthreads();
        for (int i = t; i < n; i += T) qj[i * ld] *= f;
        __syncthreads();
    }
}

// Eigenvalues near 0 before a refinement.  It works on the basis [Z, conj(Z)], so
// the halves of a vector on the even and on the odd rows (real and imaginary part
// of D q) have to be of norm 2^-1/2, and orthogonal to those of every other
// vector, each by itself, as they are for an exact lambda > 0.  An eigenvalue
// known to 2^-43 g leaves a mixture of the vectors of lambda and -lambda where
// lambda is no larger: below PAIR_TOL g the halves are scaled (and in a cluster
// orthogonalised) by themselves.  At NULL_TOL g and below, where it may be 0, the
// shift is 0, with which a solve keeps the halves apart, and the lockstep
// iteration takes single eigenvalues too.
constexpr double PAIR_TOL = 0x1p-20, NULL_TOL = 0x1.8p-43;

// Decision after an iteration: state 0 iterating, 1 all members passed (one
// more iteration), 2 done.  ff = first member that failed the growth test
// (m if none), bad = a member's norm was zero or not finite.
__device__ __forceinline__ int clu_next_state(int st, int ff, int m, int bad, int it, int maxit, bool& fin,
                                              bool& failed) {
    int nst = (st == 1) ? 2 : (ff == m ? 1 : 0);
    if (bad) nst = 0;
    fin = bad || nst == 2 || it == maxit - 1;
    failed = fin && nst == 0;
    return nst;
}

constexpr double LOST = 2.0;  // need[2 k] of a member to be started again

// One cluster (k0, m) by the CTA.
__device__ __forceinline__ void clu_body(int n, int nev, int k0, int m, const double* alpha, const double* lambda,
                                         double g, int maxit, const InvitBufs& bf, double* Q, double* need,
                                         int* fail) {
    __shared__ double red[32];
    __shared__ int redi[32];
    __shared__ int s_ff, s_bad;
    const size_t ld = (size_t)nev;
    const double eps = DBL_EPSILON, ptol = eps * g;
    const double grow = 1.0 / (100.0 * sqrt((double)n) * eps * g);
    const int t = threadIdx.x, T = blockDim.x;
    if (n == 1 || g == 0.0) {
        for (int e = t; e < m * n; e += T) {
            const int j = e / n, i = e % n;
            Q[i * ld + k0 + j] = (i == k0 + j) ? 1.0 : 0.0;
        }
        return;
    }
    if (!clu_tight(lambda, need, g, k0, m)) {
        clu_mgs(n, ld, Q, k0, m, red, redi);
        return;
    }
    // the cluster's iterations one after another; st (clu_next_state) is
    // the same in every thread
    int st = 0;
    for (int it = 0; it < maxit && st != 2; it++) {
        // the members' solves, one thread each
        for (int j = t; j < m; j += T) {
            const int k = k0 + j;
            if (it == 0 || need[2 * k] == LOST) {
                invit_lu(n, alpha, lambda[k], ptol, bf, ld, k, it == 0 ? 0.0 : ptol);
                invit_start(n, Q, ld, k);
                need[2 * k] = 1.0;
            }
            invit_solve(n, bf, Q, ld, k);
        }
        if (t == 0) {
            s_ff = m;
            s_bad = 0;
        }
        __syncthreads();
        // modified Gram-Schmidt in index order, normalisation, growth test
        for (int j = 0; j < m; j++) {
            double* qj = Q + k0 + j;
            // a second pass where the first left less than a tenth of the vector:
            // the rounding of what it took off is then not orthogonal
            double s = 0.0;
            bool lost = false;
            for (int pass = 0; pass < 2; pass++) {
                double off = 0.0;
                for (int p = 0; p < j; p++) {
                    const double* qp = Q + k0 + p;
                    double d = 0.0;
                    for (int i = t; i < n; i += T) d = fma(qp[i * ld], qj[i * ld], d);
                    d = sk_block_sum(d, red);
                    for (int i = t; i < n; i += T) qj[i * ld] = fma(-d, qp[i * ld], qj[i * ld]);
                    off = fma(d, d, off);
                    __syncthreads();
                }
                s = 0.0;
                for (int i = t; i < n; i += T) s = fma(qj[i * ld], qj[i * ld], s);
                s = sk_block_sum(s, red);
                if (!(s < 1e-2 * off)) break;  // the same in every thread
                lost = lost || s < 1e-14 * off;
            }
            // nothing left but rounding: one direction outgrows the others through
            // couplings at rounding level, so this member starts again without them
            if (lost && t == 0) {
                need[2 * (k0 + j)] = LOST;
                s_ff = min(s_ff, j);
            }
            const double nrm = sqrt(s);
            if (!(nrm > 0.0) || !isfinite(nrm)) {
                if (t == 0) {
                    s_bad = 1;
                    s_ff = min(s_ff, j);
                }
            } else {
                const double inv = 1.0 / nrm;
                for (int i = t; i < n; i += T) qj[i * ld] *= inv;
                if (t == 0 && !(nrm >= grow)) s_ff = min(s_ff, j);
            }
            __syncthreads();
        }
        bool fin, failed;
        const int nst = clu_next_state(st, s_ff, m, s_bad, it, maxit, fin, failed);
        if (failed && t == 0) atomicMin(fail, k0 + s_ff);
        if (fin) {
            // largest-modulus entry of each vector positive (lowest index on ties)
            for (int j = 0; j < m; j++) {
                double* qj = Q + k0 + j;
                const int imax = block_argmax(n, [&](int i) { return fabs(qj[i * ld]); }, red, redi);
                const bool neg = qj[imax * ld] < 0.0;  // read by all before any flip
                __syncthreads();
                if (neg)
                    for (int i = t; i < n; i += T) qj[i * ld] = -qj[i * ld];
                __syncthreads();
            }
        }
        st = fin ? 2 : nst;
        __syncthreads();
    }
}

// Vectors of the eigenvalues that are alone within ctol, and of the members
// of loose clusters.  polish: eigenvalues
// accurate to rounding; the twisted vector is followed by one step of inverse
// iteration with the same factorisation, which removes the share of the
// neighbours that the rounding of lambda leaves in it (orthogonality 3.2 n eps
// without it and 0.3 with it at n = 1001).  Otherwise eigenvalues known to
// 2^-42 g: a second factorisation at the Rayleigh quotient of the first one's
// vector (the caller refines).  A vector whose residual is above 100 sqrt(n)
// eps g (the growth test of inverse iteration) is handed to the pivoted
// inverse iteration.  About 14 FP64 instructions a row and vector, one warp a scheduler.
__device__ __forceinline__ void twist_body(int n, int nev, int kb, int lane, const double* __restrict__ as,
                                           const double* __restrict__ alpha, const double* __restrict__ lambda,
                                           const TriScalars* sc, double ctol_rel, int maxit, int polish,
                                           const InvitBufs& bf, double* Q, double* __restrict__ need,
                                           int* __restrict__ fail) {
    const int half = lane >> 4;
    const int kk = kb + (lane & 15), k = min(kk, nev - 1);
    const double g = sc->g, ctol = ctol_rel * g;
    const size_t ld = (size_t)nev;
    const bool single = starts_cluster(lambda, k, ctol) && (k + 1 >= nev || starts_cluster(lambda, k + 1, ctol));
    const double tight = TIGHT * g;
    const bool null = !polish && lambda[k] <= NULL_TOL * g;  // left to the lockstep iteration
    const bool live = kk < nev && !null && (single || (starts_cluster(lambda, k, tight) &&
                                              (k + 1 >= nev || starts_cluster(lambda, k + 1, tight))));
    if (kk < nev && !half) need[2 * k] = live ? 0.0 : 1.0;
    if (!__any_sync(0xffffffffu, live)) return;
    if (n == 1 || g == 0.0) {
        if (live && !half)
            for (int i = 0; i < n; i++) Q[i * ld + k] = (i == k) ? 1.0 : 0.0;
        return;
    }
    double* Y = half ? bf.u1 : bf.u0;
    double* L = half ? bf.ml : bf.u2;
    double lam = lambda[k] * sc->down, gam = 0.0;
    bool neg = false;
    twist_factor(n, as, lam, half, Y, L, ld, k, live);
    __syncwarp();
    int r = twist_index(n, as, lam, half, bf.u2, bf.ml, ld, k, &gam);
    double nrm = twist_vector(n, r, 1.0, false, half, L, Q, ld, k, live, &neg), res;
    __syncwarp();
    if (polish) {
        const double n0 = nrm, yr = twist_forward(n, r, half, gam, Y, L, Q, ld, k, live);
        __syncwarp();
        nrm = twist_vector(n, r, yr, true, half, L, Q, ld, k, live, &neg);
        // of an eigenvector the solve grows it by n or so; without a pivot of
        // size it can grow by any factor, and the residual below says nothing
        res = nrm <= 1e6 * n * n * n0 ? fabs(gam) * sqrt(n0 / nrm) : INFINITY;
    } else {
        const double dl = gam / nrm;
        if (fabs(dl) < 1e-9) lam += dl;
        twist_factor(n, as, lam, half, Y, L, ld, k, live);
        __syncwarp();
        r = twist_index(n, as, lam, half, bf.u2, bf.ml, ld, k, &gam);
        nrm = twist_vector(n, r, 1.0, false, half, L, Q, ld, k, live, &neg);
        res = fabs(gam) / sqrt(nrm);
    }
    const double inv = (neg ? -1.0 : 1.0) / sqrt(nrm);
    double inv_e = inv, inv_o = inv;  // of the even and the odd rows
    const bool pair = !polish && live && lambda[k] <= PAIR_TOL * g;
    if (__any_sync(0xffffffffu, pair)) {
        __syncwarp();
        double mine = 0.0;  // lane half 0 the even rows, 1 the odd ones
        for (int i = half; i < n; i += 2) {
            const double z = live ? Q[(size_t)i * ld + k] : 0.0;
            mine = fma(z, z, mine);
        }
        const double other = __shfl_xor_sync(0xffffffffu, mine, 16);
        if (pair) {
            inv_e = (neg ? -1.0 : 1.0) / sqrt(2.0 * (half ? other : mine));
            inv_o = (neg ? -1.0 : 1.0) / sqrt(2.0 * (half ? mine : other));
        }
    }
    const double gs = g * sc->down;
    // (an overflowed norm has inv = 0)
    const bool ok = maxit > 0 && inv != 0.0 && isfinite(inv_e) && isfinite(inv_o) &&
                    res <= 100.0 * sqrt((double)n) * DBL_EPSILON * gs;
    __syncwarp();
    const int h = (n + 1) / 2, lo = half ? h : 0, hi = half ? n : h;
    if (live && ok) {
        for (int i0 = lo; i0 < hi; i0 += TW_IB) {
            double z[TW_IB];
#pragma unroll
            for (int u = 0; u < TW_IB; u++)
                if (i0 + u < hi) z[u] = Q[(size_t)(i0 + u) * ld + k];
#pragma unroll
            for (int u = 0; u < TW_IB; u++)
                if (i0 + u < hi) Q[(size_t)(i0 + u) * ld + k] = z[u] * ((i0 + u) & 1 ? inv_o : inv_e);
        }
    }
    if (live && !ok && !half) need[2 * k] = 1.0;
    if (live && !ok && !half && single) invit_cluster(n, nev, alpha, lambda, g, ctol_rel, maxit, bf, Q, fail, k, true);
}

}  // namespace tri
}  // namespace sk
