// onestep_sym.cu -- the direct tridiagonalisation (onestep.cu) for orders whose
// matrix lives in memory: only the lower triangle is kept.
//
// A full matrix with whole rows per CTA needs one exchange a column, but every
// element is held, updated and moved twice.  Here the lower triangle is cut
// into units of 32 or 64 rows x 64 columns; four warps, one per scheduler, update a
// unit (A += sigma (u p^T - p u^T)) and take both of its products with x, the row sums and, negated,
// the column sums, so an element costs 4 operations and 16 bytes for its two
// places instead of 6 and 32.  The partial sums need a second exchange:
//   1. pass over the units, partial sums to memory; exchange;
//   2. the owner of 32 indices adds their partial sums (q = A x), forms p = q -
//      beta a and the next column x = a + sigma (u p_c - p u_c), and publishes
//      u, p, x and its share of |x|^2; exchange.
// p_c is one element: every CTA adds its partial sums by itself, and beta comes
// from the shares of the norm, added while the pass runs.  Two forms: FP64, and
// pairs of floats (onestep_df.cu) where the refinement follows.
#include <algorithm>
#include <cfloat>

#include "common.cuh"
#include "internal.h"
#include "onestep_dev.cuh"
#include "pairs.cuh"

namespace sk {

using namespace onestep;

namespace {

constexpr int UC = 64;  // columns of a unit and indices of a block
constexpr int ST = 512, SW = ST / 32, SG = SW / 4;  // threads, warps, groups of four warps

struct F64 {
    using V = double;
    static SK_DEV V zero() { return 0.0; }
    static SK_DEV void mac(V& a, V c, V d) { a = fma(c, d, a); }
    static SK_DEV V norm(V a) { return a; }
    static SK_DEV V sum(V a, V b) { return a + b; }
    static SK_DEV V mul(V a, V b) { return a * b; }
    static SK_DEV V prod(V a, V b) { return a * b; }
    static SK_DEV V neg(V a) { return -a; }
    static SK_DEV V scale(V a, float) { return a; }
    static SK_DEV V one() { return 1.0; }
    static SK_DEV V shfl_xor(V a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
    static SK_DEV V bcast(V a, int l) { return __shfl_sync(0xffffffffu, a, l); }
    static SK_DEV V from(double x) { return x; }
    static SK_DEV double to(V a) { return a; }
    static SK_DEV float lead(V) { return 1.f; }
    static SK_DEV bool positive(V a) { return os_tail(a); }
    static SK_DEV double prescale(unsigned long long amax) { return os_scale(amax); }
    static SK_DEV bool nonneg(V a) { return a >= 0.0; }
    static SK_DEV V root(V a) { return sqrt(a); }
    static SK_DEV V quot(V a, V b) { return a / b; }
    static constexpr bool scaled = false;
    static constexpr int UR = 32;  // rows of a unit
};
struct DfPair {
    using V = float2;
    static SK_DEV V zero() { return make_float2(0.f, 0.f); }
    static SK_DEV void mac(V& a, V c, V d) { df_mac(a, c, d); }
    static SK_DEV V norm(V a) { return df_norm(a); }
    static SK_DEV V sum(V a, V b) { return df_sum(a, b); }
    static SK_DEV V mul(V a, V b) { return df_mul2(a, b); }
    static SK_DEV V prod(V a, V b) { return df_prod(a, b); }
    static SK_DEV V neg(V a) { return df_neg2(a); }
    static SK_DEV V scale(V a, float s) { return df_scale(a, s); }
    static SK_DEV V one() { return make_float2(1.f, 0.f); }
    static SK_DEV V shfl_xor(V a, int o) { return df_shfl(a, o); }
    static SK_DEV V bcast(V a, int l) {
        return make_float2(__shfl_sync(0xffffffffu, a.x, l), __shfl_sync(0xffffffffu, a.y, l));
    }
    static SK_DEV V from(double x) { return df_from(x); }
    static SK_DEV double to(V a) { return df_to(a); }
    static SK_DEV float lead(V a) { return fabsf(a.x); }
    static SK_DEV bool positive(V a) { return a.x > 0.f; }
    static SK_DEV double prescale(unsigned long long amax) {
        const int e = (int)(amax >> 52);
        return amax == 0 ? 1.0 : ldexp(1.0, max(-1000, min(1000, 1022 - e)));
    }
    static SK_DEV bool nonneg(V a) { return a.x >= 0.f; }
    static SK_DEV V root(V a) { return df_root(a); }
    static SK_DEV V quot(V a, V b) { return df_quot(a, b); }
    static constexpr bool scaled = true;
    static constexpr int UR = 64;  // the vectors' loads of a unit take as long as 16 rows a warp
};

template <class V>
struct alignas(16) Two {
    V a, b;
};
template <class V>
SK_DEV Two<V> ld2(const V* p) {
    static_assert(sizeof(Two<V>) == 16, "two elements of 8 bytes");
    const float4 f = __ldcg(reinterpret_cast<const float4*>(p));
    Two<V> r;
    memcpy(&r, &f, 16);
    return r;
}
template <class V>
SK_DEV V ld1(const V* p) {
    const float2 f = __ldcg(reinterpret_cast<const float2*>(p));
    V r;
    memcpy(&r, &f, 8);
    return r;
}

// First unit of column block J of T; it has rb (T - J) units (rb row blocks per 64).
__host__ __device__ inline long long unit_base(int rb, int T, int J) { return (long long)J * (2 * T - J + 1) * rb / 2; }

template <class V>
struct SymArgs {
    int n, T;            // order, column blocks of 64
    V* tiles;            // units [J][I]: UR rows of 64, j < i only (0 elsewhere)
    V *x, *u, *p;        // 64 T each, 0 for retired indices
    V *prow, *pcol;      // partial sums [I][J][UR], [J][I][64]
    V* nrm;              // shares of |x|^2, one per 32 indices, scaled by the square of ...
    float* nsc;          // ... this power of two
    V* Vout;             // reflectors by columns (ld n), zeroed by the caller
    double *tau, *alpha;
    const double* scale; // A was multiplied by scale[0]
    unsigned* ctr;
    int* status;
    unsigned cap;
};

// Power of two 2^-e for |a| in [2^e, 2^(e + 1)), 0 below 2^-110.
SK_DEV float inv_pow2(float a) {
    return a > 7.7e-34f ? __int_as_float((254 << 23) - (__float_as_int(a) & 0x7f800000)) : 0.f;
}

template <class Op>
__global__ void __launch_bounds__(ST, 1) onestep_sym_kernel(SymArgs<typename Op::V> o) {
    using V = typename Op::V;
    constexpr int UR = Op::UR, RB = UC / UR, WR = UR / 4;  // row blocks per 64, rows of a warp
    __shared__ V s_grp[SW][32];
    __shared__ V s_col[2][SW][UC];  // column sums of the warps of a unit, double-buffered
    __shared__ V s_q0[2 * 256 + 4];  // the partial sums of one element (n <= 16384)
    __shared__ V s_q0v, s_beta, s_sigma, s_inv, s_u0;
    __shared__ float s_us;
    __shared__ int s_next, s_unit[2][SG];
    const int n = o.n, T = o.T, G = gridDim.x, g = blockIdx.x;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const double unscale = 1.0 / o.scale[0];
    unsigned epoch = 0;
    V sigma = Op::zero();  // of the pending update
    // publishes x_i (one index a lane of warp 0) and their share of the norm
    // without the pivot index
    auto publish_x = [&](int i, int pivot, V xi) {
        o.x[i] = xi;
        const V y = i == pivot ? Op::zero() : xi;
        float sc = 1.f;
        if (Op::scaled) {
            float mx = Op::lead(y);
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
            sc = inv_pow2(mx);
        }
        V s = Op::zero();
        const V ys = Op::scale(y, sc);
        Op::mac(s, ys, ys);
        s = Op::norm(s);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) s = Op::sum(s, Op::shfl_xor(s, d));
        if (lane == 0) {
            o.nrm[i >> 5] = s;
            o.nsc[i >> 5] = sc;
        }
    };
    // element (i, c) of the lower triangle, i > c
    auto element = [&](int i, int c) -> V {
        const int J = c / UC, I = i / UR;
        return ld1(o.tiles + ((unit_base(RB, T, J) + I - RB * J) * UR + (i & (UR - 1))) * UC + (c & (UC - 1)));
    };
    if (t == 0) s_next = 0;
    // column 0
    for (int b = g; b < 2 * T; b += G)
        if (t < 32) {
            const int i = b * 32 + t;
            publish_x(i, 1, i >= 1 && i < n ? element(i, 0) : Op::zero());
        }
    if (!sk_grid_barrier(o.ctr, epoch, o.status, o.cap)) return;
    for (int k = 0; k + 2 < n; k++) {
        const int J0 = (k + 1) / UC, Ta = T - J0;
        // ---- beta, sigma of x_k from the shares of its norm (one warp, before its
        // group takes units)
        if (warp == SW - 1) {
            const V x0 = ld1(o.x + k + 1);
            // all shares at once (one trip to L2, not one per 32 of them)
            constexpr int NS = 8;
            V s2 = Op::zero();
            float sc = 0.f;  // the scale s2 carries (0: nothing added yet)
            for (int b0 = 2 * J0; b0 < 2 * T; b0 += 32 * NS) {
                V sh[NS];
                float ss[NS];
#pragma unroll
                for (int h = 0; h < NS; h++) {
                    const int b = b0 + lane + 32 * h;
                    sh[h] = b < 2 * T ? ld1(o.nrm + b) : Op::zero();
                    ss[h] = Op::scaled && b < 2 * T ? __ldcg(o.nsc + b) : 0.f;
                }
                if (Op::scaled) {
                    // the largest entry has the smallest scale
                    float mn = sc > 0.f ? sc : 3e38f;
#pragma unroll
                    for (int h = 0; h < NS; h++)
                        if (ss[h] > 0.f) mn = fminf(mn, ss[h]);
                    const float own = inv_pow2(Op::lead(x0));
                    if (own > 0.f) mn = fminf(mn, own);
#pragma unroll
                    for (int d = 16; d > 0; d >>= 1) mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, d));
                    if (mn > 1e38f) continue;  // nothing above the floor so far
                    const float f0 = sc > 0.f ? mn / sc : 0.f;
                    s2 = Op::scale(Op::scale(s2, f0), f0);
                    sc = mn;
#pragma unroll
                    for (int h = 0; h < NS; h++) {
                        const float f = ss[h] > 0.f ? sc * (1.f / ss[h]) : 0.f;  // <= 1, powers of two
                        sh[h] = Op::scale(Op::scale(sh[h], f), f);
                    }
                } else {
                    sc = 1.f;
                }
#pragma unroll
                for (int h = 0; h < NS; h++) s2 = Op::sum(s2, sh[h]);
            }
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) s2 = Op::sum(s2, Op::shfl_xor(s2, d));
            if (lane == 0) {
                const bool zero = Op::scaled && sc == 0.f;
                if (zero) sc = 1.f;
                const V x0s = Op::scale(x0, sc);
                V bs = x0s, sg = Op::zero(), inv = sg, u0s = sg;
                if (Op::positive(s2) && !zero) {
                    Op::mac(s2, x0s, x0s);
                    bs = Op::root(Op::norm(s2));
                    if (Op::nonneg(x0s)) bs = Op::neg(bs);
                    u0s = Op::sum(x0s, Op::neg(bs));
                    sg = Op::neg(Op::quot(Op::one(), Op::mul(bs, u0s)));
                    inv = Op::neg(Op::mul(sg, bs));
                }
                s_beta = Op::scale(bs, 1.f / sc);
                s_sigma = sg;
                s_inv = inv;
                s_u0 = u0s;
                s_us = sc;
                if (g == 0) {
                    const double v = Op::to(u0s);
                    o.tau[k] = Op::to(sg) * v * v;
                    o.alpha[k] = -Op::to(bs) / (double)sc * unscale;
                }
            }
        }
        // ---- 1. the units; one warp a scheduler works on each, so the pipes stay
        // even whatever their number is.  A group takes every G-th unit from the
        // CTA's counter, one ahead of the one it works on.
        const int units = Ta * (Ta + 1) * RB / 2, grp = warp >> 2, sub = warp & 3;
        auto place = [&](int e, int& J, int& I) {
            // column block q of Ta has RB (Ta - q) units
            const int f = e * 2 / RB;
            int q = (int)((2 * Ta + 1 - sqrtf((float)((2 * Ta + 1) * (2 * Ta + 1) - 4 * f))) * 0.5f);
            q = max(0, min(q, Ta - 1));
            while (q > 0 && q * (2 * Ta - q + 1) * RB / 2 > e) q--;
            while ((q + 1) * (2 * Ta - q) * RB / 2 <= e) q++;
            J = J0 + q;
            I = RB * J + (e - q * (2 * Ta - q + 1) * RB / 2);
        };
        auto rows_of = [&](int J, int I) -> V* {
            return o.tiles + (unit_base(RB, T, J) + I - RB * J) * (UR * UC) + sub * WR * UC + 2 * lane;
        };
        int buf = 0;
        if (sub == 0 && lane == 0) s_unit[0][grp] = g + G * atomicAdd(&s_next, 1);
        asm volatile("bar.sync %0, 128;" ::"r"(grp + 1) : "memory");
        int e = s_unit[0][grp], J = 0, I = 0;
        Two<V> nxt[8];
        if (e < units) {
            place(e, J, I);
            V* tile = rows_of(J, I);
#pragma unroll
            for (int r = 0; r < 8; r++) nxt[r] = ld2(tile + r * UC);
        }
        while (e < units) {
            if (sub == 0 && lane == 0) s_unit[buf ^ 1][grp] = g + G * atomicAdd(&s_next, 1);
            V* tile = rows_of(J, I);
            const int jc = J * UC + 2 * lane, i0 = I * UR + sub * WR, ir = i0 + (lane & (WR - 1)), Jn = J, In = I;
            const Two<V> xc = ld2(o.x + jc), uc = ld2(o.u + jc), pc = ld2(o.p + jc);
            const V xr = Op::neg(ld1(o.x + ir));
            const V ur = Op::mul(sigma, ld1(o.u + ir)), pr = Op::neg(Op::mul(sigma, ld1(o.p + ir)));
            const bool diag = (I / RB) == J;
            Two<V> cs{Op::zero(), Op::zero()};
#pragma unroll 1
            for (int b = 0; b < WR / 8; b++) {
                Two<V> cur[8];
#pragma unroll
                for (int r = 0; r < 8; r++) cur[r] = nxt[r];
                if (b + 1 < WR / 8) {
#pragma unroll
                    for (int r = 0; r < 8; r++) nxt[r] = ld2(tile + (8 * (b + 1) + r) * UC);
                }
                V acc[8];
#pragma unroll
                for (int r = 0; r < 8; r++) {
                    const int row = 8 * b + r;
                    const V su = Op::bcast(ur, row), sp = Op::bcast(pr, row), nx = Op::bcast(xr, row);
                    Two<V> a = cur[r];
                    Op::mac(a.a, su, pc.a);
                    Op::mac(a.b, su, pc.b);
                    Op::mac(a.a, sp, uc.a);
                    Op::mac(a.b, sp, uc.b);
                    a.a = Op::norm(a.a);
                    a.b = Op::norm(a.b);
                    if (diag) {
                        if (jc >= i0 + row) a.a = Op::zero();
                        if (jc + 1 >= i0 + row) a.b = Op::zero();
                    }
                    *reinterpret_cast<Two<V>*>(tile + row * UC) = a;
                    acc[r] = Op::prod(a.a, xc.a);
                    Op::mac(acc[r], a.b, xc.b);
                    Op::mac(cs.a, a.a, nx);
                    Op::mac(cs.b, a.b, nx);
                }
                // row sums: halves exchanged three times, then two plain levels
#pragma unroll
                for (int lv = 0; lv < 3; lv++) {
                    const int d = 16 >> lv, h = 4 >> lv;
                    const bool up = lane & d;
#pragma unroll
                    for (int i = 0; i < 4; i++)
                        if (i < h) {
                            const V keep = up ? acc[i + h] : acc[i], send = up ? acc[i] : acc[i + h];
                            acc[i] = Op::sum(keep, Op::shfl_xor(send, d));
                        }
                }
                acc[0] = Op::sum(acc[0], Op::shfl_xor(acc[0], 2));
                acc[0] = Op::sum(acc[0], Op::shfl_xor(acc[0], 1));
                if ((lane & 3) == 0)
                    o.prow[((size_t)In * T + Jn) * UR + sub * WR + 8 * b + ((lane & 16) ? 4 : 0) +
                           ((lane & 8) ? 2 : 0) + ((lane & 4) ? 1 : 0)] = acc[0];
            }
            // column sums of the four warps; the group's next unit
            s_col[buf][warp][2 * lane] = Op::norm(cs.a);
            s_col[buf][warp][2 * lane + 1] = Op::norm(cs.b);
            asm volatile("bar.sync %0, 128;" ::"r"(grp + 1) : "memory");
            e = s_unit[buf ^ 1][grp];
            if (e < units) {
                place(e, J, I);
                V* ahead = rows_of(J, I);
#pragma unroll
                for (int r = 0; r < 8; r++) nxt[r] = ld2(ahead + r * UC);
            }
            if (sub < 2) {
                const int c = sub * 32 + lane;
                const V(*q)[UC] = &s_col[buf][grp * 4];
                o.pcol[((size_t)Jn * RB * T + In) * UC + c] =
                    Op::sum(Op::sum(q[0][c], q[1][c]), Op::sum(q[2][c], q[3][c]));
            }
            buf ^= 1;
        }
        if (!sk_grid_barrier(o.ctr, epoch, o.status, o.cap)) return;
        // ---- 2. the owners' sums, p and the next column (32 indices at a time)
        const V beta = s_beta;
        sigma = s_sigma;
        const float us = s_us;
        if (t == 0) s_next = 0;
        // a CTA takes one block of 32 indices, or one of 64 as two halves side by
        // side when there are more blocks of 32 than CTAs
        const int halves = 2 * T > G ? 2 : 1, hw = SW / halves, half = warp / hw, wh = warp - half * hw;
        for (int bb = g; bb < 2 * T / halves; bb += G) {
            const int b = bb * halves + half, bc = b >> 1;  // block of 32, column block
            if (((bb + 1) * halves - 1) >> 1 < J0) continue;  // uniform in the CTA
            const bool on = bc >= J0;
            const int i = b * 32 + lane;
            // everything this block needs from memory at once
            V xi = Op::zero(), ai = Op::zero();
            if (wh == 0 && on) {
                xi = ld1(o.x + i);
                if (i > k + 1 && i < n) ai = element(i, k + 1);
            }
            const int nr = bc - J0 + 1, nc = on ? nr + RB * (T - bc) : 0;
            auto part = [&](int ii, int cb, int nrr, int c) -> V {
                return c < nrr ? ld1(o.prow + ((size_t)(ii / UR) * T + J0 + c) * UR + (ii & (UR - 1)))
                               : ld1(o.pcol + ((size_t)cb * RB * T + RB * cb + c - nrr) * UC + (ii & 63));
            };
            const int n0 = 1 + RB * (T - J0);  // partial sums of element k + 1 (block J0)
            for (int c = t; c < n0; c += ST) s_q0[c] = part(k + 1, J0, 1, c);
            V acc = Op::zero();
#pragma unroll 1
            for (int c = wh; c < nc; c += hw * 8) {
                V v[8];
#pragma unroll
                for (int h = 0; h < 8; h++) v[h] = c + hw * h < nc ? part(i, bc, nr, c + hw * h) : Op::zero();
#pragma unroll
                for (int h = 0; h < 8; h++) acc = Op::sum(acc, v[h]);
            }
            s_grp[warp][lane] = acc;
            __syncthreads();
            if (warp == 1) {
                V s = Op::zero();
                for (int c = lane; c < n0; c += 32) s = Op::sum(s, s_q0[c]);
#pragma unroll
                for (int d = 16; d > 0; d >>= 1) s = Op::sum(s, Op::shfl_xor(s, d));
                if (lane == 0) s_q0v = s;
            }
            V qi = Op::zero();
            if (wh == 0)
                for (int w = 0; w < hw; w += 4)
                    qi = Op::sum(qi, Op::sum(Op::sum(s_grp[warp + w][lane], s_grp[warp + w + 1][lane]),
                                             Op::sum(s_grp[warp + w + 2][lane], s_grp[warp + w + 3][lane])));
            __syncthreads();
            if (wh == 0 && on) {
                const bool live = i > k && i < n;
                Op::mac(qi, Op::neg(beta), ai);
                const V pi = live ? Op::scale(Op::norm(qi), us) : Op::zero();
                const V ui = !live ? Op::zero() : i == k + 1 ? s_u0 : Op::scale(xi, us);
                const V pc = Op::mul(sigma, Op::scale(s_q0v, us)), uc = Op::neg(Op::mul(sigma, s_u0));
                V xn = ai;
                Op::mac(xn, pi, uc);
                Op::mac(xn, ui, pc);
                o.u[i] = ui;
                o.p[i] = pi;
                publish_x(i, k + 2, i > k + 1 && i < n ? Op::norm(xn) : Op::zero());
                if (live) o.Vout[(size_t)k * n + i] = i == k + 1 ? Op::one() : Op::mul(ui, s_inv);
            }
            __syncthreads();  // s_grp, s_q0 of the next block
        }
        if (!sk_grid_barrier(o.ctr, epoch, o.status, o.cap)) return;
    }
    if (g == 0 && t == 0) o.alpha[n - 2] = -Op::to(ld1(o.x + n - 1)) * unscale;
}

// Units from the strict lower triangle of A (column-major), scaled.
template <class Op>
__global__ void __launch_bounds__(256)
sym_fill_kernel(int n, int T, const double* __restrict__ A, int lda, const unsigned long long* amax,
                typename Op::V* __restrict__ tiles, double* scale, int check, int* status) {
    constexpr int UR = Op::UR, RB = UC / UR;
    __shared__ typename Op::V sh[UC][UR + 1];
    const int I = blockIdx.x, J = blockIdx.y;
    if (I < RB * J) return;
    const double s = Op::prescale(*amax);
    if (I == 0 && J == 0 && threadIdx.x == 0) scale[0] = s;
    const int tx = threadIdx.x % UR, ty = threadIdx.x / UR;
    const int i = I * UR + tx;
    bool bad = false;
    for (int c = ty; c < UC; c += 256 / UR) {
        const int j = J * UC + c;
        double v = 0.0;
        if (i < n && j < i) {
            v = A[(size_t)j * lda + i];
            if (!isfinite(v)) bad = true;
        }
        sh[c][tx] = Op::from(v * s);
    }
    __syncthreads();
    typename Op::V* out = tiles + (unit_base(RB, T, J) + I - RB * J) * (UR * UC);
    for (int q = threadIdx.x; q < UR * UC; q += 256) out[q] = sh[q & (UC - 1)][q / UC];
    if (bad && check) sk_set_error(status, SKEW_ERR_NONFINITE);
}

struct SymWs {
    void *tiles, *x, *u, *p, *prow, *pcol, *nrm;
    float* nsc;
    unsigned* ctr;  // [0] arrivals, [2..3] max |A|, [4..5] the scale
};

// (sized for units of 32 rows)
SymWs carve_sym(Carve& cv, int n) {
    const size_t T = (size_t)(n + UC - 1) / UC;
    SymWs w{};
    w.tiles = cv.take<double>(T * (T + 1) * UC * UC / 2);
    w.x = cv.take<double>(T * UC);
    w.u = cv.take<double>(T * UC);
    w.p = cv.take<double>(T * UC);
    w.prow = cv.take<double>(T * T * UC);
    w.pcol = cv.take<double>(2 * T * T * UC);
    w.nrm = cv.take<double>(2 * T);
    w.nsc = cv.take<float>(2 * T);
    w.ctr = cv.take<unsigned>(16);
    return w;
}

template <class Op>
int sym_run(cudaStream_t st, int n, const double* A, int lda, double* V, double* tau, double* alpha, const SymWs& w,
            int check, int* d_status, unsigned spin_cap) {
    using T8 = typename Op::V;
    const int T = (n + UC - 1) / UC;
    const size_t vc = (size_t)onestep_vcols(n);
    if (const cudaError_t e = cudaMemsetAsync(V, 0, sizeof(double) * vc * n, st)) return cuda_fail(e);
    if (const cudaError_t e = cudaMemsetAsync(tau, 0, sizeof(double) * vc, st)) return cuda_fail(e);
    if (const cudaError_t e = cudaMemsetAsync(w.ctr, 0, 16 * sizeof(unsigned), st)) return cuda_fail(e);
    if (const cudaError_t e = cudaMemsetAsync(w.u, 0, sizeof(double) * T * UC, st)) return cuda_fail(e);
    if (const cudaError_t e = cudaMemsetAsync(w.p, 0, sizeof(double) * T * UC, st)) return cuda_fail(e);
    auto* amax = reinterpret_cast<unsigned long long*>(w.ctr + 2);
    auto* scale = reinterpret_cast<double*>(w.ctr + 4);
    if (const int rc = onestep_amax(st, n, A, lda, amax)) return rc;
    sym_fill_kernel<Op><<<dim3(UC / Op::UR * T, T), 256, 0, st>>>(n, T, A, lda, amax, static_cast<T8*>(w.tiles), scale, check,
                                                        d_status);
    count_launch();
    SymArgs<T8> o{};
    o.n = n;
    o.T = T;
    o.tiles = static_cast<T8*>(w.tiles);
    o.x = static_cast<T8*>(w.x);
    o.u = static_cast<T8*>(w.u);
    o.p = static_cast<T8*>(w.p);
    o.prow = static_cast<T8*>(w.prow);
    o.pcol = static_cast<T8*>(w.pcol);
    o.nrm = static_cast<T8*>(w.nrm);
    o.nsc = w.nsc;
    o.Vout = reinterpret_cast<T8*>(V);
    o.tau = tau;
    o.alpha = alpha;
    o.scale = scale;
    o.ctr = w.ctr;
    o.status = d_status;
    o.cap = spin_cap ? spin_cap : SK_SPIN_CAP;
    void* args[] = {&o};
    const cudaError_t e = cudaLaunchCooperativeKernel((void*)onestep_sym_kernel<Op>, dim3((unsigned)device_sms()),
                                                      dim3(ST), args, 0, st);
    count_launch();
    if (e == cudaErrorCooperativeLaunchTooLarge) return SKEW_ERR_LAUNCH;
    if (e != cudaSuccess) return cuda_fail(e);
    return Op::scaled ? onestep_widen(st, vc * (size_t)n, V) : cuda_ok(cudaGetLastError());
}

}  // namespace

int onestep_sym_max() { return 16384; }

size_t onestep_sym_ws(int n) {
    Carve cv(nullptr, ~size_t(0));
    carve_sym(cv, n);
    return cv.off + 256;
}

int onestep_sym_reduce(cudaStream_t st, int n, const double* A, int lda, bool pairs, double* V, double* tau,
                       double* alpha, void* ws, size_t ws_bytes, int check, int* d_status, unsigned spin_cap) {
    if (n < 3 || n > onestep_sym_max()) return SKEW_ERR_UNSUPPORTED;
    Carve cv(ws, ws_bytes);
    const SymWs w = carve_sym(cv, n);
    if (!cv.ok) return SKEW_ERR_WORKSPACE;
    KtScope kt(st, KT_PANEL_QR);
    return pairs ? sym_run<DfPair>(st, n, A, lda, V, tau, alpha, w, check, d_status, spin_cap)
                 : sym_run<F64>(st, n, A, lda, V, tau, alpha, w, check, d_status, spin_cap);
}

}  // namespace sk
