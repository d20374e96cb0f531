// onestep_dev.cuh -- device routines of the direct tridiagonalisation and of its
// FP64 back-transformation, shared by the whole-GPU kernels (onestep.cu) and
// the batched ones.
#pragma once
#include "common.cuh"

namespace sk {
namespace onestep {

constexpr int GR = 256;  // rows of one Gram partial
constexpr int PB = 64;   // reflectors per panel

// Totals over the warp of N values per lane by exchanging halves: 5 levels,
// about N additions instead of 5 N.  Afterwards a[0 .. cnt) of a lane are the
// totals of the values first .. first + cnt - 1.
template <int N>
struct WarpSums {
    static constexpr int H1 = (N + 1) / 2, H2 = (H1 + 1) / 2, H3 = (H2 + 1) / 2, H4 = (H3 + 1) / 2,
                         H5 = (H4 + 1) / 2;
    int first = 0, cnt = N;
    template <int L, int H, int B>
    SK_DEV void level(double (&a)[N], int lane) {
        const bool up = lane & B;
#pragma unroll
        for (int i = 0; i < H; i++) {
            const double hi = (i + H < L) ? a[i + H < N ? i + H : 0] : 0.0;
            const double keep = up ? hi : a[i], send = up ? a[i] : hi;
            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, B);
        }
        first += up ? H : 0;
        cnt = up ? max(cnt - H, 0) : min(cnt, H);
    }
    SK_DEV void run(double (&a)[N], int lane) {
        level<N, H1, 16>(a, lane);
        level<H1, H2, 8>(a, lane);
        level<H2, H3, 4>(a, lane);
        level<H3, H4, 2>(a, lane);
        level<H4, H5, 1>(a, lane);
    }
};

// The FP64 forms work on s A, s = 1 for max |A| in [2^-400, 2^400] and else the
// power of two that brings it into [1/2, 1); a column whose tail's squares sum to
// less than 2^-1000 counts as zero (H = I, below 2^-100 max |A|).  sigma = -1 /
// (beta u_0) and A x then stay inside the double range: sigma of a plain column
// leaves it below a norm of 7.5e-155 and above 9.5e153.  The scale is set once a
// solve: a test in every column, with the column scaled where it needs it, took
// 60 us of 4.00 ms at n = 500; this takes none that the runs can tell.
constexpr unsigned TAIL_MIN = 23u << 20;  // 2^-1000
SK_DEV bool os_tail(double s2) { return (unsigned)__double2hiint(s2) >= TAIL_MIN; }  // NaN too
// amax: max |A| as the bits of a double, its finite entries
SK_DEV double os_scale(unsigned long long amax) {
    const int e = (int)(amax >> 52);
    return amax == 0 || (unsigned)(e - 623) < 800u ? 1.0 : ldexp(1.0, max(-1000, min(1000, 1022 - e)));
}
SK_DEV unsigned long long os_abs_bits(double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
    return b < 0x7ff0000000000000ull ? b : 0ull;
}
SK_DEV unsigned long long os_warp_max(unsigned long long m) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, m, o);
        m = w > m ? w : m;
    }
    return m;
}

// The rank-2 update of RC own rows (base, base + stride, ...; matrix rows i0,
// i0 + G, ...) and their products with x, columns ja + 32 seg + lane + 32 nseg t.
// coef: sigma u_i and -sigma p_i of the rows.  The row sums of this segment go
// to part[row * OCW].  GLB: rows in global memory, the next step's elements
// are loaded ahead.
constexpr int OCW = 8;  // warps of the pass, segments of a row at most

template <int RC, bool GLB>
SK_DEV void os_rows(double* base, size_t stride, int i0, int G, int n, int k, int ja, const double2* coef,
                    const double* u, const double* p, const double* x, int seg, int nseg, int lane, double* part) {
    double ui[RC], pi[RC], acc[RC];
#pragma unroll
    for (int r = 0; r < RC; r++) {
        const double2 c = coef[r];
        ui[r] = c.x;
        pi[r] = c.y;
        acc[r] = 0.0;
    }
    auto step = [&](int j, const double (&in)[RC]) {
        const double uj = u[j], pj = p[j], xj = (j > k) ? x[j] : 0.0;
        double a[RC];
#pragma unroll
        for (int r = 0; r < RC; r++) a[r] = fma(ui[r], pj, in[r]);
#pragma unroll
        for (int r = 0; r < RC; r++) {
            a[r] = fma(pi[r], uj, a[r]);
            if (j == i0 + r * G) a[r] = 0.0;
            base[r * stride + j] = a[r];
        }
#pragma unroll
        for (int r = 0; r < RC; r++) acc[r] = fma(a[r], xj, acc[r]);
    };
    const int step_j = 32 * nseg;
    int j = ja + 32 * seg + lane;
    if (GLB) {
        double nx[RC];
#pragma unroll
        for (int r = 0; r < RC; r++) nx[r] = j < n ? base[r * stride + j] : 0.0;
#pragma unroll 1
        for (; j < n; j += step_j) {
            const int jn = j + step_j;
            double in[RC];
#pragma unroll
            for (int r = 0; r < RC; r++) {
                in[r] = nx[r];
                nx[r] = jn < n ? base[r * stride + jn] : 0.0;
            }
            step(j, in);
        }
    } else {
#pragma unroll 1
        for (; j < n; j += step_j) {
            double in[RC];
#pragma unroll
            for (int r = 0; r < RC; r++) in[r] = base[r * stride + j];
            step(j, in);
        }
    }
    WarpSums<RC> ws;
    ws.run(acc, lane);
#pragma unroll
    for (int i = 0; i < WarpSums<RC>::H5; i++)
        if (i < ws.cnt) part[(ws.first + i) * OCW] = acc[i];
}

// cnt rows in chunks of at most MAXRC.
template <int MAXRC, bool GLB>
SK_DEV void os_rows_any(int cnt, double* base, size_t stride, int i0, int G, int n, int k, int ja, const double2* coef,
                        const double* u, const double* p, const double* x, int seg, int nseg, int lane,
                        double* part) {
    while (cnt > 0) {
        const int c = min(cnt, MAXRC);
        if (c == 1) {
            os_rows<1, GLB>(base, stride, i0, G, n, k, ja, coef, u, p, x, seg, nseg, lane, part);
        } else if (c == 2) {
            os_rows<2, GLB>(base, stride, i0, G, n, k, ja, coef, u, p, x, seg, nseg, lane, part);
        } else if (c == 3) {
            os_rows<3, GLB>(base, stride, i0, G, n, k, ja, coef, u, p, x, seg, nseg, lane, part);
        } else if (MAXRC <= 4 || c == 4) {
            os_rows<4, GLB>(base, stride, i0, G, n, k, ja, coef, u, p, x, seg, nseg, lane, part);
        } else if constexpr (MAXRC > 4) {
            if (c == 5) os_rows<5, GLB>(base, stride, i0, G, n, k, ja, coef, u, p, x, seg, nseg, lane, part);
            else if (c == 6) os_rows<6, GLB>(base, stride, i0, G, n, k, ja, coef, u, p, x, seg, nseg, lane, part);
            else if (c == 7) os_rows<7, GLB>(base, stride, i0, G, n, k, ja, coef, u, p, x, seg, nseg, lane, part);
            else os_rows<8, GLB>(base, stride, i0, G, n, k, ja, coef, u, p, x, seg, nseg, lane, part);
        }
        cnt -= c;
        base += (size_t)c * stride;
        i0 += c * G;
        coef += c;
        part += c * OCW;
    }
}

// A warp's share of the pass over R own rows, the first rg of them in global
// memory (from row gbase on), the others in shared memory: either kind in
// OCW / nseg groups of consecutive rows, nseg segments of the columns each.
// Few rows take all warps side by side on the columns; many rows give each
// warp rows of its own, so that a warp's row sums (5 levels of additions) come
// once per row and not eight times.  Global rows keep more segments: the warps
// then read one row's neighbouring lines together.
template <int MAXRC>
SK_DEV void os_pass(int nsg, int nss, int R, int rg, double* gbase, double* sbase, int n, int lds, int i0, int G, int k,
                    const double2* coef, const double* u, const double* p, const double* x, int warp, int lane,
                    double (*part)[OCW]) {
    const int ja = (k + 1) & ~3;
    if (rg > 0) {
        const int groups = OCW / nsg, grp = warp / nsg, seg = warp - grp * nsg;
        const int lo = rg * grp / groups, hi = rg * (grp + 1) / groups;
        if (lo < hi)
            os_rows_any<MAXRC, true>(hi - lo, gbase + (size_t)lo * G * n, (size_t)G * n, i0 + lo * G, G, n, k, ja,
                                     coef + lo, u, p, x, seg, nsg, lane, &part[lo][seg]);
    }
    if (rg < R) {
        const int groups = OCW / nss, grp = warp / nss, seg = warp - grp * nss;
        const int lo = rg + (R - rg) * grp / groups, hi = rg + (R - rg) * (grp + 1) / groups;
        if (lo < hi)
            os_rows_any<MAXRC, false>(hi - lo, sbase + (size_t)(lo - rg) * lds, lds, i0 + lo * G, G, n, k, ja,
                                      coef + lo, u, p, x, seg, nss, lane, &part[lo][seg]);
    }
}

// The row sum of the segments, in order.
SK_DEV double os_row_sum(const double* s, int nseg) {
    if (nseg == 1) return s[0];
    if (nseg == 2) return s[0] + s[1];
    if (nseg == 4) return (s[0] + s[1]) + (s[2] + s[3]);
    return ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
}

// ---- back-transformation: Z <- H_0 H_1 ... H_{n-3} Z ------------------------
// Panels of 64 reflectors (the last one padded with zero columns) act as one
// compact WY block (Eq. 7).  T is not formed: T^-1 = diag(1 / tau) + the strict
// upper triangle of V^T V, so T y is a back substitution with V^T V.

// Upper triangle of V_p^T V_p over the rows lo .. hi - 1 (GR at most), 160
// threads: 136 of them with one 4 x 4 tile each.  V: the panel's columns.
// out: 64 x 64, column-major.
SK_DEV void os_gram_body(const double* __restrict__ V, int ldv, int lo, int hi, double* __restrict__ q) {
    const int t = threadIdx.x;
    __shared__ double vs[PB][33];
    int ti = 0, tj = 0;
    if (t < 136) {
        int e = t;  // tile (ti, tj), ti <= tj
        while (e > tj) e -= ++tj;
        ti = e;
    }
    double acc[4][4] = {};
    for (int r0 = lo; r0 < hi; r0 += 32) {
        for (int e = t; e < PB * 32; e += 160) {
            const int r = e & 31, c = e >> 5;
            vs[c][r] = (r0 + r < hi) ? V[(size_t)c * ldv + r0 + r] : 0.0;
        }
        __syncthreads();
        if (t < 136) {
#pragma unroll 4
            for (int r = 0; r < 32; r++) {
                double a[4], b[4];
#pragma unroll
                for (int i = 0; i < 4; i++) a[i] = vs[4 * ti + i][r], b[i] = vs[4 * tj + i][r];
#pragma unroll
                for (int i = 0; i < 4; i++)
#pragma unroll
                    for (int j = 0; j < 4; j++) acc[i][j] = fma(a[i], b[j], acc[i][j]);
            }
        }
        __syncthreads();
    }
    if (t < 136) {
#pragma unroll
        for (int j = 0; j < 4; j++)
#pragma unroll
            for (int i = 0; i < 4; i++) q[(size_t)(4 * tj + j) * PB + 4 * ti + i] = acc[i][j];
    }
}

// Sums S partials (stride elements apart) in order, entries e0, e0 + step, ...
// scaled: Gt[i][l] = (V^T V)_{l i} tau_i for l < i, 0 elsewhere (the back
// substitution's rows); else the plain upper triangle, mirrored.
SK_DEV void os_gram_sum_body(const double* __restrict__ part, size_t stride, int S, const double* __restrict__ tau,
                             double* __restrict__ Gt, int scaled, int e0, int step) {
    for (int e = e0; e < PB * PB; e += step) {
        const int l = e % PB, i = e / PB;
        double g = 0.0;
        if (l < i || (!scaled && l == i))
            for (int s = 0; s < S; s++) g += part[(size_t)s * stride + e];
        if (scaled) {
            Gt[e] = g * tau[i];
        } else if (l <= i) {
            Gt[e] = g;
            Gt[(size_t)l * PB + i] = g;
        }
    }
}

constexpr int WT = 256;  // threads of the WY kernel

// One CTA carries E eigenvectors (C = 2 E columns: real and imaginary parts)
// through every panel without leaving the SM: the slab of Z stays in shared
// memory, V streams from L2 (read twice per panel), and nothing is exchanged
// between CTAs.  The D map is applied on the way in (Algorithm 1 step 3) and the parts
// go straight to Z_re / Z_im.  Bound by the FP64 pipe: 2 FMA per element of
// V and column.
template <int E>
SK_DEV void os_wy_body(int n, int nev, int e0, const double* __restrict__ V, const double* __restrict__ Gt,
                       const double* __restrict__ tau, const double* __restrict__ Qi, double* __restrict__ Zre,
                       double* __restrict__ Zim, int ldz, double* wy_sm) {
    constexpr int C = 2 * E, VG = C <= 8 ? 8 : 4, NP = 8 / VG;
    constexpr int NW = WT / 32;
    double* ys = wy_sm;              // [64][C]
    double* gs = ys + PB * C;        // [64][64]
    double* zs = gs + PB * PB;       // [C][n]
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    // D q: rows r mod 4 = 0, 1, 2, 3 of q are times 1, i, -1, -i
    for (int i = t; i < n; i += WT) {
#pragma unroll
        for (int e = 0; e < E; e++) {
            double q = e0 + e < nev ? Qi[(size_t)i * nev + e0 + e] : 0.0;
            if (i & 2) q = -q;
            zs[(size_t)(2 * e) * n + i] = (i & 1) ? 0.0 : q;
            zs[(size_t)(2 * e + 1) * n + i] = (i & 1) ? q : 0.0;
        }
    }
    const int P = (n - 2 + PB - 1) / PB;
    for (int p = P - 1; p >= 0; p--) {
        const int o = p * PB + 1;
        const double* Vp = V + (size_t)p * PB * n;
        for (int e = t; e < PB * PB; e += WT) gs[e] = Gt[(size_t)p * PB * PB + e];
        __syncthreads();
        // Y = V_p^T Z: a warp takes 8 columns of V, lanes the rows
#pragma unroll 1
        for (int pass = 0; pass < NP; pass++) {
            const int v0 = warp * 8 + pass * VG;
            const double* Vc = Vp + (size_t)v0 * n;
            double acc[VG * C];
#pragma unroll
            for (int i = 0; i < VG * C; i++) acc[i] = 0.0;
            double vv[VG], vn[VG];
            int r = o + lane;
#pragma unroll
            for (int i = 0; i < VG; i++) vn[i] = r < n ? Vc[(size_t)i * n + r] : 0.0;
            for (; r - lane < n; r += 32) {
#pragma unroll
                for (int i = 0; i < VG; i++) {
                    vv[i] = vn[i];
                    vn[i] = r + 32 < n ? Vc[(size_t)i * n + r + 32] : 0.0;
                }
                const int rr = r < n ? r : n - 1;
#pragma unroll
                for (int c = 0; c < C; c++) {
                    const double z = zs[(size_t)c * n + rr];
#pragma unroll
                    for (int i = 0; i < VG; i++) acc[i * C + c] = fma(vv[i], z, acc[i * C + c]);
                }
            }
            WarpSums<VG * C> ws;
            ws.run(acc, lane);
#pragma unroll
            for (int i = 0; i < WarpSums<VG * C>::H5; i++)
                if (i < ws.cnt) ys[v0 * C + ws.first + i] = acc[i];
        }
        __syncthreads();
        // y <- T y by back substitution, one warp per column
        for (int c = warp; c < C; c += NW) {
            double y0 = ys[lane * C + c], y1 = ys[(lane + 32) * C + c];
#pragma unroll 4
            for (int i = 63; i >= 32; i--) {
                const double b = __shfl_sync(0xffffffffu, y1, i - 32);
                y1 = fma(-gs[i * PB + lane + 32], b, y1);
                y0 = fma(-gs[i * PB + lane], b, y0);
            }
#pragma unroll 4
            for (int i = 31; i > 0; i--) {
                const double b = __shfl_sync(0xffffffffu, y0, i);
                y0 = fma(-gs[i * PB + lane], b, y0);
            }
            ys[lane * C + c] = -tau[p * PB + lane] * y0;
            ys[(lane + 32) * C + c] = -tau[p * PB + lane + 32] * y1;
        }
        __syncthreads();
        // Z -= V_p y: warps take blocks of 32 rows
        for (int rb = warp; o + 32 * rb < n; rb += NW) {
            const int r = o + 32 * rb + lane, rr = r < n ? r : n - 1;
            double z[C];
#pragma unroll
            for (int c = 0; c < C; c++) z[c] = zs[(size_t)c * n + rr];
            const double* Vr = Vp + rr;
            double vn[8];
#pragma unroll
            for (int i = 0; i < 8; i++) vn[i] = Vr[(size_t)i * n];
            for (int v = 0; v < PB; v += 8) {
                double vv[8];
                const int nx = v + 8 < PB ? v + 8 : v;
#pragma unroll
                for (int i = 0; i < 8; i++) {
                    vv[i] = vn[i];
                    vn[i] = Vr[(size_t)(nx + i) * n];
                }
#pragma unroll
                for (int i = 0; i < 8; i++)
#pragma unroll
                    for (int c = 0; c < C; c += 2) {
                        const double2 y = *reinterpret_cast<const double2*>(ys + (v + i) * C + c);
                        z[c] = fma(vv[i], y.x, z[c]);
                        z[c + 1] = fma(vv[i], y.y, z[c + 1]);
                    }
            }
            if (r < n) {
#pragma unroll
                for (int c = 0; c < C; c++) zs[(size_t)c * n + r] = z[c];
            }
        }
        __syncthreads();
    }
    for (int e = 0; e < E && e0 + e < nev; e++)
        for (int i = t; i < n; i += WT) {
            Zre[(size_t)(e0 + e) * ldz + i] = zs[(size_t)(2 * e) * n + i];
            Zim[(size_t)(e0 + e) * ldz + i] = zs[(size_t)(2 * e + 1) * n + i];
        }
}

inline size_t wy_smem(int n, int E) {
    return sizeof(double) * ((size_t)PB * 2 * E + PB * PB + 2 * (size_t)E * n);
}

}  // namespace onestep
}  // namespace sk
