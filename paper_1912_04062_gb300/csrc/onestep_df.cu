// onestep_df.cu -- the direct tridiagonalisation (onestep.cu) in double-float
// arithmetic, for a caller that refines the eigenpairs afterwards.
//
// The FP64 pipe issues one warp instruction per 64 clocks and scheduler on this
// part, the FP32 pipe one per clock.  An element's rank-2 update and product
// with x take 3 FP64 FMAs (about 200 clocks) or about 40 FP32 instructions on
// pairs (hi, lo), so the pair form turns the pass from arithmetic-bound to
// bound by the exchange (shared memory) or by L2.  A pair carries 2^-47 per
// operation; the refined mode's two-step reduction carries 2^-42 (six digit
// slices), and the refinement recomputes values and vectors from A.
//
// The matrix is scaled by a power of two to max |A| in [1/2, 1) (FP32 range),
// and every reflector to |u| of order one, so that nothing a pair can hold
// under- or overflows; what lies below 2^-100 of the largest entry is dropped.
#include <algorithm>
#include <cfloat>

#include "common.cuh"
#include "internal.h"
#include "onestep_dev.cuh"
#include "pairs.cuh"

namespace sk {

using namespace onestep;

namespace {

constexpr int DT = 512, DW = DT / 32;  // sixteen warps: the pass waits for L2, not for the FP32 pipe
constexpr int DMAXR = 64;
constexpr int DF_SMEM = 216 * 1024;  // dynamic shared memory at most: the static arrays take about 9.5 KB of 227

struct DfArgs {
    int n;
    float2* F;     // full skew matrix by rows, scaled
    float2* V;     // reflectors (as onestep_reduce, in pairs), zeroed by the caller
    double* tau;
    double* alpha;
    float4* qa;    // 2 n: (q, a) as pairs, double-buffered
    unsigned* ctr;
    const double* scale;  // scale[0]: the power of two A was multiplied by
    int* status;
    unsigned cap;
    int srows;
};

// os_rows (onestep_dev.cuh) on pairs.
template <int RC, bool GLB>
SK_DEV void df_rows(float2* base, size_t stride, int i0, int G, int n, int k, int ja, const float4* coef,
                    const float2* u, const float2* p, const float2* x, int seg, int nseg, int lane, float2* part) {
    float2 ui[RC], pi[RC], acc[RC];
#pragma unroll
    for (int r = 0; r < RC; r++) {
        const float4 c = coef[r];
        ui[r] = make_float2(c.x, c.y);
        pi[r] = make_float2(c.z, c.w);
        acc[r] = make_float2(0.f, 0.f);
    }
    auto step = [&](int j, float2 (&a)[RC]) {
        const float2 uj = u[j], pj = p[j];
        const float2 xj = (j > k) ? x[j] : make_float2(0.f, 0.f);
#pragma unroll
        for (int r = 0; r < RC; r++) {
            df_mac(a[r], ui[r], pj);
            df_mac(a[r], pi[r], uj);
            a[r] = df_norm(a[r]);
            if (j == i0 + r * G) a[r] = make_float2(0.f, 0.f);
            base[r * stride + j] = a[r];
            df_mac(acc[r], a[r], xj);
        }
    };
    const int step_j = 32 * nseg;
    int j = ja + 32 * seg + lane;
    if (GLB) {
        constexpr int AH = 3;  // steps loaded ahead: a step takes about 400 clocks, a load about 1000
        float2 nx[AH][RC];
#pragma unroll
        for (int h = 0; h < AH; h++)
#pragma unroll
            for (int r = 0; r < RC; r++)
                nx[h][r] = j + h * step_j < n ? base[r * stride + j + h * step_j] : make_float2(0.f, 0.f);
#pragma unroll 1
        for (; j < n; j += step_j) {
            const int jn = j + AH * step_j;
            float2 a[RC];
#pragma unroll
            for (int r = 0; r < RC; r++) {
                a[r] = nx[0][r];
#pragma unroll
                for (int h = 0; h + 1 < AH; h++) nx[h][r] = nx[h + 1][r];
                nx[AH - 1][r] = jn < n ? base[r * stride + jn] : make_float2(0.f, 0.f);
            }
            step(j, a);
        }
    } else {
#pragma unroll 1
        for (; j < n; j += step_j) {
            float2 a[RC];
#pragma unroll
            for (int r = 0; r < RC; r++) a[r] = base[r * stride + j];
            step(j, a);
        }
    }
#pragma unroll
    for (int r = 0; r < RC; r++) {
        const float2 s = df_warp_sum(acc[r]);
        if (lane == 0) part[r * DW] = s;
    }
}

template <bool GLB>
SK_DEV void df_rows_any(int cnt, float2* base, size_t stride, int i0, int G, int n, int k, int ja, const float4* coef,
                        const float2* u, const float2* p, const float2* x, int seg, int nseg, int lane,
                        float2* part) {
    while (cnt > 0) {
        const int c = min(cnt, 4);
        if (c == 4) df_rows<4, GLB>(base, stride, i0, G, n, k, ja, coef, u, p, x, seg, nseg, lane, part);
        else if (c == 3) df_rows<3, GLB>(base, stride, i0, G, n, k, ja, coef, u, p, x, seg, nseg, lane, part);
        else if (c == 2) df_rows<2, GLB>(base, stride, i0, G, n, k, ja, coef, u, p, x, seg, nseg, lane, part);
        else df_rows<1, GLB>(base, stride, i0, G, n, k, ja, coef, u, p, x, seg, nseg, lane, part);
        cnt -= c;
        base += (size_t)c * stride;
        i0 += c * G;
        coef += c;
        part += c * DW;
    }
}

// The column step of onestep_kernel; see there.
__global__ void __launch_bounds__(DT, 1) onestep_df_kernel(DfArgs o) {
    extern __shared__ __align__(16) float2 df_sm[];
    __shared__ float2 s_part[DMAXR][DW];
    __shared__ float4 s_coef[DMAXR];
    __shared__ float2 s_red[4];
    __shared__ float s_max[4];
    // of the scaled reflector u = (x - beta e_0) us; 1 / u_0 of the scaled one
    __shared__ float2 s_beta, s_sigma, s_inv, s_u0;
    __shared__ float s_us;
    __shared__ int s_ok;
    const int n = o.n, G = gridDim.x, g = blockIdx.x;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int ldn = n | 1;
    float2* u = df_sm;
    float2* p = u + ldn;
    float2* x = p + ldn;
    float2* rows = x + ldn;
    const int Rt = (n - 1 - g) / G + 1;
    const int rs0 = Rt > o.srows ? Rt - o.srows : 0;
    const int ilast = g + (Rt - 1) * G;
    for (int r = rs0; r < Rt; r++)
        for (int j = t; j < n; j += DT) rows[(size_t)(r - rs0) * ldn + j] = o.F[(size_t)(g + r * G) * n + j];
    const double unscale = 1.0 / o.scale[0];
    unsigned target = 0;
    float2 beta = make_float2(0.f, 0.f), sigma = beta;
    float us = 1.f;
    for (int k = 0; k + 1 < n; k++) {
        if (ilast < k + 1) return;
        // ---- 1. gather; p = us (q - beta a) and u <- us u of the previous
        // reflector, the updated column x
        const float4* qa = o.qa + (size_t)(k & 1) * n;
        if (k == 0) {
            for (int j = t; j < n; j += DT) {
                const float2 a = o.F[j];
                x[j] = df_neg2(a);
                u[j] = p[j] = make_float2(0.f, 0.f);
            }
        } else {
            // the first elements are under way while element k is waited for
            const float4 qk = __ldcg(qa + k);
            float4 ev[4];
#pragma unroll
            for (int h = 0; h < 4; h++) {
                const int j = k + 1 + t + h * DT;
                if (j < n) ev[h] = __ldcg(qa + j);
            }
            const float2 nb = df_neg2(beta);
            float2 pk = make_float2(qk.x, qk.y);
            df_mac(pk, nb, make_float2(qk.z, qk.w));
            pk = df_mul2(sigma, df_scale(df_norm(pk), us));
            const float2 uk = df_neg2(df_mul2(sigma, df_scale(s_u0, us)));
            auto form = [&](int j, float4 e) {
                float2 a = make_float2(e.z, e.w), pj = make_float2(e.x, e.y);
                df_mac(pj, nb, a);
                pj = df_scale(df_norm(pj), us);
                p[j] = pj;
                const float2 uj = df_scale(u[j], us);
                u[j] = uj;
                df_mac(a, pj, uk);
                df_mac(a, uj, pk);
                x[j] = df_norm(a);
            };
#pragma unroll
            for (int h = 0; h < 4; h++) {
                const int j = k + 1 + t + h * DT;
                if (j < n) form(j, ev[h]);
            }
#pragma unroll 4
            for (int j = k + 1 + t + 4 * DT; j < n; j += DT) form(j, __ldcg(qa + j));
        }
        __syncthreads();
        if (k == n - 2) {
            if (t == 0) o.alpha[k] = -df_to(x[n - 1]) * unscale;
            return;
        }
        // ---- 2. update the own rows i > k and multiply by x
        const int rf = (k + 1 > g) ? (k + 1 - g + G - 1) / G : 0;
        const int R = Rt - rf;
        const int rg = max(rs0, rf) - rf;
        for (int r = t; r < R; r += DT) {
            const int i = g + (rf + r) * G;
            const float2 c = df_mul2(sigma, u[i]), d = df_neg2(df_mul2(sigma, p[i]));
            s_coef[r] = make_float4(c.x, c.y, d.x, d.y);
        }
        __syncthreads();
        // as os_pass: the rows of global memory and those of shared memory each
        // spread over all warps
        const int rs = R - rg, i0 = g + rf * G, ja = (k + 1) & ~3;
        const int nss = rs >= 16 ? 1 : rs >= 8 ? 2 : rs >= 4 ? 4 : rs >= 2 ? 8 : 16, nsg = rg >= 16 ? 4 : rg >= 8 ? 8 : 16;
        if (rg > 0) {
            const int groups = DW / nsg, grp = warp / nsg, seg = warp - grp * nsg;
            const int lo = rg * grp / groups, hi = rg * (grp + 1) / groups;
            df_rows_any<true>(hi - lo, o.F + (size_t)(i0 + lo * G) * n, (size_t)G * n, i0 + lo * G, G, n, k, ja,
                              s_coef + lo, u, p, x, seg, nsg, lane, &s_part[lo][seg]);
        }
        if (rs > 0) {
            const int groups = DW / nss, grp = warp / nss, seg = warp - grp * nss;
            const int lo = rg + rs * grp / groups, hi = rg + rs * (grp + 1) / groups;
            df_rows_any<false>(hi - lo, rows + (size_t)(rf + lo - rs0) * ldn, ldn, i0 + lo * G, G, n, k, ja, s_coef + lo,
                               u, p, x, seg, nss, lane, &s_part[lo][seg]);
        }
        __syncthreads();
        if (warp == 0) {
            // ---- 3. publish, arrive, wait
            float4* out = o.qa + (size_t)((k + 1) & 1) * n;
            for (int r = lane; r < R; r += 32) {
                const int i = g + (rf + r) * G;
                float2 q = s_part[r][0];
                const int nseg = r < rg ? nsg : nss;
                for (int s = 1; s < nseg; s++) q = df_sum(q, s_part[r][s]);
                const float2* row = r >= rg ? rows + (size_t)(rf + r - rs0) * ldn : o.F + (size_t)i * n;
                const float2 a = row[k + 1];
                __stcg(out + i, make_float4(q.x, q.y, a.x, a.y));
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
        } else if (warp >= 4 && warp < 8) {
            // ---- meanwhile: the norm of x (scaled by a power of two near its
            // largest entry), beta, sigma
            const int q = t - 128;
            float mx = 0.f;
            for (int j = k + 1 + q; j < n; j += 128) mx = fmaxf(mx, fabsf(x[j].x));
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, d));
            if (lane == 0) s_max[warp - 4] = mx;
            asm volatile("bar.sync 1, 128;" ::: "memory");
            mx = fmaxf(fmaxf(s_max[0], s_max[1]), fmaxf(s_max[2], s_max[3]));
            // 2^-e with mx in [2^e, 2^(e+1)); entries below 2^-110 count as zero
            const bool zero = !(mx > 7.7e-34f);
            const float sc = zero ? 1.f : __int_as_float((254 << 23) - (__float_as_int(mx) & 0x7f800000));
            float2 nr = make_float2(0.f, 0.f);
            for (int j = k + 2 + q; j < n; j += 128) {
                const float2 v = df_scale(x[j], sc);
                df_mac(nr, v, v);
            }
            nr = df_warp_sum(df_norm(nr));
            if (lane == 0) s_red[warp - 4] = nr;
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (q == 0) {
                // in pairs as well: the FP64 square root and division would
                // take longer (2500 clocks) than the exchange they hide behind
                float2 s2 = df_sum(df_sum(s_red[0], s_red[1]), df_sum(s_red[2], s_red[3]));
                const float2 x0s = df_scale(x[k + 1], sc);
                float2 bs = x0s, sg = make_float2(0.f, 0.f), inv = sg, u0s = sg;
                if (s2.x > 0.f && !zero) {
                    df_mac(s2, x0s, x0s);
                    bs = df_root(df_norm(s2));
                    if (x0s.x >= 0.f) bs = df_neg2(bs);
                    u0s = df_sum(x0s, df_neg2(bs));
                    sg = df_neg2(df_quot(make_float2(1.f, 0.f), df_mul2(bs, u0s)));
                    inv = df_neg2(df_mul2(sg, bs));
                }
                const float isc = 1.f / sc;  // a power of two
                s_beta = df_scale(bs, isc);
                s_sigma = sg;
                s_us = sc;
                s_inv = inv;
                s_u0 = df_scale(u0s, isc);
                if (ilast == n - 1) {
                    const double v = df_to(u0s);
                    o.tau[k] = df_to(sg) * v * v;
                    o.alpha[k] = -df_to(bs) * (double)isc * unscale;
                }
            }
        }
        __syncthreads();
        if (!s_ok) return;
        beta = s_beta;
        sigma = s_sigma;
        us = s_us;
        for (int r = t; r < R; r += DT) {
            const int i = g + (rf + r) * G;
            o.V[(size_t)k * n + i] = (i == k + 1) ? make_float2(1.f, 0.f) : df_mul2(df_scale(x[i], us), s_inv);
        }
        if (t == 0) x[k + 1] = s_u0;  // x_0 itself is not read above
        float2* sw = u;
        u = x;
        x = sw;
        __syncthreads();
    }
}

// V from pairs to doubles, in place.
__global__ void __launch_bounds__(256) df_widen_kernel(size_t count, double* V) {
    for (size_t e = blockIdx.x * (size_t)256 + threadIdx.x; e < count; e += (size_t)gridDim.x * 256) {
        const float2 v = reinterpret_cast<const float2*>(V)[e];
        V[e] = df_to(v);
    }
}

// max |A| over the strict lower triangle, as the bits of a double (order-preserving for non-negative values)
__global__ void __launch_bounds__(256) df_amax_kernel(int n, const double* __restrict__ A, int lda,
                                                      unsigned long long* out, int check, int* status) {
    unsigned long long m = 0;
    bool bad = false;
    for (int j = blockIdx.x; j < n; j += gridDim.x)
        for (int i = j + 1 + threadIdx.x; i < n; i += 256) {
            const unsigned long long v =
                (unsigned long long)__double_as_longlong(A[(size_t)j * lda + i]) & 0x7fffffffffffffffull;
            if (v >= 0x7ff0000000000000ull) bad = true;
            else if (v > m) m = v;
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long w = __shfl_xor_sync(0xffffffffu, m, o);
        m = w > m ? w : m;
    }
    if ((threadIdx.x & 31) == 0) atomicMax(out, m);
    if (bad && check) sk_set_error(status, SKEW_ERR_NONFINITE);
}

// scale[0] = s (a power of two, s max |A| in [1/2, 1)), F = s A by rows as
// pairs (os_full_kernel's tiles)
__global__ void __launch_bounds__(256)
df_full_kernel(int n, const double* __restrict__ A, int lda, const unsigned long long* amax, float2* __restrict__ F,
               double* scale) {
    __shared__ float2 tile[32][33];
    const int bi = blockIdx.x * 32, bj = blockIdx.y * 32;
    if (bi < bj) return;
    const int e = (int)(*amax >> 52);
    const double s = *amax == 0 ? 1.0 : ldexp(1.0, max(-1000, min(1000, 1022 - e)));
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) scale[0] = s;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int jj = ty; jj < 32; jj += 8) {
        const int i = bi + tx, j = bj + jj;
        float2 v = make_float2(0.f, 0.f);
        if (i < n && j < n && i > j) v = df_from(A[(size_t)j * lda + i] * s);
        tile[jj][tx] = v;
        if (i < n && j < n && i > j) F[(size_t)j * n + i] = df_neg2(v);
        if (i < n && i == j) F[(size_t)j * n + i] = make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (int ii = ty; ii < 32; ii += 8) {
        const int i = bi + ii, j = bj + tx;
        if (i < n && j < n && i > j) F[(size_t)i * n + j] = tile[tx][ii];
    }
}

int df_srows(int n, int G) {
    const int rmax = (n + G - 1) / G;
    const size_t vec = 3 * sizeof(float2) * (size_t)(n | 1), row = sizeof(float2) * (size_t)(n | 1);
    const size_t cap = DF_SMEM;
    const int fit = vec + row > cap ? 0 : (int)((cap - vec) / row);
    return std::min(rmax, fit);
}

}  // namespace

int onestep_amax(cudaStream_t st, int n, const double* A, int lda, unsigned long long* amax) {
    df_amax_kernel<<<std::min(n, 4 * device_sms()), 256, 0, st>>>(n, A, lda, amax, 0, nullptr);
    count_launch();
    return cuda_ok(cudaGetLastError());
}

int onestep_widen(cudaStream_t st, size_t count, double* V) {
    df_widen_kernel<<<(int)std::min<size_t>((count + 255) / 256, 16384), 256, 0, st>>>(count, V);
    count_launch();
    return cuda_ok(cudaGetLastError());
}

int onestep_df_full(cudaStream_t st, int n, const double* A, int lda, void* F, int check, void* ws, size_t ws_bytes,
                    int* status) {
    Carve cv(ws, ws_bytes);
    cv.take<float4>(2 * (size_t)n);
    unsigned* ctr = cv.take<unsigned>(16);  // [0] arrivals, [2..3] max |A|, [4] the scale
    if (!cv.ok) return SKEW_ERR_WORKSPACE;
    auto* amax = reinterpret_cast<unsigned long long*>(ctr + 2);
    if (const cudaError_t e = cudaMemsetAsync(ctr, 0, 16 * sizeof(unsigned), st)) return cuda_fail(e);
    const int nb = (n + 31) / 32;
    df_amax_kernel<<<std::min(n, 4 * device_sms()), 256, 0, st>>>(n, A, lda, amax, check, status);
    df_full_kernel<<<dim3(nb, nb), 256, 0, st>>>(n, A, lda, amax, static_cast<float2*>(F),
                                                 reinterpret_cast<double*>(ctr + 4));
    count_launch(2);
    return cuda_ok(cudaGetLastError());
}

int onestep_df_reduce(cudaStream_t st, int n, void* F, double* V, double* tau, double* alpha, void* ws,
                      size_t ws_bytes, int* d_status, unsigned spin_cap) {
    if (n < 2) return 0;
    Carve cv(ws, ws_bytes);
    DfArgs o{};
    o.qa = cv.take<float4>(2 * (size_t)n);
    o.ctr = cv.take<unsigned>(16);
    if (!cv.ok) return SKEW_ERR_WORKSPACE;
    const size_t vc = (size_t)onestep_vcols(n);
    if (const cudaError_t e = cudaMemsetAsync(V, 0, sizeof(double) * vc * n, st)) return cuda_fail(e);
    if (const cudaError_t e = cudaMemsetAsync(tau, 0, sizeof(double) * vc, st)) return cuda_fail(e);
    const int G = std::min(device_sms(), (n + 1) / 2);
    if (n > DMAXR * G) return SKEW_ERR_UNSUPPORTED;
    o.n = n;
    o.F = static_cast<float2*>(F);
    o.V = reinterpret_cast<float2*>(V);
    o.tau = tau;
    o.alpha = alpha;
    o.scale = reinterpret_cast<const double*>(o.ctr + 4);
    o.status = d_status;
    o.cap = spin_cap ? spin_cap : SK_SPIN_CAP;
    o.srows = df_srows(n, G);
    const size_t dyn = sizeof(float2) * (size_t)(n | 1) * (3 + (size_t)o.srows);
    if (const cudaError_t e =
            cudaFuncSetAttribute(onestep_df_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, DF_SMEM))
        return cuda_fail(e);
    void* args[] = {&o};
    KtScope kt(st, KT_PANEL_QR);
    const cudaError_t e = cudaLaunchCooperativeKernel((void*)onestep_df_kernel, dim3(G), dim3(DT), args, dyn, st);
    count_launch();
    if (e == cudaErrorCooperativeLaunchTooLarge) return SKEW_ERR_LAUNCH;
    if (e != cudaSuccess) return cuda_fail(e);
    return onestep_widen(st, vc * (size_t)n, V);
}

}  // namespace sk
