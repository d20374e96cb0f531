// pairs.cuh -- double-float values as float2 (hi, lo), about 2^-47 an operation
// (Dekker, "A floating-point technique for extending the available precision",
// 1971; Knuth's two-sum).
#pragma once
#include "common.cuh"

namespace sk {
namespace onestep {

// a += c d on an unnormalised pair: exact product of the leading parts, exact
// sum, the rest to first order (Dekker 1971; Knuth's two-sum).
SK_DEV void df_mac(float2& a, float2 c, float2 d) {
    const float p = __fmul_rn(c.x, d.x);  // not to be fused with the sum below
    float e = fmaf(c.x, d.x, -p);
    e = fmaf(c.x, d.y, e);
    e = fmaf(c.y, d.x, e);
    const float s = a.x + p, b = s - a.x;
    a.y += ((a.x - (s - b)) + (p - b)) + e;
    a.x = s;
}
// c d, not normalised: df_mac on zero without its sum.
SK_DEV float2 df_prod(float2 c, float2 d) {
    const float p = __fmul_rn(c.x, d.x);
    float e = fmaf(c.x, d.x, -p);
    e = fmaf(c.x, d.y, e);
    return make_float2(p, fmaf(c.y, d.x, e));
}
SK_DEV float2 df_norm(float2 a) {
    const float s = a.x + a.y;
    return make_float2(s, a.y - (s - a.x));
}
SK_DEV float2 df_sum(float2 a, float2 b) {
    const float s = a.x + b.x, t = s - a.x;
    const float e = ((a.x - (s - t)) + (b.x - t)) + (a.y + b.y);
    return df_norm(make_float2(s, e));
}
SK_DEV float2 df_mul2(float2 c, float2 d) {
    const float p = __fmul_rn(c.x, d.x);
    float e = fmaf(c.x, d.x, -p);
    e = fmaf(c.x, d.y, e);
    e = fmaf(c.y, d.x, e);
    return df_norm(make_float2(p, e));
}
SK_DEV float2 df_neg2(float2 a) { return make_float2(-a.x, -a.y); }
SK_DEV float2 df_scale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }  // s a power of two
SK_DEV float2 df_from(double x) {
    const float h = (float)x;
    return make_float2(h, (float)(x - (double)h));
}
SK_DEV double df_to(float2 a) { return (double)a.x + (double)a.y; }
SK_DEV float2 df_shfl(float2 a, int o) {
    return make_float2(__shfl_xor_sync(0xffffffffu, a.x, o), __shfl_xor_sync(0xffffffffu, a.y, o));
}
SK_DEV float2 df_warp_sum(float2 a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a = df_sum(a, df_shfl(a, o));
    return a;
}

// Quotient and square root: FP32 result, corrected by its exact remainder.
SK_DEV float2 df_quot(float2 a, float2 b) {
    const float q = __fdiv_rn(a.x, b.x);
    const float r = (fmaf(-q, b.x, a.x) + a.y) - __fmul_rn(q, b.y);
    return df_norm(make_float2(q, __fdiv_rn(r, b.x)));
}
SK_DEV float2 df_root(float2 a) {
    if (!(a.x > 0.f)) return make_float2(0.f, 0.f);
    const float q = __fsqrt_rn(a.x);
    const float r = fmaf(-q, q, a.x) + a.y;
    return df_norm(make_float2(q, __fdiv_rn(r, 2.f * q)));
}

}  // namespace onestep
}  // namespace sk
