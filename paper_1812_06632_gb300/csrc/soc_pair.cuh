// soc_pair.cuh -- pairs of FP32 numbers (hi + lo, about 48 bits) for the
// Planck function where FP64, issued at 2 lanes per clock and SM, would bound
// a kernel.  Explicitly rounded operations only; every translation unit that
// includes this is compiled with -fmad=false.
#pragma once
#include <cstdint>

namespace soc {
namespace {

__device__ __forceinline__ float rcp(float v) { float r; asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(v)); return r; }

// A sum of FP32 numbers a + b = s + e exactly (Knuth's two-sum; the short
// form needs |a| >= |b| or a = 0).
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
}
__device__ __forceinline__ void quick_two_sum(float a, float b, float &s, float &e)
{
    const float t = __fadd_rn(a, b);
    e = __fsub_rn(b, __fsub_rn(t, a));
    s = t;
}

// 2^(j/32) - 1 as hi + lo, j = 0 .. 31 (Taylor series of exp(j ln2 / 32)).
struct Exp2Table { float h[32], l[32]; };
constexpr Exp2Table make_exp2_table()
{
    Exp2Table t{};
    for (int j = 0; j < 32; ++j) {
        const double a = 0.69314718055994530942 * j / 32.0;
        double term = 1.0, sum = 0.0;
        for (int n = 1; n < 24; ++n) { term = term * a / n; sum += term; }
        t.h[j] = (float)sum;
        t.l[j] = (float)(sum - (double)t.h[j]);
    }
    return t;
}
__device__ const Exp2Table g_exp2_table = make_exp2_table();

// y >= 0 on the grid of 32nds: the nearest n / 32 carries in the low bits of
// pair_grid(y), pair_index gives n (y above 2048 is taken as 2048).
__device__ __forceinline__ float pair_grid(float y) { return __fmaf_rn(fminf(y, 2048.0f), 32.0f, 12582912.0f); }
__device__ __forceinline__ int pair_index(float grid) { return __float_as_int(grid) - 0x4B400000; }

// (2^(p + pe) - 1) 2^-(n >> 5) as eh + el, grid = pair_grid(p), n its index;
// th, tl: the table's entry of this lane (the whole warp calls it).  Relative
// error below 2^-41 (1 + 1 / eh) 0.2 over p = 2^-8 .. 900, exact exponent aside.
__device__ __forceinline__ void pair_expm1(float p, float pe, float grid, int n, float th, float tl, float &eh, float &el)
{
    constexpr float kLn2H = 0x1.62e43p-1f, kLn2L = -0x1.05c61p-29f;          // ln 2, hi + lo
    // p + pe = n / 32 + s, |s| <= 1/64
    const float d = __fmaf_rn(__fsub_rn(grid, 12582912.0f), -0.03125f, p);
    float sh, sl;
    two_sum(d, pe, sh, sl);
    // a = e^(s ln2) - 1 (Taylor to the fifth power)
    const float rh = __fmul_rn(sh, kLn2H);
    const float rl = __fmaf_rn(sl, kLn2H, __fmaf_rn(sh, kLn2L, __fmaf_rn(sh, kLn2H, -rh)));
    const float r2 = __fmul_rn(rh, rh);
    const float r2l = __fmaf_rn(__fadd_rn(rh, rh), rl, __fmaf_rn(rh, rh, -r2));
    const float q = __fmul_rn(__fmul_rn(rh, r2), __fmaf_rn(rh, __fmaf_rn(rh, 0x1.111112p-7f, 0x1.555556p-5f),
                           0x1.555556p-3f));
    float ah, al;
    quick_two_sum(rh, __fmul_rn(0.5f, r2), ah, al);
    al = __fadd_rn(al, __fadd_rn(__fmaf_rn(0.5f, r2l, rl), q));
    // 2^(n/32 - k) e^(s ln2) - 1 = t + a + t a, t = 2^(j/32) - 1
    const float t1 = __shfl_sync(0xffffffffu, th, n & 31), t1l = __shfl_sync(0xffffffffu, tl, n & 31);
    const float ta = __fmul_rn(t1, ah);
    const float tal = __fmaf_rn(t1l, ah, __fmaf_rn(t1, al, __fmaf_rn(t1, ah, -ta)));
    float s1, e1, s2, e2;
    quick_two_sum(t1, ah, s1, e1);
    quick_two_sum(s1, ta, s2, e2);
    const float lo = __fadd_rn(__fadd_rn(__fadd_rn(e1, e2), __fadd_rn(al, tal)), t1l);
    // (2^y - 1) 2^-k = (1 - 2^-k) + that
    const int k = n >> 5;
    const float mk = k < 120 ? __uint_as_float((uint32_t)(127 - max(k, 0)) << 23) : 0.0f;
    const float c1 = __fsub_rn(1.0f, mk), ce = __fsub_rn(__fsub_rn(1.0f, c1), mk);
    two_sum(c1, s2, eh, el);
    // normalised: the quotient's correction is good to (el / eh)^2
    quick_two_sum(eh, __fadd_rn(el, __fadd_rn(ce, lo)), eh, el);
}

}  // namespace
}  // namespace soc
