// Two-float arithmetic: a value held as the unevaluated sum h + l of two
// binary32 numbers, |l| <= ulp(h)/2, about 48 significant bits. It stands in
// for binary64 in the per-cell sums and drag solves of the FP32 state, whose
// results are rounded to binary32 once at the end: sm_103a has 2 binary64
// lanes per SM and clock against 128 binary32 lanes, and the cell update of a
// 101^3 box spent 84 % of the binary64 pipe's cycles on those sums.
// Against the same kernels in binary64, on 1D shocks, 2D columns with
// gradients, 3D boxes and 1D ensembles of all sizes: states equal bit for bit,
// gradients 2e-10 apart, errors against 64-bit values the same in every case
// (101^3 box 762 -> 635 us, shock of 2e5 791 -> 638, 512^2 column 12.5 -> 9.4 ms,
// 24 waves 785 -> 680 us, 256 waves of a drawn ensemble 1672 -> 1227 us).
//
// Algorithms and relative error bounds (u = 2^-24): Joldes, Muller, Popescu,
// "Tight and rigorous error bounds for basic building blocks of double-word
// arithmetic", ACM TOMS 44 (2017): value + float 2u^2 (Alg. 4), value + value
// 3u^2 (Alg. 6), value x value 4u^2 (Alg. 12, with FMA), quotient about 15u^2
// (the scheme of Alg. 17, whose first quotient only has to be close). Every
// operation is an explicitly rounded intrinsic, so nothing is contracted.
//
// The exponent range is binary32's: the callers test what follows and take
// binary64 for the cell otherwise (df_drag_fits, df_vel_fits, and the lambdas
// of the cell adjoint). Sums of velocities and accelerations are not tested by
// themselves: their low parts are lost below 2^-149 only, and the velocities
// that come of them are at least 2^-80 or zero.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace tfsph {

struct df {
    float h, l;
    df() = default;
    __host__ __device__ __forceinline__ df(float hi, float lo) : h(hi), l(lo) {}
    __host__ __device__ __forceinline__ explicit df(float x) : h(x), l(0.0f) {}
    __host__ __device__ __forceinline__ explicit df(double x) : h((float)x), l(0.0f)
    {
        l = (float)(x - (double)h);
    }
    // counts: exact (both parts) for every 32-bit value
    __device__ __forceinline__ explicit df(uint32_t n)
    {
        h = __uint2float_rn(n & 0xffff0000u);
        l = __uint2float_rn(n & 0xffffu);
        const float s = __fadd_rn(h, l);
        l = __fsub_rn(l, __fsub_rn(s, h));
        h = s;
    }
    __host__ __device__ __forceinline__ explicit operator float() const { return h; }
};

// s + e = a + b exactly (fast form: |a| >= |b|, or a = 0)
__device__ __forceinline__ df df_fast_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    return df(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ df df_two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    return df(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}

__device__ __forceinline__ df operator+(df x, float y)
{
    const df s = df_two_sum(x.h, y);
    return df_fast_two_sum(s.h, __fadd_rn(x.l, s.l));
}
__device__ __forceinline__ df operator+(df x, df y)
{
    const df s = df_two_sum(x.h, y.h);
    const df t = df_two_sum(x.l, y.l);
    const df v = df_fast_two_sum(s.h, __fadd_rn(s.l, t.h));
    return df_fast_two_sum(v.h, __fadd_rn(t.l, v.l));
}
__device__ __forceinline__ df operator-(df x) { return df(-x.h, -x.l); }
__device__ __forceinline__ df operator-(df x, df y) { return x + (-y); }
__device__ __forceinline__ df operator*(df x, df y)
{
    const float c = __fmul_rn(x.h, y.h);
    const float e = __fmaf_rn(x.h, y.h, -c);
    const float t = __fmaf_rn(x.l, y.h, __fmaf_rn(x.h, y.l, __fmul_rn(x.l, y.l)));
    return df_fast_two_sum(c, __fadd_rn(e, t));
}
__device__ __forceinline__ df operator/(df x, df y)
{
    // one Newton correction of the float quotient q: x - q y is formed with
    // the error of its leading product, so q's own error only enters squared
    const float q = __fdividef(x.h, y.h);
    const float c = __fmul_rn(y.h, q);
    const float e = __fmaf_rn(y.h, q, -c);
    const float d = __fadd_rn(__fsub_rn(x.h, c), __fsub_rn(x.l, __fmaf_rn(y.l, q, e)));
    return df_fast_two_sum(q, __fdividef(d, y.h));
}
__device__ __forceinline__ df &operator+=(df &x, float y) { return x = x + y; }
__device__ __forceinline__ df &operator+=(df &x, df y) { return x = x + y; }
__device__ __forceinline__ df &operator-=(df &x, df y) { return x = x - y; }

// x nonzero and so small that a low part or a product of low parts may
// underflow (the binary64 form then keeps more digits)
__device__ __forceinline__ bool df_small(df x) { return x.h != 0.0f && !(fabsf(x.h) >= 0x1p-80f); }
// lo <= x <= hi (false for NaN)
__device__ __forceinline__ bool df_in(df x, float lo, float hi) { return x.h >= lo && x.h <= hi; }

// The scalars of a cell's drag solve: tau, the sum over the stopping times (or
// their inverses), the masses of its gas and dust, rt = tau/t* and eps*. Within
// these bounds every product and quotient that leads to rt and eps* keeps its
// low part, and inverses of stopping times beyond 2^126, which are taken as 0,
// are below 2^-46 of their sum.
__device__ __forceinline__ bool df_drag_fits(df tau, df st, df gas, df dust, df rt, df eps)
{
    return df_in(tau, 0x1p-80f, 0x1p60f) && df_in(st, 0x1p-80f, 0x1p100f) && df_in(gas, 0x1p-80f, 0x1p100f) &&
           df_in(dust, 0x1p-80f, 0x1p100f) && df_in(rt, 0x1p-60f, 0x1p24f) && df_in(eps, 0x1p-40f, 0x1p40f);
}
// One component of the solve: w', u*', v*' (|u*'|, |v*'| at most `most`).
__device__ __forceinline__ bool df_vel_fits(df wn, df un, df vn, float most)
{
    return !df_small(wn) && !df_small(un) && !df_small(vn) && df_in(un, -most, most) && df_in(vn, -most, most);
}

}  // namespace tfsph
