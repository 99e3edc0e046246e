// Pairs of floats hi + lo (|lo| <= ulp(hi) / 2, about 48 bits): GB300 has 64 FP32 operations for one of FP64, and a
// pair operation takes 6 to 12.  Sums and differences are written with the rounding intrinsics, so that no
// contraction changes their error terms.
#pragma once
#include "fv_internal.cuh"

namespace fv {

struct Pf {
    float h, l;
    Pf() = default;
    __host__ __device__ constexpr Pf(float h_, float l_) : h(h_), l(l_) {}
    __host__ __device__ constexpr explicit Pf(double v) : h((float)v), l((float)(v - (double)(float)v)) {}
};

__host__ __device__ __forceinline__ Pf pf(double v) { return Pf(v); }
__device__ __forceinline__ double pf_value(Pf a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ Pf pmul(Pf a, Pf b)
{
    const float p = __fmul_rn(a.h, b.h);
    const float e = fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p)));
    const float h = __fadd_rn(p, e);
    return Pf(h, __fadd_rn(e, -__fadd_rn(h, -p)));
}
// a + b without the last step that brings lo below hi's rounding: enough inside a few sums before a product
__device__ __forceinline__ Pf padd_raw(Pf a, Pf b)
{
    const float s = __fadd_rn(a.h, b.h), t = __fadd_rn(s, -a.h);
    return Pf(s, __fadd_rn(__fadd_rn(__fadd_rn(a.h, -__fadd_rn(s, -t)), __fadd_rn(b.h, -t)), __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ Pf padd(Pf a, Pf b)
{
    const Pf r = padd_raw(a, b);
    const float h = __fadd_rn(r.h, r.l);
    return Pf(h, __fadd_rn(r.l, -__fadd_rn(h, -r.h)));
}
__device__ __forceinline__ Pf operator-(Pf a) { return Pf(-a.h, -a.l); }
__device__ __forceinline__ Pf operator+(Pf a, Pf b) { return padd_raw(a, b); }
__device__ __forceinline__ Pf operator-(Pf a, Pf b) { return padd_raw(a, -b); }
__device__ __forceinline__ Pf operator*(Pf a, Pf b) { return pmul(a, b); }

// Pairs have a float's range.  Strengths are brought into it by a power of two, exactly, where their largest exponent
// field (key, 11 bits) leaves [2^-40, 2^30]: far enough from the float limits for tens of bits of products and sums.
__device__ __forceinline__ unsigned exponent_key(double v) { return ((unsigned)__double2hiint(v) >> 20) & 0x7ffu; }
__device__ __forceinline__ int pair_shift(unsigned key)
{
    const int e = (int)key - 1023;
    return key == 0x7ffu || (e >= -40 && e <= 30) ? 0 : -e;      // infinities and NaN pass as they are
}

// Two pairs side by side (the real and imaginary part), in packed arithmetic.
struct Pair2 { float2 h, l; };
__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float2 neg2(float2 a) { return __fmul2_rn(a, make_float2(-1.0f, -1.0f)); }
// a b: the rounded product and its error, with the low parts' cross terms
__device__ __forceinline__ Pair2 pair2_times(float2 ah, float2 al, float2 bh, float2 bl)
{
    Pair2 r;
    r.h = __fmul2_rn(ah, bh);
    r.l = __ffma2_rn(ah, bh, neg2(r.h));
    r.l = __ffma2_rn(ah, bl, r.l);
    r.l = __ffma2_rn(al, bh, r.l);
    return r;
}
// a += p (the low part is not brought below the high part's rounding)
__device__ __forceinline__ void pair2_add(Pair2 &a, const Pair2 &p)
{
    const float2 s = add2(a.h, p.h), t = sub2(s, a.h);
    a.l = add2(a.l, add2(add2(sub2(a.h, sub2(s, t)), sub2(p.h, t)), p.l));
    a.h = s;
}

// Bring the low part below the high part's rounding.  pair2_add lets it grow with the number of terms, and its own
// rounding with it: sums of 256, 4,096 and 20,000 random terms are off by 7e-14, 1.2e-12 and 4.6e-12 of their value
// without it, by 4.5e-14, 1.6e-13 and 4.5e-13 with it every 64 terms.
__device__ __forceinline__ void pair2_tidy(Pair2 &a)
{
    const float2 h = add2(a.h, a.l);
    a.l = sub2(a.l, sub2(h, a.h));
    a.h = h;
}

}  // namespace fv
