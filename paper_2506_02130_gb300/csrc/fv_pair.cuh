// Pairs of floats hi + lo (|lo| <= ulp(hi) / 2, about 48 bits): GB300 has 64 FP32 operations for one of FP64, and a
// pair operation takes 6 to 12.  Sums and differences are written with the rounding intrinsics, so that no
// contraction changes their error terms.
#pragma once
#include "fv_internal.cuh"

namespace fv {

struct Pf { float h, l; };

__host__ __device__ __forceinline__ Pf pf(double v)
{
    const float h = (float)v;
    return Pf{h, (float)(v - (double)h)};
}
__device__ __forceinline__ Pf pmul(Pf a, Pf b)
{
    const float p = __fmul_rn(a.h, b.h);
    const float e = fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p)));
    const float h = __fadd_rn(p, e);
    return Pf{h, __fadd_rn(e, -__fadd_rn(h, -p))};
}
__device__ __forceinline__ Pf padd(Pf a, Pf b)
{
    const float s = __fadd_rn(a.h, b.h), t = __fadd_rn(s, -a.h);
    const float e = __fadd_rn(__fadd_rn(__fadd_rn(a.h, -__fadd_rn(s, -t)), __fadd_rn(b.h, -t)), __fadd_rn(a.l, b.l));
    const float h = __fadd_rn(s, e);
    return Pf{h, __fadd_rn(e, -__fadd_rn(h, -s))};
}

}  // namespace fv
