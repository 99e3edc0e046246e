// One source of one FP32 slice from its per-time record: strengths with prephase, first footprint cells and
// offsets (shared by the prep kernels and the spreading that prepares its sources itself).
#pragma once
#include "fv_internal.cuh"

namespace fv {

// FP32 grids: the same strengths, prephase and grid coordinates from the per-time records tc (see
// launch_time_binning) without FP64 arithmetic.  Every channel's coordinate and prephase are the top
// channel's times r = kappa / kappa_top, formed in double-float arithmetic (an exact product by FMA plus
// the cross terms, about 2^-44 relative); the prephase is reduced by 2 pi split in two floats; the first
// footprint cell follows from the accurate offset l0 - q, which is brought into [-w/2, 1 - w/2).
__device__ __forceinline__ float2 mul_df(float ah, float al, float bh, float bl)
{
    const float p = ah * bh;
    const float e = fmaf(ah, bh, -p) + (ah * bl + al * bh);
    return make_float2(p, e);
}

// One source of one slice from its per-time record (a, b, sd) and source index n: strengths with prephase
// c[0..np), first footprint cells ci and offsets fr.
struct PrepOne {
    cpx<float> c[4];
    int np;
    int ci[3];
    float fr[3];
};

__device__ __forceinline__ void prep_tc_one(const float4 a, const float4 b, const float4 sd, long n, const void *flux,
                                            int flux_fp64, long n_src, int n_freq, int f, const SliceGeom &g,
                                            PrepOne &o)
{
    o.np = source_strengths<float, float>(g, sd.x, sd.y, sd.z, n, flux, flux_fp64, n_src, n_freq, f, o.c);
    // prephase r ph_top, reduced to about [-pi, pi]: 2 pi = 6.2831855 - 1.7484555e-7
    const float2 ph = mul_df(g.rsc_hi, g.rsc_lo, b.z, b.w);
    const float k = rintf(ph.x * 0.15915494f);
    const float phr = fmaf(-k, -1.7484555e-7f, fmaf(-k, 6.2831855f, ph.x)) + ph.y;
    float sp, cp;
    sincosf(phr, &sp, &cp);
#pragma unroll
    for (int p = 0; p < 4; ++p)
        if (p < o.np) o.c[p] = cmul(o.c[p], cmk<float>(cp, sp));
    const float hw = 0.5f * (float)g.w;
#pragma unroll
    for (int k3 = 0; k3 < 3; ++k3) {
        o.ci[k3] = 0;
        o.fr[k3] = 0.0f;
        if (k3 < g.d) {
            const float qh = k3 == 0 ? a.x : (k3 == 1 ? a.z : b.x), ql = k3 == 0 ? a.y : (k3 == 1 ? a.w : b.y);
            const float2 q = mul_df(g.rsc_hi, g.rsc_lo, qh, ql);
            float l0 = ceilf(q.x - hw);
            float off = (l0 - q.x) - q.y;                 // l0 - q
            if (off >= 1.0f - hw) { l0 -= 1.0f; off -= 1.0f; }
            else if (off < -hw) { l0 += 1.0f; off += 1.0f; }
            int c = (int)l0 + g.dim[k3].nf1 / 2;
            const int hi = g.dim[k3].nf1 - g.w;
            if (c < 0) { off -= (float)c; c = 0; }
            else if (c > hi) { off -= (float)(c - hi); c = hi; }
            o.ci[k3] = c;
            o.fr[k3] = off;
        }
    }
    if (g.K) o.fr[2] = (sd.z - g.hc_f) * g.hs_inv_f;    // height terms: the argument u of T_q
}

}  // namespace fv
