// Register DFTs of the FFT passes: e^{+2 pi i / R} butterflies of R points with compile-time twiddles
// (composite R as nested Cooley-Tukey).
#pragma once
#include "fv_internal.cuh"

namespace fv {

// ---------------------------------------------------------------- compile-time twiddles
// e^{2 pi i m / R} for 2 <= R <= 16, from Taylor series on [0, pi/4] after an
// exact reduction of the rational angle m/R to an octant (constexpr, host compiler).
namespace cx {
constexpr double kPi = 3.14159265358979323846264338327950288;
constexpr double sin_t(double a)
{
    double t = a, s = a;
    for (int n = 1; n < 12; ++n) {
        t *= -a * a / ((2.0 * n) * (2.0 * n + 1.0));
        s += t;
    }
    return s;
}
constexpr double cos_t(double a)
{
    double t = 1.0, s = 1.0;
    for (int n = 1; n < 12; ++n) {
        t *= -a * a / ((2.0 * n - 1.0) * (2.0 * n));
        s += t;
    }
    return s;
}
struct SC { double s, c; };
constexpr SC sincos2pi(int m, int R)
{
    m %= R;
    if (m < 0) m += R;
    const long t = 4L * m;
    const int k = (int)(t / R);            // quarter turns
    const long rem = t - (long)k * R;      // remaining angle (pi/2) rem / R
    double s0 = 0, c0 = 0;
    if (2 * rem <= R) {
        const double a = (kPi / 2) * (double)rem / R;
        s0 = sin_t(a);
        c0 = cos_t(a);
    } else {
        const double a = (kPi / 2) * (double)(R - rem) / R;
        s0 = cos_t(a);
        c0 = sin_t(a);
    }
    if (k == 0) return {s0, c0};
    if (k == 1) return {c0, -s0};
    if (k == 2) return {-s0, -c0};
    return {-c0, s0};
}
}  // namespace cx

// v * e^{2 pi i m / R} with compile-time m, R: exact for the quarter turns, otherwise a product by
// constants folded at compile time (no table load, no FP64 conversion in the FP32 instances)
template <class G, int M_, int R>
__device__ __forceinline__ cpx<G> twm(cpx<G> v)
{
    constexpr int m = M_ % R;
    if constexpr (m == 0) return v;
    else if constexpr (4 * m == R) return cmuli(v);
    else if constexpr (2 * m == R) return cmk<G>(-v.x, -v.y);
    else if constexpr (4 * m == 3 * R) return cmk<G>(v.y, -v.x);
    else {
        constexpr cx::SC w = cx::sincos2pi(m, R);
        return cmul(v, cmk<G>((G)w.c, (G)w.s));
    }
}

// ---------------------------------------------------------------- register DFTs (+ sign)
template <int R> struct Fac {
    static constexpr int A = (R % 4 == 0 && R != 4) ? 4 : (R % 2 == 0 && R != 2) ? 2 : (R % 3 == 0 && R != 3) ? 3 : 5;
    static constexpr int B = R / A;
};

template <class G, int R> struct Dft;

template <class G> struct Dft<G, 1> {
    static __device__ __forceinline__ void run(cpx<G> *) {}
};
template <class G> struct Dft<G, 2> {
    static __device__ __forceinline__ void run(cpx<G> *v)
    {
        cpx<G> a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    }
};
template <class G> struct Dft<G, 3> {
    static __device__ __forceinline__ void run(cpx<G> *v)
    {
        const G h = (G)0.86602540378443864676;   // sin(2 pi / 3)
        cpx<G> t = cadd(v[1], v[2]), u = cmuli(cscale(csub(v[1], v[2]), h));
        cpx<G> m = csub(v[0], cscale(t, (G)0.5));
        v[0] = cadd(v[0], t);
        v[1] = cadd(m, u);
        v[2] = csub(m, u);
    }
};
template <class G> struct Dft<G, 4> {
    static __device__ __forceinline__ void run(cpx<G> *v)
    {
        cpx<G> s02 = cadd(v[0], v[2]), d02 = csub(v[0], v[2]);
        cpx<G> s13 = cadd(v[1], v[3]), d13 = cmuli(csub(v[1], v[3]));
        v[0] = cadd(s02, s13);
        v[2] = csub(s02, s13);
        v[1] = cadd(d02, d13);
        v[3] = csub(d02, d13);
    }
};
template <class G> struct Dft<G, 5> {
    static __device__ __forceinline__ void run(cpx<G> *v)
    {
        const G c1 = (G)0.30901699437494742410, c2 = (G)-0.80901699437494742410;   // cos(2pi/5), cos(4pi/5)
        const G s1 = (G)0.95105651629515357212, s2 = (G)0.58778525229247312917;    // sin(2pi/5), sin(4pi/5)
        cpx<G> t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]);
        cpx<G> u1 = csub(v[1], v[4]), u2 = csub(v[2], v[3]);
        cpx<G> a1 = cadd(v[0], cadd(cscale(t1, c1), cscale(t2, c2)));
        cpx<G> a2 = cadd(v[0], cadd(cscale(t1, c2), cscale(t2, c1)));
        cpx<G> b1 = cmuli(cadd(cscale(u1, s1), cscale(u2, s2)));
        cpx<G> b2 = cmuli(csub(cscale(u1, s2), cscale(u2, s1)));
        v[0] = cadd(v[0], cadd(t1, t2));
        v[1] = cadd(a1, b1);
        v[4] = csub(a1, b1);
        v[2] = cadd(a2, b2);
        v[3] = csub(a2, b2);
    }
};

// Composite R = A B: with r = B r1 + r2 and q = q1 + A q2,
// w_R^{rq} = w_A^{r1 q1} w_R^{r2 q1} w_B^{r2 q2}:
// A-point DFTs over r1 for every r2, twiddles w_R^{r2 q1}, B-point DFTs over r2.
template <class G, int R, int A, int R2, int Q1>
__device__ __forceinline__ void col_twiddle(const cpx<G> *t, cpx<G> *u)
{
    if constexpr (Q1 < A) {
        u[Q1] = twm<G, R2 * Q1, R>(t[Q1]);
        col_twiddle<G, R, A, R2, Q1 + 1>(t, u);
    }
}

template <class G, int R, int A, int B, int R2>
__device__ __forceinline__ void col_pass(const cpx<G> *v, cpx<G> (*U)[A])
{
    if constexpr (R2 < B) {
        cpx<G> t[A];
#pragma unroll
        for (int r1 = 0; r1 < A; ++r1) t[r1] = v[B * r1 + R2];
        Dft<G, A>::run(t);
        col_twiddle<G, R, A, R2, 0>(t, U[R2]);
        col_pass<G, R, A, B, R2 + 1>(v, U);
    }
}

template <class G, int R> struct Dft {
    static __device__ __forceinline__ void run(cpx<G> *v)
    {
        constexpr int A = Fac<R>::A, B = Fac<R>::B;
        cpx<G> U[B][A];
        col_pass<G, R, A, B, 0>(v, U);
#pragma unroll
        for (int q1 = 0; q1 < A; ++q1) {
            cpx<G> t[B];
#pragma unroll
            for (int r2 = 0; r2 < B; ++r2) t[r2] = U[r2][q1];
            Dft<G, B>::run(t);
#pragma unroll
            for (int q2 = 0; q2 < B; ++q2) v[q1 + A * q2] = t[q2];
        }
    }
};

}  // namespace fv
