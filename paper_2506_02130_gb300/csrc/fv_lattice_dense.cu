// Lattice arrays without a grid: the mode sums of Section 2.2.1 evaluated directly.
//
// With baselines b = n_1 a_1 + n_2 a_2 (+ b_up) a slice needs, for every height term q and product,
//     W_j(n) = sum_s r_js e^{-i n_1 x_1s} e^{-i n_2 x_2s},   r_js = strength x T_q(u_s), real,
// at the few hundred modes n of the array.  The strengths are real (a polarised sky's four products follow from
// the real strengths I + Q', I - Q', U', V), so W_j(-n) = conj W_j(n) and half of the modes do.  A source costs one
// complex product per mode, shared by all terms, and one packed multiply-add per mode and term, all in registers:
// a thread holds a tile of modes x terms and walks the sources, whose phase factors e^{-i n x} and real strengths
// the CTA has put in shared memory up to 64 at a time.  Groups of threads and CTAs take different sources and
// add their sums with global reductions.  There is no spreading kernel, grid, FFT or deconvolution, and every
// channel of a time goes into one launch.
//
// Why (skies of up to 50,000 sources, or few enough modes: dense_modes_max): the type-1 transform of such an array spread each source over w^2 cells of every term's grid with
// shared-memory float atomics (each a compare-and-swap loop): 74 us of a 127-antenna slice (35,000 sources, 7 terms)
// beside 35 us for strengths, clearing, FFT passes and lookup.  The direct sum has more multiply-adds (about 290
// modes x 9 packed operations a source) but they run on the FMA pipe, about 40 % of whose rate it reaches: 17.7 us
// a slice (64 channels a launch, one stream) and 0.9 us of lookup; the rest is the waits for shared memory and at
// the chunks' barriers.  It is also more accurate (no kernel aliasing): 1.9e-7 against 7e-7 of relative L2.
//
// FP64 plans (eps >= 1e-12) use pairs of floats (hi + lo, about 2^-47 relative per operation): GB300 has 64 FP32
// multiply-adds for one of FP64, and a pair operation takes about 12.  Phases, strengths and the final sums of the
// CTAs are FP64.  A 37-antenna slice of 1,000 sources takes 29 us (172 us of FP64 spreading, 63 of preparation and
// 28 of FFT passes before) with an error against the direct sum of 1.3e-14 where the transform gave 5.8e-11.
#include "fv_lattice_dense.cuh"
#include "fv_pair.cuh"

#include <algorithm>

namespace fv {

namespace {

constexpr int kDenseThreads = 256;
constexpr int kDenseChain = 256;          // sources a thread's sum takes before it goes to the FP64 sums

// the arithmetic of one precision: values in shared memory and the thread's sums
template <class G> struct Dense;
template <> struct Dense<float> {
    static constexpr int V = 1, SW = 1;                  // float4 per phase factor, float2 per strength
    using Acc = float2;
    using E = float2;
    static __device__ __forceinline__ Acc zero() { return make_float2(0.0f, 0.0f); }
    // e: (re, re, im, im) of the n_2 factor, b: (re, im, -im, re) of the n_1 factor
    static __device__ __forceinline__ E product(const float4 *e, const float4 *b)
    {
        const float4 x = *e, y = *b;
        return __ffma2_rn(make_float2(x.z, x.w), make_float2(y.z, y.w),
                          __fmul2_rn(make_float2(x.x, x.y), make_float2(y.x, y.y)));
    }
    static __device__ __forceinline__ void add(Acc &a, const float2 *w, E e) { a = __ffma2_rn(*w, e, a); }
    static __device__ __forceinline__ void join(Acc &a, Acc b) { a = __fadd2_rn(a, b); }
    static __device__ __forceinline__ cpx<double> value(Acc a) { return cmk<double>((double)a.x, (double)a.y); }
};
template <> struct Dense<double> {
    static constexpr int V = 2, SW = 2;
    using Acc = Pair2;
    using E = Pair2;
    static __device__ __forceinline__ Acc zero() { return Pair2{make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)}; }
    static __device__ __forceinline__ E product(const float4 *e, const float4 *b)
    {
        const float4 eh = e[0], el = e[1], bh = b[0], bl = b[1];
        const Pair2 p = pair2_times(make_float2(eh.x, eh.y), make_float2(el.x, el.y), make_float2(bh.x, bh.y),
                                    make_float2(bl.x, bl.y));
        const Pair2 q = pair2_times(make_float2(eh.z, eh.w), make_float2(el.z, el.w), make_float2(bh.z, bh.w),
                                    make_float2(bl.z, bl.w));
        const float2 s = add2(p.h, q.h), t = sub2(s, p.h);
        const float2 l = add2(add2(add2(sub2(p.h, sub2(s, t)), sub2(q.h, t)), p.l), q.l);
        E r;
        r.h = add2(s, l);
        r.l = sub2(l, sub2(r.h, s));
        return r;
    }
    static __device__ __forceinline__ void add(Acc &a, const float2 *w, const E &e)
    {
        pair2_add(a, pair2_times(w[0], w[1], e.h, e.l));
    }
    static __device__ __forceinline__ void join(Acc &a, const Acc &b) { pair2_add(a, b); }
    static __device__ __forceinline__ cpx<double> value(const Acc &a)
    {
        return cmk<double>((double)a.h.x + (double)a.l.x, (double)a.h.y + (double)a.l.y);
    }
};

}  // namespace

// Channels f0 + blockIdx.y of one time, sources of CTA blockIdx.x of gridDim.x, terms and tiles of blockIdx.z.
template <class G, int JB, int TA, int TB>
__global__ void __launch_bounds__(kDenseThreads, 2)
    k_lattice_dense(const double *__restrict__ sdir, const float4 *__restrict__ tc, const int *__restrict__ sidx, const int *__restrict__ nv_ptr,
                    long n_src, const void *__restrict__ flux, int flux_fp64, int n_freq, int f0,
                    const double *__restrict__ freq, SliceGeom g0, DenseGeom dg, cpx<double> *__restrict__ out)
{
    using D = Dense<G>;
    constexpr int V = D::V, SW = D::SW;
    constexpr int BX = sizeof(G) == 4 ? 4 : 8;                            // floats of a source's phases
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int NA = dg.NA, NB = dg.NB, CS = dg.CS;
    float4 *s_e = reinterpret_cast<float4 *>(smem_raw);                  // [CS][NA][V]: n_2 factors
    float4 *s_b = s_e + (size_t)CS * NA * V;                             // [CS][NB][V]: n_1 factors
    float2 *s_w = reinterpret_cast<float2 *>(s_b + (size_t)CS * NB * V);  // [CS][JB][SW]: real strengths, twice
    // a block of sources prepared at once, one a thread: strengths x terms, and the phases (FP32: turns of x_1 and
    // x_2 as hi, lo; FP64: e^{-i x_1}, e^{-i x_2} as pairs)
    const size_t tables = max((size_t)((unsigned char *)(s_w + (size_t)CS * JB * SW) - smem_raw),
                              kDenseThreads * TB * sizeof(typename D::Acc));
    float *s_x = reinterpret_cast<float *>(smem_raw + tables);           // [kDenseThreads][BX]
    G *s_r = reinterpret_cast<G *>(s_x + kDenseThreads * BX);            // [kDenseThreads][JB]
    const int f = f0 + blockIdx.y;
    const int nv = *nv_ptr;
    const int per = (nv + (int)gridDim.x - 1) / (int)gridDim.x;
    const int first = blockIdx.x * per, last = min(nv, first + per);
    if (first >= last) return;                                            // the same on every thread of the CTA
    SliceGeom g = g0;
    g.nu = freq[f];
    g.nu_f = (float)g.nu;
    const double turns = g.nu / FV_C_LIGHT;                               // kappa / 2 pi
    const float turns_h = (float)turns, turns_l = (float)(turns - (double)turns_h);
    const int jb = blockIdx.z / dg.tile_blocks, tb = blockIdx.z - jb * dg.tile_blocks;
    const int tile0 = tb * kDenseThreads, tiles = min(kDenseThreads, dg.n_tiles - tile0);
    const int j0 = jb * JB, nj = min(JB, dg.J - j0);
    const int groups = kDenseThreads / tiles;
    const int grp = threadIdx.x / tiles, tl = threadIdx.x - grp * tiles;
    const bool work = grp < groups;
    const int tile = work ? dg.tiles[tile0 + tl] : 0;
    const int a0 = tile & 0xffff, b0 = tile >> 16;                        // first n_2 and n_1 + H_1 of the tile
    // n_1 factors: value c = n_1 + H_1 at (c mod TB)(NB / TB) + c / TB, so that the tiles of neighbouring lanes read
    // neighbouring 16 bytes
    const int nbt = NB / TB;
    auto at = [&](int c) { return (c % TB) * nbt + c / TB; };
    const int n1 = 2 * dg.H1 + 1, n2 = dg.H2 + 1;
    out += (size_t)blockIdx.y * dg.J * n1 * n2;
    typename D::Acc acc[JB][TA][TB];
#pragma unroll
    for (int j = 0; j < JB; ++j)
#pragma unroll
        for (int a = 0; a < TA; ++a)
#pragma unroll
            for (int b = 0; b < TB; ++b) acc[j][a][b] = D::zero();
    int held = 0;                                                          // sources in the thread's sums
    // FP64: the sums' power of two (pair_shift of each block of sources; a block with another one starts new sums)
    __shared__ unsigned s_key[2];
    int shift = 0, par = 0;
    double up = 1.0, down = 1.0;
    if constexpr (sizeof(G) == 8) {
        if (threadIdx.x < 2) s_key[threadIdx.x] = 0u;
        __syncthreads();
    }
    // the sums to the FP64 sums in memory: the groups' are added up through shared memory first (over the tables),
    // since every group and CTA adds to the same few hundred modes
    auto flush = [&]() {
        typename D::Acc *buf = reinterpret_cast<typename D::Acc *>(smem_raw);
#pragma unroll
        for (int j = 0; j < JB; ++j) {
            if (j >= nj) break;
#pragma unroll
            for (int i = 0; i < TA; ++i) {
                __syncthreads();
#pragma unroll
                for (int k = 0; k < TB; ++k) {
                    if (work) buf[threadIdx.x * TB + k] = acc[j][i][k];
                    acc[j][i][k] = D::zero();
                }
                __syncthreads();
                for (int o = threadIdx.x; o < tiles * TB; o += kDenseThreads) {
                    const int t = dg.tiles[tile0 + o / TB];
                    const int row = (t & 0xffff) + i, col = (t >> 16) + o % TB;
                    if (row >= n2 || col >= n1) continue;
                    typename D::Acc v = buf[o];
                    for (int q = 1; q < groups; ++q) D::join(v, buf[q * tiles * TB + o]);
                    const cpx<double> r = D::value(v);
                    cpx<double> *d = out + ((size_t)(j0 + j) * n2 + row) * n1 + col;
                    atomicAdd(&d->x, sizeof(G) == 8 ? r.x * down : r.x);
                    atomicAdd(&d->y, sizeof(G) == 8 ? r.y * down : r.y);
                }
            }
        }
    };

    for (int block = first; block < last; block += kDenseThreads) {
        const int nblk = min(kDenseThreads, last - block);
        // (the last chunk's barrier is behind every thread: s_x and s_r are free)
        if (threadIdx.x < nblk) {
            const long i = block + threadIdx.x;
            cpx<G> c[4];
            G u;
            float *x = s_x + threadIdx.x * BX;
            if constexpr (sizeof(G) == 4) {
                // the time's records: a_d . s (m) as float pairs and the direction; phases in turns by a pair product
                const float4 as = tc[2 * i], sd = tc[2 * i + 1];
                source_strengths<G, float>(g, sd.x, sd.y, sd.z, sidx[i], flux, flux_fp64, n_src, n_freq, f, c);
                u = sd.w;
#pragma unroll
                for (int d = 0; d < 2; ++d) {
                    const float ah = d == 0 ? as.x : as.z, al = d == 0 ? as.y : as.w;
                    const float ph = turns_h * ah, pl = fmaf(turns_h, ah, -ph) + (turns_h * al + turns_l * ah);
                    x[2 * d] = ph - rintf(ph);
                    x[2 * d + 1] = pl;
                }
            } else {
                const double s0 = sdir[i], s1 = sdir[n_src + i], s2 = sdir[2 * n_src + i];
                source_strengths<G>(g, s0, s1, s2, sidx[i], flux, flux_fp64, n_src, n_freq, f, c);
                u = (G)(2.0 * s2 - 1.0);
#pragma unroll
                for (int d = 0; d < 2; ++d) {
                    double v = turns * (dg.a[d][0] * s0 + dg.a[d][1] * s1);
                    v -= rint(v);
                    double sn, cn;
                    sincospi(2.0 * v, &sn, &cn);
                    const Pf re = pf(cn), im = pf(-sn);
                    x[4 * d] = re.h;
                    x[4 * d + 1] = re.l;
                    x[4 * d + 2] = im.h;
                    x[4 * d + 3] = im.l;
                }
            }
            G r[4] = {c[0].x, (G)0, (G)0, (G)0};
            if (g.n_pol == 4) {
                r[1] = c[3].x;                    // I - Q'
                r[2] = c[1].x;                    // U'
                r[3] = c[1].y;                    // V
            }
            if constexpr (sizeof(G) == 8) {
                const unsigned e = max(max(exponent_key(r[0]), exponent_key(r[1])),
                                       max(exponent_key(r[2]), exponent_key(r[3])));
                const unsigned lanes = __activemask();
                const unsigned m = __reduce_max_sync(lanes, e);
                if ((threadIdx.x & 31) == __ffs(lanes) - 1) atomicMax(&s_key[par], m);
            }
            int p = j0 / dg.K, q = j0 - p * dg.K;
            G tm = u, t = (G)1;                   // T_{-1} = T_1, T_0
            for (int k = 0; k < q; ++k) {
                const G tn = k == 0 ? u : (G)2 * u * t - tm;
                tm = t;
                t = tn;
            }
#pragma unroll
            for (int j = 0; j < JB; ++j) {
                const G rp = p == 0 ? r[0] : (p == 1 ? r[1] : (p == 2 ? r[2] : r[3]));
                s_r[threadIdx.x * JB + j] = j < nj ? rp * t : (G)0;
                if (++q == dg.K) {
                    q = 0;
                    ++p;
                    tm = u;
                    t = (G)1;
                } else {
                    const G tn = q == 1 ? u : (G)2 * u * t - tm;
                    tm = t;
                    t = tn;
                }
            }
        }
        __syncthreads();
        if constexpr (sizeof(G) == 8) {
            const int sh = pair_shift(s_key[par]);
            par ^= 1;
            if (threadIdx.x == 0) s_key[par] = 0u;       // last read before the chunks' barriers of the block before
            if (sh != shift) {                           // the same on every thread
                if (held > 0) {
                    flush();
                    held = 0;
                    __syncthreads();                     // the sums have been read: the tables may be written
                }
                shift = sh;
                up = scalbn(1.0, sh);
                down = scalbn(1.0, -sh);
            }
        }
        for (int base = 0; base < nblk; base += CS) {
            const int n = min(CS, nblk - base);
            // the chunk's tables: strengths, n_2 factors as (re, re, im, im), n_1 factors as (re, im, -im, re)
            for (int k = threadIdx.x; k < n * JB; k += kDenseThreads) {
                const G v = s_r[base * JB + k];
                float2 *w = s_w + (size_t)k * SW;
                if constexpr (sizeof(G) == 4) {
                    w[0] = dup((float)v);
                } else {
                    const Pf y = pf((double)v * up);
                    w[0] = dup(y.h);
                    w[1] = dup(y.l);
                }
            }
            if constexpr (sizeof(G) == 4) {
                // every factor from its own reduced phase, m (hi + lo) turns; n_1 < 0 by conjugation
                const int nbp = NB - dg.H1, per_src = NA + nbp;           // n_1 = 0 .. NB - 1 - H_1
                for (int k = threadIdx.x; k < n * per_src; k += kDenseThreads) {
                    const int s = k / per_src, v = k - s * per_src;
                    const bool e2 = v < NA;
                    const int m = e2 ? v : v - NA;                         // power
                    const float *x = s_x + (base + s) * BX + (e2 ? 2 : 0);
                    const float fm = (float)m, ph = fm * x[0];
                    const float fr = (ph - rintf(ph)) + (fmaf(fm, x[0], -ph) + fm * x[1]);
                    float sn, cn;
                    sincospif(2.0f * fr, &sn, &cn);
                    if (m > (e2 ? dg.H2 : dg.H1)) sn = cn = 0.0f;          // padding
                    if (e2) {
                        s_e[(size_t)s * NA + m] = make_float4(cn, cn, -sn, -sn);
                    } else {
                        float4 *row = s_b + (size_t)s * NB;
                        row[at(dg.H1 + m)] = make_float4(cn, -sn, sn, cn);
                        if (m > 0 && m <= dg.H1) row[at(dg.H1 - m)] = make_float4(cn, sn, -sn, cn);
                    }
                }
                __syncthreads();
            } else {
                // powers by doubling: z^n = z^m z^(n - m), n in (m, 2m], for both axes
                for (int k = threadIdx.x; k < n; k += kDenseThreads) {
                    const float *x = s_x + (base + k) * BX;
                    float4 *e = s_e + (size_t)k * NA * V, *b = s_b + ((size_t)k * NB + at(dg.H1)) * V;
                    e[0] = make_float4(1.0f, 1.0f, 0.0f, 0.0f);
                    b[0] = make_float4(1.0f, 0.0f, 0.0f, 1.0f);
                    e[1] = b[1] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    if (NA > 1) {
                        e[V] = make_float4(x[4], x[4], x[6], x[6]);
                        e[V + 1] = make_float4(x[5], x[5], x[7], x[7]);
                    }
                    if (dg.H1 > 0) {
                        b = s_b + ((size_t)k * NB + at(dg.H1 + 1)) * V;
                        b[0] = make_float4(x[0], x[2], -x[2], x[0]);
                        b[1] = make_float4(x[1], x[3], -x[3], x[1]);
                    }
                }
                const int HA = NA - 1, HB = dg.H1;
                for (int m = 1; m < max(HA, HB); m *= 2) {
                    __syncthreads();
                    const int na = max(0, min(2 * m, HA) - m), nb = max(0, min(2 * m, HB) - m);
                    for (int k = threadIdx.x; k < n * (na + nb); k += kDenseThreads) {
                        const int s = k / (na + nb), v = k - s * (na + nb);
                        const bool e2 = v < na;
                        const int step = e2 ? v + 1 : v - na + 1;          // n = m + step
                        float4 *zb = e2 ? s_e + (size_t)s * NA * V : s_b + (size_t)s * NB * V;
                        const float4 *zx = zb + (e2 ? m : at(dg.H1 + m)) * V, *zy = zb + (e2 ? step : at(dg.H1 + step)) * V;
                        const float4 xh = zx[0], xl = zx[1], yh = zy[0], yl = zy[1];
                        const Pf xr{xh.x, xl.x}, yr{yh.x, yl.x};
                        const Pf xi = e2 ? Pf{xh.z, xl.z} : Pf{xh.y, xl.y}, yi = e2 ? Pf{yh.z, yl.z} : Pf{yh.y, yl.y};
                        const Pf ii = pmul(xi, yi);
                        const Pf re = padd(pmul(xr, yr), Pf{-ii.h, -ii.l}), im = padd(pmul(xr, yi), pmul(xi, yr));
                        float4 *o = zb + (e2 ? m + step : at(dg.H1 + m + step)) * V;
                        if (e2) {
                            o[0] = make_float4(re.h, re.h, im.h, im.h);
                            o[1] = make_float4(re.l, re.l, im.l, im.l);
                        } else {
                            o[0] = make_float4(re.h, im.h, -im.h, re.h);
                            o[1] = make_float4(re.l, im.l, -im.l, re.l);
                        }
                    }
                }
                __syncthreads();
                // negative n_1 by conjugation, and zeros in the padding
                for (int k = threadIdx.x; k < n * NB; k += kDenseThreads) {
                    const int s = k / NB, v = k - s * NB;
                    float4 *row = s_b + (size_t)s * NB * V;
                    if (v < dg.H1) {
                        const float4 *z = row + at(2 * dg.H1 - v) * V;
                        const float4 h = z[0], l = z[1];
                        row[at(v) * V] = make_float4(h.x, -h.y, -h.z, h.w);
                        row[at(v) * V + 1] = make_float4(l.x, -l.y, -l.z, l.w);
                    } else if (v > 2 * dg.H1) {
                        row[at(v) * V] = row[at(v) * V + 1] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                    }
                }
                __syncthreads();
            }
            if (work) {
                for (int s = grp; s < n; s += groups) {
                    const float4 *e = s_e + ((size_t)s * NA + a0) * V, *b = s_b + ((size_t)s * NB + b0 / TB) * V;
                    const float2 *w = s_w + (size_t)s * JB * SW;
                    typename D::E E[TA][TB];
#pragma unroll
                    for (int i = 0; i < TA; ++i)
#pragma unroll
                        for (int k = 0; k < TB; ++k) E[i][k] = D::product(e + i * V, b + k * nbt * V);
                    // the strengths by 16 bytes (two in FP32, one pair in FP64)
                    float2 wr[JB * SW];
                    if constexpr (JB * SW % 2 == 0) {
#pragma unroll
                        for (int j = 0; j < JB * SW; j += 2) {
                            const float4 v = *reinterpret_cast<const float4 *>(w + j);
                            wr[j] = make_float2(v.x, v.y);
                            wr[j + 1] = make_float2(v.z, v.w);
                        }
                    } else {
                        wr[0] = w[0];
                    }
#pragma unroll
                    for (int j = 0; j < JB; ++j)
#pragma unroll
                        for (int i = 0; i < TA; ++i)
#pragma unroll
                            for (int k = 0; k < TB; ++k) D::add(acc[j][i][k], wr + j * SW, E[i][k]);
                }
            }
            held += (n + groups - 1) / groups;
            // at the end, and before a sum grows long: its rounding grows with the number of its terms (pairs: 7e-14 of
            // the sum after 256, 1.2e-12 after 4,096, 4.6e-12 after 20,000)
            if (block + base + CS >= last || held >= kDenseChain) {
                held = 0;
                flush();
            }
            __syncthreads();                          // the chunk's tables have been read
        }
    }
}

// Visibilities of the baselines (bl_list, or all) of channels f0 + blockIdx.y from the mode sums: the height terms
// with the weights wq[f][b][q] (nullptr: one term of weight 1), the products from the real strengths' sums.
template <class G>
__global__ void __launch_bounds__(128) k_dense_gather(const cpx<double> *__restrict__ modes, const int *__restrict__ bln,
                                                      const int *__restrict__ bl_list, int n_bl, int n_bl_all,
                                                      int n_pol, DenseGeom dg, int f0,
                                                      const cpx<double> *__restrict__ wq, char *__restrict__ out0,
                                                      long slice_stride)
{
    const int jb = blockIdx.x * blockDim.x + threadIdx.x;
    if (jb >= n_bl) return;
    const long b = bl_list ? bl_list[jb] : jb;
    int nx = bln[2 * b], ny = bln[2 * b + 1];
    const bool flip = ny < 0 || (ny == 0 && nx < 0);      // W(-n) = conj W(n)
    if (flip) {
        nx = -nx;
        ny = -ny;
    }
    const int n1 = 2 * dg.H1 + 1, n2 = dg.H2 + 1;
    const size_t msize = (size_t)n1 * n2;
    const cpx<double> *m = modes + (size_t)blockIdx.y * dg.J * msize + (size_t)ny * n1 + nx + dg.H1;
    const cpx<double> *wb = wq ? wq + ((size_t)(f0 + blockIdx.y) * n_bl_all + b) * dg.K : nullptr;
    cpx<double> r[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        r[p] = cmk<double>(0.0, 0.0);
        if (p < n_pol) {
            for (int q = 0; q < dg.K; ++q) {
                const cpx<double> t = m[(size_t)(p * dg.K + q) * msize];
                const cpx<double> v = cmk<double>(t.x, flip ? -t.y : t.y);
                r[p] = wb ? cadd(r[p], cmul(wb[q], v)) : v;
            }
        }
    }
    cpx<G> *o = reinterpret_cast<cpx<G> *>(out0 + (size_t)blockIdx.y * slice_stride);
    if (n_pol == 1) {
        o[b] = cmk<G>((G)r[0].x, (G)r[0].y);
    } else {
        // r: I + Q', I - Q', U', V; products 00, 01 = U' + i V, 10 = U' - i V, 11
        o[4 * b] = cmk<G>((G)r[0].x, (G)r[0].y);
        o[4 * b + 1] = cmk<G>((G)(r[2].x - r[3].y), (G)(r[2].y + r[3].x));
        o[4 * b + 2] = cmk<G>((G)(r[2].x + r[3].y), (G)(r[2].y - r[3].x));
        o[4 * b + 3] = cmk<G>((G)r[1].x, (G)r[1].y);
    }
}

static void dense_shape(int J, int elem, int &JB, int &TA, int &TB)
{
    if (J == 1) {
        JB = 1;
        TA = elem == 4 ? 4 : 2;
        TB = 4;
    } else {
        JB = elem == 4 && J > 4 ? 8 : 4;
        TA = TB = 2;
    }
}

static size_t dense_smem(const DenseGeom &dg, int elem)
{
    int JB, TA, TB;
    dense_shape(dg.J, elem, JB, TA, TB);
    const size_t cs = dg.CS, v = elem == 4 ? 1 : 2;
    // tables (or the groups' sums of one row of tiles), then the prepared sources
    return std::max(cs * ((size_t)(dg.NA + dg.NB) * 16 * v + (size_t)JB * 8 * v), (size_t)kDenseThreads * TB * 8 * v) +
           (size_t)kDenseThreads * ((elem == 4 ? 4 : 8) * 4 + (size_t)JB * elem);
}

// Modes up to which J sums a mode are faster than the type-1 transform of a w-point kernel, for skies of more than
// kDenseFew sources.  FP32: a source costs the direct sums modes (2 + J) multiply-adds and the grid about J (1,000 + 33 w^2)
// of them.  FP64 (pairs): the sums of 4 terms go together, so the cost goes by the terms rounded up to fours (one term
// alone: two of them), against J (70 + 1.85 w^2) and the FP64 preparation.  Measured per slice (200,000 sources, 16
// channels), direct sums against the grid: FP32, one term: 325 modes 36.5 / 37.3 us (w = 4), 861 modes 53.5 / 39.9 (w = 4)
// and 53.7 / 49.2 (w = 7: kept, its error is a quarter of the grid's), 1,431 modes 69.5 / 41.9 (w = 4), 69.6 / 51.1 (w = 7);
// 5 terms, w = 4: 861 modes 112 / 111, 1,431 modes 157 / 119.  FP64, one term: 861 modes 274 / 187 (w = 4), 274 / 264 (w = 7),
// 1,431 modes 440 / 269 (w = 7), 440 / 399 (w = 11); 5 terms, w = 4: 325 modes 408 / 453, 861 modes 1,013 / 633; 7 terms,
// w = 7: 1,431 modes 1,383 / 1,235.
static double dense_modes_max(int elem, int w, int J)
{
    if (elem == 4) return J * (1000.0 + 33.0 * w * w) / (J + 2.0);
    const int slots = J == 1 ? 2 : (J + 3) / 4 * 4;
    return (95.0 + J * (70.0 + 1.85 * w * w)) / (0.14 * slots);
}

bool dense_plan(int elem, double eps, int w, long n_src, int K, int n_pol, int H1, int H2, int n_bl, const int *bln, DenseGeom &dg,
                std::vector<int> &tiles)
{
    if (elem == 8 && eps < 1e-12) return false;
    dg.H1 = H1;
    dg.H2 = H2;
    dg.K = K;
    dg.J = K * n_pol;
    int JB, TA, TB;
    dense_shape(dg.J, elem, JB, TA, TB);
    dg.NA = (H2 + 1 + TA - 1) / TA * TA;
    dg.NB = (2 * H1 + 1 + TB - 1) / TB * TB;
    // sources a chunk: as many as two CTAs an SM hold tables for, 64 at most (fewer barriers)
    dg.CS = 64;
    while (dg.CS > 8 && dense_smem(dg, elem) > 100 * 1024) dg.CS /= 2;
    const long modes = (long)(2 * H1 + 1) * (H2 + 1);
    if (modes > kDenseModes || dense_smem(dg, elem) > 100 * 1024) return false;
    if (n_src > kDenseFew && (double)modes > dense_modes_max(elem, w, dg.J)) return false;
    // the tiles that hold a mode of some baseline
    const int ta = dg.NA / TA, tb = dg.NB / TB;
    std::vector<char> need((size_t)ta * tb, 0);
    for (int b = 0; b < n_bl; ++b) {
        int nx = bln[2 * b], ny = bln[2 * b + 1];
        if (ny < 0 || (ny == 0 && nx < 0)) {
            nx = -nx;
            ny = -ny;
        }
        need[(size_t)(ny / TA) * tb + (nx + H1) / TB] = 1;
    }
    tiles.clear();
    for (int i = 0; i < ta; ++i)
        for (int k = 0; k < tb; ++k)
            if (need[(size_t)i * tb + k]) tiles.push_back(i * TA | (k * TB) << 16);
    if (tiles.empty()) tiles.push_back(0);
    dg.n_tiles = (int)tiles.size();
    dg.tile_blocks = (dg.n_tiles + kDenseThreads - 1) / kDenseThreads;
    return true;
}

template <class G, int JB, int TA, int TB>
static cudaError_t dense_go(const double *sdir, const float4 *tc, const int *sidx, const int *nv_ptr, long n_src, const void *flux,
                            int flux_fp64, int n_freq, int f0, int nch, const double *freq, const SliceGeom &g,
                            const DenseGeom &dg, cpx<double> *modes, cudaStream_t st)
{
    static bool attr[64] = {};
    static int sms[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr[dev]) {
        e = cudaFuncSetAttribute(k_lattice_dense<G, JB, TA, TB>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        attr[dev] = true;
    }
    const int z = (dg.J + JB - 1) / JB * dg.tile_blocks;
    // two waves of two CTAs an SM over all the channels of the launch, each CTA with at least two chunks of sources
    const long want = std::max(1L, (4L * sms[dev] + (long)nch * z - 1) / ((long)nch * z));
    const long most = std::max(1L, n_src / 64);
    const dim3 blocks((unsigned)std::min(want, most), (unsigned)nch, (unsigned)z);
    k_lattice_dense<G, JB, TA, TB><<<blocks, kDenseThreads, dense_smem(dg, sizeof(G)), st>>>(
        sdir, tc, sidx, nv_ptr, n_src, flux, flux_fp64, n_freq, f0, freq, g, dg, modes);
    return cudaGetLastError();
}

template <class G>
cudaError_t launch_lattice_dense(const double *sdir, const float4 *tc, const int *sidx, const int *nv_ptr, long n_src, const void *flux,
                                 int flux_fp64, int n_freq, int f0, int nch, const double *freq, const SliceGeom &g,
                                 const DenseGeom &dg, cpx<double> *modes, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(modes, 0, (size_t)nch * dense_modes(dg) * sizeof(cpx<double>), st);
    if (e != cudaSuccess || n_src <= 0 || nch <= 0) return e;
#define FV_DENSE_ARGS sdir, tc, sidx, nv_ptr, n_src, flux, flux_fp64, n_freq, f0, nch, freq, g, dg, modes, st
    if constexpr (sizeof(G) == 4) {
        if (dg.J == 1) return dense_go<G, 1, 4, 4>(FV_DENSE_ARGS);
        if (dg.J <= 4) return dense_go<G, 4, 2, 2>(FV_DENSE_ARGS);
        return dense_go<G, 8, 2, 2>(FV_DENSE_ARGS);
    } else {
        if (dg.J == 1) return dense_go<G, 1, 2, 4>(FV_DENSE_ARGS);
        return dense_go<G, 4, 2, 2>(FV_DENSE_ARGS);
    }
#undef FV_DENSE_ARGS
}

template <class G>
cudaError_t launch_dense_gather(const cpx<double> *modes, const int *bln, const int *bl_list, int n_bl, int n_bl_all,
                                int n_pol, const DenseGeom &dg, int f0, int nch, const cpx<double> *wq, void *out0,
                                long slice_stride, cudaStream_t st)
{
    if (n_bl <= 0 || nch <= 0) return cudaSuccess;
    const dim3 blocks((unsigned)((n_bl + 127) / 128), (unsigned)nch);
    k_dense_gather<G><<<blocks, 128, 0, st>>>(modes, bln, bl_list, n_bl, n_bl_all, n_pol, dg, f0, wq, (char *)out0,
                                              slice_stride);
    return cudaGetLastError();
}

#define FV_DENSE_INST(G)                                                                                              \
    template cudaError_t launch_lattice_dense<G>(const double *, const float4 *, const int *, const int *, long, const void *, int,   \
                                                 int, int, int, const double *, const SliceGeom &, const DenseGeom &, \
                                                 cpx<double> *, cudaStream_t);                                        \
    template cudaError_t launch_dense_gather<G>(const cpx<double> *, const int *, const int *, int, int, int,              \
                                                const DenseGeom &, int, int, const cpx<double> *, void *, long,       \
                                                cudaStream_t);
FV_DENSE_INST(float)
FV_DENSE_INST(double)
#undef FV_DENSE_INST

}  // namespace fv
