// Spreading and interpolation of FP64 type-3 slices in pairs of floats (Section 2.2, steps 1 and 3b).
//
// GB300 has 64 FP32 multiply-adds for one of FP64, so an FP64 slice was bound by the FP64 pipe in every step: on the
// 127-antenna workload (35,000 sources, 10 height terms, 12-point kernel) 1,050 us of spreading, 515 + 420 us of FFT
// passes and 400 us of interpolation (now 210, 90 + 74 and 62 us).  A pair of floats carries 48 bits, and a multiply-add
// of pairs takes about 13 operations.  FP64 plans take this path at sigma = 2 and kernels of at most 13 points (at 13
// points, own error 1.7e-12, only up to kPairTermsMax terms a cell), where the transform's own error stays above the
// pairs' (about 1e-14 an operation, and growing with the length of the cells' sums); wider kernels and other sigma keep
// FP64 throughout.
// FP64 remains in the per-time directions, the strengths, coordinates and phases (k_prep), the per-target set-up and
// the tables.
#include "fv_pairs.cuh"

#include <algorithm>
#include <cmath>
#include <math.h>

namespace fv {

// Interpolation at the Chebyshev nodes, degree 13: with degree 13 to 21 the transform's error is the same to three
// digits for every w <= 13 (the kernel's own error dominates).
PairPoly pair_polynomials(int w, double beta)
{
    PairPoly es;
    constexpr int n = 2 * kPairTerms;
    for (int j = 0; j < kPairHalf; ++j) {
        double p[n] = {};
        if (2 * j < w) {
            double v[n], c[n], t0[n] = {}, t1[n] = {};
            for (int k = 0; k < n; ++k) {
                const double s = std::cos(M_PI * (k + 0.5) / n);
                const double z = (2.0 / w) * (0.5 * (s + 1.0) + j - 0.5 * w), t = 1.0 - z * z;
                v[k] = t >= 0.0 ? std::exp(beta * (std::sqrt(t) - 1.0)) : 0.0;
            }
            for (int q = 0; q < n; ++q) {
                c[q] = 0.0;
                for (int k = 0; k < n; ++k) c[q] += v[k] * std::cos(M_PI * q * (k + 0.5) / n);
                c[q] *= (q == 0 ? 1.0 : 2.0) / n;
            }
            t0[0] = 1.0;
            t1[1] = 1.0;
            for (int q = 0; q < n; ++q) {
                double t2[n];
                for (int k = 0; k < n; ++k) {
                    p[k] += c[q] * t0[k];
                    t2[k] = (k > 0 ? 2.0 * t1[k - 1] : 0.0) - t0[k];
                }
                for (int k = 0; k < n; ++k) {
                    t0[k] = t1[k];
                    t1[k] = t2[k];
                }
            }
        }
        for (int k = 0; k < kPairTerms; ++k) {
            es.v[j * kPairTerms + k] = pf(p[2 * k]);
            es.v[(kPairHalf + j) * kPairTerms + k] = pf(p[2 * k + 1]);
        }
    }
    return es;
}

namespace {

constexpr int kPsTileX = 16, kPsTileY = 8, kPsPatchX = kPsTileX / 8;    // a warp: 8 x 4 cells
constexpr int kPsPatches = kPsPatchX * (kPsTileY / 4), kPsThreads = 32 * kPsPatches, kPsChunk = 64;
constexpr int kPsTidy = 64;                             // sources a warp's sums take between two pair2_tidy

// Horner in pairs; value p (even + s odd) and its mirror (even - s odd)
__device__ __forceinline__ void pair_kernel(const Pf *es, int p, Pf s, Pf s2, Pf &v, Pf &mirror)
{
    const Pf *e = es + p * kPairTerms, *o = es + (kPairHalf + p) * kPairTerms;
    Pf a = e[kPairTerms - 1], b = o[kPairTerms - 1];
#pragma unroll
    for (int k = kPairTerms - 2; k >= 0; --k) {
        a = padd(pmul(a, s2), e[k]);
        b = padd(pmul(b, s2), o[k]);
    }
    b = pmul(b, s);
    v = padd(a, b);
    mirror = padd(a, -b);
}

}  // namespace

// A CTA of 4 warps owns a 16 x 8 tile of (x, y) columns, a warp an 8 x 4 patch, a lane one column with its NZ planes x
// NP products in registers (as the FP64 register gather).  The sources of the tile's bins that reach it (about half) are taken
// kPsChunk at a time: their kernel values and height terms are computed once per chunk into shared memory, each is
// listed for the patches its footprint meets, and every warp adds its list's sources.  The warps of a CTA wait for the
// longest list of a chunk, so small tiles win although a source's values are computed in more of them (12-point kernel,
// 10 height terms): 208 us a slice, 246 with 32 x 8, 225 with 8 x 8, 231 with 16 x 4 and 16 x 16 cells; chunks of 32
// instead of 64 sources 222.  Every cell is stored once.
template <int NP, int NZ>
__global__ void __launch_bounds__(kPsThreads, 512 / kPsThreads) k_spread_pairs(const int *__restrict__ offsets,
                                                                const SrcRec<double> *__restrict__ rec,
                                                                const cpx<double> *__restrict__ cs, SliceGeom g, TimeBin tb,
                                                                double r0, double r1, PairPoly es,
                                                                const unsigned *__restrict__ key, cpx<Pf> *__restrict__ grid)
{
    __shared__ Pf s_es[kPairPoly];
    __shared__ Pf s_w[2][kPsChunk][kPairW];
    __shared__ float4 s_wz[NZ > 1 ? kPsChunk : 1][NZ];               // (h, h, l, l)
    __shared__ float4 s_c[kPsChunk][NP];                              // (re h, im h, re l, im l)
    __shared__ Pf s_s[2][kPsChunk], s_z[NZ > 1 ? kPsChunk : 1];
    __shared__ int s_cz[NZ > 1 ? kPsChunk : 1];
    __shared__ int s_list[kPsPatches][kPsChunk], s_cnt[kPsPatches];
    __shared__ int s_row0[32], s_pre[32], s_total, s_bins[4], s_idx[kPsChunk + kPsThreads], s_have;
    __shared__ double s_up;
    const int nx = g.dim[0].nf1, ny = g.dim[1].nf1, nz = g.d == 3 || g.K ? g.dim[2].nf1 : 1;
    const int w = g.w;
    const int x0 = blockIdx.x * kPsTileX, y0 = blockIdx.y * kPsTileY;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gx = x0 + warp % kPsPatchX * 8 + (lane & 7), gy = y0 + warp / kPsPatchX * 4 + (lane >> 3);
    Pair2 acc[NP][NZ];
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
        for (int z = 0; z < NZ; ++z) acc[p][z] = Pair2{make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)};
    int held = 0;                               // sources since the warp's last pair2_tidy
    for (int k = threadIdx.x; k < kPairPoly; k += kPsThreads) s_es[k] = es.v[k];
    if (threadIdx.x < kPsPatches) s_cnt[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        s_have = 0;
        s_up = scalbn(1.0, pair_shift(*key));
        // bins whose sources can reach the tile (one top cell of margin)
        const double qx_lo = (x0 - nx / 2 - 0.5 * w) / r0, qx_hi = (x0 + kPsTileX - nx / 2 + 0.5 * w - 1) / r0;
        const double qy_lo = (y0 - ny / 2 - 0.5 * w) / r1, qy_hi = (y0 + kPsTileY - ny / 2 + 0.5 * w - 1) / r1;
        s_bins[0] = top_cell(qx_lo - 1.0, tb.nf1_top[0]) / tb.T[0];
        s_bins[1] = top_cell(qx_hi + 1.0, tb.nf1_top[0]) / tb.T[0];
        s_bins[2] = top_cell(qy_lo - 1.0, tb.nf1_top[1]) / tb.T[1];
        s_bins[3] = top_cell(qy_hi + 1.0, tb.nf1_top[1]) / tb.T[1];
    }
    __syncthreads();
    const int bx_lo = s_bins[0], bx_hi = s_bins[1], by_lo = s_bins[2], by_hi = s_bins[3];
    const int half = (w + 1) / 2;
    const double up = s_up;
    for (int r0w = by_lo; r0w <= by_hi; r0w += 32) {
        const int nrows = min(32, by_hi - r0w + 1);
        if (warp == 0) {
            int start = 0, len = 0;
            if (lane < nrows) {
                const int row = (r0w + lane) * tb.nbx;
                start = offsets[row + bx_lo];
                len = offsets[row + bx_hi + 1] - start;
            }
            int incl = len;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += v;
            }
            s_row0[lane] = start;
            s_pre[lane] = incl - len;
            if (lane == 31) s_total = incl;
        }
        __syncthreads();
        const int total = s_total;
        int base = 0, have = 0;
        while (true) {
            // the bins' sources that reach the tile, until there is a chunk of them
            while (have < kPsChunk && base < total) {
                const int v = base + threadIdx.x;
                if (v < total) {
                    int r = 0;                          // the last row whose prefix is <= v
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1)
                        if (r + step < nrows && s_pre[r + step] <= v) r += step;
                    const int i = s_row0[r] + (v - s_pre[r]);
                    const unsigned cell = rec[i].cell;
                    const int cx = (int)(cell & 0x3fffu) - x0, cy = (int)((cell >> 14) & 0x3fffu) - y0;
                    if (cx < kPsTileX && cx + w > 0 && cy < kPsTileY && cy + w > 0) s_idx[atomicAdd(&s_have, 1)] = i;
                }
                base += kPsThreads;
                __syncthreads();
                have = s_have;
                __syncthreads();
            }
            const int n = min(kPsChunk, have);
            if (n == 0) break;
            have -= n;
            if (threadIdx.x < n) {
                const int t = threadIdx.x;
                const long i = s_idx[have + t];
                const SrcRec<double> rr = rec[i];
                const int cx = (int)(rr.cell & 0x3fffu), cy = (int)((rr.cell >> 14) & 0x3fffu);
                s_s[0][t] = pf(2.0 * rr.fx + (double)(w - 1));
                s_s[1][t] = pf(2.0 * rr.fy + (double)(w - 1));
                if (NZ > 1) {
                    s_cz[NZ > 1 ? t : 0] = (int)(rr.cell >> 28);
                    s_z[NZ > 1 ? t : 0] = g.K ? pf(rr.fz) : pf(2.0 * rr.fz + (double)(w - 1));
                }
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    const cpx<double> c = cs[(size_t)i * NP + p];
                    const Pf re = pf(c.x * up), im = pf(c.y * up);
                    s_c[t][p] = make_float4(re.h, im.h, re.l, im.l);
                }
                const int ax = max(cx - x0, 0), bx = min(cx + w - 1 - x0, kPsTileX - 1);
                const int ay = max(cy - y0, 0), by2 = min(cy + w - 1 - y0, kPsTileY - 1);
                for (int qy = ay / 4; qy <= by2 / 4; ++qy)
                    for (int qx = ax / 8; qx <= bx / 8; ++qx) {
                        const int q = qy * kPsPatchX + qx, pos = atomicAdd(&s_cnt[q], 1);
                        s_list[q][pos] = t | ((cx - x0 + 16) << 8) | ((cy - y0 + 16) << 16);
                    }
            }
            if (threadIdx.x == 0) s_have = have;
            __syncthreads();
            // kernel values: (source fastest, axis, mirrored pair)
            for (int v = threadIdx.x; v < kPsChunk * 2 * half; v += kPsThreads) {
                const int t = v % kPsChunk, q = v / kPsChunk, axis = q & 1, p = q >> 1;
                if (t < n) {
                    const Pf s = s_s[axis][t];
                    Pf a, b;
                    pair_kernel(s_es, p, s, pmul(s, s), a, b);
                    s_w[axis][t][p] = a;
                    if (w - 1 - p != p) s_w[axis][t][w - 1 - p] = b;
                }
            }
            if (NZ > 1 && g.K) {
                for (int t = threadIdx.x; t < n; t += kPsThreads) {
                    const Pf u = s_z[t], u2 = Pf(2.0f * u.h, 2.0f * u.l);
                    Pf tm = u, tq = Pf(1.0f, 0.0f);              // T_{-1} = T_1, T_0
#pragma unroll
                    for (int q = 0; q < NZ; ++q) {
                        s_wz[t][q] = q < g.K ? make_float4(tq.h, tq.h, tq.l, tq.l) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                        const Pf tn = q == 0 ? u : padd(pmul(u2, tq), -tm);
                        tm = tq;
                        tq = tn;
                    }
                }
            } else if (NZ > 1) {
                for (int v = threadIdx.x; v < n * NZ; v += kPsThreads) {
                    const int t = v / NZ, z = v - t * NZ, jz = z - s_cz[t];
                    Pf a(0.0f, 0.0f), b;
                    if (jz >= 0 && jz < w) {
                        const Pf s = s_z[t];
                        pair_kernel(s_es, min(jz, w - 1 - jz), s, pmul(s, s), a, b);
                        if (jz > w - 1 - jz) a = b;
                    }
                    s_wz[t][z] = make_float4(a.h, a.h, a.l, a.l);
                }
            }
            __syncthreads();
            const int cnt = s_cnt[warp];
            const int lx16 = gx - x0 + 16, ly16 = gy - y0 + 16;
            for (int e = 0; e < cnt; ++e) {
                const int ent = s_list[warp][e];
                const int t = ent & 0xff;
                const unsigned dx = (unsigned)(lx16 - ((ent >> 8) & 0xff)), dy = (unsigned)(ly16 - (ent >> 16));
                if (dx < (unsigned)w && dy < (unsigned)w) {
                    const Pf k = pmul(s_w[0][t][dx], s_w[1][t][dy]);
                    const float2 kh = dup(k.h), kl = dup(k.l);
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        const float4 c = s_c[t][p];
                        const Pair2 cw = pair2_times(kh, kl, make_float2(c.x, c.y), make_float2(c.z, c.w));
                        if (NZ == 1) {
                            pair2_add(acc[p][0], cw);
                        } else {
#pragma unroll
                            for (int z = 0; z < NZ; ++z) {
                                const float4 q = s_wz[t][z];
                                pair2_add(acc[p][z], pair2_times(make_float2(q.x, q.y), make_float2(q.z, q.w), cw.h, cw.l));
                            }
                        }
                    }
                }
            }
            held += cnt;
            if (held >= kPsTidy) {
                held = 0;
#pragma unroll
                for (int p = 0; p < NP; ++p)
#pragma unroll
                    for (int z = 0; z < NZ; ++z) pair2_tidy(acc[p][z]);
            }
            __syncthreads();
            if (threadIdx.x < kPsPatches) s_cnt[threadIdx.x] = 0;
            __syncthreads();
        }
        __syncthreads();
    }
    if (gx < nx && gy < ny) {
        const Pf sc = pmul(pf(((const double *)g.pre_x)[gx]), pf(((const double *)g.pre_y)[gy]));
#pragma unroll
        for (int p = 0; p < NP; ++p)
#pragma unroll
            for (int z = 0; z < NZ; ++z)
                if (z < nz) {
                    const Pair2 a = acc[p][z];
                    grid[(((size_t)p * nz + z) * ny + gy) * nx + gx] =
                        cmk<Pf>(pmul(padd(Pf(a.h.x, 0.0f), Pf(a.l.x, 0.0f)), sc), pmul(padd(Pf(a.h.y, 0.0f), Pf(a.l.y, 0.0f)), sc));
                }
    }
}

bool pairs_fit(int w, int n_pol, int nz)
{
    return w <= kPairW && ((n_pol == 1 && nz >= 1 && nz <= 16) || (n_pol == 4 && nz == 1));
}

cudaError_t launch_spread_pairs(const int *offsets, const SrcRec<double> *rec, const cpx<double> *cs, const SliceGeom &g,
                                const TimeBin &tb, double r0, double r1, const PairPoly &es, const unsigned *key, cpx<Pf> *grid,
                                cudaStream_t st)
{
    const int nz = g.d == 3 || g.K ? g.dim[2].nf1 : 1;
    if (!pairs_fit(g.w, g.n_pol, nz) || !g.pre_x || !g.pre_y) return cudaErrorInvalidValue;
    const dim3 blocks((g.dim[0].nf1 + kPsTileX - 1) / kPsTileX, (g.dim[1].nf1 + kPsTileY - 1) / kPsTileY);
#define FV_PS(NP, NZ) k_spread_pairs<NP, NZ><<<blocks, kPsThreads, 0, st>>>(offsets, rec, cs, g, tb, r0, r1, es, key, grid)
    if (g.n_pol == 4) FV_PS(4, 1);
    else if (nz == 1) FV_PS(1, 1);
    else if (nz <= 8) FV_PS(1, 8);
    else if (nz <= 10) FV_PS(1, 10);
    else if (nz <= 12) FV_PS(1, 12);
    else FV_PS(1, 16);
#undef FV_PS
    return cudaGetLastError();
}

// ---------------------------------------------------------------- interpolation
// Per-target constants in FP64, one thread a target (a warp per target would spend the FP64 pipe's 16 cycles a warp
// instruction on one value each): first footprint cell and offset, postphase x deconvolution (with the height terms'
// common phase), and the weights of the target's planes (height terms, or K(l_z) of a short up axis).  Bessel series
// with reciprocals from a table: a division is about ten FP64 operations.
__global__ void __launch_bounds__(64) k_pair_targets(const double *__restrict__ bu, int n_u, const double *__restrict__ dec,
                                                     SliceGeom g, const double *__restrict__ prez,
                                                     const cpx<double> *__restrict__ twz, PairTarget *__restrict__ tgt,
                                                     cpx<Pf> *__restrict__ wz)
{
    constexpr int kRecip = 96;                                  // m + q < 80 + 16
    __shared__ double s_r[kRecip];
    for (int k = threadIdx.x; k < kRecip; k += 64) s_r[k] = k > 0 ? 1.0 / k : 0.0;
    __syncthreads();
    const int nz = g.d == 3 || g.K ? g.dim[2].nf1 : 1;
    const int u = blockIdx.x * 64 + threadIdx.x;
    const int z0 = blockIdx.y;                                  // plane z0 - 1, or the target's constants
    if (u >= n_u) return;
    const int w = g.w;
    const double b_up = bu[3 * (size_t)u + 2];
    if (z0 == 0) {
        double x[3] = {0.0, 0.0, 0.0}, s[2], ph = 0.0;
        int m[2];
#pragma unroll
        for (int i = 0; i < 3; ++i)
            if (i < g.d) {
                x[i] = -g.kappa * bu[3 * (size_t)u + i];
                ph += x[i] * g.dim[i].C;
            }
        if (g.K) ph -= g.kappa * b_up * g.hc;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const double p = (x[i] - g.dim[i].D) * g.dim[i].pscale, c = ceil(p - 0.5 * w);
            m[i] = (int)c;
            s[i] = (double)(w - 1) - 2.0 * (p - c);             // 2 (l0 - q + w/2) - 1 with l0 - q = c - p
        }
        double sn, cn;
        sincos(ph, &sn, &cn);
        PairTarget t;
        t.m0 = m[0] + g.dim[0].H;
        t.m1 = m[1] + g.dim[1].H;
        t.pad0 = t.pad1 = 0;
        t.sx = pf(s[0]);
        t.sy = pf(s[1]);
        t.post = cmk<Pf>(pf(cn * dec[u]), pf(sn * dec[u]));
        tgt[u] = t;
        return;
    }
    const int z = z0 - 1;
    cpx<double> k = cmk<double>(0.0, 0.0);
    if (g.K) {
        // eps_q (-i)^q J_q(k b_up hs)
        const double h = 0.5 * g.kappa * b_up * g.hs, h2 = -h * h;
        double term = z == 0 ? 1.0 : 2.0;
        for (int i = 1; i <= z; ++i) term *= h * s_r[i];
        double sum = term;
        for (int i = 1; i < 80; ++i) {
            term *= h2 * (s_r[i] * s_r[i + z]);
            sum += term;
            if (fabs(term) <= 1e-18 * fabs(sum)) break;
        }
        const double j = (z & 2) ? -sum : sum;
        k = (z & 1) ? cmk<double>(0.0, -j) : cmk<double>(j, 0.0);
    } else {
        const int Mz = g.dim[2].M, lc = z - nz / 2;
        const double p = (-g.kappa * b_up - g.dim[2].D) * g.dim[2].pscale, c = ceil(p - 0.5 * w);
        int a = (lc * (int)c) % Mz, step = lc % Mz;
        if (a < 0) a += Mz;
        if (step < 0) step += Mz;
        for (int j = 0; j < w; ++j) {
            k = cadd(k, cscale(twz[a], es_k<double>((2.0 / w) * (p - c - j), g.beta)));
            a += step;
            if (a >= Mz) a -= Mz;
        }
        k = cscale(k, prez[z]);
    }
    wz[(size_t)u * nz + z] = cmk<Pf>(pf(k.x), pf(k.y));
}

// One warp per target; lane L sums the values L, L + 32, ... (four at a time) of the footprint rows, w P consecutive
// values each, with the rows' y weights, then applies the x weights, the planes' weights and the sum over the lanes.
template <int NP>
__global__ void __launch_bounds__(128) k_interp_pairs(const cpx<Pf> *__restrict__ band, int n_u, SliceGeom g,
                                                      PairPoly es, const unsigned *__restrict__ key,
                                                      const PairTarget *__restrict__ tgt,
                                                      const cpx<Pf> *__restrict__ wz, SliceOut so)
{
    constexpr int kR = 4;
    __shared__ Pf s_es[kPairPoly];
    for (int k = threadIdx.x; k < kPairPoly; k += 128) s_es[k] = es.v[k];
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int u = (int)(blockIdx.x * 4 + (threadIdx.x >> 5));
    if (u >= n_u) return;                       // whole warps
    const int b0 = so.u_off[so.u_base + u], nb = so.u_off[so.u_base + u + 1] - b0;
    const int w = g.w, nz = g.d == 3 || g.K ? g.dim[2].nf1 : 1, P = NP * nz, row_n = w * P;
    const PairTarget t = tgt[u];
    // lane j < w: the j-th x and y kernel values
    Pf wx(0.0f, 0.0f), wy(0.0f, 0.0f);
    if (lane < w) {
        const int p = min(lane, w - 1 - lane);
        Pf a, b;
        pair_kernel(s_es, p, t.sx, pmul(t.sx, t.sx), a, b);
        wx = lane == p ? a : b;
        pair_kernel(s_es, p, t.sy, pmul(t.sy, t.sy), a, b);
        wy = lane == p ? a : b;
    }
    const cpx<Pf> *base = band + ((size_t)t.m1 * g.dim[0].B + t.m0) * P;
    const size_t rstride = (size_t)g.dim[0].B * P;
    cpx<Pf> sum[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) sum[p] = cmk<Pf>(Pf(0.0f, 0.0f), Pf(0.0f, 0.0f));
    for (int v0 = 0; v0 < row_n; v0 += 32 * kR) {
        Pair2 acc[kR];
#pragma unroll
        for (int r = 0; r < kR; ++r) acc[r] = Pair2{make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)};
        const float4 *row = reinterpret_cast<const float4 *>(base);
        for (int y = 0; y < w; ++y, row += rstride) {
            const float2 yh = dup(__shfl_sync(0xffffffffu, wy.h, y)), yl = dup(__shfl_sync(0xffffffffu, wy.l, y));
#pragma unroll
            for (int r = 0; r < kR; ++r) {
                if (v0 + 32 * r >= row_n) break;               // the same on every lane
                const float4 c = __ldg(row + min(v0 + lane + 32 * r, row_n - 1));      // (re h, re l, im h, im l)
                pair2_add(acc[r], pair2_times(yh, yl, make_float2(c.x, c.z), make_float2(c.y, c.w)));
            }
        }
#pragma unroll
        for (int r = 0; r < kR; ++r) {
            if (v0 + 32 * r >= row_n) break;
            const int v = min(v0 + lane + 32 * r, row_n - 1), c = v / P, pl = v - c * P;
            const int pol = NP == 1 ? 0 : pl / nz, z = pl - pol * nz;
            const Pf k(__shfl_sync(0xffffffffu, wx.h, c), __shfl_sync(0xffffffffu, wx.l, c));
            if (v0 + lane + 32 * r < row_n) {
                cpx<Pf> a = cmk<Pf>(pmul(padd(Pf(acc[r].h.x, 0.0f), Pf(acc[r].l.x, 0.0f)), k),
                                    pmul(padd(Pf(acc[r].h.y, 0.0f), Pf(acc[r].l.y, 0.0f)), k));
                if (nz > 1) {
                    const cpx<Pf> q = wz[(size_t)u * nz + z];
                    a = cmk<Pf>(padd(pmul(a.x, q.x), -pmul(a.y, q.y)), padd(pmul(a.x, q.y), pmul(a.y, q.x)));
                }
#pragma unroll
                for (int p = 0; p < NP; ++p)
                    if (NP == 1 || p == pol) sum[p] = cmk<Pf>(padd(sum[p].x, a.x), padd(sum[p].y, a.y));
            }
        }
    }
    const double down = scalbn(1.0, -pair_shift(*key));
    double vx[NP], vy[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        for (int o = 16; o > 0; o >>= 1) {
            const Pf x(__shfl_xor_sync(0xffffffffu, sum[p].x.h, o), __shfl_xor_sync(0xffffffffu, sum[p].x.l, o));
            const Pf y(__shfl_xor_sync(0xffffffffu, sum[p].y.h, o), __shfl_xor_sync(0xffffffffu, sum[p].y.l, o));
            sum[p] = cmk<Pf>(padd(sum[p].x, x), padd(sum[p].y, y));
        }
        const cpx<Pf> s = sum[p], q = t.post;
        vx[p] = pf_value(padd(pmul(s.x, q.x), -pmul(s.y, q.y))) * down;
        vy[p] = pf_value(padd(pmul(s.x, q.y), pmul(s.y, q.x))) * down;
    }
    write_target<double, NP>(so, b0, nb, vx, vy, lane);
}

cudaError_t launch_interp_pairs(const cpx<Pf> *band, const double *bu, int n_u, const double *dec, const SliceGeom &g,
                                const double *prez, const cpx<double> *twz, const PairPoly &es, const unsigned *key, int chunk,
                                PairTarget *tgt, cpx<Pf> *wz, const SliceOut &so, cudaStream_t st)
{
    const int nz = g.d == 3 || g.K ? g.dim[2].nf1 : 1;
    if (!pairs_fit(g.w, g.n_pol, nz) || !so.out || chunk < 1) return cudaErrorInvalidValue;
    for (int u0 = 0; u0 < n_u; u0 += chunk) {
        const int n = std::min(chunk, n_u - u0);
        SliceOut o = so;
        o.u_base += u0;
        k_pair_targets<<<dim3((n + 63) / 64, nz > 1 ? nz + 1 : 1), 64, 0, st>>>(bu + 3 * (size_t)u0, n, dec + u0, g, prez,
                                                                               twz, tgt, wz);
        const unsigned blocks = (unsigned)((n + 3) / 4);
        if (g.n_pol == 4) k_interp_pairs<4><<<blocks, 128, 0, st>>>(band, n, g, es, key, tgt, wz, o);
        else k_interp_pairs<1><<<blocks, 128, 0, st>>>(band, n, g, es, key, tgt, wz, o);
    }
    return cudaGetLastError();
}

}  // namespace fv
