// Preparation and spreading of FP32 slices in one pass over the sources (Section 2.2, step 1).
//
// The per-time sort orders the visible sources by strips of a few columns of the top channel's grid and,
// within a strip, row by row.  A warp takes one contiguous run of the sorted sources: 32 at a time its
// lanes compute one source each (beam x flux strengths with the prephase, grid coordinates, kernel values)
// into shared memory, then the warp adds them one after another to a window of 16 columns x 8 rows of the
// grid that it holds in registers (lane = column x half of the rows, 4 rows a lane).  Rows and columns live
// at their grid index modulo 8 and 16, and a source's kernel values are stored at those places (zero
// elsewhere), so a source costs its shared-memory reads and the multiply-adds, with no index arithmetic and
// no branches.  As the sources advance, the rows they have left are added to the grid (red.global,
// 16 bytes a lane: a cell's planes are adjacent) and their registers start again at zero.  A source outside the window
// (the next strip, a jump in the rows) empties the window and moves it, so any order of the sources gives
// the same sums; the order only decides how often that happens.  A channel's rows are the top channel's
// times r <= 1, so the sources of one top row differ by at most one row, which the window's eighth row
// holds for w <= 7.
//
// Why this form: each source is prepared and added once (the gather forms copy it to every tile it meets and
// walk it once per 8 x 4 block: about 170 warp instructions a source on the 350-antenna workload, beside a
// preparation pass that writes 112 bytes a source and the gather that reads them back); here a source takes
// about 74, of which 30 add it, 22 are its share of the preparation and 20 of the rows that leave the window.
// Bound by instruction issue (56 % busy, 16 warps an SM).  Measured per slice, one stream: 350-antenna workload
// (443,000 sources above the horizon, four products, 1500 x 750 cells) 54 us and 8 us to clear the grid, against
// 33 + 117 us for the preparation pass and the ring gather; 127-antenna workload (35,000 sources, 8 height terms)
// 28 + 7 against 8 + 48 us with the register gather.
#include "fv_staged.cuh"
#include "fv_prep.cuh"

#include <algorithm>
#include <cmath>

namespace fv {

namespace {

constexpr int kStripThreads = 128;                     // four warps, independent of one another
constexpr int kWinX = 16, kWinY = 8;
// least sources of a warp's run: 8 (a nearly empty grid takes them; the warp's latency is its run's length), with eight
// planes 32 (each run ends with a window of 128 cells x 8 planes to add to the grid)
// (hex array of 127 antennas, 128 channels x 8 terms, 31.0 -> 28.1 ms; with fewer planes 32 leaves SMs idle)
__host__ __device__ constexpr int strip_min(int npl) { return npl == 8 ? 32 : 8; }

// resident CTAs per SM (without spills in the loop over the sources)
__host__ __device__ constexpr int strip_ctas(int npl) { return npl == 8 ? 4 : (npl == 4 ? 5 : 6); }

// words per source in shared memory: 16 column values, 8 row values twice (for packed products), the
// strengths; an odd number of 16-byte rows, so that the lanes' 16-byte stores fall on distinct banks
template <int NPL> struct StripRec {
    static constexpr int words = NPL == 8 ? 52 : (NPL == 4 ? 44 : 36);
};

// *p += v where on (16-byte aligned for four values)
__device__ __forceinline__ void red_add2(cpx<float> *p, float2 v, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %3, 0;\n\t@q red.global.add.v2.f32 [%0], {%1, %2};\n\t}" ::"l"(p),
                 "f"(v.x), "f"(v.y), "r"((int)on)
                 : "memory");
}
__device__ __forceinline__ void red_add4(cpx<float> *p, float2 v, float2 u, bool on)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %5, 0;\n\t@q red.global.add.v4.f32 [%0], {%1, %2, %3, %4};\n\t}" ::"l"(p),
                 "f"(v.x), "f"(v.y), "f"(u.x), "f"(u.y), "r"((int)on)
                 : "memory");
}

// The grid a warp adds to: its first plane of cell 0, complex values per cell, planes of the warp in use.
struct Grid {
    cpx<float> *p;
    int nx, ny, stride, npl;
};

// The window of one warp.  acc[k][p]: plane p of row slot 4 half + k, column slot col.
template <int NPL, bool POL4> struct Window {
    float2 acc[4][NPL];
    int X0, wb;                  // first column and row; columns [X0, X0 + 16), rows [wb, wb + 8)
    int col, half, x;            // this lane's column slot, row half, and column of the grid

    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int p = 0; p < NPL; ++p) acc[k][p] = make_float2(0.0f, 0.0f);
    }
    // add this lane's row in slot 4 half + K, row y of the grid, and start it again at zero
    template <int K> __device__ __forceinline__ void emit(int y, bool mine, const Grid &gr)
    {
        const bool in = mine && (unsigned)x < (unsigned)gr.nx && (unsigned)y < (unsigned)gr.ny;
        cpx<float> *o = gr.p + (long)(y * gr.nx + x) * gr.stride;
        if constexpr (NPL == 1) {
            red_add2(o, acc[K][0], in);
        } else {
#pragma unroll
            for (int q = 0; q < NPL; q += 2) red_add4(o + q, acc[K][q], acc[K][q + 1], in && (POL4 || q < gr.npl));
        }
#pragma unroll
        for (int p = 0; p < NPL; ++p) {
            acc[K][p].x = mine ? 0.0f : acc[K][p].x;
            acc[K][p].y = mine ? 0.0f : acc[K][p].y;
        }
    }
    // row y leaves the window
    __device__ __forceinline__ void flush_row(int y, const Grid &gr)
    {
        const bool mine = ((y >> 2) & 1) == half;
        switch (y & 3) {                              // the same on every lane
        case 0: emit<0>(y, mine, gr); break;
        case 1: emit<1>(y, mine, gr); break;
        case 2: emit<2>(y, mine, gr); break;
        default: emit<3>(y, mine, gr); break;
        }
    }
    // every row leaves the window: slot s holds row wb + ((s - wb) mod 8)
    __device__ __forceinline__ void flush(const Grid &gr)
    {
        emit<0>(wb + ((4 * half - wb) & 7), true, gr);
        emit<1>(wb + ((4 * half + 1 - wb) & 7), true, gr);
        emit<2>(wb + ((4 * half + 2 - wb) & 7), true, gr);
        emit<3>(wb + ((4 * half + 3 - wb) & 7), true, gr);
    }
    __device__ __forceinline__ void set_x(int x0)
    {
        X0 = x0;
        x = x0 + ((col - x0) & (kWinX - 1));
    }
    // one source: c psi_x psi_y into the window (packed multiply-adds: 54.4 us a 350-antenna slice, 56.8 scalar)
    __device__ __forceinline__ void add(const float *r)
    {
        const float wx = r[col];
        const float4 ya = *reinterpret_cast<const float4 *>(r + kWinX + 8 * half);
        const float4 yb = *reinterpret_cast<const float4 *>(r + kWinX + 8 * half + 4);
        const float2 y[4] = {make_float2(ya.x, ya.y), make_float2(ya.z, ya.w), make_float2(yb.x, yb.y),
                             make_float2(yb.z, yb.w)};
        const float *cp = r + kWinX + 2 * kWinY;
        if constexpr (NPL == 1) {
            const float2 c = *reinterpret_cast<const float2 *>(cp);
            const float2 cw = make_float2(c.x * wx, c.y * wx);
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[k][0] = __ffma2_rn(y[k], cw, acc[k][0]);
        } else {
            const float2 w2 = make_float2(wx, wx);
            float2 kk[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) kk[k] = __fmul2_rn(y[k], w2);
#pragma unroll
            for (int q = 0; q < NPL / 2; ++q) {
                const float4 c = *reinterpret_cast<const float4 *>(cp + 4 * q);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    acc[k][2 * q] = __ffma2_rn(kk[k], make_float2(c.x, c.y), acc[k][2 * q]);
                    acc[k][2 * q + 1] = __ffma2_rn(kk[k], make_float2(c.z, c.w), acc[k][2 * q + 1]);
                }
            }
        }
    }
};

}  // namespace

// Planes [blockIdx.y NPL, + NPL) of product blockIdx.z (POL4: all four products of a flat grid at once).
// nz: planes per product (1, the up planes, or the height terms).
template <int NPL, bool POL4>
__global__ void __launch_bounds__(kStripThreads, strip_ctas(NPL))
    k_spread_strip(const float4 *__restrict__ tc, const int *__restrict__ sidx, const int *__restrict__ nv_ptr,
                   long n_src, const void *__restrict__ flux, int flux_fp64, int n_freq, int f, SliceGeom g,
                   EsPoly es, int nz, cpx<float> *__restrict__ grid)
{
    constexpr int W = StripRec<NPL>::words;
    __shared__ __align__(16) float s_rec[kStripThreads / 32][32 * W];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nv = *nv_ptr;
    // contiguous runs of equally many sources, one per warp (at least strip_min), cut into equal batches of at most 32
    const int warps = gridDim.x * (kStripThreads / 32), wid = blockIdx.x * (kStripThreads / 32) + warp;
    const int per = max(strip_min(NPL), (nv + warps - 1) / warps);
    const int first = wid * per, last = min(nv, first + per);
    if (first >= last) return;                      // whole warps; nothing below synchronises the CTA
    const int batches = (last - first + 31) / 32, step = (last - first + batches - 1) / batches;
    float *rec = s_rec[warp];
    const int w = g.w;
    const float *pre_x = (const float *)g.pre_x, *pre_y = (const float *)g.pre_y;
    const int z0 = POL4 ? 0 : blockIdx.y * NPL, pz = POL4 ? 0 : blockIdx.z;
    const int nzp = strip_planes(nz);
    const Grid gr{grid + pz * nzp + z0, g.dim[0].nf1, g.dim[1].nf1, g.n_pol * nzp, min(NPL, nz - z0)};
    const int slack = kWinY - w, room = kWinX - w;

    Window<NPL, POL4> win;
    win.clear();
    win.col = lane & (kWinX - 1);
    win.half = lane >> 4;
    win.wb = 0;
    win.set_x(-(1 << 20));                          // holds no source yet

    for (int base = first; base < last; base += step) {
        const int n = min(step, last - base);
        int cx = 0, cy = -(1 << 28);
        if (lane < n) {
            const long i = base + lane;
            PrepOne o;
            prep_tc_one(tc[3 * i], tc[3 * i + 1], tc[3 * i + 2], sidx[i], flux, flux_fp64, n_src, n_freq, f, g, o);
            cx = o.ci[0];
            cy = o.ci[1];
            float *r = rec + lane * W;
            float4 *r4 = reinterpret_cast<float4 *>(r);
#pragma unroll
            for (int k = 0; k < (kWinX + 2 * kWinY) / 4; ++k) r4[k] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            // kernel values of both axes by the plan's polynomials, with the axes' prescales
            const float hw = 0.5f * (float)w;
            const float2 s = make_float2(2.0f * (o.fr[0] + hw) - 1.0f, 2.0f * (o.fr[1] + hw) - 1.0f);
            const float2 s2 = __fmul2_rn(s, s);
            auto put = [&](int j, float2 v) {
                r[(cx + j) & (kWinX - 1)] = v.x * pre_x[cx + j];
                const float vy = v.y * pre_y[cy + j];
                *reinterpret_cast<float2 *>(r + kWinX + 2 * ((cy + j) & (kWinY - 1))) = make_float2(vy, vy);
            };
#pragma unroll
            for (int j = 0; j < kWinY / 2; ++j) {
                if (2 * j < w) {
                    float2 e = es.e[j][kEsTerms - 1], od = es.o[j][kEsTerms - 1];
#pragma unroll
                    for (int k = kEsTerms - 2; k >= 0; --k) {
                        e = __ffma2_rn(e, s2, es.e[j][k]);
                        od = __ffma2_rn(od, s2, es.o[j][k]);
                    }
                    put(j, __ffma2_rn(od, s, e));
                    if (w - 1 - j != j) put(w - 1 - j, __ffma2_rn(make_float2(-od.x, -od.y), s, e));
                }
            }
            float2 *c2 = reinterpret_cast<float2 *>(r + kWinX + 2 * kWinY);
            if constexpr (POL4) {
#pragma unroll
                for (int p = 0; p < 4; ++p) c2[p] = make_float2(o.c[p].x, o.c[p].y);
            } else {
                cpx<float> c = o.c[0];
                if (pz == 1) c = o.c[1];
                else if (pz == 2) c = o.c[2];
                else if (pz == 3) c = o.c[3];
                if (g.K) {
                    // height terms: plane q takes c T_q(u) (three-term recurrence)
                    const float u = o.fr[2];
                    float tm = u, t = 1.0f;                     // T_{-1} = T_1
                    for (int q = 0; q < z0; ++q) {
                        const float tn = q == 0 ? u : 2.0f * u * t - tm;
                        tm = t;
                        t = tn;
                    }
#pragma unroll
                    for (int q = 0; q < NPL; ++q) {
                        c2[q] = make_float2(c.x * t, c.y * t);
                        const float tn = z0 + q == 0 ? u : 2.0f * u * t - tm;
                        tm = t;
                        t = tn;
                    }
                } else if (nz > 1) {
                    // up planes: c phi_z at absolute z, zero outside the footprint
                    const float two_over_w = 2.0f / (float)w;
#pragma unroll
                    for (int q = 0; q < NPL; ++q) {
                        const int jz = z0 + q - o.ci[2];
                        const float v = jz >= 0 && jz < w ? es_kernel_f(two_over_w * (o.fr[2] + (float)jz), g.beta_f) : 0.0f;
                        c2[q] = make_float2(c.x * v, c.y * v);
                    }
                } else {
                    c2[0] = make_float2(c.x, c.y);
                }
            }
        }
        __syncwarp();
        for (int i = 0;;) {
            // From source i on: `top` is the largest row start the window holds now and m the largest of the
            // sources before each lane's; a source past both makes rows leave (adv), one more than `slack` rows
            // below them, or outside the columns, has to wait for the window to be emptied and moved (bad)
            const int top = win.wb + slack;
            int m = lane >= i ? cy : -(1 << 28);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) m = max(m, __shfl_up_sync(0xffffffffu, m, o));   // a lane below o: its own
            m = __shfl_up_sync(0xffffffffu, m, 1);
            m = max(lane > 0 ? m : -(1 << 28), top);
            const bool here = lane >= i && lane < n;
            const bool fits = cx >= win.X0 && cx <= win.X0 + room && cy >= m - slack;
            const unsigned bad = __ballot_sync(0xffffffffu, here && !fits);
            unsigned adv = __ballot_sync(0xffffffffu, here && cy > m);
            const int e = bad ? __ffs(bad) - 1 : n;
            while (i < e) {
                if ((adv >> i) & 1u) {
                    const int nb = __shfl_sync(0xffffffffu, cy, i) - slack;
                    if (nb >= win.wb + kWinY) {
                        win.flush(gr);
                        win.wb = nb;
                    } else {
                        for (; win.wb < nb; ++win.wb) win.flush_row(win.wb, gr);
                    }
                    adv &= ~(1u << i);
                }
                const unsigned later = adv & (0xffffffffu << i);
                const int s = min(e, later ? __ffs(later) - 1 : 32);
                const float *r = rec + i * W;
                const int cnt = s - i;
#pragma unroll 2
                for (int k = 0; k < cnt; ++k) win.add(r + k * W);
                i = s;
            }
            if (e >= n) break;
            // empty the window and move it over the sources near this one
            win.flush(gr);
            const int c0 = __shfl_sync(0xffffffffu, cx, e);
            const bool near = lane >= e && lane < n && abs(cx - c0) <= room;
            int lo = __reduce_min_sync(0xffffffffu, near ? cx : c0), hi = __reduce_max_sync(0xffffffffu, near ? cx : c0);
            if (hi - lo > room) {
                lo = max(lo, c0 - room / 2);
                hi = lo + room;
            }
            win.set_x(lo - (room - (hi - lo)) / 2);
            win.wb = __shfl_sync(0xffffffffu, cy, e) - slack;
        }
        __syncwarp();                               // the records are read before the next batch overwrites them
    }
    win.flush(gr);
}

// The kernel values phi((2/w)(l0 - q + j)), j < w, as polynomials of s = 2 (l0 - q + w/2) - 1 in [-1, 1)
// (piecewise polynomial kernels as in Barnett, Magland & af Klinteberg 2019): value j is E_j(s^2) + s O_j(s^2)
// and, the kernel being even, value w - 1 - j is E_j - s O_j.  Interpolation at the Chebyshev nodes in FP64.  Of
// degree 9 the values differ from the kernel's by at most half its jump e^-beta at |z| = 1, next to that jump,
// and by less than FP32 rounding elsewhere; the transform's error is the same to three digits for every w <= 8.
// It takes 10 packed FMAs a pair of values for both axes against about 25 instructions a value for the square
// root and the exponential.
EsPoly es_polynomials(int w, double beta)
{
    EsPoly r{};
    constexpr int n = 2 * kEsTerms;                 // nodes = coefficients
    for (int j = 0; 2 * j < w && j < kWinY / 2; ++j) {
        double v[n], c[n];
        for (int k = 0; k < n; ++k) {
            const double s = std::cos(M_PI * (k + 0.5) / n);
            const double z = (2.0 / w) * (0.5 * (s + 1.0) + j - 0.5 * w);
            const double t = 1.0 - z * z;
            v[k] = t >= 0.0 ? std::exp(beta * (std::sqrt(t) - 1.0)) : 0.0;
        }
        for (int q = 0; q < n; ++q) {
            c[q] = 0.0;
            for (int k = 0; k < n; ++k) c[q] += v[k] * std::cos(M_PI * q * (k + 0.5) / n);
            c[q] *= (q == 0 ? 1.0 : 2.0) / n;
        }
        // Chebyshev to powers of s
        double p[n] = {}, t0[n] = {}, t1[n] = {};
        t0[0] = 1.0;
        t1[1] = 1.0;
        for (int q = 0; q < n; ++q) {
            for (int k = 0; k < n; ++k) p[k] += c[q] * t0[k];
            double t2[n];
            for (int k = 0; k < n; ++k) t2[k] = (k > 0 ? 2.0 * t1[k - 1] : 0.0) - t0[k];
            for (int k = 0; k < n; ++k) {
                t0[k] = t1[k];
                t1[k] = t2[k];
            }
        }
        for (int k = 0; k < kEsTerms; ++k) {
            r.e[j][k] = make_float2((float)p[2 * k], (float)p[2 * k]);
            r.o[j][k] = make_float2((float)p[2 * k + 1], (float)p[2 * k + 1]);
        }
    }
    return r;
}

bool spread_strip_fits(int w, int n_pol, int nz)
{
    return w <= kWinY && (n_pol == 1 || n_pol == 4) && nz >= 1 && nz <= 16;
}

cudaError_t launch_spread_strip(const float4 *tc, const int *sidx, const int *nv_ptr, long n_src, const void *flux,
                                int flux_fp64, int n_freq, int f, const SliceGeom &g, const EsPoly &es,
                                cpx<float> *grid, cudaStream_t st)
{
    if (n_src <= 0) return cudaSuccess;
    const int nz = g.d == 3 || g.K ? g.dim[2].nf1 : 1;      // up planes or height terms
    if (!spread_strip_fits(g.w, g.n_pol, nz)) return cudaErrorInvalidValue;
    static int sms[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!sms[dev]) {
        e = cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
    }
    const bool pol4 = g.n_pol == 4 && nz == 1;
    const int npl = pol4 ? 4 : (nz == 1 ? 1 : (nz <= 4 ? 4 : 8));
    // one wave of CTAs, each warp one run of at least strip_min sources
    const int min_cta = strip_min(npl) * (kStripThreads / 32);
    const long want = (n_src + min_cta - 1) / min_cta;
    const unsigned groups = pol4 ? 1u : (unsigned)((nz + npl - 1) / npl), pols = pol4 ? 1u : (unsigned)g.n_pol;
    const long slots = (long)strip_ctas(npl) * sms[dev];
    const unsigned gx = (unsigned)std::min<long>(want, std::max<long>(1, slots / (groups * pols)));
    const dim3 blocks(gx, groups, pols);
#define FV_STRIP_ARGS tc, sidx, nv_ptr, n_src, flux, flux_fp64, n_freq, f, g, es, nz, grid
    if (pol4) k_spread_strip<4, true><<<blocks, kStripThreads, 0, st>>>(FV_STRIP_ARGS);
    else if (npl == 4) k_spread_strip<4, false><<<blocks, kStripThreads, 0, st>>>(FV_STRIP_ARGS);
    else if (npl == 1) k_spread_strip<1, false><<<blocks, kStripThreads, 0, st>>>(FV_STRIP_ARGS);
    else k_spread_strip<8, false><<<blocks, kStripThreads, 0, st>>>(FV_STRIP_ARGS);
#undef FV_STRIP_ARGS
    return cudaGetLastError();
}

}  // namespace fv
