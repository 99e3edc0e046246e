// Hand-written mixed-radix FFT pass for the oversampled grid (Section 2.2,
// step 2: "Oversampled FFT").
//
// One pass transforms every row of its input along the row's contiguous axis:
//   load the N grid values of the row, multiply by the deconvolution prescale
//   1/Phihat(l w pi / M) of this axis (Section 2.2, step 3a, applied on the
//   grid side of the inner transform; pre = nullptr when the spreading kernel
//   already applied it), place them at l - N/2 (mod M) of a
//   zero-padded length-M vector, run a Stockham autosort FFT with the sign
//   e^{+2 pi i l m / M}, and keep only the band m in [-H, B-1-H] that the
//   interpolation reads, written transposed as out[b][row].
// The transposed write rotates the axes so that the next pass again reads
// contiguous rows.
//
// GB300 mapping.  M is chosen as a product of at most three (four beyond
// 4096) radices from {2,3,4,5,6,8,9,10,12,15,16}, so a row takes at most
// three trips through shared memory; each radix-R butterfly runs in
// registers (composite R as nested Cooley-Tukey with compile-time twiddles).
// A CTA holds R_rows consecutive rows in two padded shared buffers (one
// complex of padding per 16, which breaks the bank conflicts of the
// stride-R stores of the first stage); index arithmetic uses
// multiply-high division by the per-stage constants prepared on the host.
#include "fv_dft.cuh"
#include "fv_pair.cuh"

namespace fv {

static constexpr int kThreads = 256;

// ---------------------------------------------------------------- stages
__device__ __forceinline__ unsigned fdiv(unsigned n, unsigned mul, unsigned sh)
{
    return (__umulhi(n, mul) + n) >> sh;
}
__device__ __forceinline__ int pad(int i) { return i + (i >> 4); }

// Where a stage's input and output live.  The first stage reads the
// zero-padded row without the padding ever being stored: positions in
// [zlo, zhi) are zeros.  The last stage (Ns = M / RD, so j = k and its
// outputs are the frequencies m = k + q Ns) writes only the band, straight to
// global memory, transposed: out[b][row] with b = m + H (mod M), every b < B.
template <class G> struct StageIO {
    int zlo, zhi;                 // first stage: zero positions of the input row
    cpx<G> *out;                  // last stage: band output (nullptr: write y)
    long rows, row0;
    int nr, B, H;
    float inv_nrows;
};

template <class G, int RD>
__device__ __forceinline__ void stage(const cpx<G> *__restrict__ x, cpx<G> *__restrict__ y, const DimGeom &dg,
                                      int s, int nrows, int Ns, const cpx<G> *__restrict__ tw, bool first,
                                      StageIO<G> io)
{
    const int M = dg.M;
    const int MR = M / RD;
    const int per = nrows * MR;
    const int twstep = M / (Ns * RD);
    const bool last = io.out != nullptr;
    for (int bi = threadIdx.x; bi < per; bi += kThreads) {
        int row, j;
        if (last) {
            // row fastest, so that consecutive threads write consecutive rows of one band index
            j = (int)(((float)bi + 0.5f) * io.inv_nrows);
            row = bi - j * nrows;
        } else {
            row = (int)fdiv((unsigned)bi, dg.mr_mul[s], dg.mr_sh[s]);
            j = bi - row * MR;
        }
        const int jq = last ? 0 : (int)fdiv((unsigned)j, dg.ns_mul[s], dg.ns_sh[s]);
        const int k = j - jq * Ns;
        const int base = row * M;
        cpx<G> v[RD];
        if (first) {
#pragma unroll
            for (int q = 0; q < RD; ++q) {
                const int pos = j + q * MR;
                v[q] = (pos >= io.zlo && pos < io.zhi) ? cmk<G>((G)0, (G)0) : x[pad(base + pos)];
            }
        } else {
#pragma unroll
            for (int q = 0; q < RD; ++q) v[q] = x[pad(base + j + q * MR)];
        }
        if (Ns > 1) {
            if constexpr (sizeof(G) == 4) {
                // FP32: twiddles w^q, w = e^{2 pi i k / (Ns RD)}, from one table load and RD - 2 products
                // (the FMA pipe has room, the load pipe less; the products add a few ulps, measured
                // 9.2e-7 -> 9.4e-7 of relative L2 on the mixed 127-antenna workload)
                const cpx<G> w1 = tw[k * twstep];
                cpx<G> wq = w1;
#pragma unroll
                for (int q = 1; q < RD; ++q) {
                    v[q] = cmul(v[q], wq);
                    if (q + 1 < RD) wq = cmul(wq, w1);
                }
            } else {
                // FP64: products would run on the narrow FP64 pipe, so every twiddle comes from the table
#pragma unroll
                for (int q = 1; q < RD; ++q) v[q] = cmul(v[q], tw[q * k * twstep]);
            }
        }
        Dft<G, RD>::run(v);
        if (last) {
            if (row < io.nr) {
#pragma unroll
                for (int q = 0; q < RD; ++q) {
                    int b = k + q * Ns + io.H;
                    while (b >= M) b -= M;
                    for (; b < io.B; b += M) io.out[(size_t)b * io.rows + io.row0 + row] = v[q];
                }
            }
        } else {
            const int o = base + jq * Ns * RD + k;
#pragma unroll
            for (int q = 0; q < RD; ++q) y[pad(o + q * Ns)] = v[q];
        }
    }
    __syncthreads();
}

template <class G, int MAXRD>
__device__ __forceinline__ void run_stage(int rd, const cpx<G> *x, cpx<G> *y, const DimGeom &dg, int s, int nrows,
                                          int Ns, const cpx<G> *tw, bool first, StageIO<G> io)
{
    switch (rd) {
    case 2: stage<G, 2>(x, y, dg, s, nrows, Ns, tw, first, io); break;
    case 3: stage<G, 3>(x, y, dg, s, nrows, Ns, tw, first, io); break;
    case 4: stage<G, 4>(x, y, dg, s, nrows, Ns, tw, first, io); break;
    case 5: stage<G, 5>(x, y, dg, s, nrows, Ns, tw, first, io); break;
    case 6: stage<G, 6>(x, y, dg, s, nrows, Ns, tw, first, io); break;
    case 8: stage<G, 8>(x, y, dg, s, nrows, Ns, tw, first, io); break;
    default:
        if constexpr (MAXRD > 8) {
            switch (rd) {
            case 9: stage<G, 9>(x, y, dg, s, nrows, Ns, tw, first, io); break;
            case 10: stage<G, 10>(x, y, dg, s, nrows, Ns, tw, first, io); break;
            case 12: stage<G, 12>(x, y, dg, s, nrows, Ns, tw, first, io); break;
            case 15: stage<G, 15>(x, y, dg, s, nrows, Ns, tw, first, io); break;
            default: stage<G, 16>(x, y, dg, s, nrows, Ns, tw, first, io); break;
            }
        }
        break;
    }
}

// kRowsElems: the input values of one row block held in registers (prefetch); kSmemElems: the
// transform points of one row block in shared memory (rows per CTA = kSmemElems / M).  FP32: 6,144
// points, i.e. two rows of 3,072 (measured 16 % faster x passes than one row per CTA: three butterflies
// per thread and stage instead of one or two), the prefetch covering their 2 x 1,500 inputs.
template <class G> struct FftCfg;
template <> struct FftCfg<float> { static constexpr int kRowsElems = 4096, kSmemElems = 6144; };
template <> struct FftCfg<double> { static constexpr int kRowsElems = 2048, kSmemElems = 2048; };

int fft_rows_per_cta(int M, int elem_bytes)
{
    const int cap = elem_bytes == 4 ? FftCfg<float>::kSmemElems : FftCfg<double>::kSmemElems;
    int R = cap / M;
    return R < 1 ? 1 : (R > 8 ? 8 : R);
}

__host__ __device__ __forceinline__ size_t buf_elems(int R, int M) { return (size_t)R * M + ((size_t)R * M >> 4) + 1; }

size_t fft_pass_smem_bytes(int M, int elem_bytes)
{
    return 2 * buf_elems(fft_rows_per_cta(M, elem_bytes), M) * 2 * elem_bytes;
}

// longest row: two padded buffers of one row within 200 KB of shared memory
int fft_max_M(int elem_bytes) { return elem_bytes == 4 ? 12000 : 6000; }

// Input of one row block, held in registers between blocks so that the
// global loads of block i+1 are in flight while block i runs its stages.
template <class G> struct Prefetch {
    static constexpr int kMax = FftCfg<G>::kRowsElems / kThreads;   // values per thread
    cpx<G> v[kMax];
};

template <class G>
__device__ __forceinline__ void prefetch_rows(Prefetch<G> &pf, const cpx<G> *__restrict__ in, long rows, long row0,
                                              int R, int N)
{
    const int tot = R * N;
#pragma unroll
    for (int k = 0; k < Prefetch<G>::kMax; ++k) {
        const int idx = threadIdx.x + k * kThreads;
        const long r = row0 + idx / N;
        pf.v[k] = (idx < tot && r < rows) ? in[row0 * N + idx] : cmk<G>((G)0, (G)0);
    }
}

// resident CTAs per SM the register allocation must allow (FP32 radix <= 8: 3 CTAs at <= 80 registers
// without spills; the wider instances need more registers per thread)
template <class G, int MAXRD> struct FftMinBlocks {
    static constexpr int value = sizeof(G) == 4 ? (MAXRD <= 8 ? 3 : 2) : 1;
};

template <class G, int MAXRD>
__global__ void __launch_bounds__(kThreads, (FftMinBlocks<G, MAXRD>::value)) k_fft_rows(const cpx<G> *__restrict__ in, cpx<G> *__restrict__ out,
                                                       long rows, DimGeom dg, const G *__restrict__ pre,
                                                       const cpx<G> *__restrict__ tw, int R)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int M = dg.M, N = dg.nf1, B = dg.B, H = dg.H;
    cpx<G> *buf0 = reinterpret_cast<cpx<G> *>(smem_raw);
    cpx<G> *buf1 = buf0 + buf_elems(R, M);
    const int half = N / 2;
    const long stride = (long)gridDim.x * R;
    Prefetch<G> pf;
    long row0 = (long)blockIdx.x * R;
    if (row0 < rows) prefetch_rows(pf, in, rows, row0, R, N);
    for (; row0 < rows; row0 += stride) {
        const int nr = (int)((rows - row0) < R ? (rows - row0) : R);
        // the prefetched row values with the prescale: l -> slot (l - N/2) mod M; the other slots are
        // zeros that are never stored (the first stage knows where they are)
#pragma unroll
        for (int k = 0; k < Prefetch<G>::kMax; ++k) {
            const int idx = threadIdx.x + k * kThreads;
            if (idx < R * N) {
                const int r = idx / N;
                const int l = idx - r * N;
                int m = l - half;
                if (m < 0) m += M;
                buf0[pad(r * M + m)] = pre ? cscale(pf.v[k], pre[l]) : pf.v[k];
            }
        }
        // a row longer than the prefetch holds (then R = 1): the rest of it straight from memory
        for (int idx = Prefetch<G>::kMax * kThreads + threadIdx.x; idx < R * N; idx += kThreads) {
            const int r = idx / N;
            const int l = idx - r * N;
            int m = l - half;
            if (m < 0) m += M;
            const cpx<G> v = row0 + r < rows ? in[row0 * N + idx] : cmk<G>((G)0, (G)0);
            buf0[pad(r * M + m)] = pre ? cscale(v, pre[l]) : v;
        }
        __syncthreads();
        // issue the next block's loads before the stages
        if (row0 + stride < rows) prefetch_rows(pf, in, rows, row0 + stride, R, N);
        cpx<G> *x = buf0, *y = buf1;
        int Ns = 1;
        StageIO<G> io{N - half, M - half, nullptr, rows, row0, nr, B, H, 1.0f / (float)R};
        for (int s = 0; s < dg.nstages; ++s) {
            const int rd = dg.radix[s];
            io.out = s == dg.nstages - 1 ? out : nullptr;
            run_stage<G, MAXRD>(rd, x, y, dg, s, R, Ns, tw, s == 0, io);
            cpx<G> *t = x; x = y; y = t;
            Ns *= rd;
        }
    }
}

template <class G, int MAXRD>
static cudaError_t launch_rows(const cpx<G> *in, cpx<G> *out, long rows, const DimGeom &dg, const G *pre,
                               const cpx<G> *tw, cudaStream_t st)
{
    const int R = fft_rows_per_cta(dg.M, sizeof(G));
    const size_t smem = 2 * buf_elems(R, dg.M) * sizeof(cpx<G>);
    static bool attr_set[64] = {};
    static int max_ctas[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_set[dev]) {
        e = cudaFuncSetAttribute(k_fft_rows<G, MAXRD>, cudaFuncAttributeMaxDynamicSharedMemorySize, 210000);
        if (e != cudaSuccess) return e;
        attr_set[dev] = true;
    }
    // persistent CTAs: as many as fit on the device for the largest configuration (each keeps a
    // row block of prefetch in registers)
    if (!max_ctas[dev]) {
        int sms = 0;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        max_ctas[dev] = sms;
    }
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fft_rows<G, MAXRD>, kThreads, smem);
    if (e != cudaSuccess) return e;
    const long cap = (long)max_ctas[dev] * (per_sm > 0 ? per_sm : 1);
    const long ctas = (rows + R - 1) / R;
    const unsigned grid = (unsigned)(ctas < cap ? ctas : cap);
    k_fft_rows<G, MAXRD><<<grid, kThreads, smem, st>>>(in, out, rows, dg, pre, tw, R);
    return cudaGetLastError();
}

template <class G>
cudaError_t launch_fft_pass(const cpx<G> *in, cpx<G> *out, long rows, const DimGeom &dg, const G *pre,
                            const cpx<G> *tw, cudaStream_t st)
{
    if (rows <= 0) return cudaSuccess;
    if (dg.M > fft_max_M(sizeof(G)) || dg.nstages < 1) return cudaErrorInvalidValue;
    int maxrd = 1;
    for (int s = 0; s < dg.nstages; ++s) maxrd = dg.radix[s] > maxrd ? dg.radix[s] : maxrd;
    if (maxrd <= 8) return launch_rows<G, 8>(in, out, rows, dg, pre, tw, st);
    return launch_rows<G, 16>(in, out, rows, dg, pre, tw, st);
}

template cudaError_t launch_fft_pass<double>(const cpx<double> *, cpx<double> *, long, const DimGeom &,
                                             const double *, const cpx<double> *, cudaStream_t);
template cudaError_t launch_fft_pass<float>(const cpx<float> *, cpx<float> *, long, const DimGeom &, const float *,
                                            const cpx<float> *, cudaStream_t);

// ---------------------------------------------------------------- compile-time lengths (fv_fft_fixed.cuh)
#define FV_FIXED_ARGS(G) const cpx<G> *in, cpx<G> *out, int rows, const DimGeom &dg, int P, int sP, int nz, int nzp, \
                         const cpx<G> *twB, cpx<G> *clr, cudaStream_t st
cudaError_t fft_fixed_a(FV_FIXED_ARGS(float));      // lengths up to 864
cudaError_t fft_fixed_b(FV_FIXED_ARGS(float));      // up to 1728
cudaError_t fft_fixed_c(FV_FIXED_ARGS(float));      // up to 2560
cudaError_t fft_fixed_d(FV_FIXED_ARGS(float));      // up to 4096
cudaError_t fft_pairs_a(FV_FIXED_ARGS(Pf));
cudaError_t fft_pairs_b(FV_FIXED_ARGS(Pf));
cudaError_t fft_pairs_c(FV_FIXED_ARGS(Pf));
cudaError_t fft_pairs_d(FV_FIXED_ARGS(Pf));

struct FixedLength { short M, R2, R3; };
// every product 16 R2 R3 from 256 to 4096 of the radices 4, 5, 6, 8, 9, 10, 12, 15, 16, at most 17 % apart above 480, and
// 16 R2 below (two stages), for the short axis of a thin array: with nothing below 256 an axis that needs 20 points had
// a band of 139 values in place of 27.  East-west line of 60 antennas, 760 m, 0.4 m of scatter across: four products x 7
// height terms 76 -> 25 MB a stream and 124 -> 103 us a slice, FP64 with 16 up planes 91 -> 36 MB and 463 -> 400 us
// (general lengths and the spreading that goes with them: 260 and 1,123 us).
static const FixedLength kFixed[] = {
    {32, 2, 1}, {48, 3, 1}, {64, 4, 1}, {80, 5, 1}, {96, 6, 1}, {128, 8, 1}, {160, 10, 1}, {192, 12, 1},
    {256, 4, 4}, {320, 5, 4}, {384, 6, 4}, {400, 5, 5}, {480, 6, 5}, {512, 8, 4},
    {576, 6, 6}, {640, 8, 5}, {720, 9, 5}, {768, 8, 6}, {800, 10, 5}, {864, 9, 6},
    {960, 10, 6}, {1024, 8, 8}, {1152, 9, 8}, {1200, 15, 5}, {1280, 10, 8}, {1296, 9, 9},
    {1440, 10, 9}, {1536, 12, 8}, {1600, 10, 10}, {1728, 12, 9}, {1920, 12, 10}, {2048, 16, 8},
    {2160, 15, 9}, {2304, 12, 12}, {2400, 15, 10}, {2560, 16, 10}, {2880, 15, 12}, {3072, 16, 12},
    {3600, 15, 15}, {3840, 16, 15}, {4096, 16, 16}};

bool fft_choose_fixed(int target, int *radix, int &nstages, int &M)
{
    for (const FixedLength &l : kFixed)
        if (l.M >= target) {
            M = l.M;
            radix[0] = 16;
            radix[1] = l.R2;
            radix[2] = l.R3;
            nstages = l.R3 > 1 ? 3 : 2;
            return true;
        }
    return false;
}

size_t fft_fixed_table(const DimGeom &dg) { return (size_t)16 * dg.radix[1] + dg.M; }

// tb[q 16 + m1] = e^{2 pi i q m1 / (16 R2)}, then tc[q 16 R2 + c] = e^{2 pi i q c / M}
template <class G> __global__ void k_fixed_twiddles(cpx<G> *tw, int M, int R2)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int nB = 16 * R2;
    if (k >= nB + M) return;
    double s, c;
    if (k < nB) {
        sincospi(2.0 * (double)((k / 16) * (k % 16)) / (double)nB, &s, &c);
    } else {
        const int j = k - nB;
        sincospi(2.0 * (double)((j / nB) * (j % nB)) / (double)M, &s, &c);
    }
    tw[k] = cmk<G>((G)c, (G)s);
}

template <class G> cudaError_t launch_fixed_twiddles(cpx<G> *tw, const DimGeom &dg, cudaStream_t st)
{
    const int n = (int)fft_fixed_table(dg);
    k_fixed_twiddles<G><<<(n + 255) / 256, 256, 0, st>>>(tw, dg.M, dg.radix[1]);
    return cudaGetLastError();
}
template cudaError_t launch_fixed_twiddles<float>(cpx<float> *, const DimGeom &, cudaStream_t);
template cudaError_t launch_fixed_twiddles<Pf>(cpx<Pf> *, const DimGeom &, cudaStream_t);

template <class G>
cudaError_t launch_fft_fixed(const cpx<G> *in, cpx<G> *out, long rows, const DimGeom &dg, int P, int sP, int nz, int nzp,
                             const cpx<G> *tw, cudaStream_t st, cpx<G> *clr)
{
    if (rows <= 0) return cudaSuccess;
    if (rows > (1L << 30) || P < 1 || nz < 1) return cudaErrorInvalidValue;
    const int r = (int)rows;
    if constexpr (sizeof(G) == 4) {
        if (dg.M <= 864) return fft_fixed_a(in, out, r, dg, P, sP, nz, nzp, tw, clr, st);
        if (dg.M <= 1728) return fft_fixed_b(in, out, r, dg, P, sP, nz, nzp, tw, clr, st);
        if (dg.M <= 2560) return fft_fixed_c(in, out, r, dg, P, sP, nz, nzp, tw, clr, st);
        return fft_fixed_d(in, out, r, dg, P, sP, nz, nzp, tw, clr, st);
    } else {
        if (dg.M <= 864) return fft_pairs_a(in, out, r, dg, P, sP, nz, nzp, tw, clr, st);
        if (dg.M <= 1728) return fft_pairs_b(in, out, r, dg, P, sP, nz, nzp, tw, clr, st);
        if (dg.M <= 2560) return fft_pairs_c(in, out, r, dg, P, sP, nz, nzp, tw, clr, st);
        return fft_pairs_d(in, out, r, dg, P, sP, nz, nzp, tw, clr, st);
    }
}
template cudaError_t launch_fft_fixed<float>(const cpx<float> *, cpx<float> *, long, const DimGeom &, int, int, int, int,
                                             const cpx<float> *, cudaStream_t, cpx<float> *);
template cudaError_t launch_fft_fixed<Pf>(const cpx<Pf> *, cpx<Pf> *, long, const DimGeom &, int, int, int, int,
                                          const cpx<Pf> *, cudaStream_t, cpx<Pf> *);

// ---------------------------------------------------------------- host planning
static const int kRadices[] = {16, 15, 12, 10, 9, 8, 6, 5, 4, 3, 2};

static bool factor_into(int M, int maxStages, int maxRadix, int *rad, int &n)
{
    if (M == 1) return true;
    if (maxStages == 0) return false;
    for (int r : kRadices)
        if (r <= maxRadix && M % r == 0) {
            rad[n++] = r;
            if (factor_into(M / r, maxStages - 1, maxRadix, rad, n)) return true;
            --n;
        }
    return false;
}

// multiply-high division by d: q = (umulhi(n, mul) + n) >> sh for n < 2^31
void fft_magic(unsigned d, unsigned &mul, unsigned &sh)
{
    unsigned s = 0;
    while ((1ull << s) < d) ++s;
    sh = s;
    mul = (unsigned)((((1ull << 32) * ((1ull << s) - d)) / d) + 1);
}

int fft_choose_length(int target, int *radix, int &nstages, int maxRadix)
{
    if (maxRadix < 2) maxRadix = 16;
    // stage budget: enough stages of maxRadix to reach the target, at least 3
    int maxStages = 3;
    for (long span = (long)maxRadix * maxRadix * maxRadix; span < target && maxStages < FV_MAX_STAGES; span *= maxRadix)
        ++maxStages;
    for (int M = target + (target & 1); M <= 4 * target + 64; M += 2) {
        int n = 0;
        if (factor_into(M, maxStages, maxRadix, radix, n)) {
            nstages = n;
            return M;
        }
    }
    return -1;
}

void fft_stage_constants(DimGeom &dg)
{
    int Ns = 1;
    for (int s = 0; s < dg.nstages; ++s) {
        fft_magic((unsigned)(dg.M / dg.radix[s]), dg.mr_mul[s], dg.mr_sh[s]);
        fft_magic((unsigned)Ns, dg.ns_mul[s], dg.ns_sh[s]);
        Ns *= dg.radix[s];
    }
}

}  // namespace fv
