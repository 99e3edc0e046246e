// FFT passes of FP32 grids, and of grids of float pairs (G = Pf: FP64 plans), with compile-time lengths
// M = 16 R2 R3 (R3 = 1 below 256: the third stage only stores; M >= 2 N, no prescale): the same transform as k_fft_rows (zero-padded rows of N values at l - N/2 mod M, sign +, band of outputs m in [-H, B-1-H], written
// transposed as out[b][row]).
//
// With n = n1 R2 R3 + n2 R3 + n3 and m = m1 + 16 m2 + 16 R2 m3 the transform is three stages of register DFTs,
// over n1, n2 and n3, with the twiddles e^{2 pi i m1 n2 / (16 R2)} and e^{2 pi i (m1 + 16 m2) n3 / M} before the
// second and third.  Every stage reads and writes the same places, so one buffer of R rows in shared memory and
// two barriers do: the first stage reads the rows from memory (only the eight of its 16 points that can hold
// data: the row fills at most half of M), the last one writes its outputs to memory (only those that can lie in
// the band, M / 4 and a few points on either side of zero).  A row's place is [m1][n2][n3] with odd strides and
// rows 4 (R = 4) or 8 (R = 2) complex values apart modulo 16, which keeps every stage's accesses free of bank
// conflicts; consecutive lanes take the R rows of one point, so that a transposed store fills a 32-byte sector
// and a load of interleaved planes is contiguous.
//
// What bounds it: instruction issue (52-58 % busy), with half of the multi-length kernel's instructions (15.1 M
// against 29.1 M for 3,000 rows of 3,072: no index divisions by variables, no products for the twiddles, half of
// the first stage's inputs and of the last one's outputs left out), then the waits for the rows.  Packed FP32 x 2
// sums (one instruction for a complex sum) changed nothing: 22.2 against 21.6 us, the operands' moves take the slots.
// Measured per slice, one stream, against the multi-length kernel: 350-antenna workload 22 + 21 us (x and y) against
// 55 + 50, 127-antenna workload with 8 height terms 17 + 16 against 38 + 36.
#pragma once
#include "fv_dft.cuh"
#include "fv_pair.cuh"

namespace fv {

template <class G, int R2, int R3> struct FixedFft {
    static constexpr bool P = sizeof(G) == 8;                    // pairs: 16 bytes a value, twice the registers
    static constexpr int M = 16 * R2 * R3;
    static constexpr int R = P ? (M <= 2304 ? 2 : 1) : (M <= 3072 ? 4 : 2);     // rows a CTA (32 bytes of a transposed store)
    static constexpr int S3 = R3 | 1, S1 = (R2 * S3) | 1;       // strides of n2 and m1
    static constexpr int kOff = R == 4 || P ? 4 : 8;             // pairs move 8 lanes at a time, others 16
    static constexpr int S0 = (16 * S1 + 15 - kOff) / 16 * 16 + kOff;   // of a row: kOff modulo 16
    static constexpr int items = R * M / 16;
    static constexpr int rounds = items <= 320 ? 1 : (items <= 768 ? 2 : 3);
    static constexpr int T = (items + 32 * rounds - 1) / (32 * rounds) * 32;
    static constexpr int smem = R * S0 * 2 * (int)sizeof(G);
    // registers a thread: pairs 160, above 1,152 points 128 (a second CTA per SM: 1,728 and 1,920 points 102 -> 92 us;
    // at 576 to 864 points 128 is slower, 77 against 74 us)
    static constexpr int regs = P ? (M > 1152 ? 128 : 160) : 80;
    static constexpr int by_smem = 225000 / (smem + 1024), by_regs = 65536 / (T * regs);
    static constexpr int blocks = by_smem < by_regs ? (by_smem > 0 ? by_smem : 1) : (by_regs > 0 ? by_regs : 1);
    static constexpr int keep = R3 / 4;                          // outputs m3 <= keep and m3 >= R3 - 1 - keep
};

// first-stage DFT of 16 points of which 4..11 are zero: v[0..3] = points 0..3, v[4..7] = points 12..15
template <class G> __device__ __forceinline__ void dft16_half(const cpx<G> *v, cpx<G> *o)
{
    using C = cpx<G>;
    C U[4][4];
    auto column = [&](const int r2, C a, C d) {
        // points r2 (r1 = 0) and 12 + r2 (r1 = 3): a + d e^{2 pi i 3 q / 4}
        U[r2][0] = cadd(a, d);
        U[r2][1] = cmk<G>(a.x + d.y, a.y - d.x);
        U[r2][2] = csub(a, d);
        U[r2][3] = cmk<G>(a.x - d.y, a.y + d.x);
    };
    column(0, v[0], v[4]);
    column(1, v[1], v[5]);
    column(2, v[2], v[6]);
    column(3, v[3], v[7]);
    U[1][1] = twm<G, 1, 16>(U[1][1]);
    U[1][2] = twm<G, 2, 16>(U[1][2]);
    U[1][3] = twm<G, 3, 16>(U[1][3]);
    U[2][1] = twm<G, 2, 16>(U[2][1]);
    U[2][2] = twm<G, 4, 16>(U[2][2]);
    U[2][3] = twm<G, 6, 16>(U[2][3]);
    U[3][1] = twm<G, 3, 16>(U[3][1]);
    U[3][2] = twm<G, 6, 16>(U[3][2]);
    U[3][3] = twm<G, 9, 16>(U[3][3]);
#pragma unroll
    for (int q1 = 0; q1 < 4; ++q1) {
        C t[4] = {U[0][q1], U[1][q1], U[2][q1], U[3][q1]};
        Dft<G, 4>::run(t);
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2) o[q1 + 4 * q2] = t[q2];
    }
}

// rows (y, p), y = row / P, p = row % P: value l at in[(y N + l) sP + (p / nz) nzp + p % nz].  CLEAR: read from clr
// (the same rows), which is left zero for the next slice's spreading (with its padding plane): a memset launch less,
// for small grids (a 22 MB grid costs the pass more, 22 -> 33 us, than its memset, 8 us).
template <class G, int R2, int R3, bool CLEAR>
__global__ void __launch_bounds__((FixedFft<G, R2, R3>::T), (FixedFft<G, R2, R3>::blocks))
    k_fft_fixed(const cpx<G> *__restrict__ in, cpx<G> *clr, cpx<G> *__restrict__ out, int rows, int N, int H, int B, int P,
                int sP, int nz, int nzp, const cpx<G> *__restrict__ twB, const cpx<G> *__restrict__ twC)
{
    using F = FixedFft<G, R2, R3>;
    using C = cpx<G>;
    constexpr int M = F::M, R = F::R, T = F::T, S0 = F::S0, S1 = F::S1, S3 = F::S3, MB = R2 * R3;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *buf = reinterpret_cast<C *>(smem_raw);
    const int tid = threadIdx.x;
    const int row = blockIdx.x * R + tid % R;            // T is a multiple of R: a thread keeps its row
    const bool live = row < rows;
    C *mine = buf + (tid % R) * S0;
    {
        const int half = N / 2;
        const int y = live ? row / P : 0, p = live ? row - y * P : 0;
        const size_t at = (size_t)y * N * sP + (p / nz) * nzp + p % nz;
        const C *src = in + at;
        C *own = CLEAR ? clr + at : nullptr;
        const bool pad = CLEAR && nzp > nz && p % nz == nz - 1;
        const C zero = cmk<G>((G)0.0, (G)0.0);
#pragma unroll
        for (int k = 0; k < (R * MB + T - 1) / T; ++k) {
            const int j = tid / R + k * (T / R);
            if ((R * MB) % T != 0 && j >= MB) break;
            C v[8], o[16];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int pos = j + q * MB;                                     // l - N/2
                const bool in_row = live && pos < N - half;
                const size_t l = (size_t)(pos + half) * sP;
                v[q] = in_row ? (CLEAR ? own[l] : src[l]) : zero;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int l = j + (q - 4) * MB + half;
                v[4 + q] = live && l >= 0 ? (CLEAR ? own[(size_t)l * sP] : src[(size_t)l * sP]) : zero;
            }
            if constexpr (CLEAR) {
                if (live) {
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int l = j + (q < 4 ? q : q - 8) * MB + half;
                        if (q < 4 ? l < N : l >= 0) {
                            own[(size_t)l * sP] = zero;
                            if (pad) own[(size_t)l * sP + 1] = zero;
                        }
                    }
                }
            }
            dft16_half(v, o);
            C *d = mine + (j / R3) * S3 + j % R3;
#pragma unroll
            for (int q = 0; q < 16; ++q) d[q * S1] = o[q];
        }
    }
    __syncthreads();
    {
        constexpr int items = 16 * R3;
#pragma unroll
        for (int k = 0; k < (R * items + T - 1) / T; ++k) {
            const int j = tid / R + k * (T / R);
            if ((R * items) % T != 0 && j >= items) break;
            const int m1 = j / R3, n3 = j % R3;
            C *d = mine + m1 * S1 + n3;
            C v[R2];
            v[0] = d[0];
#pragma unroll
            for (int q = 1; q < R2; ++q) v[q] = cmul(d[q * S3], twB[q * 16 + m1]);
            Dft<G, R2>::run(v);
#pragma unroll
            for (int q = 0; q < R2; ++q) d[q * S3] = v[q];
        }
    }
    __syncthreads();
    {
        constexpr int items = 16 * R2;
#pragma unroll
        for (int k = 0; k < (R * items + T - 1) / T; ++k) {
            const int c = tid / R + k * (T / R);
            if ((R * items) % T != 0 && c >= items) break;
            const C *d = mine + (c % 16) * S1 + (c / 16) * S3;
            C v[R3];
            v[0] = d[0];
#pragma unroll
            for (int q = 1; q < R3; ++q) v[q] = cmul(d[q], twC[q * items + c]);
            Dft<G, R3>::run(v);
            if (!live) continue;
#pragma unroll
            for (int q = 0; q <= F::keep; ++q) {
                const int b = c + q * items + H;                                // m + H
                if (b < B) out[(size_t)b * rows + row] = v[q];
            }
#pragma unroll
            for (int q = R3 - 1 - F::keep; q < R3; ++q) {
                const int b = c + q * items + H - M;
                if (b >= 0) out[(size_t)b * rows + row] = v[q];
            }
        }
    }
}

template <class G, int R2, int R3>
cudaError_t fft_fixed_go(const cpx<G> *in, cpx<G> *out, int rows, const DimGeom &dg, int P, int sP, int nz, int nzp,
                         const cpx<G> *twB, cpx<G> *clr, cudaStream_t st)
{
    using F = FixedFft<G, R2, R3>;
    static_assert(F::T % F::R == 0 && F::T <= 1024, "a thread keeps one row");
    // what the kernel leaves out has to be empty: the row within half of M, the band within the kept outputs
    constexpr int third = 16 * R2;
    if (2 * dg.nf1 > F::M || dg.H >= (F::keep + 1) * third || dg.B - 1 - dg.H >= (F::keep + 1) * third)
        return cudaErrorInvalidValue;
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!attr_set[dev]) {
        e = cudaFuncSetAttribute(k_fft_fixed<G, R2, R3, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, F::smem);
        if constexpr (!F::P)
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(k_fft_fixed<G, R2, R3, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, F::smem);
        if (e != cudaSuccess) return e;
        attr_set[dev] = true;
    }
    const unsigned blocks = (unsigned)((rows + F::R - 1) / F::R);
    if constexpr (!F::P) {
        if (clr) {
            k_fft_fixed<G, R2, R3, true><<<blocks, F::T, F::smem, st>>>(nullptr, clr, out, rows, dg.nf1, dg.H, dg.B, P, sP, nz,
                                                                       nzp, twB, twB + 16 * R2);
            return cudaGetLastError();
        }
    }
    k_fft_fixed<G, R2, R3, false><<<blocks, F::T, F::smem, st>>>(in, nullptr, out, rows, dg.nf1, dg.H, dg.B, P, sP, nz, nzp,
                                                                twB, twB + 16 * R2);
    return cudaGetLastError();
}

}  // namespace fv
