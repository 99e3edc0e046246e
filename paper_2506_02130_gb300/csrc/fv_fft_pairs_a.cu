// Instances of the compile-time-length FFT pass on pairs of floats, lengths 32 to 864 (one translation unit of several, so
// that they compile side by side).
#include "fv_fft_fixed.cuh"

namespace fv {

cudaError_t fft_pairs_a(const cpx<Pf> *in, cpx<Pf> *out, int rows, const DimGeom &dg, int P, int sP, int nz,
                        int nzp, const cpx<Pf> *twB, cpx<Pf> *clr, cudaStream_t st)
{
    switch (dg.M) {
    case 32: return fft_fixed_go<Pf, 2, 1>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 48: return fft_fixed_go<Pf, 3, 1>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 64: return fft_fixed_go<Pf, 4, 1>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 80: return fft_fixed_go<Pf, 5, 1>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 96: return fft_fixed_go<Pf, 6, 1>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 128: return fft_fixed_go<Pf, 8, 1>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 160: return fft_fixed_go<Pf, 10, 1>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 192: return fft_fixed_go<Pf, 12, 1>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 256: return fft_fixed_go<Pf, 4, 4>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 320: return fft_fixed_go<Pf, 5, 4>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 384: return fft_fixed_go<Pf, 6, 4>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 400: return fft_fixed_go<Pf, 5, 5>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 480: return fft_fixed_go<Pf, 6, 5>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 512: return fft_fixed_go<Pf, 8, 4>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 576: return fft_fixed_go<Pf, 6, 6>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 640: return fft_fixed_go<Pf, 8, 5>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 720: return fft_fixed_go<Pf, 9, 5>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 768: return fft_fixed_go<Pf, 8, 6>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 800: return fft_fixed_go<Pf, 10, 5>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 864: return fft_fixed_go<Pf, 9, 6>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace fv
