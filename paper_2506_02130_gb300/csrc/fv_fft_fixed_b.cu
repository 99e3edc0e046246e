// Instances of the compile-time-length FFT pass, lengths 960 to 1728 (one translation unit of several, so
// that they compile side by side).
#include "fv_fft_fixed.cuh"

namespace fv {

cudaError_t fft_fixed_b(const cpx<float> *in, cpx<float> *out, int rows, const DimGeom &dg, int P, int sP, int nz,
                        int nzp, const cpx<float> *twB, cpx<float> *clr, cudaStream_t st)
{
    switch (dg.M) {
    case 960: return fft_fixed_go<float, 10, 6>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 1024: return fft_fixed_go<float, 8, 8>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 1152: return fft_fixed_go<float, 9, 8>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 1200: return fft_fixed_go<float, 15, 5>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 1280: return fft_fixed_go<float, 10, 8>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 1296: return fft_fixed_go<float, 9, 9>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 1440: return fft_fixed_go<float, 10, 9>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 1536: return fft_fixed_go<float, 12, 8>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 1600: return fft_fixed_go<float, 10, 10>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 1728: return fft_fixed_go<float, 12, 9>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace fv
