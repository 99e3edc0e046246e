// Instances of the compile-time-length FFT pass, lengths 1920 to 2560 (one translation unit of several, so
// that they compile side by side).
#include "fv_fft_fixed.cuh"

namespace fv {

cudaError_t fft_fixed_c(const cpx<float> *in, cpx<float> *out, int rows, const DimGeom &dg, int P, int sP, int nz,
                        int nzp, const cpx<float> *twB, cpx<float> *clr, cudaStream_t st)
{
    switch (dg.M) {
    case 1920: return fft_fixed_go<float, 12, 10>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 2048: return fft_fixed_go<float, 16, 8>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 2160: return fft_fixed_go<float, 15, 9>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 2304: return fft_fixed_go<float, 12, 12>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 2400: return fft_fixed_go<float, 15, 10>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 2560: return fft_fixed_go<float, 16, 10>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace fv
