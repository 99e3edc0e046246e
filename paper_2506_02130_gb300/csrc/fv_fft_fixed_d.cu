// Instances of the compile-time-length FFT pass, lengths 2880 to 4096 (one translation unit of several, so
// that they compile side by side).
#include "fv_fft_fixed.cuh"

namespace fv {

cudaError_t fft_fixed_d(const cpx<float> *in, cpx<float> *out, int rows, const DimGeom &dg, int P, int sP, int nz,
                        int nzp, const cpx<float> *twB, cpx<float> *clr, cudaStream_t st)
{
    switch (dg.M) {
    case 2880: return fft_fixed_go<float, 15, 12>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 3072: return fft_fixed_go<float, 16, 12>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 3600: return fft_fixed_go<float, 15, 15>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 3840: return fft_fixed_go<float, 16, 15>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    case 4096: return fft_fixed_go<float, 16, 16>(in, out, rows, dg, P, sP, nz, nzp, twB, clr, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace fv
