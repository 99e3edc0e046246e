// FP64 type-3 slices in pairs of floats (fv_pairs.cu).
#pragma once
#include "fv_pair.cuh"
#include "fv_staged.cuh"

namespace fv {

// Kernel values phi((2/w)(l0 - q + j)) of a w <= kPairW point kernel as polynomials of s = 2 (l0 - q + w/2) - 1:
// es[0][p][k] even and es[1][p][k] odd coefficients of value p and, mirrored, of value w - 1 - p.
constexpr int kPairW = 13, kPairTerms = 7, kPairHalf = (kPairW + 1) / 2;
constexpr int kPairPoly = 2 * kPairHalf * kPairTerms;
struct PairPoly { Pf v[kPairPoly]; };
PairPoly pair_polynomials(int w, double beta);

// A target of one slice: first footprint cell, s of both axes, postphase x deconvolution.
struct __align__(16) PairTarget {
    int m0, m1, pad0, pad1;
    Pf sx, sy;
    cpx<Pf> post;
};
static_assert(sizeof(PairTarget) == 48, "three 16-byte rows");

// Whether the pair kernels hold a slice: w <= 13, one or four products, planes the gather kernel has sums for.
bool pairs_fit(int w, int n_pol, int nz);

// Gather spreading of staged FP64 records onto a grid of pairs [n_pol][nz][ny][nx], prescaled.  key: the strengths'
// largest exponent (launch_prep_staged); the grid is scaled by 2^pair_shift(*key), which the interpolation takes back.
cudaError_t launch_spread_pairs(const int *offsets, const SrcRec<double> *rec, const cpx<double> *cs, const SliceGeom &g,
                                const TimeBin &tb, double r0, double r1, const PairPoly &es, const unsigned *key, cpx<Pf> *grid, cudaStream_t st);
// Interpolation of the band of pairs [b_y][b_x][n_pol][nz] at the n_u targets bu, written to their baselines (so).
// tgt [chunk] and wz [chunk][nz] are scratch: chunk targets at a time.
cudaError_t launch_interp_pairs(const cpx<Pf> *band, const double *bu, int n_u, const double *dec, const SliceGeom &g,
                                const double *prez, const cpx<double> *twz, const PairPoly &es, const unsigned *key, int chunk,
                                PairTarget *tgt, cpx<Pf> *wz, const SliceOut &so, cudaStream_t st);

}  // namespace fv
