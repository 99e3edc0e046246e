// The lattice route without a grid (fv_lattice_dense.cu): direct sums at the array's modes.
#pragma once
#include "fv_internal.cuh"

#include <vector>

namespace fv {

// Largest (2 H_1 + 1)(H_2 + 1) evaluated directly, for skies of up to kDenseFew sources: the grid's clearing, FFT passes
// and launches cost twice a small sky's direct sums (2,000 sources, 1,431 modes, one term, 16 channels: 6.6 against
// 16.6 us a slice in FP32, 12.6 against 32.7 in FP64).  Larger skies: dense_modes_max.
constexpr int kDenseModes = 1600;
constexpr long kDenseFew = 50000;

struct DenseGeom {
    double a[2][2];          // lattice vectors (east, north), m
    int H1, H2, K, J;        // largest |n_1| and |n_2|, height terms, real strengths x terms
    int CS;                  // sources a chunk in shared memory
    int NA, NB;              // phase factors held per source: n_2 = 0..NA-1, n_1 = -H_1..NB-1-H_1 (whole tiles)
    int n_tiles, tile_blocks;
    const int *tiles;        // device: first n_2 | (first n_1 + H_1) << 16 of every tile with a mode in use
};

inline size_t dense_modes(const DenseGeom &dg) { return (size_t)dg.J * (2 * dg.H1 + 1) * (dg.H2 + 1); }

// Host: the geometry (without a and tiles) and its tile list, or false where the grid has to do it.
bool dense_plan(int elem, double eps, int w, long n_src, int K, int n_pol, int H1, int H2, int n_bl, const int *bln, DenseGeom &dg,
                std::vector<int> &tiles);

// Mode sums (FP64) [nch][J][H_2 + 1][2 H_1 + 1] of channels f0 .. f0 + nch of one time from its sources above the horizon
// (FP64: sdir; FP32: records tc of launch_time_compact; sidx, *nv_ptr).  g: any channel's geometry with the group's beams (the channel's frequency comes from freq).
template <class G>
cudaError_t launch_lattice_dense(const double *sdir, const float4 *tc, const int *sidx, const int *nv_ptr, long n_src, const void *flux,
                                 int flux_fp64, int n_freq, int f0, int nch, const double *freq, const SliceGeom &g,
                                 const DenseGeom &dg, cpx<double> *modes, cudaStream_t st);

// Visibilities of baselines bl_list[0..n_bl) (nullptr: all n_bl) of channels f0 .. f0 + nch from those sums; channel
// f0 + k is written at out0 + k slice_stride bytes.
template <class G>
cudaError_t launch_dense_gather(const cpx<double> *modes, const int *bln, const int *bl_list, int n_bl, int n_bl_all,
                                int n_pol, const DenseGeom &dg, int f0, int nch, const cpx<double> *wq, void *out0,
                                long slice_stride, cudaStream_t st);

}  // namespace fv
