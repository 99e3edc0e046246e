"""The one-pass preparation and spreading of FP32 slices (sources sorted by strips, a register window of the
grid per warp) and the compile-time-length FFT passes, against the paths that use neither.

Both sides are within the mixed path's error of the direct sum (about eps plus FP32 rounding, 1.2e-6 at eps 1e-6),
so they differ by at most a few times that: 1e-5 at eps 1e-6, ten times eps where eps is larger.
"""
import numpy as np
import pytest

from oracle.oracle import OracleProblem, oracle_vis, rel_l2
from paper_2506_02130_gb300 import fv, workloads as W

pytestmark = pytest.mark.gpu


def _run(prob, eps, **kw):
    p = fv.Plan.from_problem(prob, precision=fv.FV_MIXED, eps=eps, transform="type3", **kw)
    try:
        p.set_sky(prob.sky.ra, prob.sky.dec, prob.sky.flux)
        return p.run(), p.info()
    finally:
        p.close()


def _prob(n_src, polarised=False, seed=3, radius=3, n_chan=2, z_sigma=0.0):
    rng = np.random.default_rng(seed)
    make = W.config_hex350_pol if polarised else W.config_hex127
    kw = dict(n_keep=None) if polarised else {}
    prob = make(seed=seed, n_chan=n_chan, n_time=1, n_point=n_src, nside=0, radius=radius, **kw)
    prob.ant_enu = W.hex_array(radius)
    prob.ant_enu[:, :2] += rng.normal(0.0, 0.3, (len(prob.ant_enu), 2))
    if z_sigma:
        prob.ant_enu[:, 2] = rng.normal(0.0, z_sigma, len(prob.ant_enu))
    return prob


@pytest.mark.parametrize("polarised", [False, True])
@pytest.mark.parametrize("n_src", [1, 2, 9, 65, 700, 40000])
def test_source_counts(n_src, polarised):
    """One source, less than a batch, a batch and a rest, several runs of sources per warp."""
    prob = _prob(n_src, polarised)
    if n_src <= 2:            # above the horizon
        prob.sky.dec[:] = prob.latitude_rad + 0.3
        prob.sky.ra[:] = prob.lsts_rad[0]
    out, info = _run(prob, 1e-6)
    assert info["spread"] == "gather"
    assert rel_l2(out, oracle_vis(OracleProblem.from_workload(prob), "factored")) <= 2e-5


@pytest.mark.parametrize("polarised", [False, True])
@pytest.mark.parametrize("eps", [1e-2, 1e-3, 1e-4, 1e-5, 1e-6])
def test_kernel_widths_against_the_atomic_spreading(eps, polarised):
    """Kernels of 3 to 7 points: the window's room beside the footprint, and the polynomial kernel values."""
    prob = _prob(3000, polarised)
    out, info = _run(prob, eps)
    assert info["kernel_width"] <= 7
    ref, _ = _run(prob, eps, spread="atomic")
    assert rel_l2(out, ref) <= max(1e-5, eps)


@pytest.mark.parametrize("bins", [(1, 1), (64, 64), (3, 7), (33, 2)])
def test_any_order_of_the_sources(bins):
    """Bins far from the strips the spreading prefers: sources leave the window in every direction."""
    prob = _prob(6000, True)
    out, _ = _run(prob, 1e-6, bin_size=bins)
    ref, _ = _run(prob, 1e-6)
    assert rel_l2(out, ref) <= 2e-6


@pytest.mark.parametrize("z_sigma,heights,polarised", [(0.002, "terms", False), (0.02, "terms", True),
                                                      (0.05, "terms", False), (0.3, "terms", False),
                                                      (0.02, "grid", True), (0.3, "grid", False)])
def test_planes(z_sigma, heights, polarised):
    """Up planes and height terms of 3 to 16, odd and even, one and two groups of eight."""
    prob = _prob(2500, polarised, radius=2, z_sigma=z_sigma)
    out, info = _run(prob, 1e-6, heights=heights)
    assert (info["height_terms"] > 0) == (heights == "terms")
    assert rel_l2(out, oracle_vis(OracleProblem.from_workload(prob), "factored")) <= 2e-5


@pytest.mark.parametrize("scale", list(np.geomspace(0.6, 11.0, 24)))
def test_fft_lengths_against_the_general_passes(scale):
    """Compile-time FFT lengths (radix cap 16, the default) against the general kernel (radix cap 8)."""
    prob = _prob(1500, n_chan=3)
    prob.ant_enu = prob.ant_enu * [scale, 0.7 * scale, 0.0]
    out, info = _run(prob, 1e-6)
    ref, _ = _run(prob, 1e-6, fft_max_radix=8)
    assert rel_l2(out, ref) <= 1e-5, info["nf2_max"]


@pytest.mark.parametrize("z_sigma,polarised,kw", [(0.05, False, dict(heights="terms")), (0.02, True, dict(heights="terms")),
                                                 (0.1, False, dict(heights="grid")), (0.02, True, dict(heights="grid")),
                                                 (0.02, False, dict(heights="terms", kernel_width=11)),
                                                 (0.05, False, dict(heights="grid", kernel_width=14))])
def test_plane_interpolation_writes_every_copy_of_a_baseline(z_sigma, polarised, kw):
    """Antennas in pairs of equal offset, so that targets have several baselines, with planes to sum."""
    prob = _prob(900, polarised, radius=2, z_sigma=z_sigma)
    n = len(prob.ant_enu)
    prob.ant_enu = np.concatenate([prob.ant_enu, prob.ant_enu + [512.0, 256.0, 0.0]]) * [0.25, 0.25, 1.0]
    prob.ant_enu = np.round(prob.ant_enu * 1024) / 1024          # exact differences
    prob.pairs = W.cross_pairs(2 * n)
    out, info = _run(prob, 1e-6, **kw)
    assert info["n_unique"] < info["n_bl"]
    assert rel_l2(out, oracle_vis(OracleProblem.from_workload(prob), "factored")) <= 2e-5
