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


@pytest.mark.parametrize("n_chan", [1, 2, 3, 31, 33])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("polarised", [False, True])
def test_flux_layouts(n_chan, dtype, polarised):
    """The channel-major copy of the fluxes: one channel to more than a tile's, both types, host and borrowed."""
    torch = pytest.importorskip("torch")
    prob = _prob(1500, polarised, radius=1, n_chan=n_chan)
    prob.sky.flux = np.ascontiguousarray(prob.sky.flux.astype(dtype))
    out, _ = _run(prob, 1e-6)
    assert rel_l2(out, oracle_vis(OracleProblem.from_workload(prob), "factored")) <= 2e-5
    dev = torch.from_numpy(prob.sky.flux).cuda()
    p = fv.Plan.from_problem(prob, precision=fv.FV_MIXED, eps=1e-6, transform="type3")
    p.set_sky(prob.sky.ra, prob.sky.dec, dev)
    assert rel_l2(p.run(), out) <= 2e-6
    dev *= 2.0                                   # rewritten in place between executions
    torch.cuda.synchronize()
    assert rel_l2(p.run(), 2.0 * out) <= 2e-6
    p.close()


def test_sources_on_the_horizon_are_cut_as_in_fp64():
    """Sources within a few FP64 roundings of the horizon: the pair arithmetic of the sort must not decide them."""
    prob = _prob(400, False, radius=2, n_chan=1)
    lst, lat = prob.lsts_rad[0], prob.latitude_rad
    az = np.linspace(0.0, 2 * np.pi, 400, endpoint=False)
    alt = np.repeat([0.0, 1e-17, -1e-17, 1e-16, -1e-16, 1e-15, -1e-15, 1e-13], 50)
    e, n, u = np.cos(alt) * np.sin(az), np.cos(alt) * np.cos(az), np.sin(alt)
    z = n * np.cos(lat) + u * np.sin(lat)
    r = -n * np.sin(lat) + u * np.cos(lat)
    prob.sky.dec = np.arcsin(np.clip(z, -1, 1))
    prob.sky.ra = (lst + np.arctan2(e, r)) % (2 * np.pi)
    prob.beam, prob.beam_param = "uniform", ()          # a beam that reaches the horizon
    mixed, _ = _run(prob, 1e-6)
    p = fv.Plan.from_problem(prob, precision=fv.FV_FP64, eps=1e-9, transform="type3")
    p.set_sky(prob.sky.ra, prob.sky.dec, prob.sky.flux)
    assert rel_l2(mixed, p.run()) <= 2e-5
    p.close()


@pytest.mark.parametrize("z_sigma,heights,polarised", [(0.0, "auto", True), (0.002, "terms", True), (0.05, "terms", False),
                                                      (0.02, "grid", True)])
def test_grid_left_clear_between_slices(z_sigma, heights, polarised):
    """The x pass leaves the grid clear for the next slice: channels of growing and shrinking grids, odd planes and
    their padding, one stream, against every channel in a plan of its own (the same sums in another order)."""
    prob = _prob(1500, polarised, n_chan=6, z_sigma=z_sigma)
    order = [3, 0, 5, 1, 4, 2]
    prob.freqs_hz = prob.freqs_hz[order]
    prob.sky.flux = np.ascontiguousarray(prob.sky.flux[:, :, order])
    flux, freqs = prob.sky.flux, prob.freqs_hz
    out, _ = _run(prob, 1e-6, heights=heights, n_streams=1)
    for f in range(6):
        prob.freqs_hz, prob.sky.flux = freqs[f:f + 1], np.ascontiguousarray(flux[:, :, f:f + 1])
        one, _ = _run(prob, 1e-6, heights=heights, n_streams=1)
        assert rel_l2(out[f], one[0]) <= 1e-5
