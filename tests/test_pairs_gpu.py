"""FP64 type-3 slices in pairs of floats, against the direct sum and the FP64 path (the same plan with FFT radices
up to 8, which the pair kernels do not take).

A pair holds 47 bits and a slice takes some tens of dependent operations, so the pair path adds at most about 3e-13 of
relative L2 to the transform's own error, which both paths share (the polynomial kernel values are within the kernel's
truncation): its error is at most 1.2 times the FP64 path's plus 3e-13.
"""
import numpy as np
import pytest

from oracle.oracle import OracleProblem, oracle_vis, rel_l2
from paper_2506_02130_gb300 import fv, workloads as W

pytestmark = pytest.mark.gpu


def _run(prob, eps, transform="type3", scale=1.0, **kw):
    p = fv.Plan.from_problem(prob, precision=fv.FV_FP64, eps=eps, transform=transform, **kw)
    try:
        if prob.beams is not None:
            p.set_beams(prob.beams, prob.beam_of_ant)
        p.set_sky(prob.sky.ra, prob.sky.dec, prob.sky.flux.astype(np.float64) * scale)
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


def _check(prob, eps, **kw):
    exact = oracle_vis(OracleProblem.from_workload(prob), "factored")
    out, info = _run(prob, eps, **kw)
    ref, _ = _run(prob, eps, fft_max_radix=8, **kw)
    e, e0 = rel_l2(out, exact), rel_l2(ref, exact)
    print(f"w {info['kernel_width']} error {e:.3e} (FP64 path {e0:.3e})")
    assert e <= 1.2 * e0 + 3e-13
    return out, info


@pytest.mark.parametrize("polarised", [False, True])
@pytest.mark.parametrize("eps", [1e-2, 1e-4, 1e-6, 1e-7, 1e-8, 1e-9, 1e-10, 1e-11, 1e-12, 1e-13])
def test_kernel_widths(eps, polarised):
    _check(_prob(900, polarised), eps)


@pytest.mark.parametrize("n_src", [20, 63, 64, 65, 5000])
def test_source_counts(n_src):
    """Chunks of 64 candidates, whole and with a rest."""
    _check(_prob(n_src), 1e-11)


@pytest.mark.parametrize("z_sigma,heights", [(0.002, "terms"), (0.02, "terms"), (0.1, "terms"), (0.05, "grid"),
                                             (0.3, "grid")])
def test_planes(z_sigma, heights):
    """Height terms and up planes of every number the sums are compiled for."""
    _, info = _check(_prob(400, z_sigma=z_sigma), 1e-8, heights=heights)
    assert (info["height_terms"] > 0) == (heights == "terms")


def test_radius_and_bins():
    """A longer array (other FFT lengths), and bins unlike the tile."""
    _check(_prob(300, radius=7), 1e-9)
    _check(_prob(300, radius=2), 1e-9, bin_size=(33, 2))


@pytest.mark.parametrize("transform", ["type3", "lattice"])
@pytest.mark.parametrize("power", [-700, -120, 120, 700])
def test_strengths_beyond_a_floats_range(power, transform):
    """Fluxes scaled by powers of two scale the visibilities, also far outside a float's range."""
    prob = _prob(300)
    if transform == "lattice":
        prob.ant_enu = W.hex_array(3)
    prob.sky.flux[::3] *= 1e-9
    one, _ = _run(prob, 1e-9, transform=transform)
    out, _ = _run(prob, 1e-9, transform=transform, scale=2.0**power)
    assert rel_l2(out * 2.0**-power, one) <= 1e-12
