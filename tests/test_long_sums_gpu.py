"""FP64 plans whose sums in pairs of floats take tens of thousands of terms: many sources on few cells or modes.

A pair sum whose low part is not kept below the high part's rounding loses accuracy in proportion to its length (4.6e-12
of the sum after 20,000 terms).  The direct sums go to FP64 after 256 sources: 7e-14 a chain, which adds up as the sums
do, and a few 2^-47 each for phases and strengths, so 4e-13 in all.  The type-3 spreading's cells are tidied as they
grow: the pair path stays within 1.2 times the FP64 path's error plus 3e-13, as for small skies.
"""
import dataclasses

import numpy as np
import pytest

from oracle.oracle import OracleProblem, oracle_vis, rel_l2
from paper_2506_02130_gb300 import fv, workloads as W

pytestmark = pytest.mark.gpu


def _run(prob, eps, **kw):
    p = fv.Plan.from_problem(prob, precision=fv.FV_FP64, eps=eps, **kw)
    try:
        p.set_sky(prob.sky.ra, prob.sky.dec, prob.sky.flux)
        return p.run()
    finally:
        p.close()


def _small_array(seed, n_src, z_sigma):
    prob = W.config_hex127(seed=seed, n_chan=1, n_time=1, n_point=n_src, nside=0, radius=1)
    rng = np.random.default_rng(seed)
    prob.ant_enu = W.hex_array(1)
    prob.ant_enu[:, :2] += rng.normal(0.0, 0.4, (7, 2))
    prob.ant_enu[:, 2] = rng.normal(0.0, z_sigma, 7) if z_sigma else 0.0
    return prob


@pytest.mark.parametrize("height", [0.0, 0.05])
def test_direct_sums_of_many_sources(height):
    """Fluxes of both signs through a flat beam (sums that grow as a random walk), 64 channels a launch, so that a channel
    gets few CTAs."""
    prob = W.config_hex127(seed=3, n_chan=64, n_time=1, n_point=300000, nside=0, radius=6)
    prob.beam, prob.beam_param = "uniform", ()
    prob.ant_enu[:, 2] = np.random.default_rng(4).normal(0.0, height, len(prob.ant_enu)) if height else 0.0
    prob.sky.flux *= np.random.default_rng(5).choice([-1.0, 1.0], prob.sky.flux.shape[1])[None, :, None]
    out = _run(prob, 1e-12, transform="lattice")
    one = dataclasses.replace(prob, freqs_hz=prob.freqs_hz[:1],
                              sky=dataclasses.replace(prob.sky, flux=prob.sky.flux[:, :, :1]))
    e = rel_l2(out[:1], oracle_vis(OracleProblem.from_workload(one), "factored"))
    print(f"error {e:.3e}")
    assert e <= 4e-13


@pytest.mark.parametrize("z_sigma", [0.0, 0.05])
@pytest.mark.parametrize("seed", [1, 2])
def test_type3_cells_of_many_sources(seed, z_sigma):
    """1.5 million visible sources on a grid of about 9,000 cells: some 25,000 terms a cell."""
    prob = _small_array(seed, 3000000, z_sigma)
    exact = oracle_vis(OracleProblem.from_workload(prob), "factored")
    e = rel_l2(_run(prob, 1e-11, transform="type3"), exact)
    e0 = rel_l2(_run(prob, 1e-11, transform="type3", fft_max_radix=8), exact)
    print(f"error {e:.3e} (FP64 path {e0:.3e})")
    assert e <= 1.2 * e0 + 3e-13


@pytest.mark.parametrize("z_sigma", [0.0, 0.05])
@pytest.mark.parametrize("seed,n_src", [(1, 300000), (1, 1500000), (2, 1500000)])
def test_long_sums_with_the_widest_pair_kernel_stay_in_fp64(seed, n_src, z_sigma):
    """At eps 1e-12 the kernel's own error leaves no room for the pairs' rounding in sums of thousands of terms."""
    prob = _small_array(seed, n_src, z_sigma)
    exact = oracle_vis(OracleProblem.from_workload(prob), "factored")
    e = rel_l2(_run(prob, 1e-12, transform="type3"), exact)
    e0 = rel_l2(_run(prob, 1e-12, transform="type3", fft_max_radix=8), exact)
    print(f"error {e:.3e} (FP64 path {e0:.3e})")
    assert e <= 1.02 * e0
