"""Large lattices at a loose tolerance: the direct sums up to 50,000 sources, the grid for larger skies, seen by their
errors against the direct sum: the sums' own rounding (2e-6 in FP32, 1e-11 in pairs), or the grid's (up to ten times eps,
and far above the sums')."""
import numpy as np
import pytest

from oracle.oracle import OracleProblem, oracle_vis, rel_l2
from paper_2506_02130_gb300 import fv, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,eps,sums", [(fv.FV_MIXED, 1e-3, 2e-6), (fv.FV_FP64, 1e-3, 1e-11)])
@pytest.mark.parametrize("radius,n_src,direct", [(13, 50000, True), (13, 50001, False), (4, 60000, True)])
def test_grid_or_direct_sums(radius, n_src, direct, precision, eps, sums):
    prob = W.config_hex127(seed=6, n_chan=1, n_time=1, n_point=n_src, nside=0, radius=1)
    prob.ant_enu = W.hex_array(radius)
    pairs = W.cross_pairs(len(prob.ant_enu))
    prob.pairs = pairs[np.random.default_rng(7).permutation(len(pairs))[:3000]]
    p = fv.Plan.from_problem(prob, precision=precision, eps=eps, transform="lattice")
    sky = prob.sky
    flux = sky.flux * np.random.default_rng(8).choice([-1.0, 1.0], n_src)[None, :, None]
    sky.flux = flux
    p.set_sky(sky.ra, sky.dec, flux)
    e = rel_l2(p.run(), oracle_vis(OracleProblem.from_workload(prob), "factored"))
    p.close()
    print(f"error {e:.3e}")
    assert e <= sums if direct else 10 * sums < e <= 10 * eps
