"""Skies whose sources meet in one bin of the per-time sort: whole warps, parts of warps and scattered sources of it,
against the direct sum (mixed path: 2e-5)."""
import numpy as np
import pytest

from oracle.oracle import OracleProblem, oracle_vis, rel_l2
from paper_2506_02130_gb300 import fv, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("polarised", [False, True])
@pytest.mark.parametrize("n_src,every", [(3, 1), (33, 1), (20000, 1), (20000, 2), (20000, 7), (20000, 15)])
def test_sources_of_one_bin(n_src, every, polarised):
    """Every `every`-th source of a sky in a field far smaller than a bin."""
    make = W.config_hex350_pol if polarised else W.config_hex127
    prob = make(seed=2, n_chan=2, n_time=2, n_point=max(n_src, 20), nside=0, radius=2,
                **(dict(n_keep=None) if polarised else {}))
    prob.ant_enu = W.hex_array(2)
    prob.ant_enu[:, :2] += np.random.default_rng(3).normal(0.0, 0.3, (len(prob.ant_enu), 2))
    prob.pairs = W.cross_pairs(len(prob.ant_enu))
    sky = prob.sky
    sky.ra, sky.dec, sky.flux = sky.ra[:n_src].copy(), sky.dec[:n_src].copy(), sky.flux[:, :n_src].copy()
    k = slice(None, None, every)
    rng = np.random.default_rng(4)
    sky.ra[k] = prob.lsts_rad[0] + 0.1 + rng.normal(0.0, 1e-5, len(sky.ra[k]))
    sky.dec[k] = prob.latitude_rad + 0.2 + rng.normal(0.0, 1e-5, len(sky.ra[k]))
    p = fv.Plan.from_problem(prob, precision=fv.FV_MIXED, eps=1e-6, transform="type3")
    p.set_sky(sky.ra, sky.dec, sky.flux)
    assert p.info()["spread"] == "gather"
    assert rel_l2(p.run(), oracle_vis(OracleProblem.from_workload(prob), "factored")) <= 2e-5
    p.close()
