"""Direct mode sums of lattice arrays (no grid) against the oracle and the type-3 route: tile edges of the modes, one
and several blocks of height terms, four products, beams by pair, chunks of sources and of channels.

Tolerances: the mixed path's 2e-5 and FP64's 1e-9 relative L2 against the direct sum; pairs of floats hold about 2^-47
per operation, so an FP64 plan's sums are within 1e-12 of the oracle's, whatever eps (from 1e-12 up) asks for.
"""
import numpy as np
import pytest

from oracle.oracle import OracleProblem, oracle_vis, rel_l2
from paper_2506_02130_gb300 import fv, workloads as W

pytestmark = pytest.mark.gpu


def _run(prob, precision, eps, **kw):
    p = fv.Plan.from_problem(prob, precision=precision, eps=eps, transform="lattice", **kw)
    try:
        if prob.beams is not None:
            p.set_beams(prob.beams, prob.beam_of_ant)
        p.set_sky(prob.sky.ra, prob.sky.dec, prob.sky.flux)
        return p.run(), p.info()
    finally:
        p.close()


@pytest.mark.parametrize("precision,eps,tol", [(fv.FV_FP64, 1e-7, 1e-12), (fv.FV_FP64, 1e-12, 1e-12),
                                               (fv.FV_FP64, 1e-13, 1e-9), (fv.FV_MIXED, 1e-6, 2e-6)])
@pytest.mark.parametrize("radius,n_src", [(1, 1), (1, 40), (2, 500), (3, 33), (4, 700), (7, 300)])
def test_flat_lattices(radius, n_src, precision, eps, tol):
    prob = W.config_hex127(seed=radius, n_chan=3, n_time=2, n_point=max(n_src, 20), nside=0, radius=radius)
    prob.ant_enu = W.hex_array(radius)
    prob.pairs = W.cross_pairs(len(prob.ant_enu))
    out, info = _run(prob, precision, eps)
    assert info["lattice_terms"] == 1
    assert rel_l2(out, oracle_vis(OracleProblem.from_workload(prob), "factored")) <= tol


@pytest.mark.parametrize("precision,eps,tol", [(fv.FV_FP64, 1e-11, 1e-9), (fv.FV_MIXED, 1e-6, 2e-5)])
@pytest.mark.parametrize("z_sigma,polarised", [(0.002, False), (0.05, False), (0.4, False), (0.0, True), (0.03, True)])
def test_terms_and_products(z_sigma, polarised, precision, eps, tol):
    make = W.config_hex350_pol if polarised else W.config_hex127
    kw = dict(n_keep=None) if polarised else {}
    prob = make(seed=5, n_chan=2, n_time=2, n_point=400, nside=4, radius=3, **kw)
    prob.ant_enu = W.hex_array(3)
    if z_sigma:
        prob.ant_enu[:, 2] = np.random.default_rng(6).normal(0.0, z_sigma, len(prob.ant_enu))
    out, info = _run(prob, precision, eps)
    assert (info["lattice_terms"] > 1) == (z_sigma > 0)
    assert rel_l2(out, oracle_vis(OracleProblem.from_workload(prob), "factored")) <= tol


@pytest.mark.parametrize("precision,eps,tol", [(fv.FV_FP64, 1e-11, 1e-9), (fv.FV_MIXED, 1e-6, 2e-5)])
def test_lines_and_pairs_in_both_directions(precision, eps, tol):
    """A line of antennas (no second lattice direction), and pairs (j, i) beside (i, j)."""
    prob = W.config_hex127(seed=9, n_chan=2, n_time=1, n_point=300, nside=0, radius=1)
    prob.ant_enu = np.array([[14.6 * k, 0.0, 0.0] for k in (0, 1, 3, 7, 12, 20)])
    i, j = np.meshgrid(np.arange(6), np.arange(6), indexing="ij")
    prob.pairs = np.stack([i.ravel(), j.ravel()], axis=1).astype(np.int32)
    out, _ = _run(prob, precision, eps)
    assert rel_l2(out, oracle_vis(OracleProblem.from_workload(prob), "factored")) <= tol


def test_many_channels_and_windows_of_a_batch():
    """More channels than one launch takes, and a window of channels and times of a batch."""
    torch = pytest.importorskip("torch")
    prob = W.config_hex127(seed=11, n_chan=150, n_time=2, n_point=60, nside=0, radius=2)
    prob.ant_enu = W.hex_array(2)
    prob.pairs = W.cross_pairs(len(prob.ant_enu))
    ref = oracle_vis(OracleProblem.from_workload(prob), "factored")
    p = fv.Plan.from_problem(prob, precision=fv.FV_MIXED, eps=1e-6, transform="lattice")
    p.set_sky(prob.sky.ra, prob.sky.dec, prob.sky.flux)
    assert rel_l2(p.run(), ref) <= 2e-6
    out = torch.zeros((90, 1) + ref.shape[2:], dtype=torch.complex64, device="cuda")
    b = fv.Batch()
    b.add(p, out, (1, 2), (40, 130), window=(40, 1, 1))
    b.execute()
    torch.cuda.synchronize()
    assert rel_l2(out.cpu().numpy(), ref[40:130, 1:2]) <= 2e-6
    b.close()
    p.close()


@pytest.mark.parametrize("precision,eps,tol", [(fv.FV_FP64, 1e-11, 1e-9), (fv.FV_MIXED, 1e-6, 2e-5)])
def test_lattices_too_large_for_direct_sums_keep_the_grid(precision, eps, tol):
    prob = W.config_hex127(seed=12, n_chan=2, n_time=1, n_point=200, nside=0, radius=1)
    prob.ant_enu = np.array([[0.5 * k, 0.0, 0.0] for k in (0, 1, 3, 850)])      # 1,701 modes along the line
    prob.pairs = W.cross_pairs(4)
    out, info = _run(prob, precision, eps)
    assert info["lattice_modes"][0] == 1701
    assert rel_l2(out, oracle_vis(OracleProblem.from_workload(prob), "factored")) <= tol
