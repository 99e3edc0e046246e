"""Arrays that are short along one axis: FFT lengths from 32 points on, and the static scratch.

Mixed plans stay within the mixed path's 2e-5 of the direct sum.  FP64 plans (pairs of floats) are within 1.2 times the
error of the FP64 path (the same plan with FFT radices up to 8) plus 3e-13.  The static scratch runs the same kernels as
fv_execute: 3e-6 (mixed) and 1e-11 (FP64) for the order of the sources' sums.
"""
import math

import numpy as np
import pytest

from oracle.oracle import OracleProblem, oracle_vis, rel_l2
from paper_2506_02130_gb300 import fv, workloads as W

pytestmark = pytest.mark.gpu

NU = 200e6


def _prob(ant, polarised=False, n_src=2000, nu=NU):
    make = W.config_hex350_pol if polarised else W.config_hex127
    prob = make(seed=3, n_chan=1, n_time=1, n_point=n_src, nside=0, radius=1, **(dict(n_keep=None) if polarised else {}))
    prob.freqs_hz = np.array([nu])
    prob.ant_enu = ant
    prob.pairs = W.cross_pairs(len(ant))
    return prob


def _plan(prob, precision, eps, **kw):
    p = fv.Plan.from_problem(prob, precision=precision, eps=eps, transform="type3", **kw)
    p.set_sky(prob.sky.ra, prob.sky.dec, prob.sky.flux)
    return p


def _run(prob, precision, eps, **kw):
    p = _plan(prob, precision, eps, **kw)
    out, info = p.run(), p.info()
    p.close()
    return out, info


def _line(M, w, z_sigma):
    """An east-west line of 12 antennas whose north-south extent needs just under M / 2 grid cells."""
    rng = np.random.default_rng(M)
    half = (M / 2 - 1.5 - w) * math.pi / (4 * 2 * math.pi * NU / 299792458.0)
    ant = np.zeros((12, 3))
    ant[:, 0] = np.sort(rng.uniform(0, 150.0, 12))
    ant[:, 1] = rng.uniform(0, half, 12)
    ant[[3, 7], 1] = 0.0, half                     # baselines i < j: (3, 7) and its opposite below
    ant[[2, 9], 1] = half, 0.0
    ant[:, 2] = rng.normal(0.0, z_sigma, 12) if z_sigma else 0.0
    return ant


@pytest.mark.parametrize("polarised,z_sigma", [(False, 0.0), (True, 0.0), (False, 0.02), (True, 0.02)])
@pytest.mark.parametrize("M", [32, 48, 64, 80, 96, 128, 160, 192])
def test_short_lengths_mixed(M, polarised, z_sigma):
    prob = _prob(_line(M, 7, z_sigma), polarised)
    out, info = _run(prob, fv.FV_MIXED, 1e-6)
    assert info["nf2_max"][1] == M
    assert rel_l2(out, oracle_vis(OracleProblem.from_workload(prob), "factored")) <= 2e-5


@pytest.mark.parametrize("z_sigma", [0.0, 0.02])
@pytest.mark.parametrize("M", [32, 48, 64, 80, 96, 128, 160, 192])
def test_short_lengths_in_pairs(M, z_sigma):
    prob = _prob(_line(M, 11, z_sigma))
    exact = oracle_vis(OracleProblem.from_workload(prob), "factored")
    out, info = _run(prob, fv.FV_FP64, 1e-10)
    ref, _ = _run(prob, fv.FV_FP64, 1e-10, fft_max_radix=8)
    assert info["nf2_max"][1] == M
    assert rel_l2(out, exact) <= 1.2 * rel_l2(ref, exact) + 3e-13


def _east_west(z_sigma):
    rng = np.random.default_rng(5)
    ant = np.zeros((60, 3))
    ant[:, 0] = np.sort(rng.uniform(0, 760.0, 60))
    ant[:, 1] = rng.normal(0.0, 0.4, 60)
    ant[:, 2] = rng.normal(0.0, z_sigma, 60) if z_sigma else 0.0
    return ant


def _wall(L):
    """Antennas spread over L m east-west and L m in height."""
    rng = np.random.default_rng(1)
    ant = np.zeros((20, 3))
    ant[:, 0] = rng.uniform(0, L, 20)
    ant[:, 2] = rng.uniform(0, L, 20)
    ant[:2, 0] = 0, L
    ant[2:4, 2] = 0, L
    return ant


@pytest.mark.parametrize("ant,precision,polarised,eps,n_src,nu", [
    (_east_west(0.05), fv.FV_MIXED, True, 1e-6, 50000, NU), (_east_west(0.3), fv.FV_FP64, False, 1e-10, 50000, NU),
    (_wall(30.0), fv.FV_MIXED, True, 1e-6, 500, 150e6), (_wall(60.0), fv.FV_MIXED, True, 1e-6, 500, 150e6),
    (_wall(60.0), fv.FV_MIXED, False, 1e-7, 500, 150e6), (_wall(130.0), fv.FV_MIXED, False, 1e-7, 500, 150e6)])
def test_the_static_scratch_takes_what_the_general_form_fits(ant, precision, polarised, eps, n_src, nu):
    """Plans whose grid, bands and records at the general FFT lengths fit the static scratch: it takes them, whatever
    form their slices have (the last one only with the general lengths themselves)."""
    torch = pytest.importorskip("torch")
    prob = _prob(ant, polarised, n_src, nu)
    p = _plan(prob, precision, eps)
    ref = p.run()
    out = torch.zeros(ref.shape, dtype=torch.from_numpy(ref[:0]).dtype, device="cuda")
    fv.fv_execute_static(p.handle, out)
    torch.cuda.synchronize()
    assert rel_l2(out.cpu().numpy(), ref) <= (3e-6 if precision == fv.FV_MIXED else 1e-11)
    p.close()


def test_a_thin_array_holds_about_what_the_general_lengths_do():
    prob = _prob(_east_west(0.05), True, 50000)
    _, info = _run(prob, fv.FV_MIXED, 1e-6)
    _, general = _run(prob, fv.FV_MIXED, 1e-6, fft_max_radix=8)
    assert info["workspace_bytes"] <= 1.5 * general["workspace_bytes"]
