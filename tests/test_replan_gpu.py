"""One plan whose sky or array changes the route of its slices, against a fresh plan of the same inputs.

Both plans run the same kernels on the same inputs; only the order of the sources' sums differs (atomics), so they
agree to a few roundings: 3e-6 relative L2 in mixed precision, 1e-11 in FP64 (pairs of floats, chains of a few hundred
terms).
"""
import numpy as np
import pytest

from paper_2506_02130_gb300 import fv, workloads as W

pytestmark = pytest.mark.gpu

TOL = {fv.FV_MIXED: 3e-6, fv.FV_FP64: 1e-11}


def _plan(prob, precision, eps):
    return fv.Plan.create(prob.freqs_hz, prob.lsts_rad, prob.latitude_rad, prob.beam, prob.beam_param, precision, eps,
                          prob.polarized)


def _fresh(prob, precision, eps, ant, pairs, sky):
    p = _plan(prob, precision, eps)
    p.set_array(ant, pairs)
    p.set_sky(*sky)
    out, info = p.run(), p.info()
    p.close()
    return out, info


def _same(out, ref, precision):
    assert np.linalg.norm(ref) > 0
    assert np.linalg.norm(out - ref) <= TOL[precision] * np.linalg.norm(ref)


@pytest.mark.parametrize("precision,eps", [(fv.FV_MIXED, 1e-6), (fv.FV_MIXED, 1e-7), (fv.FV_FP64, 1e-9),
                                           (fv.FV_FP64, 1e-13)])
def test_a_larger_sky_moves_a_polarised_lattice_to_type3(precision, eps):
    """1,000 sources go by the lattice, 40,000 by the type-3 route, and back; the batch's lanes as well."""
    torch = pytest.importorskip("torch")
    prob = W.config_hex350_pol(seed=4, n_chan=2, n_time=1, n_point=40000, nside=0, radius=3, n_keep=None)
    ant = W.hex_array(3)
    sky = (prob.sky.ra, prob.sky.dec, prob.sky.flux)
    small = (prob.sky.ra[:1000], prob.sky.dec[:1000], np.ascontiguousarray(prob.sky.flux[:, :1000]))
    p = _plan(prob, precision, eps)
    p.set_array(ant)
    batch = fv.Batch()
    for s, lattice in ((small, True), (sky, False), (small, True)):
        p.set_sky(*s)
        ref, _ = _fresh(prob, precision, eps, ant, None, s)
        assert (p.info()["transform"] == "lattice") == lattice
        _same(p.run(), ref, precision)
        out = torch.zeros(ref.shape, dtype=torch.from_numpy(ref[:0]).dtype, device="cuda")
        batch.clear()
        batch.add(p, out)
        batch.execute()
        torch.cuda.synchronize()
        _same(out.cpu().numpy(), ref, precision)
    batch.close()
    p.close()


@pytest.mark.parametrize("precision,eps", [(fv.FV_MIXED, 1e-6), (fv.FV_MIXED, 1e-7), (fv.FV_FP64, 1e-9),
                                           (fv.FV_FP64, 1e-13)])
@pytest.mark.parametrize("height", [0.0, 0.05])
def test_an_array_that_is_no_lattice_replaces_one(height, precision, eps):
    prob = W.config_hex127(seed=5, n_chan=2, n_time=1, n_point=3000, nside=0, radius=3)
    rng = np.random.default_rng(6)
    lattice = W.hex_array(3)
    lattice[:, 2] = rng.normal(0.0, height, len(lattice)) if height else 0.0
    moved = lattice.copy()
    moved[:, :2] += rng.normal(0.0, 0.3, (len(moved), 2))
    sky = (prob.sky.ra, prob.sky.dec, prob.sky.flux)
    p = _plan(prob, precision, eps)
    p.set_array(lattice)
    p.set_sky(*sky)
    for ant in (lattice, moved, lattice):
        p.set_array(ant)
        ref, info = _fresh(prob, precision, eps, ant, None, sky)
        assert p.info()["transform"] == info["transform"] == ("type3" if ant is moved else "lattice")
        _same(p.run(), ref, precision)
    p.close()
