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


def _halves():
    """Two baseline lists of a hexagon of equal length: one baseline of every longest vector (along the lattice axes, east
    and north), and half of the other vectors, in different corners of the mode plane."""
    ant = W.hex_array(3)
    pairs = W.cross_pairs(len(ant))
    _, k, _ = fv.fv_lattice_detect(ant)
    n = k[pairs[:, 0]] - k[pairs[:, 1]]
    n[(n[:, 1] < 0) | ((n[:, 1] == 0) & (n[:, 0] < 0))] *= -1
    vec, first = np.unique(n, axis=0, return_index=True)
    enu = (ant[pairs[:, 0]] - ant[pairs[:, 1]])[first, :2]
    edge = (np.abs(vec) == np.abs(vec).max(axis=0)).any(axis=1)
    edge |= (np.isclose(enu, enu.max(axis=0)) | np.isclose(enu, enu.min(axis=0))).any(axis=1)
    ends, rest = first[edge], first[~edge]
    m = len(rest) // 2
    return ant, pairs[np.concatenate([ends, rest[:m]])], pairs[np.concatenate([ends, rest[-m:]])]


@pytest.mark.parametrize("precision,eps", [(fv.FV_MIXED, 1e-6), (fv.FV_FP64, 1e-9)])
def test_other_baselines_of_the_same_lattice(precision, eps):
    """Baseline lists of equal length and extent with other modes."""
    prob = W.config_hex127(seed=7, n_chan=2, n_time=1, n_point=2000, nside=0, radius=3)
    ant, a, b = _halves()
    sky = (prob.sky.ra, prob.sky.dec, prob.sky.flux)
    p = _plan(prob, precision, eps)
    p.set_array(ant, a)
    p.set_sky(*sky)
    infos = []
    for pairs in (a, b, a):
        p.set_array(ant, pairs)
        ref, info = _fresh(prob, precision, eps, ant, pairs, sky)
        infos.append((info["n_bl"], info["n_unique"], info["lattice_modes"]))
        assert info["transform"] == "lattice"
        _same(p.run(), ref, precision)
    assert infos[0] == infos[1]
    p.close()


@pytest.mark.parametrize("precision,eps", [(fv.FV_MIXED, 1e-6), (fv.FV_FP64, 1e-9), (fv.FV_FP64, 1e-13)])
def test_other_heights_on_the_same_lattice(precision, eps):
    """The same lattice and number of height terms with other heights (direct sums, and the grid at 1e-13)."""
    prob = W.config_hex127(seed=8, n_chan=2, n_time=1, n_point=2000, nside=0, radius=3)
    rng = np.random.default_rng(9)
    one = W.hex_array(3)
    one[:, 2] = rng.normal(0.0, 0.05, len(one))
    two = one.copy()
    two[:, 2] = -one[::-1, 2]                       # the same largest difference
    sky = (prob.sky.ra, prob.sky.dec, prob.sky.flux)
    p = _plan(prob, precision, eps)
    p.set_array(one)
    p.set_sky(*sky)
    for ant in (one, two):
        p.set_array(ant)
        ref, info = _fresh(prob, precision, eps, ant, None, sky)
        assert info["transform"] == "lattice" and info["lattice_terms"] > 1
        _same(p.run(), ref, precision)
    p.close()
