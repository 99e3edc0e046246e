"""fv_set_sky checks the coordinates on the device, before it touches the sky that the plan holds."""
import numpy as np
import pytest

from paper_2506_02130_gb300 import fv, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_streams", [1, 4])
@pytest.mark.parametrize("where", ["ra", "dec"])
@pytest.mark.parametrize("at", [0, 256, -1])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_a_bad_coordinate_is_refused_and_leaves_the_sky(value, at, where, n_streams):
    prob = W.config_small(seed=5, n_src=700)
    p = fv.Plan.from_problem(prob, precision=fv.FV_FP64, eps=1e-9, n_streams=n_streams)
    p.set_sky(prob.sky.ra, prob.sky.dec, prob.sky.flux)
    before = p.run()
    ra, dec = prob.sky.ra[:600].copy(), prob.sky.dec[:600].copy()
    (ra if where == "ra" else dec)[at] = value
    with pytest.raises(fv.FvError) as e:
        p.set_sky(ra, dec, np.ascontiguousarray(2 * prob.sky.flux[:, :600]))
    assert e.value.status == fv.FV_ERR_ARG and "non-finite" in str(e.value)
    after = p.run()
    assert np.linalg.norm(after - before) <= 1e-12 * np.linalg.norm(before)
    p.close()
