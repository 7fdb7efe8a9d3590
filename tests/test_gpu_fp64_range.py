"""All-FP64 pairs at the ends of the range of s = |d|^2 + eps^2: s = inf adds 0, and an
s whose power -3/2 overflows gives the infinite field that FP64 arithmetic has there."""
import numpy as np
import pytest

import oracle
from paper_2502_10640_gb300 import capi, workloads as wl

pytestmark = pytest.mark.gpu


def fields(pos, eps):
    with capi.Simulation(len(pos), 10.0, 1e-15, eps, acc=capi.PP_ACC_FP64_FULL) as sim:
        sim.load(pos)
        return sim.fields()


@pytest.mark.parametrize("n", [2, 33, 1500])
def test_infinite_softened_distance_adds_nothing(n):
    pos = wl.gaussian_bunch(n, 1e-5, seed=83)
    assert np.all(oracle.fields(pos, 10.0, 1e160) == 0.0)
    assert np.all(fields(pos, 1e160) == 0.0)


@pytest.mark.parametrize("gap", np.geomspace(1e-109, 1e-140, 16).tolist())
def test_overflowing_pair_term_is_infinite_with_its_sign(gap):
    p = np.round(wl.gaussian_bunch(49, 1e-5, seed=84) * 2.0 ** 50) / 2.0 ** 50
    pos = np.zeros((100, 3))
    pos[1:-1:2], pos[2:-1:2] = p, -p        # the centroid is exactly gap / 100
    pos[0] = gap, -gap, gap
    ref, got = oracle.fields(pos, 10.0, 0.0), fields(pos, 0.0)
    assert np.all(np.isinf(ref[[0, 99]]))
    assert np.array_equal(got[[0, 99]], ref[[0, 99]])
    assert np.isfinite(got[1:-1]).all()
