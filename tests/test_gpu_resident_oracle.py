"""The resident kernel with two targets per thread (N >= 5000) against the oracle, each
particle inside its own a-priori bound: one far source lost from a sum would show."""
import numpy as np
import pytest

import oracle
from tests._bounds import field_error_bound
from tests.test_gpu_pair_symmetric import K_E
from paper_2502_10640_gb300 import capi, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,mode,weighted", [
    (5000, capi.PP_POS_SINGLE, False), (5001, capi.PP_POS_SINGLE, False),
    (7777, capi.PP_POS_SINGLE, True), (12288, capi.PP_POS_SINGLE, False),
    (5001, capi.PP_POS_SPLIT, False), (6144, capi.PP_POS_SPLIT, False)])
def test_two_targets_per_thread_match_the_oracle(n, mode, weighted):
    pos = wl.uniform_sphere(n, 3e-6, seed=n)
    w, eps = 2.0, 1e-8
    wts = w * (0.5 + wl.uniform(99, 3, n))
    with capi.Simulation(n, w, 1e-16, eps, positions=mode) as sim:
        sim.set_option(capi.PP_OPT_RESIDENT, capi.PP_RESIDENT_ON)
        if weighted:
            sim.set_weights(wts)
        sim.load(pos)
        assert sim.get_option(capi.PP_OPT_RESIDENT_ACTIVE) == 1
        sim.step(2)
        p, v, a = sim.state()[:3]
    c = oracle.constants()
    idx = np.unique(np.r_[0:4, np.arange(0, n, 13), n - 4:n])
    ref = oracle.fields_subset(p, wts if weighted else w, eps, idx)
    got = a[idx] * (c["me"] / -c["e"])
    bound = field_error_bound(p, w, eps, idx, K_E, tile=512, split=mode == capi.PP_POS_SPLIT)
    err = np.linalg.norm(got - ref, axis=1)
    assert np.all(err <= (1.5 if weighted else 1.0) * bound)
