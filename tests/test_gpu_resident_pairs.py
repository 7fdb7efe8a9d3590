"""The resident kernel with two targets per thread (N >= 5000) at its edges: either side of
the change, an odd tail, the largest N of each form; against the per-launch kernels, which
sum in another order (both within FP32 summation error of the same staged positions)."""
import numpy as np
import pytest

from paper_2502_10640_gb300 import capi, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,mode,weighted", [
    (4999, capi.PP_POS_SINGLE, False), (5000, capi.PP_POS_SINGLE, False),
    (5001, capi.PP_POS_SINGLE, False), (7777, capi.PP_POS_SINGLE, True),
    (12288, capi.PP_POS_SINGLE, False), (5001, capi.PP_POS_SPLIT, False),
    (6144, capi.PP_POS_SPLIT, False)])
def test_two_targets_per_thread_match_the_per_launch_kernels(n, mode, weighted):
    pos = wl.gaussian_bunch(n, 3e-6, seed=n)
    w = 2.0 * (0.5 + wl.uniform(95, 3, n))
    out = []
    for resident in (capi.PP_RESIDENT_ON, capi.PP_RESIDENT_OFF):
        with capi.Simulation(n, 2.0, 1e-16, 1e-8, positions=mode) as sim:
            sim.set_option(capi.PP_OPT_RESIDENT, resident)
            if weighted:
                sim.set_weights(w)
            sim.load(pos)
            assert sim.get_option(capi.PP_OPT_RESIDENT_ACTIVE) == int(resident != capi.PP_RESIDENT_OFF)
            sim.step(3)
            out.append(sim.state()[:3])
    # a target's sum of one-signed partial sums of at most 512 FP32 terms each, plus the
    # rounding of a pair term, relative to the largest acceleration
    tol = (512 + 16) * 2.0 ** -24
    for a, b in zip(*out):
        assert np.max(np.abs(a - b)) <= tol * np.max(np.linalg.norm(b, axis=1))
