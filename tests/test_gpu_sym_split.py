"""PP_OPT_SPLIT on the pair-symmetric default plan only shortens the ranges of a row: small
values change nothing, large ones the FP64 grouping of the partial sums."""
import numpy as np
import pytest

from paper_2502_10640_gb300 import capi, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,acc", [(262145, capi.PP_ACC_FP64FOLD), (20001, capi.PP_ACC_KAHAN),
                                   (9001, capi.PP_ACC_FP64_FULL)])
def test_split_only_shortens_the_ranges(n, acc):
    pos = wl.uniform_sphere(n, 5e-5, seed=n)
    out = []
    with capi.Simulation(n, 10.0, 1e-15, 1e-9, acc=acc, positions=capi.PP_POS_SINGLE) as sim:
        sim.load(pos)
        assert ".sym" in capi.variants()[sim.get_option(capi.PP_OPT_VARIANT)]
        for split in (0, 1, 2, 64):
            sim.set_option(capi.PP_OPT_SPLIT, split)
            out.append(sim.fields())
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2])
    assert np.max(np.abs(out[3] - out[0])) <= 1e-13 * np.linalg.norm(out[0], axis=1).max()
