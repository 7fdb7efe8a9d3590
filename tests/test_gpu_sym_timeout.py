"""The bounded wait of the pair-symmetric kernels: a completion that never comes makes it run
out after the limit set, the call returns PP_ERR_TIMEOUT, and the context works again, bitwise
as before (the queue words are zero), after a reload."""
import time

import numpy as np
import pytest

from paper_2502_10640_gb300 import capi, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,acc,mode", [
    (16385, capi.PP_ACC_FP64FOLD, capi.PP_POS_SINGLE),
    (30001, capi.PP_ACC_KAHAN, capi.PP_POS_SINGLE),
    (40001, capi.PP_ACC_FP64FOLD, capi.PP_POS_GUARDED),
    (40, capi.PP_ACC_FP64_FULL, capi.PP_POS_SINGLE),
    (5001, capi.PP_ACC_FP64_FULL, capi.PP_POS_SINGLE)])
def test_symmetric_wait_runs_out_and_the_context_recovers(n, acc, mode):
    pos = wl.uniform_sphere(n, 1e-5, seed=n)
    with capi.Simulation(n, 1.0, 1e-15, 1e-9, acc=acc, positions=mode) as sim:
        sim.set_option(capi.PP_OPT_TIMEOUT_NS, 20_000_000)
        sim.load(pos)
        assert ".sym" in capi.variants()[sim.get_option(capi.PP_OPT_VARIANT)]
        before = sim.fields()
        for _ in range(2):
            sim.set_option(capi.PP_OPT_TEST_SKIP_COPY, 1)
            t0 = time.perf_counter()
            with pytest.raises(capi.PPError) as e:
                sim.step(1)
            # the pass itself takes milliseconds; the minimum of an ordinary pass is 1 s
            assert 0.02 <= time.perf_counter() - t0 < 0.9
            assert e.value.status == capi.PP_ERR_TIMEOUT
            with pytest.raises(capi.PPError) as e:
                sim.step(1)
            assert e.value.status == capi.PP_ERR_STATE
            sim.load(pos)
            assert np.array_equal(sim.fields(), before)
        # a limit far below the length of an item is no limit for an ordinary pass
        sim.set_option(capi.PP_OPT_TIMEOUT_NS, 100_000)
        sim.step(3)
