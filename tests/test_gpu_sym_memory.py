"""The partial sums of the pair-symmetric passes: at most a quarter of the free memory, the
one-sided kernels without it, the symmetric ones again once there is room."""
import numpy as np
import pytest

from paper_2502_10640_gb300 import capi, workloads as wl

pytestmark = pytest.mark.gpu
GB = 1 << 30


@pytest.fixture
def torch():
    return pytest.importorskip("torch")


def plan(sim):
    return capi.variants()[sim.get_option(capi.PP_OPT_VARIANT)]


def test_a_fine_split_falls_back_to_the_automatic_ranges(torch):
    """N = 2^21 cut into 64-source ranges would keep 109 GB of sums, the automatic plan 14."""
    n = 1 << 21
    before = torch.cuda.mem_get_info()[0]
    if before < 80 * GB or before > 400 * GB:
        pytest.skip("sized for a card with 80 to 400 GB free")
    pos = wl.uniform_sphere(n, 5e-5, seed=8)
    with capi.Simulation(n, 10.0, 1e-15, 1e-9, positions=capi.PP_POS_SINGLE) as sim:
        sim.set_option(capi.PP_OPT_SPLIT, 4096)
        sim.load(pos)
        fine = sim.fields()
        assert ".sym" in plan(sim)
        assert before - torch.cuda.mem_get_info()[0] < 30 * GB
        sim.set_option(capi.PP_OPT_SPLIT, 0)
        assert before - torch.cuda.mem_get_info()[0] < 10 * GB    # the sums are given back
        assert np.array_equal(sim.fields(), fine)


def test_little_free_memory_means_one_sided_until_there_is_more(torch):
    n = 131072   # 0.6 GB of sums
    pos = wl.uniform_sphere(n, 5e-5, seed=9)
    out = []
    with capi.Simulation(n, 10.0, 1e-15, 1e-9, positions=capi.PP_POS_SINGLE) as sim:
        hold = torch.empty(torch.cuda.mem_get_info()[0] - 2 * GB, dtype=torch.uint8, device="cuda")
        try:
            sim.load(pos)
            assert ".sym" not in plan(sim)
            assert torch.cuda.mem_get_info()[0] > 1.8 * GB        # left to whoever needs it
            sim.step(1)
            out.append(sim.fields())
        finally:
            del hold
            torch.cuda.empty_cache()
        sim.set_option(capi.PP_OPT_SPLIT, 0)
        out.append(sim.fields())
        assert ".sym" in plan(sim)
        sim.load(pos)
        assert ".sym" in plan(sim)
    scale = np.linalg.norm(out[0], axis=1).max()
    # the same staged positions, another summation order: 256 FP32 terms of a tile
    assert np.max(np.abs(out[0] - out[1])) <= 256 * 2.0 ** -24 * scale
