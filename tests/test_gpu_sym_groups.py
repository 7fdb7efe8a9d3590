"""Pair-symmetric passes with several target blocks to a group (N > 128 blocks), where the
sums of the sources are added onto a row that another block has started: every form of the
kernels against the oracle on sampled targets, odd N."""
import numpy as np
import pytest

import oracle
from tests._bounds import field_error_bound
from tests.test_gpu_pair_symmetric import K_E, run, sym_variants
from paper_2502_10640_gb300 import capi, workloads as wl

pytestmark = pytest.mark.gpu


def sample(n):
    """Targets spread over the blocks, the first and the last ones among them."""
    return np.unique(np.r_[0:3, np.arange(5, n, n // 97), n - 3:n])


@pytest.mark.parametrize("n", [70001, 98305])
def test_every_form_with_several_blocks_to_a_group(n):
    pos = wl.uniform_sphere(n, 2e-5, seed=n)
    pos[n - 2] = pos[7]                # a coincident pair across groups: hi/lo where guarded
    eps = 2e-9
    wts = 10.0 * (0.5 + wl.uniform(97, 3, n))
    idx = sample(n)
    ref = oracle.fields_subset(pos, 10.0, eps, idx)
    ref_w = oracle.fields_subset(pos, wts, eps, idx)
    bound = field_error_bound(pos, 10.0, eps, idx, K_E, tile=512)
    for name in sym_variants():
        E, weighted, _ = run(name, pos, eps, wts)
        err = np.linalg.norm(E[idx] - (ref_w if weighted else ref), axis=1)
        assert np.all(err <= (1.5 if weighted else 1.0) * bound), name


@pytest.mark.parametrize("n", [4097, 8193, 20481])
@pytest.mark.parametrize("weighted", [False, True])
def test_fp64_with_several_blocks_to_a_group(n, weighted):
    """FP64 level: n u on the sum of the terms' sizes and a few u on each term (u = 2^-53),
    close pairs by the rounding of their scaled positions; weights as float32 ratios."""
    pos = wl.gaussian_bunch(n, 1e-6, seed=n)
    eps = 1e-8
    wts = 10.0 * (0.5 + wl.uniform(98, 3, n)).astype(np.float32).astype(np.float64)
    idx = sample(n)
    with capi.Simulation(n, 10.0, 1e-15, eps, acc=capi.PP_ACC_FP64_FULL) as sim:
        if weighted:
            sim.set_weights(wts)
        sim.load(pos)
        E = sim.fields()
    w = wts if weighted else np.full(n, 10.0)
    ref = oracle.fields_subset(pos, w, eps, idx)
    d = pos[idx, None, :] - pos[None, :, :]
    d2 = np.einsum("ijk,ijk->ij", d, d)
    mag = np.sqrt(d2) / (d2 + eps * eps) ** 1.5
    far = np.abs(pos).max()
    ratio = np.where(d2 > 0, far / np.sqrt(np.maximum(d2, 1e-300)), 0.0)
    rel = (n + 40) * 2.0 ** -53 + (2.0 ** -24 if weighted else 0.0)
    bound = K_E * ((mag * (rel + 32 * 2.0 ** -53 * ratio)) @ w)
    assert np.all(np.linalg.norm(E[idx] - ref, axis=1) <= bound)
