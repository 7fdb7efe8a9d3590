"""Pair-symmetric tiles whose two halves of packs take different forms: a zero-distance
pair in the first or in the second half of a warp's targets sends that half through the
slow form while the other runs fast, both adding to the same sums of the sources."""
import numpy as np
import pytest

import oracle
from tests._bounds import field_error_bound
from tests.test_gpu_pair_symmetric import K_E, run, sym_variants
from paper_2502_10640_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def test_slow_and_fast_halves_of_a_tile_share_the_source_sums():
    n = 3000
    pos = wl.gaussian_bunch(n, 1e-6, seed=71)
    pos[2600] = pos[5]      # first half of the packs of the first block
    pos[2900] = pos[300]    # second half of 8 packs, a later block with 4
    pos[1700] = pos[700]    # second half of the second block of 8 packs
    wts = 10.0 * (0.5 + wl.uniform(96, 3, n))
    ref, ref_w = oracle.fields(pos, 10.0, 0.0), oracle.fields(pos, wts, 0.0)
    bound = field_error_bound(pos, 10.0, 0.0, np.arange(n), K_E)
    for name in sym_variants():
        E, weighted, _ = run(name, pos, 0.0, wts, lambda s: [s.fields() for _ in range(4)])
        err = np.linalg.norm(E[0] - (ref_w if weighted else ref), axis=1)
        assert np.all(err <= (1.5 if weighted else 1.0) * bound), name
        assert all(np.array_equal(E[0], e) for e in E[1:]), name
