"""pp_fields_noalloc at the edges of its kernels: blocks of 64 and 256 targets, one and
several blocks in the reductions of the staging frame, refused input."""
import numpy as np
import pytest

import oracle
from tests._bounds import field_error_bound
from tests.test_zz_no_alloc import K_E, noalloc, torch  # noqa: F401 (fixture)
from paper_2502_10640_gb300 import capi, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 64, 65, 257, 4096, 4097])
def test_noalloc_at_the_edges_of_its_blocks(torch, n):
    pos = wl.uniform_sphere(n, 5e-6, seed=61 + n) + 3e-6
    got = noalloc(torch, pos, 10.0, 1e-8)
    if n == 1:
        assert np.all(got == 0.0)
        return
    bound = field_error_bound(pos, 10.0, 1e-8, np.arange(n), K_E, split=True)
    assert np.all(np.linalg.norm(got - oracle.fields(pos, 10.0, 1e-8), axis=1) <= bound)


def test_noalloc_refuses_non_finite_input_and_leaves_the_output(torch):
    pos_d = torch.zeros((70, 3), device="cuda", dtype=torch.float64)
    pos_d[69, 1] = float("inf")
    out_d = torch.full((70, 3), 7.0, device="cuda", dtype=torch.float64)
    with pytest.raises(capi.PPError) as e:
        capi.pp_fields_noalloc(70, 1.0, 0.0, pos_d, out_d)
    assert e.value.status == capi.PP_ERR_ARG
    assert bool((out_d == 7.0).all())
