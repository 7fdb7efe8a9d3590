"""The potential energy's pass over unordered pairs (pp_potential.cu) against the FP64
oracle at its edges: one particle, either side of a block of 64, one and two blocks (the
antipodal block of an even ring), an odd ring, the change to blocks of 256 at 16384, and
zero-distance pairs inside a block and across blocks."""
import math

import numpy as np
import pytest

import oracle
from paper_2502_10640_gb300 import capi, workloads as wl

pytestmark = pytest.mark.gpu

R = 1e-6
# all terms are positive, so the sum's relative error is at most a term's: the FP32 sum of
# 256 terms, rsqrt.approx (2^-22.9) and the separation's rounding, 2 sqrt(3) 2^-24 |p| / eps
# with |p| <= 2 L0 and eps = 0.1 R >= 0.05 L0
TOL = 256 * 2.0 ** -24 + 2.0 ** -22 + 2 * math.sqrt(3) * 2.0 ** -24 * 2 / 0.05


@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 128, 129, 192, 1000, 16383, 16384, 16641])
@pytest.mark.parametrize("weighted", [False, True])
def test_potential_matches_oracle(n, weighted):
    pos = wl.uniform_sphere(n, R, seed=n)
    w = 3.0 * (0.5 + wl.uniform(17, 3, n)) if weighted else 3.0
    with capi.Simulation(n, 3.0, 1e-18, 0.1 * R) as sim:
        if weighted:
            sim.set_weights(w)
        sim.load(pos)
        pe = sim.diagnostics()["pe"]
    ref = oracle.potential_energy(pos, w, 0.1 * R)
    assert abs(pe - ref) <= TOL * abs(ref)


def test_zero_distance_pairs_add_nothing():
    n = 700
    pos = wl.uniform_sphere(n, R, seed=5)
    pos[40] = pos[3]       # inside a block
    pos[699] = pos[3]      # across blocks
    with capi.Simulation(n, 3.0, 1e-18, 0.0, positions=capi.PP_POS_SINGLE) as sim:
        sim.load(pos)
        pe = sim.diagnostics()["pe"]
    d = np.linalg.norm(pos[:, None] - pos[None], axis=2)
    inv = np.zeros_like(d)
    inv[d > 0] = 1.0 / d[d > 0]
    k = oracle.constants()["k"] * oracle.constants()["e"] ** 2
    # the separations' rounding, pair by pair
    err = 0.5 * k * 9.0 * float((inv * (258 * 2.0 ** -24 + 2.0 ** -22
                                        + 2 * math.sqrt(3) * 2.0 ** -24 * 2 * R * inv)).sum())
    assert abs(pe - 0.5 * k * 9.0 * float(inv.sum())) <= err
