"""How many FP32 terms a partial sum takes before it is folded, seen from the outside: a
target far from thousands of coincident (softened) sources adds equal terms t, t, ..., whose
rounding errors do not average out but grow with the length of the chain.  The error expected
of chains of 64 and of 128 terms is computed here by adding floats; the default kernels of
these sizes have to stay on the 64-term side."""
import numpy as np
import pytest

import oracle
from paper_2502_10640_gb300 import capi, workloads as wl

pytestmark = pytest.mark.gpu

U32 = 2.0 ** -24
FOLD, KAHAN = capi.PP_ACC_FP64FOLD, capi.PP_ACC_KAHAN
SINGLE, GUARDED = capi.PP_POS_SINGLE, capi.PP_POS_GUARDED


def chain_rms(length):
    """RMS relative error of `length` equal FP32 terms added one after the other."""
    t = (0.5 + 1.5 * wl.uniform(17, 1, 4096)).astype(np.float32)
    s = np.zeros_like(t)
    for _ in range(length):
        s = s + t
    exact = length * t.astype(np.float64)
    return float(np.sqrt(np.mean(((s - exact) / exact) ** 2)))


# the pair terms add about 3 u of their own (staging, reciprocal root); half way between the
# two lengths on a logarithmic scale leaves room for that
LIMIT = float(np.sqrt(chain_rms(64) * chain_rms(128)))


def test_the_model_separates_the_lengths():
    assert 7 * U32 < chain_rms(64) < 9 * U32 < LIMIT < 13 * U32 < chain_rms(128)


@pytest.mark.parametrize("n,acc,mode,weighted", [
    (14336, FOLD, SINGLE, False), (28673, FOLD, SINGLE, False), (32768, FOLD, SINGLE, False),
    (49151, FOLD, SINGLE, False), (15361, KAHAN, SINGLE, False), (28673, KAHAN, SINGLE, False),
    (32767, KAHAN, SINGLE, False), (16385, FOLD, SINGLE, True), (32767, FOLD, SINGLE, True),
    (16384, FOLD, GUARDED, False), (40001, FOLD, GUARDED, False), (98303, FOLD, GUARDED, False),
    (32767, KAHAN, GUARDED, False), (20001, FOLD, GUARDED, True), (32767, FOLD, GUARDED, True)])
def test_fields_add_at_most_64_terms_in_fp32(n, acc, mode, weighted):
    m, eps = 4096, 1e-8
    pos = np.zeros((n, 3))       # the targets first, then the sources, all at one point
    d = wl.gaussian_bunch(m, 1.0, seed=n)
    r = 1e-5 * (0.5 + 1.5 * wl.uniform(18, 1, m))
    pos[:m] = d / np.linalg.norm(d, axis=1)[:, None] * r[:, None]
    w = np.full(n, 12.0)
    with capi.Simulation(n, 10.0 if weighted else 12.0, 1e-16, eps, acc=acc, positions=mode) as sim:
        if weighted:
            sim.set_weights(w)
        sim.load(pos)
        E = sim.fields()
    idx = np.arange(0, m, 4)
    ref = oracle.fields_subset(pos, w, eps, idx)
    err = np.linalg.norm(E[idx] - ref, axis=1) / np.linalg.norm(ref, axis=1)
    rms = float(np.sqrt(np.mean(err ** 2)))
    assert rms <= LIMIT, f"rms error {rms / U32:.1f} u"


def two_clusters(n, gap):
    pos = np.zeros((n, 3))
    pos[n // 2:] = gap * np.array([0.48, 0.6, 0.64])
    return pos


@pytest.mark.parametrize("n", [16384, 24001, 32767])
def test_potential_energy_adds_at_most_128_terms_in_fp32(n):
    """Two clusters of coincident particles: the potential energy is n_A n_B equal terms (the
    zero-distance pairs add nothing).  The limit lies half way between chains of 128 and 256."""
    limit = float(np.sqrt(chain_rms(128) * chain_rms(256)))
    c = oracle.constants()
    err = []
    with capi.Simulation(n, 12.0, 1e-16, 0.0, positions=SINGLE) as sim:
        for gap in 1e-5 * (0.5 + 1.5 * wl.uniform(19, 1, 32)):
            pos = two_clusters(n, gap)
            sim.load(pos)
            got = sim.diagnostics()["pe"]
            pairs = float(n // 2) * (n - n // 2)
            want = c["k"] * c["e"] ** 2 * 12.0 ** 2 * pairs / np.linalg.norm(pos[-1])
            err.append((got - want) / want)
    rms = float(np.sqrt(np.mean(np.square(err))))
    assert rms <= limit, f"rms error {rms / U32:.1f} u of {limit / U32:.1f}"
