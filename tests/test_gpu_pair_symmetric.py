"""The pair-symmetric force kernels (pp_sym.cuh) against the FP64 oracle at the sizes where
their decomposition can go wrong: one particle, an odd tail, either side of a warp's block
of targets (256, 512) and of a tile, a partly filled last group, coincident particles."""
import numpy as np
import pytest

import oracle
from tests._bounds import field_error_bound
from paper_2502_10640_gb300 import capi, workloads as wl

pytestmark = pytest.mark.gpu

K_E = oracle.constants()["k"] * oracle.constants()["e"]
MODES = {"f32x2.": capi.PP_POS_SINGLE, "f32x2w.": capi.PP_POS_SINGLE,
         "f32x2split.": capi.PP_POS_SPLIT, "f32x2wsplit.": capi.PP_POS_SPLIT,
         "f32x2guard.": capi.PP_POS_GUARDED, "f32x2wguard.": capi.PP_POS_GUARDED,
         "f32x2bguard.": capi.PP_POS_GUARDED, "f32x2wbguard.": capi.PP_POS_GUARDED}


def sym_variants():
    out = [v for v in capi.variants() if ".sym" in v and not v.startswith("f64")]
    assert len(out) >= 15
    return out


def run(name, pos, eps, wts=None, fn=lambda s: s.fields()):
    acc = capi.PP_ACC_KAHAN if ".kahan." in name else capi.PP_ACC_FP64FOLD
    mode = MODES[name[:name.index(".") + 1]]
    weighted = name.startswith("f32x2w")
    with capi.Simulation(len(pos), 10.0, 1e-15, eps, acc=acc, positions=mode) as sim:
        sim.set_option(capi.PP_OPT_VARIANT, capi.variants().index(name))
        if weighted:
            sim.set_weights(wts)
        sim.load(pos)
        assert sim.get_option(capi.PP_OPT_VARIANT) == capi.variants().index(name)
        return fn(sim), weighted, mode


@pytest.mark.parametrize("n", [1, 2, 33, 255, 257, 513, 1025, 2047, 5000])
def test_every_symmetric_variant_matches_oracle(n):
    pos = wl.uniform_sphere(n, 5e-6, seed=700 + n)
    wts = 10.0 * (0.5 + wl.uniform(91, 3, n))
    eps = 1e-8
    ref, ref_w = oracle.fields(pos, 10.0, eps), oracle.fields(pos, wts, eps)
    bound = field_error_bound(pos, 10.0, eps, np.arange(n), K_E)
    for name in sym_variants():
        E, weighted, _ = run(name, pos, eps, wts)
        if n == 1:
            assert np.all(E == 0.0), name
            continue
        err = np.linalg.norm(E - (ref_w if weighted else ref), axis=1)
        # weights are at most 1.5 times the common one the bound is computed with
        assert np.all(err <= (1.5 if weighted else 1.0) * bound), name


def test_coincident_particles_add_nothing():
    """Zero-distance pairs without softening, within a warp's block (3, 17) and across
    blocks (0, 2999), through the slow form of a tile."""
    pos = wl.gaussian_bunch(3000, 1e-6, seed=34)
    pos[17] = pos[3]
    pos[2999] = pos[0]
    wts = 10.0 * (0.5 + wl.uniform(92, 3, 3000))
    ref, ref_w = oracle.fields(pos, 10.0, 0.0), oracle.fields(pos, wts, 0.0)
    bound = field_error_bound(pos, 10.0, 0.0, np.arange(3000), K_E)
    for name in sym_variants():
        E, weighted, _ = run(name, pos, 0.0, wts)
        err = np.linalg.norm(E - (ref_w if weighted else ref), axis=1)
        assert np.all(err <= (1.5 if weighted else 1.0) * bound), name


@pytest.mark.parametrize("n,mode", [(20481, capi.PP_POS_SINGLE), (36865, capi.PP_POS_GUARDED),
                                    (13001, capi.PP_POS_SPLIT)])
def test_default_plan_steps_and_ranges(n, mode):
    """The default plan is symmetric from these sizes on; steps are bitwise the same with
    and without graph blocks; cutting the rows into other ranges (PP_OPT_SPLIT) changes
    the FP64 grouping of the partial sums only."""
    pos = wl.uniform_sphere(n, 1e-5, seed=n)
    idx = np.arange(0, n, 97)
    ref = oracle.fields_subset(pos, 10.0, 1e-9, idx)
    runs, fields = [], []
    for gb, split in ((0, 0), (4, 0), (4, 3)):
        with capi.Simulation(n, 10.0, 1e-16, 1e-9, positions=mode) as sim:
            sim.set_option(capi.PP_OPT_GRAPH_BLOCK, gb)
            sim.set_option(capi.PP_OPT_SPLIT, split)
            sim.load(pos)
            assert ".sym" in capi.variants()[sim.get_option(capi.PP_OPT_VARIANT)]
            fields.append(sim.fields())
            sim.step(6)
            runs.append(sim.state())
    for x, y in zip(runs[0][:3], runs[1][:3]):
        assert np.array_equal(x, y)
    scale = np.linalg.norm(fields[0], axis=1).max()
    assert np.max(np.abs(fields[2] - fields[0])) <= 1e-13 * scale
    bound = field_error_bound(pos, 10.0, 1e-9, idx, K_E)
    assert np.all(np.linalg.norm(fields[0][idx] - ref, axis=1) <= bound)


@pytest.mark.parametrize("n", [1, 2, 31, 33, 64, 1023, 1025, 3001])
@pytest.mark.parametrize("eps", [0.0, 1e-8])
def test_fp64_pairs_match_oracle(n, eps):
    """All-FP64 pairs, equal and per-particle weights, coincident particles included: the
    recursive-summation bound n u on sums of same-scale terms, with room for the few
    roundings of a pair term (u = 2^-53)."""
    pos = wl.gaussian_bunch(n, 1e-6, seed=900 + n)
    if n > 40:
        pos[37] = pos[3]
        pos[n - 1] = pos[0]
    wts = 10.0 * (0.5 + wl.uniform(94, 3, n))
    for w in (None, wts):
        with capi.Simulation(n, 10.0, 1e-15, eps, acc=capi.PP_ACC_FP64_FULL) as sim:
            if w is not None:
                sim.set_weights(w)
            sim.load(pos)
            assert "f64" in capi.variants()[sim.get_option(capi.PP_OPT_VARIANT)]
            E = sim.fields()
        ref = oracle.fields(pos, 10.0 if w is None else w, eps)
        d = pos[:, None, :] - pos[None, :, :]
        s = np.einsum("ijk,ijk->ij", d, d) + eps * eps
        with np.errstate(divide="ignore", invalid="ignore"):
            mag = np.where(s > 0, np.sqrt(np.maximum(s - eps * eps, 0.0)) / s ** 1.5, 0.0)
            # the separation of a close pair carries the rounding of the scaled positions
            ratio = np.where(s > eps * eps, 1e-5 / np.sqrt(np.maximum(s - eps * eps, 1e-300)), 0.0)
        wj = np.full(n, 10.0) if w is None else w
        # weights enter as float32 ratios
        rel = (n + 40) * 2.0 ** -53 + (2.0 ** -24 if w is not None else 0.0)
        bound = K_E * ((mag * (rel + 8 * 2.0 ** -53 * ratio)) @ wj)
        assert np.all(np.linalg.norm(E - ref, axis=1) <= bound + 1e-300), (n, eps)
