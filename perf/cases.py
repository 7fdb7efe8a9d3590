"""The work this framework is measured on: direct Coulomb sums and Velocity-Verlet runs of
electron bunches, through the calls a user's program makes.

Kinds of case:

* ``steps``    a program that owns a context restores a bunch (pp_set_state with the saved
               staging frame, device arrays), advances it by ``steps`` time steps and reads the
               state back: the time loop of every expansion run.
* ``analyse``  a new bunch is loaded (which decides the staging), its field is read and its
               diagnostics with the potential energy are taken: a parameter scan's work on
               each sample.
* ``noalloc``  one allocation-free field evaluation of a small bunch at device positions, as a
               host framework's inner loop calls it.
* ``serve``    a batch of expansion requests served to completion by the continuous-batching
               server: host arrays in, final states out.

The fields, and the states a run reaches, are sums of single-precision pair terms that the
ABI hands over in double containers; the programs modelled here keep their snapshots as
float32.  Runs with the all-FP64 pair arithmetic keep float64.
"""
import math

import numpy as np
import torch

from paper_2502_10640_gb300 import capi, serve

E_CHARGE = 1.602176634e-19
M_ELECTRON = 9.1093837015e-31
COULOMB = 1.0 / (4.0 * math.pi * 8.8541878128e-12)

ACC = {"fp64fold": capi.PP_ACC_FP64FOLD, "kahan": capi.PP_ACC_KAHAN,
       "fp64": capi.PP_ACC_FP64_FULL}
POSITIONS = {"auto": None, "guarded": capi.PP_POS_GUARDED, "split": capi.PP_POS_SPLIT}


def _steps(name, profile, n, scale, w, eps, dt, steps, acc="fp64fold", weights=False,
           positions="auto"):
    return {"name": name, "kind": "steps", "profile": profile, "n": n, "scale": scale, "w": w,
            "eps": eps, "dt": dt, "steps": steps, "acc": acc, "weights": weights,
            "positions": positions}


def listed():
    return [
        # one field call on a handful of electrons: launch and synchronisation latency
        {"name": "noalloc_900", "kind": "noalloc", "n": 900, "scale": 1e-6, "w": 1.0, "eps": 0.0},
        # 2048 real electrons, cold Gaussian of 1 um, no softening, the whole 200-step run
        _steps("gaussian_2048", "gaussian", 2048, 1e-6, 1.0, 0.0, 1e-16, 200),
        # the paper's 16^3 cube lattice (0.1 mm, w = 12.2, dt = 1e-13 s), warm, a stretch of its run
        _steps("lattice_4096", "lattice", 4096, 1e-4, 12.207, 0.0, 1e-13, 100),
        # the all-FP64 comparison path of the Gaussian runs, ragged N
        _steps("fp64_16385", "gaussian", 16385, 1e-5, 1e8 / 16385, 1e-9, 1e-14, 2, acc="fp64"),
        # macro-electrons of unequal weight, ragged N
        _steps("weights_24001", "sphere", 24001, 2e-5, 1000.0, 2e-9, 1e-14, 8, weights=True),
        # the 32^3 lattice of the particle-number sweep
        _steps("lattice_32768", "lattice", 32768, 1e-4, 1.526, 0.0, 1e-13, 16),
        # a ball whose user asks for guarded staging because pairs may come close, ragged N
        _steps("guarded_40001", "sphere", 40001, 2e-5, 10.0, 1e-9, 1e-14, 8,
               positions="guarded"),
        # N = 65536 Gaussian of 10 um carrying 1e8 electrons, 1 nm softening
        _steps("gaussian_65536", "gaussian", 65536, 1e-5, 1e8 / 65536, 1e-9, 1e-14, 8),
        # scan sample: load, field, diagnostics with the potential energy
        {"name": "analyse_100003", "kind": "analyse", "profile": "sphere", "n": 100003,
         "scale": 5e-5, "w": 5952.4, "eps": 5e-9, "dt": 2e-14},
        # compensated FP32 accumulation, mid-size ball
        _steps("kahan_200001", "sphere", 200001, 5e-5, 5952.4, 5e-9, 2e-14, 1, acc="kahan"),
        # N = 2^20 uniform ball of 1 nC (the benchmark's bunch), one step
        _steps("sphere_1m", "sphere", 1 << 20, 5e-5, 5952.4, 5e-9, 2e-14, 1),
        # eight served runs of 4096 to 65536 macro-electrons, joining and leaving
        {"name": "serve_8", "kind": "serve", "count": 8, "n_min": 4096, "n_max": 65536,
         "steps_min": 4, "steps_max": 24},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps"] * 6 + ["analyse", "noalloc", "serve"])
    if kind == "noalloc":
        return {"kind": "noalloc", "n": _log_int(rng, 500, 16384), "scale": 1e-6, "w": 1.0,
                "eps": rng.choice([0.0, 1e-9])}
    if kind == "serve":
        return {"kind": "serve", "count": rng.randint(3, 8), "n_min": 4096,
                "n_max": _log_int(rng, 8192, 65536), "steps_min": 4,
                "steps_max": rng.randint(8, 24)}
    profile = rng.choice(["gaussian", "sphere"])
    scale = math.exp(rng.uniform(math.log(1e-6), math.log(5e-5)))
    eps = rng.choice([0.0, 1e-5, 1e-4]) * scale
    if kind == "analyse":
        n = _log_int(rng, 2048, 262144)
    else:
        n = _log_int(rng, 1024, 524288)
    # a common charge of 0.1 nC keeps dt well inside the bunch's expansion time
    w = 1e-10 / (E_CHARGE * n)
    rate = COULOMB * E_CHARGE ** 2 * n * w / (M_ELECTRON * scale ** 3)
    dt = 0.01 / math.sqrt(2.0 * rate)
    if kind == "analyse":
        return {"kind": "analyse", "profile": profile, "n": n, "scale": scale, "w": w,
                "eps": eps, "dt": dt}
    mode = rng.choice(["fp64fold"] * 4 + ["kahan", "weights", "fp64"])
    if mode == "fp64":
        n = min(n, 32768)
    steps = max(1, min(100, int(4e10 / (float(n) * n * (20.0 if mode == "fp64" else 1.0)))))
    c = _steps("", profile, n, scale, w, eps, dt, steps,
               acc="fp64fold" if mode == "weights" else mode, weights=mode == "weights",
               positions="auto" if mode == "fp64" else rng.choice(["auto"] * 4 +
                                                                  ["guarded", "split"]))
    del c["name"]
    return c


# ---- inputs --------------------------------------------------------------------

def _positions(profile, n, scale, g):
    if profile == "lattice":
        m = round(n ** (1.0 / 3.0))
        a = (torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) * (scale / m) - scale / 2
        x, y, z = torch.meshgrid(a, a, a, indexing="ij")
        return torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], dim=1).contiguous()
    p = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
    if profile == "gaussian":
        p = p * scale
    else:
        u = torch.rand(n, 1, generator=g, device="cuda", dtype=torch.float64)
        p = p / p.norm(dim=1, keepdim=True) * (scale * u ** (1.0 / 3.0))
    return (p - p.mean(dim=0, keepdim=True)).contiguous()


def _inputs(case, seed):
    """Positions, velocities and per-particle weights (None: equal) of a bunch."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    pos = _positions(case["profile"], case["n"], case["scale"], g)
    vel = torch.zeros_like(pos)
    if case["profile"] == "lattice":   # a thermal spread of the emitted electrons
        vel = torch.randn(case["n"], 3, generator=g, device="cuda", dtype=torch.float64) * 1e4
    wts = None
    if case.get("weights"):
        u = torch.rand(case["n"], generator=g, device="cuda", dtype=torch.float64)
        wts = case["w"] * (0.5 + u)
    return pos, vel, wts


def _requests(case, seed):
    """The (n, steps, positions) of a served trace; N spread over its range by rank."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for k in range(case["count"]):
        f = k / max(1, case["count"] - 1)
        n = int(round(case["n_min"] * (case["n_max"] / case["n_min"]) ** f)) - (k % 2)
        steps = case["steps_min"] + (case["steps_max"] - case["steps_min"]) * (k * 3 % 8) // 7
        out.append((n, steps, _positions("sphere", n, 5e-5, g)))
    return out


SERVE_W, SERVE_EPS, SERVE_DT = 5952.4, 5e-9, 2e-14


def prepare(case, seed):
    if case["kind"] == "noalloc":
        g = torch.Generator(device="cuda").manual_seed(seed)
        pos = _positions("gaussian", case["n"], case["scale"], g)
        return {"case": case, "pos": pos, "out": torch.empty_like(pos)}
    if case["kind"] == "serve":
        reqs = [serve.ServeRequest(k, 0.0, n, SERVE_W, SERVE_DT, SERVE_EPS, steps,
                                   pos.cpu().numpy())
                for k, (n, steps, pos) in enumerate(_requests(case, seed))]
        return {"case": case, "requests": reqs}
    pos, vel, wts = _inputs(case, seed)
    sim = capi.Simulation(case["n"], case["w"], case["dt"], case["eps"],
                          acc=ACC[case["acc"]] if "acc" in case else None,
                          positions=POSITIONS[case.get("positions", "auto")])
    state = {"case": case, "sim": sim, "pos": pos, "out": torch.empty_like(pos)}
    if case["kind"] == "analyse":
        return state
    if wts is not None:
        sim.set_weights(wts)
    sim.load(pos, vel)
    state["vel"], state["acc"] = vel, torch.empty_like(pos)
    _, _, _, _, state["frame"] = capi.pp_get_state(sim.ctx, None, None, state["acc"])
    state["outs"] = [torch.empty_like(pos) for _ in range(3)]
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "noalloc":
        capi.pp_fields_noalloc(case["n"], case["w"], case["eps"], state["pos"], state["out"])
        return {"fields": state["out"].float()}
    if case["kind"] == "serve":
        server = serve.Server(budget_bytes=16 << 30)
        server.run(state["requests"])
        results = sorted(server.results, key=lambda r: r.rid)
        server.close()
        return {k: np.concatenate([getattr(r, k) for r in results]).astype(np.float32)
                for k in ("positions", "velocities", "accelerations")}
    sim = state["sim"]
    if case["kind"] == "analyse":
        sim.load(state["pos"])
        fields = sim.fields(state["out"])
        d = sim.diagnostics()
        return {"fields": fields.float(),
                "moments": [d[k] for k in ("rms_radius", "pe", "x_rms", "x_max")]}
    capi.pp_set_state(sim.ctx, state["pos"], state["vel"], state["acc"], 0, state["frame"])
    sim.step(case["steps"])
    p, v, a = state["outs"]
    capi.pp_get_state(sim.ctx, p, v, a)
    if case["acc"] != "fp64":
        p, v, a = p.float(), v.float(), a.float()
    return {"positions": p, "velocities": v, "accelerations": a}


# ---- what a pass cannot do without ---------------------------------------------

def _pair_flops(n):
    """One force evaluation: each unordered pair's separation (3 subtractions, 6 flops for the
    softened square), reciprocal root and its cube (3), and the term added to both (12)."""
    return 24.0 * n * (n - 1) / 2


def work(case):
    if case["kind"] == "noalloc":
        return {"bytes": 48.0 * case["n"], "flops": _pair_flops(case["n"])}
    if case["kind"] == "serve":
        b = f = 0.0
        for k in range(case["count"]):
            x = k / max(1, case["count"] - 1)
            n = int(round(case["n_min"] * (case["n_max"] / case["n_min"]) ** x)) - (k % 2)
            steps = case["steps_min"] + (case["steps_max"] - case["steps_min"]) * (k * 3 % 8) // 7
            b += n * (24.0 + 72.0)
            f += (steps + 1) * _pair_flops(n)
        return {"bytes": b, "flops": f}
    n = case["n"]
    if case["kind"] == "analyse":
        # the field once (it serves the initial acceleration too) and the potential's pairs
        return {"bytes": 48.0 * n, "flops": _pair_flops(n) + 11.0 * n * (n - 1) / 2}
    # positions, velocities and accelerations in and out, each once
    return {"bytes": 144.0 * n, "flops": case["steps"] * _pair_flops(n)}


# ---- the same in 64 bits --------------------------------------------------------

def _sums(pos, w, eps, want_phi=False):
    """sum_j w_j (r_i - r_j) / s^(3/2) and, if asked, sum_j w_j / s^(1/2), j != i."""
    n = pos.shape[0]
    x, y, z = (pos[:, k].contiguous() for k in range(3))
    out = torch.empty_like(pos)
    phi = torch.empty_like(x) if want_phi else None
    rows = max(1, min(n, (1 << 25) // n))
    for i in range(0, n, rows):
        j = min(n, i + rows)
        dx, dy, dz = (c[i:j, None] - c[None, :] for c in (x, y, z))
        s = dx * dx
        s.addcmul_(dy, dy).addcmul_(dz, dz)
        s += eps * eps
        inv = torch.where(s > 0, s.rsqrt(), torch.zeros_like(s))
        if want_phi:
            k = torch.arange(i, j, device=pos.device)
            own = inv[k - i, k] * w[k]
            phi[i:j] = inv @ w - own
        f = inv * inv * inv * w[None, :]
        out[i:j, 0] = (f * dx).sum(1)
        out[i:j, 1] = (f * dy).sum(1)
        out[i:j, 2] = (f * dz).sum(1)
    return (out, phi) if want_phi else out


def _verlet(pos, vel, w, eps, dt, steps):
    c = COULOMB * E_CHARGE ** 2 / M_ELECTRON
    r, v = pos.clone(), vel.clone()
    a = c * _sums(r, w, eps)
    for _ in range(steps):
        r = r + v * dt + a * (dt * dt / 2)
        b = c * _sums(r, w, eps)
        v = v + (a + b) * (dt / 2)
        a = b
    return r, v, a


def exact(case, seed):
    if case["kind"] == "noalloc":
        g = torch.Generator(device="cuda").manual_seed(seed)
        pos = _positions("gaussian", case["n"], case["scale"], g)
        w = torch.full_like(pos[:, 0], case["w"])
        return {"fields": -COULOMB * E_CHARGE * _sums(pos, w, case["eps"])}
    if case["kind"] == "serve":
        got = []
        for n, steps, pos in _requests(case, seed):
            w = torch.full_like(pos[:, 0], SERVE_W)
            got.append(_verlet(pos, torch.zeros_like(pos), w, SERVE_EPS, SERVE_DT, steps))
        return {k: torch.cat([t[i] for t in got])
                for i, k in enumerate(("positions", "velocities", "accelerations"))}
    n = case["n"]
    if (case.get("steps", 1) + 1) * float(n) * n > 2.5e11:   # too long in 64 bits
        return None
    pos, vel, wts = _inputs(case, seed)
    w = torch.full_like(pos[:, 0], case["w"]) if wts is None else wts
    if case["kind"] == "analyse":
        s, phi = _sums(pos, w, case["eps"], want_phi=True)
        pe = 0.5 * COULOMB * E_CHARGE ** 2 * float((w * phi).sum())
        rms = math.sqrt(float(((pos - pos.mean(dim=0)) ** 2).sum(1).mean()))
        x = pos[:, 0]
        return {"fields": -COULOMB * E_CHARGE * s,
                "moments": [rms, pe, math.sqrt(float((x * x).mean())), float(x.max())]}
    r, v, a = _verlet(pos, vel, w, case["eps"], case["dt"], case["steps"])
    return {"positions": r, "velocities": v, "accelerations": a}
