"""Measured workloads of the filament library, each through its public calls.

A case is a dict of plain values. ``prepare`` makes what a program holds before
the call (device inputs from the seed, the context or network), ``run`` does one
pass and returns the whole result, ``work`` states the bytes and operations the
pass cannot do without, and ``exact`` gives the same result in plain 64-bit
torch where the call is a direct formula. Kinds:

* ``apply``   one mobility apply (``fil_mobility_apply``): random-walk
  filaments at 5% (small) or 2% volume fraction, N(0, 1) forces and torques;
* ``residual``  one residual f(X) at a perturbed state of a straight cloud,
  optionally with the steric barrier (``fil_residual``);
* ``j0_solve``  one solve with the factored approximate Jacobian of a step in
  progress (``fil_j0_solve``);
* ``steps``   a simulation segment: straight filaments set up
  (``fil_init_straight``), a few whole timesteps (``fil_step``) and the state
  read back (``fil_get_state``);
* ``mlp_forward``, ``mlp_gradients``  the warm-start network.

Results of the forms whose pair sums or history are FP32 (FIL_MIXED,
FIL_PAIR32) carry FP32 accuracy and are kept in float32, as a program that
stores velocities or trajectory frames of those forms does; FP64 forms and
FP64-accurate solves stay in float64.
"""
from __future__ import annotations

import math

import torch

from paper_1903_12609_gb300 import fil
from paper_1903_12609_gb300.inputs import box_side, workload_params

PRECISION = {"fp64": fil.FIL_FP64, "mixed": fil.FIL_MIXED, "pair32": fil.FIL_PAIR32}
J0_MODEL = {"drag": fil.FIL_J0_DRAG, "rpy": fil.FIL_J0_FILAMENT_RPY}
F64 = torch.float64
PAIR_FLOPS = 84          # operations of one ordered pair of the far form


def listed():
    return [
        # the smallest system of the workloads: one 20-segment filament, FP64 (latency)
        dict(name="apply_single_fp64", kind="apply", precision="fp64", n_sys=1, fil_lo=1, fil_hi=1,
             seg_lo=20, seg_hi=20, vf=0.05),
        # the mobility workload: 100 random-walk filaments of 32 segments
        dict(name="apply_3200_pair32", kind="apply", precision="pair32", n_sys=1, fil_lo=100,
             fil_hi=100, seg_lo=32, seg_hi=32, vf=0.05),
        # the same workload in the parity form, every operation in FP64
        dict(name="apply_3200_fp64", kind="apply", precision="fp64", n_sys=1, fil_lo=100,
             fil_hi=100, seg_lo=32, seg_hi=32, vf=0.05),
        # a mid-size suspension of unequal filaments (about 9 600 segments, no round size)
        dict(name="apply_ragged_mixed", kind="apply", precision="mixed", n_sys=1, fil_lo=301,
             fil_hi=301, seg_lo=16, seg_hi=48, vf=0.02),
        # the full suspension, 32 000 segments: the apply that every Broyden iteration makes
        dict(name="apply_32000_pair32", kind="apply", precision="pair32", n_sys=1, fil_lo=1000,
             fil_hi=1000, seg_lo=32, seg_hi=32, vf=0.02),
        # one residual with the steric barrier on: a user's own nonlinear solver calls this
        dict(name="residual_steric_8000", kind="residual", precision="pair32", n_fil=250, seg=32,
             steric=20.0),
        # the FP64-accurate J0 solve of the full suspension (filament-RPY blocks)
        dict(name="j0_solve_32000", kind="j0_solve", precision="pair32", model="rpy", n_fil=1000,
             seg_lo=32, seg_hi=32),
        # the single sedimenting filament, tolerance 1e-8, FP64: launches and host round trips
        dict(name="steps_single_fp64", kind="steps", precision="fp64", model="drag", n_sys=1,
             fil_lo=1, fil_hi=1, seg_lo=20, seg_hi=20, steps=10, tol=1e-8, dt_frac=0.01, reuse=1,
             memory=0, adaptive=False),
        # the flagship: 32 000-segment suspension with J0 kept and Broyden memory carried
        dict(name="steps_suspension_32000", kind="steps", precision="pair32", model="rpy", n_sys=1,
             fil_lo=1000, fil_hi=1000, seg_lo=32, seg_hi=32, steps=4, tol=1e-4, dt_frac=0.005,
             reuse=10, memory=48, adaptive=True),
        # a parameter sweep: 256 independent small suspensions in one context, mixed form
        dict(name="steps_ensemble_256", kind="steps", precision="mixed", model="drag", n_sys=256,
             fil_lo=1, fil_hi=64, seg_lo=16, seg_hi=48, steps=2, tol=1e-4, dt_frac=0.005, reuse=10,
             memory=0, adaptive=True),
        # the warm-start network's prediction for every filament of the suspension
        dict(name="mlp_forward_1000", kind="mlp_forward", batch=1000),
        # loss and gradient of one training batch of the network
        dict(name="mlp_gradients_1024", kind="mlp_gradients", batch=1024),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.499)))))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "residual", "j0_solve", "steps", "steps",
                       "mlp_forward", "mlp_gradients"])
    if kind == "apply":
        precision = rng.choice(["fp64", "mixed", "pair32"])
        total = _log_int(rng, 16, 4000 if precision == "fp64" else 32000)
        if rng.random() < 0.3:           # equal filaments
            lo = hi = rng.randint(1, min(64, total))
        else:
            lo, hi = sorted((rng.randint(1, min(48, total)), rng.randint(1, min(64, total))))
        n_sys = 1 if rng.random() < 0.7 or total < 200 else rng.randint(2, min(64, total // 100))
        m = max(1, int(2 * total / (lo + hi) / n_sys))
        return dict(kind="apply", precision=precision, n_sys=n_sys, fil_lo=m if n_sys == 1 else
                    max(1, m // 2), fil_hi=m, seg_lo=lo, seg_hi=hi,
                    vf=rng.choice([0.02, 0.05]))
    if kind == "residual":
        precision = rng.choice(["fp64", "pair32", "mixed"])
        seg = rng.randint(2, 48)
        m = max(1, _log_int(rng, 20, 2500 if precision == "fp64" else 16000) // seg)
        return dict(kind="residual", precision=precision, n_fil=m, seg=seg,
                    steric=rng.choice([0.0, 20.0]))
    if kind == "j0_solve":
        model = rng.choice(["rpy", "rpy", "drag"])
        lo, hi = sorted((rng.randint(2, 38 if model == "rpy" else 64),
                         rng.randint(2, 38 if model == "rpy" else 64)))
        return dict(kind="j0_solve", precision=rng.choice(["fp64", "mixed", "pair32"])
                    if model == "drag" else rng.choice(["mixed", "pair32"]), model=model,
                    n_fil=_log_int(rng, 1, 300 if model == "drag" else 1000), seg_lo=lo, seg_hi=hi)
    if kind == "steps":
        form = rng.choice(["single", "suspension", "ensemble"])
        if form == "single":
            n = rng.randint(8, 40)
            return dict(kind="steps", precision="fp64", model="drag", n_sys=1, fil_lo=1, fil_hi=1,
                        seg_lo=n, seg_hi=n, steps=rng.randint(3, 10), tol=1e-8, dt_frac=0.01,
                        reuse=1, memory=0, adaptive=False)
        if form == "suspension":
            m = _log_int(rng, 8, 700)
            n = rng.randint(16, 32)
            return dict(kind="steps", precision=rng.choice(["pair32", "mixed"]), model="rpy",
                        n_sys=1, fil_lo=m, fil_hi=m, seg_lo=n, seg_hi=n, steps=rng.randint(2, 4),
                        tol=1e-4, dt_frac=0.005, reuse=10, memory=48, adaptive=True)
        return dict(kind="steps", precision=rng.choice(["mixed", "pair32"]), model="drag",
                    n_sys=_log_int(rng, 4, 160), fil_lo=1, fil_hi=rng.randint(4, 32), seg_lo=16,
                    seg_hi=rng.randint(20, 40), steps=2, tol=1e-4, dt_frac=0.005,
                    reuse=rng.choice([1, 10]), memory=0, adaptive=True)
    if kind == "mlp_forward":
        return dict(kind=kind, batch=_log_int(rng, 1, 4096))
    return dict(kind=kind, batch=_log_int(rng, 16, 2048))


# ---- inputs -----------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _randn(g, *shape):
    return torch.randn(*shape, dtype=F64, device="cuda", generator=g)


def _rand(g, *shape):
    return torch.rand(*shape, dtype=F64, device="cuda", generator=g)


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _layout(case):
    """Filaments per system and segments per filament (host lists): part of the
    case, so the same for every seed."""
    g = torch.Generator().manual_seed(7919)

    def ints(lo, hi, n):
        return torch.randint(lo, hi + 1, (n,), generator=g).tolist()

    if "n_fil" in case:
        fps = [case["n_fil"]]
    else:
        fps = ints(case["fil_lo"], case["fil_hi"], case["n_sys"])
    if "seg" in case:
        return fps, [case["seg"]] * sum(fps)
    return fps, ints(case["seg_lo"], case["seg_hi"], sum(fps))


def _segment_tables(fps, segs):
    """Device tables: filament and index in the filament of every segment, and
    the system of every filament."""
    n = torch.tensor(segs, device="cuda")
    fil_of = torch.repeat_interleave(torch.arange(len(segs), device="cuda"), n)
    start = torch.cumsum(n, 0) - n
    idx = torch.arange(int(sum(segs)), device="cuda") - start[fil_of]
    sys_of = torch.repeat_interleave(torch.arange(len(fps), device="cuda"),
                                     torch.tensor(fps, device="cuda"))
    return n, fil_of, idx, sys_of


def _sides(fps, segs, vf):
    out, f = [], 0
    for m in fps:
        out.append(box_side(sum(segs[f:f + m]), vf))
        f += m
    return torch.tensor(out, dtype=F64, device="cuda")


def _walks(fps, segs, vf, g):
    """Random-walk filaments (bond 2.2) centred uniformly in each system's cube."""
    n, fil_of, idx, sys_of = _segment_tables(fps, segs)
    bond = _unit(_randn(g, len(segs), max(segs), 3)) * 2.2
    bond[:, 0] = 0.0
    walk = torch.cumsum(bond, 1)
    live = (torch.arange(max(segs), device="cuda")[None] < n[:, None]).to(F64)[..., None]
    centre = _rand(g, len(segs), 3) * _sides(fps, segs, vf)[sys_of][:, None]
    walk = walk - (walk * live).sum(1, keepdim=True) / n[:, None, None] + centre[:, None]
    return walk[fil_of, idx].contiguous()


def _axis_distance2(p, d, L, q, e, K):
    """Squared distance of the segments p + s d (0 <= s <= L) and q + t e (0 <= t <= K)."""
    r = p - q
    b, c, f = (d * e).sum(-1), (d * r).sum(-1), (e * r).sum(-1)
    s = torch.minimum(((b * f - c) / (1.0 - b * b).clamp_min(1e-12)).clamp_min(0.0), L)
    t = torch.minimum((b * s + f).clamp_min(0.0), K)
    s = torch.minimum((b * t - c).clamp_min(0.0), L)
    x = r + s[..., None] * d - t[..., None] * e
    return (x * x).sum(-1)


def _cloud(fps, segs, vf, dL, g):
    """Isotropic clouds of straight filaments without overlaps: base points
    uniform in each system's cube, frames uniform on SO(3); of two filaments
    that come closer than a diameter the later one is drawn again."""
    n, _, _, sys_of = _segment_tables(fps, segs)
    ns, m = len(fps), max(fps)
    live = torch.arange(m, device="cuda")[None] < torch.tensor(fps, device="cuda")[:, None]
    side = _sides(fps, segs, vf)[:, None, None]
    L = torch.zeros(ns, m, dtype=F64, device="cuda")
    L[live] = (n - 1).to(F64) * dL
    below = torch.tril(torch.ones(m, m, dtype=torch.bool, device="cuda"), -1)
    pair = below[None] & live[:, :, None] & live[:, None, :]
    base = t = None
    redraw = live
    for _ in range(400):
        nb, nt = _rand(g, ns, m, 3) * side, _unit(_randn(g, ns, m, 3))
        pick = redraw[..., None]
        base = nb if base is None else torch.where(pick, nb, base)
        t = nt if t is None else torch.where(pick, nt, t)
        d2 = _axis_distance2(base[:, :, None], t[:, :, None], L[:, :, None], base[:, None],
                             t[:, None], L[:, None])
        redraw = (pair & (d2 < 4.0)).any(-1)
        if not bool(redraw.any()):
            break
    else:
        raise RuntimeError("could not place the filaments")
    base, t = base[live].contiguous(), t[live].contiguous()
    mu = _randn(g, len(segs), 3)
    mu = _unit(mu - (mu * t).sum(-1, keepdim=True) * t).contiguous()
    return base, t, mu


def _suspension(case, fps, segs, g):
    """Straight cloud with the loads of the suspension workload: in every system
    the first half of the filaments sediment, the rest carry a follower force."""
    n_ref = segs[0] if len(set(segs)) == 1 else 32
    wl = workload_params(1, n_ref, B=1000.0, dt_over_T=case.get("dt_frac", 0.005),
                         tol=case.get("tol", 1e-4), max_iter=60)
    base, t, mu = _cloud(fps, segs, 0.02, wl.dL, g)
    n, fil_of, _, sys_of = _segment_tables(fps, segs)
    count = torch.tensor(fps, device="cuda")
    first = torch.cumsum(count, 0) - count
    rank = torch.arange(len(segs), device="cuda") - first[sys_of]
    passive = (rank < count[sys_of] // 2) if len(segs) > 1 else torch.ones(1, dtype=torch.bool,
                                                                           device="cuda")
    Fext = torch.zeros(int(n.sum()), 3, dtype=F64, device="cuda")
    Fext[:, 2] = torch.where(passive[fil_of], -wl.W * wl.dL, 0.0)
    follower = torch.where(passive, 0.0, 100.0 * wl.KB / (n.to(F64) * wl.dL) ** 2).to(F64)
    return wl, base, t, mu, Fext, follower.contiguous()


def _context(case, wl, fps, segs):
    kw = dict(precision=PRECISION[case["precision"]],
              fil_per_sys=fps if len(fps) > 1 else None)
    if wl is not None:
        kw.update(a=wl.a, eta=wl.eta, dL=wl.dL, KB=wl.KB, KT=wl.KT, dt=wl.dt, tol=wl.tol,
                  max_iter=wl.max_iter, j0_model=J0_MODEL[case.get("model", "drag")])
    return fil.Filaments(segs, **kw)


def _perturbed_X(case, segs, base, g):
    """X = (Y_1, u, Lambda) near a straight state: small rotations, O(1) multipliers."""
    m, n = len(segs), segs[0]
    X = torch.cat([base + 0.05 * _randn(g, m, 3), 0.02 * _randn(g, m, 3 * n),
                   _randn(g, m, 3 * (n - 1))], 1)
    return X.reshape(-1).contiguous()


def _mlp_inputs(case, g, train):
    B = case["batch"]

    def f32(x):
        return x.to(torch.float32).contiguous()

    dims = [(fil.MLP_IN, 256), (256, 256), (256, 256), (256, fil.MLP_OUT)]
    params = f32(torch.cat([torch.cat([_randn(g, i * o) * math.sqrt(2.0 / i), 0.1 * _randn(g, o)])
                            for i, o in dims]))
    norm = [f32(0.1 * _randn(g, fil.MLP_IN)), f32(0.5 + _rand(g, fil.MLP_IN)),
            f32(0.1 * _randn(g, fil.MLP_OUT)), f32(0.5 + _rand(g, fil.MLP_OUT))]
    x = f32(norm[0] + norm[1] * _randn(g, B, fil.MLP_IN))
    target = f32(norm[2] + norm[3] * _randn(g, B, fil.MLP_OUT)) if train else None
    return params, norm, x, target


class _Network:
    """Owns one network handle."""

    def __init__(self, batch, params, norm):
        self.handle = fil.fil_mlp_create(batch)
        fil.fil_mlp_set_params(self.handle, params)
        fil.fil_mlp_set_norm(self.handle, *norm)

    def __del__(self):
        fil.fil_mlp_destroy(self.handle)


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    s = {"case": case}
    if kind in ("mlp_forward", "mlp_gradients"):
        params, norm, s["x"], s["target"] = _mlp_inputs(case, g, kind == "mlp_gradients")
        s["net"] = _Network(case["batch"], params, norm)
        s["out"] = (torch.empty(case["batch"], fil.MLP_OUT, device="cuda")
                    if kind == "mlp_forward" else torch.empty(fil.MLP_NPARAM, device="cuda"))
        return s
    fps, segs = _layout(case)
    S = sum(segs)
    if kind == "apply":
        s["Y"] = _walks(fps, segs, case["vf"], g)
        s["FT"] = _randn(g, S, 6)
        s["VW"] = torch.empty(S, 6, dtype=F64, device="cuda")
        s["m"] = _context(case, None, fps, segs)
        return s
    wl, base, t, mu, Fext, follower = _suspension(case, fps, segs, g)
    s["m"] = m = _context(case, wl, fps, segs)
    m.set_external(Fext, None, follower)
    if kind == "steps":
        m.set_j0_reuse(case["reuse"])
        m.set_broyden_memory(case["memory"])
        if case["adaptive"]:
            m.set_extrapolation(fil.FIL_EXTRAP_ADAPTIVE)
        xi = 1e-3 * _randn(g, S, 3)
        s["init"] = (base, t, mu, xi)
        s["state"] = {"Y": torch.empty(S, 3, dtype=F64, device="cuda"),
                      "q": torch.empty(S, 4, dtype=F64, device="cuda"),
                      "Yprev": torch.empty(S, 3, dtype=F64, device="cuda"),
                      "u": torch.empty(S, 3, dtype=F64, device="cuda"),
                      "Lambda": torch.empty(max(1, S - len(segs)), 3, dtype=F64, device="cuda")}
        return s
    m.init_straight(base, t, mu, None)
    if kind == "residual":
        if case["steric"]:
            m.set_steric(case["steric"])
        s["X"] = _perturbed_X(case, segs, base, g)
        s["f"] = torch.empty(6 * S, dtype=F64, device="cuda")
        return s
    m.broyden_begin()
    s["b"] = _randn(g, 6 * S)
    s["x"] = torch.empty(6 * S, dtype=F64, device="cuda")
    return s


def _kept(case, v):
    """Results in the type their form's accuracy fills."""
    return v if case["precision"] == "fp64" else v.to(torch.float32)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "apply":
        state["m"].mobility_apply(state["Y"], state["FT"], state["VW"])
        return _kept(case, state["VW"])
    if kind == "residual":
        norm = state["m"].residual(state["X"], state["f"])
        return {"f": _kept(case, state["f"]), "finf": norm}
    if kind == "j0_solve":
        state["m"].j0_solve(state["b"], state["x"])
        # FIL_PAIR32 solves J0 as FIL_FP64 does; FIL_MIXED in FP32
        return state["x"].to(torch.float32) if case["precision"] == "mixed" else state["x"]
    if kind == "steps":
        m, st = state["m"], state["state"]
        m.init_straight(*state["init"])
        for _ in range(case["steps"]):
            m.step()
        m.get_state(st["Y"], st["q"], st["Yprev"], st["u"], st["Lambda"])
        return {k: _kept(case, v) for k, v in st.items()}
    if kind == "mlp_forward":
        fil.fil_mlp_forward(state["net"].handle, state["x"], state["out"], case["batch"])
        return state["out"]
    loss = fil.fil_mlp_gradients(state["net"].handle, state["x"], state["target"], case["batch"],
                                 state["out"])
    return {"grad": state["out"], "loss": loss}


def work(case):
    kind = case["kind"]
    if kind in ("mlp_forward", "mlp_gradients"):
        B, P = case["batch"], fil.MLP_NPARAM
        if kind == "mlp_forward":
            return {"bytes": 4.0 * (B * (fil.MLP_IN + fil.MLP_OUT) + P), "flops": 2.0 * B * P}
        return {"bytes": 4.0 * (B * (fil.MLP_IN + fil.MLP_OUT) + 2 * P),
                "flops": 2.0 * B * (3 * P - 256 * fil.MLP_IN)}
    if "n_fil" in case:
        fils, segs = float(case["n_fil"]), (case["seg"] if "seg" in case else
                                            0.5 * (case["seg_lo"] + case["seg_hi"]))
        S, pairs = fils * segs, (fils * segs) ** 2
    else:
        lo, hi, ns = case["fil_lo"], case["fil_hi"], case["n_sys"]
        segs = 0.5 * (case["seg_lo"] + case["seg_hi"])
        S = ns * 0.5 * (lo + hi) * segs
        m2 = sum(m * m for m in range(lo, hi + 1)) / (hi - lo + 1)
        pairs = ns * m2 * segs * segs
    if kind == "apply":
        return {"bytes": 8.0 * 15 * S, "flops": PAIR_FLOPS * pairs}
    if kind == "residual":
        # X, Y^j, q^j, loads in; f out
        return {"bytes": 8.0 * (6 + 3 + 4 + 3 + 6) * S, "flops": PAIR_FLOPS * pairs}
    if kind == "j0_solve":
        if case["model"] == "rpy":       # one product with each filament's dense inverse
            return {"bytes": 4.0 * 36 * segs * S + 8.0 * 12 * S, "flops": 2.0 * 36 * segs * S}
        word = 4.0 if case["precision"] == "mixed" else 8.0
        return {"bytes": word * 25 * 6 * S + 8.0 * 12 * S, "flops": 2.0 * 24 * 6 * S}
    # a step evaluates f at its guess and at one further iterate at least
    return {"bytes": 8.0 * (9 + 16) * S + 8.0 * 26 * S * case["steps"],
            "flops": 2.0 * case["steps"] * PAIR_FLOPS * pairs}


# ---- the same results in plain 64-bit torch ------------------------------------

def _cross(a, b):
    return torch.linalg.cross(a, b, dim=-1)


def _rpy(Y, F, T, a=1.0, eta=1.0):
    """(V, Omega) of the equal-radius RPY tensors over all pairs of one system."""
    V, W = torch.empty_like(F), torch.empty_like(F)
    S = Y.shape[0]
    step = max(1, 8_000_000 // S)
    for i in range(0, S, step):
        d = Y[i:i + step, None] - Y[None]
        dx, dy, dz = d.unbind(-1)
        r2 = dx * dx + dy * dy + dz * dz
        r = r2.sqrt()
        ri = torch.where(r > 0, 1.0 / r, torch.zeros_like(r))
        far = r2 >= 4.0 * a * a
        i3 = ri * ri * ri
        i5 = i3 * ri * ri
        A = torch.where(far, ri + (2 * a * a / 3) * i3, 4 / (3 * a) * (1 - 9 * r / (32 * a)))
        B = torch.where(far, i3 - 2 * a * a * i5, ri / (8 * a * a))
        C = torch.where(far, -0.5 * i3,
                        (1 - 27 * r / (32 * a) + 5 * r * r2 / (64 * a ** 3)) / a ** 3)
        D = torch.where(far, 1.5 * i5, (9 * ri / (32 * a) - 3 * r / (64 * a ** 3)) / a ** 3)
        G = torch.where(far, i3, (1 - 3 * r / (8 * a)) / (2 * a ** 3))
        bF = B * (dx * F[:, 0] + dy * F[:, 1] + dz * F[:, 2])
        dT = D * (dx * T[:, 0] + dy * T[:, 1] + dz * T[:, 2])
        e = (G * dx, G * dy, G * dz)
        dd = (dx, dy, dz)
        for c in range(3):
            p, q = (c + 1) % 3, (c + 2) % 3
            V[i:i + step, c] = (A * F[:, c] + bF * dd[c] + (T[:, p] * e[q] - T[:, q] * e[p])).sum(1)
            W[i:i + step, c] = (C * T[:, c] + dT * dd[c] + (F[:, p] * e[q] - F[:, q] * e[p])).sum(1)
    k = 1.0 / (8.0 * math.pi * eta)
    return k * V, k * W


def _qmul(p, q):
    w = p[..., :1] * q[..., :1] - (p[..., 1:] * q[..., 1:]).sum(-1, keepdim=True)
    v = p[..., :1] * q[..., 1:] + q[..., :1] * p[..., 1:] + _cross(p[..., 1:], q[..., 1:])
    return torch.cat([w, v], -1)


def _qconj(q):
    return torch.cat([q[..., :1], -q[..., 1:]], -1)


def _qsqrt(p):
    s = torch.sqrt(2.0 * (p[..., :1] + 1.0))
    return torch.cat([(p[..., :1] + 1.0) / s, p[..., 1:] / s], -1)


def _qexp(u):
    x = u.norm(dim=-1, keepdim=True)
    f = 0.5 * torch.sinc(x / (2.0 * math.pi))
    return torch.cat([torch.cos(0.5 * x), f * u], -1)


def _rotate(q, v):
    t = 2.0 * _cross(q[..., 1:], v)
    return v + q[..., :1] * t + _cross(q[..., 1:], t)


def _exact_residual(case, seed):
    g = _gen(seed)
    fps, segs = _layout(case)
    wl, base, t, mu, Fext, follower = _suspension(case, fps, segs, g)
    X = _perturbed_X(case, segs, base, g)
    M, N = len(segs), segs[0]
    X = X.reshape(M, 2 * N, 3)
    Y1, u, lam = X[:, 0], X[:, 1:N + 1], X[:, N + 1:]
    # the frame (t, mu, t x mu) as a quaternion: e_x -> t, then about t onto mu
    zero = torch.zeros_like(t[:, :1])
    p1 = _qsqrt(torch.cat([t[:, :1], zero, -t[:, 2:], t[:, 1:2]], -1))
    ey = torch.tensor([0.0, 1.0, 0.0], dtype=F64, device="cuda").expand_as(t)
    n1 = _rotate(p1, ey)
    q0 = _qmul(_qsqrt(torch.cat([(n1 * mu).sum(-1, keepdim=True), _cross(n1, mu)], -1)), p1)
    q = _qmul(_qexp(u), q0[:, None].expand(M, N, 4))
    ex = torch.tensor([1.0, 0.0, 0.0], dtype=F64, device="cuda").expand(M, N, 3)
    tan = _rotate(q, ex)

    def arm(start, tang):
        inc = torch.cat([torch.zeros_like(tang[:, :1]), 0.5 * wl.dL * (tang[:, :-1] + tang[:, 1:])],
                        1)
        return start[:, None] + torch.cumsum(inc, 1)

    Y, Yj = arm(Y1, tan), arm(base, t[:, None].expand(M, N, 3))
    pad = torch.zeros(M, 1, 3, dtype=F64, device="cuda")
    right, left = torch.cat([lam, pad], 1), torch.cat([pad, lam], 1)
    qa, qb = q[:, :-1], q[:, 1:]
    qh = _qmul(_qsqrt(_qmul(qb, _qconj(qa))), qa)
    strain = 2.0 * _qmul(_qconj(qh), (qb - qa) / wl.dL)[..., 1:]
    mom = _rotate(qh, strain * torch.tensor([wl.KT, wl.KB, wl.KB], dtype=F64, device="cuda"))
    F = right - left + Fext.reshape(M, N, 3)
    F[:, -1] -= follower[:, None] * tan[:, -1]
    T = (torch.cat([mom, pad], 1) - torch.cat([pad, mom], 1)
         + 0.5 * wl.dL * _cross(tan, right + left))
    Yf, F, T = Y.reshape(-1, 3), F.reshape(-1, 3), T.reshape(-1, 3)
    if case["steric"]:
        chi, S = 1.1, Yf.shape[0]
        n = torch.arange(S, device="cuda")
        for i in range(0, S, 500):
            d = Yf[i:i + 500, None] - Yf[None]
            r2 = (d * d).sum(-1)
            hit = r2 < 4.0 * chi * chi
            near = (n[i:i + 500, None] - n[None]).abs() <= 1
            hit &= ~(near & (n[i:i + 500, None] // N == n[None] // N))
            x = torch.where(hit, (4 * chi * chi - r2) / (4 * (chi * chi - 1)), 0.0)
            F[i:i + 500] += (case["steric"] * x ** 4 / 2.0)[..., None].mul(d).sum(1)
    V, W = _rpy(Yf, F, T, wl.a, wl.eta)
    V, W = V.reshape(M, N, 3), W.reshape(M, N, 3)
    x = u.norm(dim=-1, keepdim=True)
    c = torch.where(x < 1e-2, -1 / 12 - x * x / 720 - x ** 4 / 30240,
                    (x / torch.tan(0.5 * x) - 2) / (2 * x * x))
    uW = _cross(u, W)
    pos = Y - Yj - wl.dt * V
    rot = u - wl.dt * (W - 0.5 * uW - c * _cross(u, uW))
    f = torch.cat([pos[:, :1], rot, pos[:, 1:]], 1).reshape(-1)
    return {"f": f, "finf": float(f.abs().max())}


def _exact_mlp(case, seed):
    params, norm, x, target = _mlp_inputs(case, _gen(seed), case["kind"] == "mlp_gradients")
    p = params.to(F64).requires_grad_(target is not None)
    in_mean, in_std, out_mean, out_std = (v.to(F64) for v in norm)
    h = (x.to(F64) - in_mean) / in_std
    at = 0
    dims = [(fil.MLP_IN, 256), (256, 256), (256, 256), (256, fil.MLP_OUT)]
    for k, (i, o) in enumerate(dims):
        h = h @ p[at:at + i * o].reshape(o, i).T + p[at + i * o:at + i * o + o]
        at += i * o + o
        if k < 3:
            h = torch.relu(h)
    if target is None:
        return out_mean + out_std * h
    loss = ((h - (target.to(F64) - out_mean) / out_std) ** 2).sum() / (2 * case["batch"])
    loss.backward()
    return {"grad": p.grad, "loss": float(loss.detach())}


def exact(case, seed):
    kind = case["kind"]
    if kind == "apply":
        fps, segs = _layout(case)
        g = _gen(seed)
        Y = _walks(fps, segs, case["vf"], g)
        FT = _randn(g, sum(segs), 6)
        out, f, s = [], 0, 0
        for m in fps:
            n = sum(segs[f:f + m])
            V, W = _rpy(Y[s:s + n], FT[s:s + n, :3], FT[s:s + n, 3:])
            out.append(torch.cat([V, W], 1))
            f, s = f + m, s + n
        return torch.cat(out)
    if kind == "residual":
        return _exact_residual(case, seed)
    if kind in ("mlp_forward", "mlp_gradients"):
        return _exact_mlp(case, seed)
    return None      # iterates and approximate-Jacobian solves: no direct formula
