"""Cases that stand for what a program does with this framework: force evaluations, cyclotronic
steps of one crystal, steps of an ensemble of crystals, and Metropolis-Hastings scans.

Each case is a dict of plain values; ``kind`` says which entry point it calls:

  forces    Plan.forces(pos, q): field and potential of n ions uniform in a sphere of density
            2e14 m^-3 with 1 % jitter (the single-evaluation sweep), automatic depth.
  step      Plan.step(state, trap, laser, dt, steps): a crystal at the rigid-rotor density in a
            spheroid of the given aspect, 10 mK rotating Maxwellian, with or without the cooling
            beams; returns the whole state after the call.
  ensemble  Ensemble.step + sync: independent cooled crystals of log-uniform ion count, each
            with its own plan; returns the state of all of them (one buffer per component).
  mh        mh_scans: Metropolis-Hastings scans of a crystal started on a jittered lattice;
            returns positions, accepted moves and the energy change.
"""
import math

import numpy as np
import torch

import paper_2405_13973_gb300 as pt

AMU, E_CHARGE, EPS0, K_B = 1.66053906660e-27, 1.602176634e-19, 8.8541878128e-12, 1.380649e-23
HBAR, K_E = 1.054571817e-34, 1.0 / (4.0 * math.pi * 8.8541878128e-12)
MASS, B_FIELD, OMEGA_Z, DELTA = 9.0 * AMU, 4.46, 2 * math.pi * 1.58e6, 0.01
GAMMA0, K_313, DT, DENSITY = 2 * math.pi * 18e6, 2 * math.pi / 313e-9, 1e-9, 2e14
TEMPERATURE, MH_DX = 10e-3, 1e-6


def listed():
    return [
        # the smallest request of the serving loop: launches and latency are all there is
        {"name": "step_bf16x3_300", "kind": "step", "precision": "bf16x3", "n": 300, "p": 12,
         "aspect": 0.7, "cooling": True, "steps": 10},
        # the plain FP64 method on the 1,000-ion spherical crystal, cooling off
        {"name": "step_fp64_1k", "kind": "step", "precision": "fp64", "n": 1000, "p": 8,
         "aspect": 1.0, "cooling": False, "steps": 10},
        # the cooled 10,000-ion spheroid at the order that meets the 1e-6 force error
        {"name": "step_bf16x3_10k", "kind": "step", "precision": "bf16x3", "n": 10000, "p": 12,
         "aspect": 0.3, "cooling": True, "steps": 10},
        # the same crystal on the FP64 path that the mixed one is measured against
        {"name": "step_fp64_10k", "kind": "step", "precision": "fp64", "n": 10000, "p": 12,
         "aspect": 0.3, "cooling": True, "steps": 2},
        # the 3xTF32 option, an odd ion count between the sizes of the sweep
        {"name": "step_tf32x3_23k", "kind": "step", "precision": "tf32x3", "n": 23457, "p": 10,
         "aspect": 0.5, "cooling": True, "steps": 10},
        # single evaluations of the sweep: FP64 at the middle size, FP64 at the largest
        {"name": "forces_fp64_1e5", "kind": "forces", "precision": "fp64", "n": 100000, "p": 12},
        {"name": "forces_fp64_1e6", "kind": "forces", "precision": "fp64", "n": 1000000, "p": 8},
        # FP32 on the CUDA cores
        {"name": "forces_fp32_1e5", "kind": "forces", "precision": "fp32", "n": 100003, "p": 12},
        # the tensor-core path at the middle and the largest size
        {"name": "forces_bf16x3_1e5", "kind": "forces", "precision": "bf16x3", "n": 100000, "p": 12},
        {"name": "forces_bf16x3_1e6", "kind": "forces", "precision": "bf16x3", "n": 1000000, "p": 12},
        # the batched ensemble: 256 crystals of 100 to 20,000 ions
        {"name": "ensemble_bf16x3_256", "kind": "ensemble", "precision": "bf16x3", "members": 256,
         "n_lo": 100, "n_hi": 20000, "p": 12, "steps": 1},
        # the Metropolis-Hastings initialisation of 1,000 ions
        {"name": "mh_fp64_1k", "kind": "mh", "n": 1000, "scans": 2},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    u = rng.random()
    if u < 0.45:
        precision = rng.choice(["fp64", "fp32", "bf16x3", "tf32x3"])
        p = rng.choice([4, 6, 8, 10, 12, 16] if precision in ("fp64", "fp32") else [6, 8, 10, 12])
        # FP64 sizes are bounded so that no draw outweighs the 1e6-ion evaluation at p = 8
        hi = min(1000000, int(1e6 * (9.0 / (p + 1)) ** 4)) if precision == "fp64" else 1000000
        return {"kind": "forces", "precision": precision, "n": _log_uniform(rng, 1000, hi), "p": p}
    if u < 0.80:
        precision = rng.choice(["fp64", "bf16x3", "bf16x3", "tf32x3", "fp32"])
        p = rng.choice([8, 10, 12])
        n = _log_uniform(rng, 200, 20000 if precision == "fp64" else 50000)
        return {"kind": "step", "precision": precision, "n": n, "p": p,
                "aspect": round(rng.uniform(0.1, 1.0), 3), "cooling": rng.random() < 0.7,
                "steps": 2 if precision == "fp64" and n > 3000 else 10}
    if u < 0.88:
        return {"kind": "ensemble", "precision": "bf16x3", "members": _log_uniform(rng, 4, 200),
                "n_lo": 100, "n_hi": _log_uniform(rng, 1000, 20000), "p": rng.choice([10, 12]),
                "steps": 1}
    return {"kind": "mh", "n": _log_uniform(rng, 200, 4000), "scans": rng.choice([1, 2])}


# ---- inputs -------------------------------------------------------------------------------
def _trap(aspect):
    """Trap whose rigid-rotor spheroid has the given aspect, and that spheroid's density."""
    a = float(aspect)
    if abs(a - 1.0) < 1e-12:
        nz = 1.0 / 3.0
    else:
        e = math.sqrt(1.0 - a * a)
        nz = (1.0 - a * math.asin(e) / e) / (e * e)
    beta, wc = (1.0 - nz) / (2.0 * nz), E_CHARGE * B_FIELD / MASS
    wr = 0.5 * (wc - math.sqrt(wc * wc - 4.0 * (beta + 0.5) * OMEGA_Z * OMEGA_Z))
    trap = {"B": B_FIELD, "omega_z": OMEGA_Z, "omega_r": wr, "delta": DELTA, "mass": MASS,
            "charge": E_CHARGE}
    return trap, 2.0 * EPS0 * MASS * wr * (wc - wr) / (E_CHARGE * E_CHARGE)


def _beams():
    """Two uniform axial beams and one planar beam along x."""
    return [{"s0": 5e-3, "detuning": -0.5 * GAMMA0, "k": (0.0, 0.0, K_313), "uniform": True},
            {"s0": 5e-3, "detuning": -0.5 * GAMMA0, "k": (0.0, 0.0, -K_313), "uniform": True},
            {"s0": 9e-3, "detuning": 2 * math.pi * 13.6e6, "k": (K_313, 0.0, 0.0),
             "uniform": False, "waist_y": 2.48e-6, "waist_z": 1e-3, "offset_d": 5e-6}]


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _ball(gen, n):
    """(3, n) points uniform in the unit ball."""
    v = torch.randn(3, n, generator=gen, device="cuda", dtype=torch.float64)
    r = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)
    return v / v.norm(dim=0) * r.pow(1.0 / 3.0)


def _sweep_positions(n, seed):
    gen = _generator(seed)
    a_ws = (3.0 / (4.0 * math.pi * DENSITY)) ** (1.0 / 3.0)
    jitter = torch.randn(3, n, generator=gen, device="cuda", dtype=torch.float64)
    return (_ball(gen, n) * (a_ws * n ** (1.0 / 3.0)) + jitter * (0.01 * a_ws)).contiguous()


def _crystal(gen, n, aspect):
    """Positions and velocities (6, n) of a crystal, and its trap."""
    trap, n0 = _trap(aspect)
    a_r = (3.0 * n / (4.0 * math.pi * n0 * aspect)) ** (1.0 / 3.0)
    x = _ball(gen, n) * torch.tensor([[a_r], [a_r], [aspect * a_r]], device="cuda", dtype=torch.float64)
    v = torch.randn(3, n, generator=gen, device="cuda", dtype=torch.float64)
    v *= math.sqrt(K_B * TEMPERATURE / MASS)
    v[0] += trap["omega_r"] * x[1]
    v[1] -= trap["omega_r"] * x[0]
    return torch.cat([x, v]), trap


def _members(case):
    """Ion counts and aspects: those of the case, whatever the seed."""
    m = case["members"]
    rng = np.random.default_rng([m, case["n_hi"]])
    ns = np.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), m)).astype(int)
    return [int(n) for n in ns], [float(a) for a in rng.uniform(0.1, 1.0, m)]


def _lattice(n, seed):
    """The n sites of a simple-cubic lattice nearest the origin at the spherical crystal's
    rigid-rotor density, each jittered by 5 % of the spacing."""
    trap, n0 = _trap(1.0)
    a = n0 ** (-1.0 / 3.0)
    m = int(math.ceil((3.0 * n / (4.0 * math.pi)) ** (1.0 / 3.0))) + 2
    g = np.arange(-m, m + 1, dtype=np.float64)
    pts = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    r = np.linalg.norm(pts, axis=1) + 1e-9 * (pts @ np.array([1.0, 1e-3, 1e-6]))
    pts = pts[np.argsort(r, kind="stable")[:n]]
    pts = (pts + np.random.default_rng(seed).normal(size=pts.shape) * 0.05) * a
    return np.ascontiguousarray(pts.T), trap


def _charges(n):
    return torch.full((n,), E_CHARGE, device="cuda", dtype=torch.float64)


def _state(buf, q):
    return pt.State(buf[0], buf[1], buf[2], buf[3], buf[4], buf[5], q)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "forces":
        plan = pt.Plan(case["n"], p=case["p"], precision=case["precision"])
        return {"kind": kind, "plan": plan, "pos": _sweep_positions(case["n"], seed),
                "q": _charges(case["n"])}
    if kind == "step":
        plan = pt.Plan(case["n"], p=case["p"], precision=case["precision"])
        buf, trap = _crystal(_generator(seed), case["n"], case["aspect"])
        laser = pt.make_laser(_beams(), seed=seed, gamma0=GAMMA0) if case["cooling"] else None
        return {"kind": kind, "plan": plan, "state": _state(buf, _charges(case["n"])), "buf": buf,
                "trap": trap, "laser": laser, "steps": case["steps"]}
    if kind == "ensemble":
        ns, aspects = _members(case)
        gen = _generator(seed)
        buf = torch.empty(6, sum(ns), device="cuda", dtype=torch.float64)
        plans, states, traps, lasers, at = [], [], [], [], 0
        for k, (n, a) in enumerate(zip(ns, aspects)):
            part = buf[:, at:at + n]
            xv, trap = _crystal(gen, n, a)
            part.copy_(xv)
            plans.append(pt.Plan(n, p=case["p"], precision=case["precision"]))
            states.append(_state(part, _charges(n)))
            traps.append(trap)
            lasers.append(pt.make_laser(_beams(), seed=seed + k, gamma0=GAMMA0))
            at += n
        return {"kind": kind, "ens": pt.Ensemble(plans), "states": states, "traps": traps,
                "lasers": lasers, "dts": [DT] * len(ns), "buf": buf, "steps": case["steps"]}
    pos, trap = _lattice(case["n"], seed)
    buf = torch.zeros(6, case["n"], device="cuda", dtype=torch.float64)
    buf[:3] = torch.from_numpy(pos).cuda()
    return {"kind": kind, "state": _state(buf, _charges(case["n"])), "buf": buf, "trap": trap,
            "seed": seed, "scan": 0, "scans": case["scans"]}


def run(state):
    kind = state["kind"]
    if kind == "forces":
        E, phi = state["plan"].forces(state["pos"], state["q"])
        return {"E": E, "phi": phi}
    if kind == "step":
        state["plan"].step(state["state"], state["trap"], state["laser"], DT, state["steps"])
        return {"pos": state["buf"][:3], "vel": state["buf"][3:]}
    if kind == "ensemble":
        state["ens"].step(state["states"], state["traps"], state["lasers"], state["dts"], state["steps"])
        state["ens"].sync()
        return {"pos": state["buf"][:3], "vel": state["buf"][3:]}
    accepted, de = pt.mh_scans(state["state"], state["trap"], TEMPERATURE, MH_DX, state["seed"],
                               state["scan"], state["scans"])
    state["scan"] += state["scans"]
    return {"pos": state["buf"][:3], "accepted": accepted, "de": de}


# ---- work ---------------------------------------------------------------------------------
def _field_flops(n, p):
    """The fast multipole method on n ions at about 12 ions a leaf: 20 flops per near pair, about
    130 translations a cell (8/7 cells per leaf) at the O(p^3) cost of the rotated form, and four
    expansions' worth of flops per ion for P2M and L2P."""
    leaf = 12.0
    shift = 2.0 * (2.0 * sum((2 * k + 1) ** 2 for k in range(p + 1)) + (p + 1) ** 3 * 2.0 / 3.0)
    near = 20.0 * n * min(n, 27.0 * leaf)
    far = 0.0 if n < 64 * leaf else (8.0 / 7.0) * n / leaf * 130.0 * shift + 8.0 * n * (p + 1) ** 2 * 4.0
    return near + far


def work(case):
    if case["kind"] == "forces":
        return {"bytes": 64.0 * case["n"], "flops": _field_flops(case["n"], case["p"])}
    if case["kind"] == "step":
        k = case["steps"]
        return {"bytes": 104.0 * case["n"], "flops": k * (_field_flops(case["n"], case["p"]) + 150.0 * case["n"])}
    if case["kind"] == "ensemble":
        span = math.log(case["n_hi"] / case["n_lo"])
        n = case["members"] * (case["n_hi"] - case["n_lo"]) / span  # the mean of the log-uniform counts
        one = _field_flops(n / case["members"], case["p"])
        return {"bytes": 104.0 * n, "flops": case["steps"] * (case["members"] * one + 150.0 * n)}
    n, scans = case["n"], case["scans"]
    return {"bytes": 56.0 * n, "flops": 24.0 * n * n * scans}


# ---- the same in 64 bits ------------------------------------------------------------------
def _direct(x, q, rows=1 << 27):
    """Coulomb field (3, n) and potential (n,) by the plain pair sum."""
    n = x.shape[1]
    E, phi = torch.empty_like(x), torch.empty_like(q)
    step = max(1, rows // n)
    for i in range(0, n, step):
        j = min(n, i + step)
        d = [x[a, i:j, None] - x[a, None, :] for a in range(3)]
        r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
        at = torch.arange(i, j, device=x.device)
        r2[at - i, at] = math.inf
        w = q[None, :] / r2.sqrt()
        phi[i:j] = K_E * w.sum(1)
        w /= r2
        for a in range(3):
            E[a, i:j] = K_E * (w * d[a]).sum(1)
    return E, phi


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on arrays of counters."""
    c = [np.asarray(v, dtype=np.uint64) for v in np.broadcast_arrays(c0, c1, c2, c3)]
    k0, k1, low = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF, np.uint64(0xFFFFFFFF)
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
        a, b = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(b >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), b & low,
             (a >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), a & low]
    return c


def _u01(a, b):
    return (((a >> np.uint64(5)) << np.uint64(26)) | (b >> np.uint64(6))).astype(np.float64) * 2.0 ** -53


def _disc(ion, field, step, seed, slot):
    """The disc pick that starts at `slot`: (v1, v2, s) and the slot after it."""
    for _ in range(64):
        w = _philox(ion, field | (slot << 8), step & 0xFFFFFFFF, step >> 32, seed)
        slot += 1
        v1, v2 = 2.0 * float(_u01(w[0], w[1])) - 1.0, 2.0 * float(_u01(w[2], w[3])) - 1.0
        s = v1 * v1 + v2 * v2
        if s < 1.0:
            break
    return v1, v2, s, slot


def _kicks(x, v, seed, step):
    """Recoil velocity change (3, n) of the cooling beams at the mid-step state (numpy)."""
    n, dv, rk = x.shape[1], np.zeros_like(v), HBAR / MASS
    ions = np.arange(n)
    for l, b in enumerate(_beams()):
        S = b["s0"] if b["uniform"] else b["s0"] * np.exp(
            -((x[1] - b["offset_d"]) ** 2 / b["waist_y"] ** 2 + x[2] ** 2 / b["waist_z"] ** 2))
        g2, det = (0.5 * GAMMA0) ** 2, b["detuning"] - sum(b["k"][a] * v[a] for a in range(3))
        lam = S * GAMMA0 * g2 / (g2 * (1.0 + 2.0 * S) + det * det) * DT
        w = _philox(ions, l, step & 0xFFFFFFFF, step >> 32, seed)
        u, prob = _u01(w[0], w[1]), np.exp(-lam)
        for i in np.nonzero(u >= prob)[0]:
            pr = F = float(prob[i])
            count = 0
            while u[i] >= F and count < 64:
                count += 1
                pr = pr * float(lam[i]) / count
                F += pr
            slot = 1
            dv[:, i] += count * rk * np.array(b["k"])
            for _ in range(count):
                v1, v2, s, slot = _disc(int(i), l, step, seed, slot)
                f = 2.0 * math.sqrt(1.0 - s)
                dv[:, i] += rk * math.sqrt(sum(k * k for k in b["k"])) * np.array([v1 * f, v2 * f, 1.0 - 2.0 * s])
    return dv


def _steps(xv, q, trap, cooling, seed, steps):
    """`steps` cyclotronic steps from t = 0 with the plain pair sum; (6, n) in and out."""
    x, v = xv[:3].clone(), xv[3:].clone()
    wc, wr = E_CHARGE * B_FIELD / MASS, trap["omega_r"]
    kz = MASS * OMEGA_Z ** 2 / E_CHARGE
    C, S = math.cos(0.5 * wc * DT), math.sin(0.5 * wc * DT)

    def drift():
        ux, uy = v[0].clone(), v[1].clone()
        x[0] += (ux * S + uy * (1.0 - C)) / wc
        x[1] += (uy * S - ux * (1.0 - C)) / wc
        x[2] += v[2] * (0.5 * DT)
        v[0], v[1] = ux * C + uy * S, uy * C - ux * S

    for k in range(steps):
        drift()
        E, _ = _direct(x, q)
        c, s = math.cos(2.0 * wr * (k * DT + 0.5 * DT)), math.sin(2.0 * wr * (k * DT + 0.5 * DT))
        kw = 0.5 * kz * DELTA
        E[0] += 0.5 * kz * x[0] - kw * (x[0] * c - x[1] * s)
        E[1] += 0.5 * kz * x[1] + kw * (x[1] * c + x[0] * s)
        E[2] -= kz * x[2]
        dv = torch.from_numpy(_kicks(x.cpu().numpy(), v.cpu().numpy(), seed, k)).to(x) if cooling else 0.0
        v += q / MASS * E * DT + dv
        drift()
    return {"pos": x, "vel": v}


def exact(case, seed):
    kind = case["kind"]
    if kind == "forces":
        if case["n"] > 150000:  # the pair sum takes minutes there
            return None
        E, phi = _direct(_sweep_positions(case["n"], seed), _charges(case["n"]))
        return {"E": E, "phi": phi}
    if kind == "step":
        xv, trap = _crystal(_generator(seed), case["n"], case["aspect"])
        return _steps(xv, _charges(case["n"]), trap, case["cooling"], seed, case["steps"])
    if kind == "ensemble":
        ns, aspects = _members(case)
        gen, out = _generator(seed), []
        for k, (n, a) in enumerate(zip(ns, aspects)):
            xv, trap = _crystal(gen, n, a)
            out.append(_steps(xv, _charges(n), trap, True, seed + k, case["steps"]))
        return {key: torch.cat([o[key] for o in out], 1) for key in ("pos", "vel")}
    x, trap = _lattice(case["n"], seed)
    wr, kz = trap["omega_r"], MASS * OMEGA_Z ** 2 / E_CHARGE

    def external(r):
        r2 = r[0] * r[0] + r[1] * r[1]
        return (0.25 * E_CHARGE * kz * (2.0 * r[2] * r[2] - r2)
                + 0.5 * (E_CHARGE * B_FIELD * wr - MASS * wr * wr) * r2
                + 0.25 * E_CHARGE * kz * DELTA * (r[0] * r[0] - r[1] * r[1]))

    accepted, total = 0, 0.0
    for scan in range(case["scans"]):
        for i in range(case["n"]):
            w = _philox(i, 0xFF, scan, 0, seed)
            v1, v2, s, _ = _disc(i, 0xFF, scan, seed, 1)
            f, r = 2.0 * math.sqrt(1.0 - s), MH_DX * float(_u01(w[0], w[1]))
            a = x[:, i].copy()
            b = a + r * np.array([v1 * f, v2 * f, 1.0 - 2.0 * s])
            far = [np.sqrt(((x - p[:, None]) ** 2).sum(0)) for p in (b, a)]
            far[0][i] = far[1][i] = math.inf
            de = external(b) - external(a) + K_E * E_CHARGE * E_CHARGE * float((1.0 / far[0] - 1.0 / far[1]).sum())
            if de < 0.0 or float(_u01(w[2], w[3])) < math.exp(min(0.0, -de / (K_B * TEMPERATURE))):
                x[:, i] = b
                accepted += 1
                total += de
    return {"pos": torch.from_numpy(x).cuda(), "accepted": accepted, "de": total}
