"""Performance cases: what programs have this library do, through its public entry points.

One pass of a case is what a program does per energy grid: hand over the incident energies (host), solve
every (partial wave, energy) pair and read the collision strengths Omega back into page-locked host memory
(and, where K-matrices are asked for, leave them on the device). Loading the pole sets belongs to
prepare(): a program loads a partial wave once and solves many grids against it.

A case is a dict of plain values:
  call      "solve"  rm_solve_energies + rm_collision_strengths on one wave
            "qdt"    rm_solve_energies_qdt (coarse-mesh interpolation) on one wave
            "prop"   as "solve", on a wave propagated through the outer region (rm_set_multipoles)
            "batch"  rm_solve_batch over several waves of one target (lanes, captured graph)
            "lanes"  one request per lane (rm_lane_solve_energies), read back lane by lane
  precision "fp64" (the library's default), "bf16x3" or "tf32x3" (tensor-core formation, FP32 solve)
  mode      "direct" or "mqdt"
  channels, poles (per channel), energies, z, and per call: waves, steps, spacing, k (K-matrices out)
"""
import math

import numpy as np
import torch

from paper_1909_07321_gb300 import rmgb

# Energy range, radius, pole range, amplitude and threshold range of the waves,
# by size: the repository's 4-channel, 64-channel and 1000-channel workloads.
FLAVOURS = ((16, dict(a=20.0, poles=(-1.0, 40.0), sigma=0.1, thr=1.5, emax=3.0, per_level=1, lmax=4)),
            (96, dict(a=15.0, poles=(-2.0, 60.0), sigma=0.05, thr=2.0, emax=2.5, per_level=1, lmax=8)),
            (1 << 20, dict(a=20.0, poles=(-5.0, 200.0), sigma=0.03, thr=6.0, emax=8.0, per_level=4, lmax=8)))
PRECISION = {"fp64": dict(precision=rmgb.RM_FP64, solve_precision=rmgb.RM_FP64),
             "bf16x3": dict(precision=rmgb.RM_BF16X3, solve_precision=rmgb.RM_FP32),
             "tf32x3": dict(precision=rmgb.RM_FP32, solve_precision=rmgb.RM_FP32)}
MODE = {"direct": rmgb.RM_DIRECT, "mqdt": rmgb.RM_MQDT}


def listed():
    def c(name, call, precision, mode, channels, poles, energies, z=2, **more):
        return dict(name=name, call=call, precision=precision, mode=mode, channels=channels, poles=poles,
                    energies=energies, z=z, **more)

    return [
        # a handful of energies of a light ion, K-matrices wanted: call latency
        c("few-energies-4ch", "solve", "fp64", "direct", 4, 20, 16, z=1, k=True),
        # the 4-channel workload as it is shipped: FP64, K and Omega
        c("small-4ch", "solve", "fp64", "direct", 4, 20, 2000, z=1, k=True),
        # one partial wave of a mid-size ion, a whole fine mesh: the benchmark's workload
        c("ion-64ch", "solve", "bf16x3", "direct", 64, 30, 20000),
        # the same wave through the default FP64 path, the reference other results are checked against
        c("ion-64ch-fp64", "solve", "fp64", "direct", 64, 30, 4000),
        # the same wave by quantum-defect theory at every energy
        c("ion-64ch-mqdt", "solve", "bf16x3", "mqdt", 64, 30, 4000),
        # ... and with the quantum-defect solve on a coarse mesh only, interpolated onto a fine one
        c("interpolated-64ch", "qdt", "bf16x3", "mqdt", 64, 30, 8000, spacing=25),
        # a neutral target (no Coulomb tables), odd sizes
        c("neutral-41ch", "solve", "bf16x3", "direct", 41, 27, 1777, z=0),
        # a mid-size target in FP64 by quantum-defect theory: too wide for the shared-memory solver
        c("wide-132ch-fp64", "solve", "fp64", "mqdt", 132, 30, 200),
        # long-range dipole and quadrupole couplings, propagated through the outer region
        c("multipole-32ch", "prop", "fp64", "direct", 32, 30, 304, steps=600),
        # the partial waves of one target on one grid, as one batch
        c("batch-5waves", "batch", "bf16x3", "direct", 203, 30, 500, z=3, waves=5),
        # requests of a served mix, one per lane, half by quantum-defect theory
        c("served-3requests", "lanes", "bf16x3", "mqdt", 431, 28, 512, waves=3),
        # the widest target: 1000 channels and 30000 poles
        c("wide-1000ch", "solve", "bf16x3", "direct", 1000, 30, 256),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    call = rng.choice(["solve", "solve", "solve", "solve", "solve", "qdt", "prop", "batch", "lanes"])
    z = rng.choice([1, 2, 2, 3])
    poles = rng.randint(20, 35)
    mode = rng.choice(["direct", "mqdt"])
    mixed = rng.choice(["bf16x3", "bf16x3", "tf32x3"])
    if call == "prop":
        return dict(call=call, precision="fp64", mode=mode, channels=rng.randint(5, 40), poles=poles,
                    energies=log(16, 200), z=z, steps=rng.randint(200, 600))
    if call == "qdt":
        return dict(call=call, precision=mixed, mode="mqdt", channels=rng.randint(8, 80), poles=poles,
                    energies=log(500, 8000), z=z, spacing=rng.randint(8, 40))
    if call in ("batch", "lanes"):
        n = log(40, 300)
        return dict(call=call, precision=mixed, mode="direct" if call == "batch" else mode, channels=n,
                    poles=poles, energies=min(log(64, 2000), max(64, int(5e9 / n ** 3))), z=z,
                    waves=rng.randint(2, 5))
    if rng.random() < 0.4:
        n = log(3, 160)
        return dict(call=call, precision="fp64", mode=mode, channels=n, poles=poles,
                    energies=min(log(8, 4000), max(8, int(1e9 / n ** 3))), z=z, k=n < 16)
    n = log(8, 900)
    z = rng.choice([0, 1, 2, 2, 3])
    return dict(call=call, precision=mixed, mode=mode if z else "direct", channels=n, poles=poles,
                energies=min(log(64, 20000), max(32, int(1.5e10 / n ** 3))), z=z, k=n < 16)


# ---- inputs -----------------------------------------------------------------

def _sizes(case):
    """Channel counts of the case's waves (the largest first named, the others smaller)."""
    n, m = case["channels"], case.get("waves", 1)
    return [max(3, int(round(n * (0.3 + 0.7 * (w + 1) / m))) if m > 1 else n) for w in range(m)]


def _flavour(n):
    return next(f for top, f in FLAVOURS if n <= top)


def _wave(rng, n, case, f):
    """One partial wave: poles jittered on a grid, Gaussian amplitudes, `per_level` channels a level."""
    N = n * case["poles"]
    lo, hi = f["poles"]
    h = (hi - lo) / N
    E_k = np.sort(lo + (np.arange(N) + 0.5 + rng.uniform(-0.1, 0.1, N)) * h)
    W = rng.standard_normal((n, N))
    W *= f["sigma"]
    levels = -(-_sizes(case)[-1] // f["per_level"])
    level = np.arange(n, dtype=np.int32) // f["per_level"]
    l = np.concatenate([rng.permutation(f["lmax"] + 1)[:f["per_level"]] for _ in range(level[-1] + 1)])[:n]
    return dict(E_k=E_k, W=W, a=f["a"], b=0.0, e_thr=np.linspace(0.0, f["thr"], levels)[level],
                l=l.astype(np.int32), z=float(case["z"]), level=level, n_levels=levels,
                g=float(rng.integers(1, 9)) / 2)


def _inputs(case, seed):
    rng = np.random.default_rng(seed)
    f = _flavour(_sizes(case)[-1])
    waves = [_wave(rng, n, case, f) for n in _sizes(case)]
    m, lo = case["energies"], 0.01
    E = lo + (np.arange(m) + rng.uniform(0.25, 0.75)) * ((f["emax"] - lo) / m)
    couplings = None
    if case["call"] == "prop":
        n = case["channels"]
        couplings = rng.normal(0.0, 0.3, (2, n, n))
        couplings = 0.5 * (couplings + couplings.transpose(0, 2, 1))
    return waves, E, couplings


def prepare(case, seed):
    waves, E, couplings = _inputs(case, seed)
    call, m = case["call"], case["energies"]
    more = dict(lanes=len(waves), mem_budget=8 << 30) if call in ("batch", "lanes") else {}
    ctx = rmgb.Context(**PRECISION[case["precision"]], **more)
    for w, wave in enumerate(waves):
        ctx.load_pw(w, wave)
    if couplings is not None:
        a = waves[0]["a"]
        ctx.set_multipoles(0, couplings, a + 10.0, case["steps"])
    tri = waves[0]["n_levels"] * (waves[0]["n_levels"] + 1) // 2
    reads = len(waves) if call == "lanes" else 1
    state = dict(case=case, ctx=ctx, E=E, waves=len(waves),
                 omega=[torch.empty((m, tri), dtype=torch.float64, pin_memory=True).numpy() for _ in range(reads)])
    if call not in ("batch", "lanes"):
        n = case["channels"]
        state["n_open"] = torch.zeros(m, dtype=torch.int32, device="cuda")
        state["status"] = torch.zeros(m, dtype=torch.int32, device="cuda")
        state["K"] = torch.zeros((m, n, n), dtype=torch.float64, device="cuda") if case.get("k") else None
    return state


def run(state):
    case, ctx, E, omega = state["case"], state["ctx"], state["E"], state["omega"]
    mode = MODE[case["mode"]]
    if case["call"] == "batch":
        ctx.solve_batch(list(range(state["waves"])), E, mode)
        ctx.collision_strengths(omega[0], reset=True)
        return {"omega": omega[0]}
    if case["call"] == "lanes":
        for w in range(state["waves"]):
            ctx.lane_solve_energies(w, w, E, mode if w % 2 == 0 else rmgb.RM_DIRECT)
        for w in range(state["waves"]):
            ctx.lane_collision_strengths(w, omega[w], reset=True)
        return {"omega": list(omega)}
    if case["call"] == "qdt":
        ctx.solve_energies_qdt(0, E, -case["spacing"], n_open_out=state["n_open"], status_out=state["status"])
    else:
        ctx.solve_energies(0, E, mode, K_out=state["K"], n_open_out=state["n_open"], status_out=state["status"])
    ctx.collision_strengths(omega[0], reset=True)
    out = {"omega": omega[0], "n_open": state["n_open"], "status": state["status"]}
    if state["K"] is not None:
        out["K"] = state["K"]
    return out


def work(case):
    """Bytes: amplitudes, poles, energies in; Omega (and K) out. Flops: per energy the upper triangle of R
    (n(n+1)N), the matching solve (2/3 n^3 + n^2 n_o + n_o^2 n), the T step (4 n_o^3), with n_o averaged over
    the grid; interpolation solves its nodes and eliminates at the fine energies; propagation 4 n^3 a step."""
    m = case["energies"]
    f = _flavour(_sizes(case)[-1])
    levels = -(-_sizes(case)[-1] // f["per_level"])
    open_share = 1.0 - 0.5 * f["thr"] / f["emax"]
    reads = case.get("waves", 1) if case["call"] == "lanes" else 1
    b = 8.0 * m * (1 + reads * levels * (levels + 1) / 2)
    fl = 0.0
    for n in _sizes(case):
        N, no = n * case["poles"], open_share * n
        b += 8.0 * (n + 1) * N + (8.0 * m * n * n if case.get("k") else 0.0)
        solves = m / case["spacing"] if case["call"] == "qdt" else m
        fl += solves * (n * (n + 1.0) * N + 2.0 / 3.0 * n ** 3 + n * n * no + no * no * n)
        fl += m * 4.0 * no ** 3
        if case["call"] == "prop":
            fl += m * case["steps"] * 4.0 * n ** 3
    return {"bytes": b, "flops": fl}


# ---- the same results in plain 64-bit torch -------------------------------------

def _open_pairs(l, eta, rho):
    """F, F', G, G' (derivatives in rho) of the Coulomb wave equation, elementwise: Steed's method. F'/F by
    its continued fraction in l, H+'/H+ by its own at l = 0, G carried up to l, F_l from the Wronskian."""
    def cf1(L0, depth):
        v, s = torch.zeros_like(rho), torch.ones_like(rho)
        for j in range(depth, -1, -1):
            L1, L2 = L0 + j + 1.0, L0 + j + 2.0
            v = torch.sqrt(1 + (eta / L1) ** 2) / (L1 / rho + eta / L1 + L2 / rho + eta / L2
                                                   - torch.sqrt(1 + (eta / L2) ** 2) * v)
            s = torch.where(v < 0, -s, s)
        L1 = L0 + 1.0
        return L1 / rho + eta / L1 - torch.sqrt(1 + (eta / L1) ** 2) * v, s

    depth = 128 + 2 * int(rho.max())
    fl, sl = cf1(l, depth)
    f0, s0 = cf1(torch.zeros_like(l), depth)
    v = _fraction(lambda j, eta, rho: (j + 1j * eta) * (j - 1 + 1j * eta),
                  lambda j, eta, rho: 2 * (rho - eta) + 2j * j, (eta, rho), 128)
    p, q = -v.imag / rho, 1.0 - eta / rho + v.real / rho
    F0 = s0 * torch.sqrt(q / ((f0 - p) ** 2 + q * q))
    G = (f0 - p) * F0 / q
    Gp = p * G - q * F0
    for L in range(1, int(l.max()) + 1):
        S, R = L / rho + eta / L, torch.sqrt(1 + (eta / L) ** 2)
        up = (S * G - Gp) / R
        G, Gp = torch.where(l >= L, up, G), torch.where(l >= L, R * G - S * up, Gp)
    F = 1.0 / (fl * G - Gp)
    return F, fl * F, G, Gp


def _closed_slope(l, nu, x):
    """d/dx ln W_{nu, l+1/2}(x), elementwise: from the recurrence of Kummer's U in its first argument at a
    low l (no centrifugal barrier), carried to l by the Coulomb ladder operator."""
    ls = torch.where(nu <= l + 0.5, torch.minimum(torch.clamp(torch.ceil(nu - 0.5), min=0.0), l), torch.zeros_like(l))
    r = _fraction(lambda j, nu, x, ls: -((j > 1) * ((ls - nu + j) * (j - nu - ls - 1.0) - 1.0) + 1.0),
                  lambda j, nu, x, ls: 2.0 * (nu - j) - x, (nu, x, ls), 256)
    al = ls + 1.0 - nu
    y = -0.5 + (ls + 1.0) / x - (al / x) * (1.0 + (ls + nu) * r)
    for L in range(int(l.max())):
        T, c = (L + 1.0) / x - nu / (2.0 * (L + 1.0)), -0.25 + nu * nu / (4.0 * (L + 1.0) ** 2)
        y = torch.where((ls <= L) & (L < l), c / (T - y) - T, y)
    return y


def _fraction(a, b, args, depth):
    """a(1)/(b(1) + a(2)/(b(2) + ...)), elementwise and bottom-up, the depth doubled for each element until
    two doublings agree (near a threshold that takes 1e5 terms: the few such elements go through numpy)."""
    def at(depth, args):
        if args[0].numel() > 2048 or depth < 1024:
            v = 0.0
            for j in range(depth, 0, -1):
                v = a(j, *args) / (b(j, *args) + v)
            return v
        host = [t.cpu().numpy()[None, :] for t in args]
        v = 0.0
        for top in range(depth, 0, -1024):
            j = np.arange(top, max(0, top - 1024), -1, dtype=np.float64)[:, None]
            for num, den in zip(a(j, *host), b(j, *host)):
                v = num / (den + v)
        return torch.as_tensor(v, device=args[0].device)

    out = at(depth, args)
    idx = torch.arange(out.numel(), device=out.device)
    quiet = torch.zeros_like(idx)
    while idx.numel() and depth < 1 << 18:
        depth *= 2
        new = at(depth, [t[idx] for t in args])
        same = (new - out[idx]).abs() <= 1e-14 * new.abs()
        out[idx] = new
        quiet = torch.where(same, quiet + 1, torch.zeros_like(quiet))
        idx, quiet = idx[quiet < 2], quiet[quiet < 2]
    return out


def _exact_wave(pw, E, dev):
    """K (closed rows and columns zero) and |T|^2 by level of one wave in direct mode (the quantum-defect
    elimination gives the same physical K): R by its sum, matching and T by LU, all in 64 bits."""
    n, a = pw["e_thr"].size, pw["a"]
    t = lambda v: torch.as_tensor(np.asarray(v, dtype=np.float64), device=dev)  # noqa: E731
    W, Ek, l, e = t(pw["W"]), t(pw["E_k"]), t(pw["l"]), t(E)
    eps = e[:, None] - t(pw["e_thr"])[None, :]
    lb = l[None, :].expand_as(eps)
    op = eps > 0
    s, sp, g, gp = (torch.zeros_like(eps) for _ in range(4))
    if op.any():
        k = torch.sqrt(eps[op])
        F, Fp, G, Gp = _open_pairs(lb[op], -pw["z"] / k, k * a)
        s[op], sp[op], g[op], gp[op] = F / k.sqrt(), Fp * k.sqrt(), G / k.sqrt(), Gp * k.sqrt()
    if (~op).any():
        kap = torch.sqrt(-eps[~op])
        L = 2 * kap * _closed_slope(lb[~op], pw["z"] / kap, 2 * kap * a)
        nrm = 1.0 / torch.sqrt(1.0 + (a * L) ** 2)
        g[~op], gp[~op] = nrm, L * nrm
    eye = torch.eye(n, dtype=torch.float64, device=dev)
    lev = torch.zeros((n, pw["n_levels"]), dtype=torch.float64, device=dev)
    lev[torch.arange(n, device=dev), torch.as_tensor(pw["level"], device=dev, dtype=torch.long)] = 1.0
    up = torch.triu_indices(pw["n_levels"], pw["n_levels"], device=dev)
    Ks, rows = [], []
    step = max(1, min(512, int(2e9 / (8.0 * n * Ek.numel()))))
    for i in range(0, E.size, step):
        b = slice(i, i + step)
        R = (W[None] * (1.0 / (Ek[None, :] - e[b, None]))[:, None, :]) @ W.T / (2.0 * a)
        A = eye * g[b, None, :] - R * (a * gp[b])[:, None, :]
        B = (R * (a * sp[b])[:, None, :] - eye * s[b, None, :]) * op[b, None, :]
        K = torch.linalg.solve(A, B) * op[b, :, None] * op[b, None, :]
        T = 2j * K @ torch.linalg.inv(eye - 1j * K)
        rows.append(pw["g"] * (lev.T @ (T.abs() ** 2) @ lev)[:, up[0], up[1]])
        Ks.append(K)
    return torch.cat(Ks), torch.cat(rows)


def exact(case, seed):
    """None for interpolated and propagated results (approximations of their own) and beyond some seconds of
    64-bit arithmetic."""
    if case["call"] in ("qdt", "prop") or work(case)["flops"] > 4e12:
        return None
    waves, E, _ = _inputs(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    got = [_exact_wave(pw, E, dev) for pw in waves]
    if case["call"] == "lanes":
        return {"omega": [o for _, o in got]}
    out = {"omega": sum(o for _, o in got)}
    if case.get("k"):
        out["K"] = got[0][0]
    return out
