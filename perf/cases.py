"""The workloads that the timestep library's speed is measured on.

Each case is work that a program using the library has it do, through its
Python entry points: advancing clusters from a checkpoint (``Cluster``), the
diagnostics taken between steps, and the single-step calls on device arrays
(``stage_*``).  Sizes come from the repository's own workloads: Plummer
spheres of 10^4 to 10^7 stars, equal or Salpeter masses, ensembles of
clusters of 10^4 to 2 10^5 stars; the smallest and the odd sizes are those of
its tests.

A pass of a stepping case sets the cluster back to its checkpoint (as a
program does that resumes a run or starts a member of a parameter study),
advances it a few timesteps and reads the new state into device arrays.
Starting every pass from the same state keeps the model in the regime its
inputs describe, however many passes are timed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1206_5878_gb300 as cmc

A_PLUMMER = 3.0 * math.pi / 16.0  # Plummer scale in Henon units (E = -1/4)
FRACTIONS = (0.01, 0.05, 0.1, 0.25, 0.5, 0.75, 0.9)
KEYS = ("r", "vr", "vt", "m", "id")


# ------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest clusters anybody advances (the size of brute-force
        # checks): nothing but launches and latencies
        _step("step_1021_mixed", 1021, 10, "mixed"),
        # the smallest named workload: 10^4 equal masses, FP64, ten steps
        _step("step_1e4_fp64", 10_000, 10, "fp64"),
        # 10^5 stars, mixed: the size long runs to core collapse are made at
        _step("step_1e5_mixed", 100_000, 10, "mixed"),
        # 10^6 stars with a Salpeter mass spectrum, mixed
        _step("step_1e6_salpeter_mixed", 1_000_000, 4, "mixed", masses="salpeter"),
        # 64 independent clusters of uneven size advanced together
        _step("ensemble64_mixed", 10_000, 4, "mixed", clusters=64, nmax=200_000),
        # the headline: 10^7 stars, mixed
        _step("step_1e7_mixed", 10_000_000, 4, "mixed"),
        # the same step in FP64 throughout
        _step("step_1e7_fp64", 10_000_000, 3, "fp64"),
        # stars with radii and binaries: collisions and the binary timesteps
        # on, a ragged size, a mass spectrum
        _step("step_physics_200003_fp64", 200_003, 2, "fp64", masses="salpeter", physics=True),
        # the diagnostics between steps: energies, Lagrangian radii, core
        {"name": "diagnose_1e6", "kind": "diagnose", "n": 1_000_000, "masses": "salpeter"},
        # the single-step calls on a program's own device arrays
        {"name": "sort_999983", "kind": "sort", "n": 999_983},
        {"name": "potential_4000037", "kind": "potential", "n": 4_000_037, "masses": "salpeter"},
        {"name": "orbit_100003_fp64", "kind": "orbit", "n": 100_003, "precision": "fp64"},
    ]


def _step(name, n, steps, precision, masses="equal", clusters=1, nmax=0, physics=False):
    c = {"kind": "step", "n": n, "steps": steps, "precision": precision, "masses": masses,
         "clusters": clusters, "nmax": nmax, "physics": physics}
    if name:
        c["name"] = name
    return c


def _log_uniform(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi], any residue."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("step", "step", "step", "step", "ensemble", "ensemble", "diagnose",
                       "sort", "potential", "orbit"))
    masses = rng.choice(("equal", "salpeter"))
    precision = rng.choice(("mixed", "mixed", "fp64"))
    if kind == "step":
        n = _log_uniform(rng, 1000, 8_000_000)
        budget = 30_000_000 if precision == "mixed" else 20_000_000
        few = precision == "fp64" and n < 150_000 and rng.random() < 0.5
        steps = max(1, min(rng.randint(1, 3) if few else rng.randint(2, 10), budget // n))
        return _step(None, n, steps, precision, masses, physics=n < 500_000 and rng.random() < 0.25)
    if kind == "ensemble":
        nmax = _log_uniform(rng, 20_000, 200_000)
        clusters = rng.randint(2, 64)
        return _step(None, rng.randint(1000, nmax), rng.randint(1, 4), precision, masses, clusters,
                     nmax)
    if kind == "diagnose":
        return {"kind": kind, "n": _log_uniform(rng, 10_000, 8_000_000), "masses": "salpeter"}
    if kind == "sort":
        return {"kind": kind, "n": _log_uniform(rng, 1000, 8_000_000)}
    if kind == "potential":
        return {"kind": kind, "n": _log_uniform(rng, 1000, 8_000_000), "masses": masses}
    return {"kind": kind, "n": _log_uniform(rng, 1000, 1_000_000), "precision": precision}


def _sizes(case):
    """Stars per cluster: one size, or sizes spread over [n, nmax]."""
    if case["clusters"] == 1:
        return [case["n"]]
    golden = 0.6180339887498949
    return [case["n"] + int(((c + 1) * golden) % 1.0 * (case["nmax"] - case["n"] + 1))
            for c in range(case["clusters"])]


# ----------------------------------------------------------------- inputs
def _plummer(n, seed, masses, device):
    """A Plummer sphere in Henon units (G = M = 1): radii from the enclosed
    mass, speeds v = q v_esc with q^2 ~ Beta(3/2, 9/2) (the distribution
    q^2 (1 - q^2)^(7/2)), isotropic directions; unsorted."""
    g = torch.Generator(device=device)
    g.manual_seed(seed)

    def u():
        return 1.0 - torch.rand(n, generator=g, device=device, dtype=torch.float64)

    def z():
        return torch.randn(n, generator=g, device=device, dtype=torch.float64)

    X = torch.clamp(u(), 1e-12, 1.0 - 1e-12)
    r = A_PLUMMER / torch.sqrt(X ** (-2.0 / 3.0) - 1.0)
    g1 = -torch.log(u()) + 0.5 * z() ** 2
    g2 = -torch.log(u() * u() * u() * u()) + 0.5 * z() ** 2
    q = torch.sqrt(g1 / (g1 + g2))
    v = q * (math.sqrt(2.0 / A_PLUMMER) * (1.0 + (r / A_PLUMMER) ** 2) ** -0.25)
    ct = 2.0 * u() - 1.0
    d = {"r": r, "vr": v * ct, "vt": v * torch.sqrt(torch.clamp(1.0 - ct * ct, min=0.0))}
    if masses == "salpeter":  # dN/dm ~ m^-2.35 on [0.1, 100]
        e, lo, hi = -1.35, 0.1 ** -1.35, 100.0 ** -1.35
        m = (lo + u() * (hi - lo)) ** (1.0 / e)
        # (a fixed order of summation: the same masses on every run)
        d["m"] = m / float(np.sum(m.cpu().numpy()))
    else:
        d["m"] = torch.full((n,), 1.0 / n, dtype=torch.float64, device=device)
    d["id"] = torch.arange(n, dtype=torch.int32, device=device)
    return d


def _clusters(case, seed, device):
    parts = [_plummer(nc, 1000 * seed + c, case["masses"], device)
             for c, nc in enumerate(_sizes(case))]
    return {k: torch.cat([p[k] for p in parts]) if len(parts) > 1 else parts[0][k] for k in KEYS}


def _sorted(d):
    p = torch.argsort(d["r"], stable=True)
    return {k: v[p].contiguous() for k, v in d.items()}


def _attributes(case, n, seed):
    """Stellar radii and semi-major axes by star id (every tenth a binary)."""
    ids = np.arange(n)
    R = 2e-5 * (1.0 + (ids * 7 + seed) % 11 / 10.0)
    A = np.where(ids % 10 == 3, 1e-4 * (1.0 + (ids + seed) % 7 / 6.0), 0.0)
    return R, A


def _phi_host(r, m):
    """Henon's shell potential (Eqs. 1-5) of sorted host arrays."""
    x = 1.0 / r
    mx = m * x
    return -(np.cumsum(m) * x + (np.cumsum(mx[::-1])[::-1] - mx))


def _orbit_inputs(case, seed):
    d = {k: v.cpu().numpy() for k, v in _sorted(_plummer(case["n"], seed, "equal", "cuda")).items()}
    d["phi"] = _phi_host(d["r"], d["m"])
    return d


PRECISION = {"fp64": 0, "mixed": 1}


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("step", "diagnose"):
        whole = dict(case)
        whole.setdefault("clusters", 1)
        sizes = _sizes(whole)
        d = _clusters(whole, seed, "cuda")
        cfg = {"precision": PRECISION[case.get("precision", "mixed")]}
        if case.get("physics"):
            cfg.update(collisions=1, binaries=1)
        c = cmc.Cluster(d, [1000 * seed + k for k in range(len(sizes))], sizes=sizes, **cfg)
        n = sum(sizes)
        if kind == "diagnose":
            return {"case": case, "cluster": c}

        def arrays():
            a = {k: torch.empty(n, dtype=torch.float64, device="cuda")
                 for k in ("r", "vr", "vt", "m", "phi")}
            a["id"] = torch.empty(n, dtype=torch.int32, device="cuda")
            return a

        checkpoint = c.get_state(arrays())
        s = {"case": case, "cluster": c, "checkpoint": checkpoint, "out": arrays()}
        if case.get("physics"):
            by_id = checkpoint["id"].cpu().numpy()
            s["radii"], s["axes"] = (a[by_id] for a in _attributes(case, n, seed))
        return s
    if kind == "sort":
        d = _plummer(case["n"], seed, "equal", "cuda")
        return {"case": case, "r": d["r"], "id": d["id"]}
    if kind == "potential":
        d = _sorted(_plummer(case["n"], seed, case["masses"], "cuda"))
        return {"case": case, "r": d["r"], "m": d["m"]}
    d = _orbit_inputs(case, seed)
    return {"case": case, "seed": 1000 * seed, "precision": PRECISION[case["precision"]],
            **{k: torch.from_numpy(d[k]).cuda() for k in ("r", "phi", "vr", "vt", "id")}}


def run(state):
    kind = state["case"]["kind"]
    if kind == "step":
        c = state["cluster"]
        c.set_state(state["checkpoint"], 0)
        if "radii" in state:
            c.set_radii(state["radii"])
            c.set_binaries(state["axes"])
        c.step(state["case"]["steps"])
        return c.get_state(state["out"])
    if kind == "diagnose":
        c = state["cluster"]
        return {"energy": c.energy(), "lagrange": c.lagrange_radii(FRACTIONS), "core": c.core(),
                "escaped": c.escaped()}
    if kind == "sort":
        return cmc.stage_sort_radius(state["r"], state["id"])
    if kind == "potential":
        return cmc.stage_potential(state["r"], state["m"], want_M=True)
    return cmc.stage_orbit(state["r"], state["phi"], state["vr"], state["vt"], state["id"],
                           state["seed"], 1, precision=state["precision"])


def work(case):
    """Bytes and operations that a pass cannot do without.  A timestep reads
    the state (r, v_r, v_t, m, Phi: 8 bytes each, id: 4) and writes it once;
    its formulas, each +, -, x, / and square root counted once, come to about
    49 for the relaxation, 28 for the turning points, 21 x 14 for the
    envelope, 2 x 20 for the trials, 20 for the new velocities, 6 for the
    potential, 15 for the correction and 10 for the timestep per star."""
    kind = case["kind"]
    if kind == "step":
        n, steps = sum(_sizes(case)), case["steps"]
        # the checkpoint read, the steps, the state read out
        return {"bytes": n * (36 + steps * 88 + 44), "flops": n * steps * 462}
    n = case["n"]
    return {"diagnose": {"bytes": 32 * n, "flops": 30 * n},   # r, v_r, v_t, m
            "sort": {"bytes": 16 * n, "flops": 0},            # r, id -> permutation
            "potential": {"bytes": 32 * n, "flops": 6 * n},   # r, m -> Phi, M
            "orbit": {"bytes": 96 * n, "flops": 382 * n},     # 36 in, 60 out
            }[kind]


# ---------------------------------------------------- the same in 64 bits
# A plain numpy statement of the method (one cluster at a time, sums in
# extended precision where numpy has it), for the cases whose results are
# one value: FP64 steps and orbits, the potential, the diagnostics.  Mixed
# mode draws its orbits under an FP32 envelope of its own, so no other
# arithmetic gives its new radii: it has no exact value.
EXACT_MOST = 450_000  # star-steps: about 20 seconds of numpy
# a rounding grows a hundredfold a step (close encounters, orbits that barely
# reach a shell) until two neighbours change places, and with them every
# later pair: three steps still have one value, ten have not
EXACT_STEPS = 3


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        sizes = _sizes(case)
        if (case["precision"] != "fp64" or case["steps"] > EXACT_STEPS or
                sum(sizes) * case["steps"] > EXACT_MOST):
            return None
        d = {k: v.cpu().numpy() for k, v in _clusters(case, seed, "cuda").items()}
        at, outs = 0, []
        for c, nc in enumerate(sizes):
            s = {k: v[at:at + nc].copy() for k, v in d.items()}
            if case.get("physics"):
                s["R"], s["A"] = (a[s["id"]] for a in _attributes(case, nc, seed))
            outs.append(_run_steps(s, 1000 * seed + c, case["steps"]))
            at += nc
        out = {k: np.concatenate([o[k] for o in outs]) for k in ("r", "vr", "vt", "m", "phi")}
        out["id"] = out["step"] = None
        return out
    if kind == "diagnose":
        d = _sorted(_plummer(case["n"], 1000 * seed, case["masses"], "cuda"))
        return _diagnostics({k: v.cpu().numpy() for k, v in d.items()})
    if kind == "potential":
        d = _sorted(_plummer(case["n"], seed, case["masses"], "cuda"))
        M, phi = _potential(d["r"].cpu().numpy(), d["m"].cpu().numpy())
        return phi, M
    if kind == "orbit" and case["precision"] == "fp64" and case["n"] <= EXACT_MOST:
        d = _orbit_inputs(case, seed)
        o = _orbits(d["r"], d["phi"], d["vr"], d["vt"], d["id"], 1000 * seed, 1)
        o["code"] = None
        return o
    return None


def _potential(r, m):
    L = np.longdouble
    x = 1.0 / r
    M = np.cumsum(m.astype(L))
    mx = m.astype(L) * x
    S = np.cumsum(mx[::-1])[::-1] - mx
    return M.astype(float), (-(M * x + S)).astype(float)


def _diagnostics(s):
    L = np.longdouble
    r, m = s["r"], s["m"]
    M = np.cumsum(m.astype(L))
    K = 0.5 * np.sum(m.astype(L) * (s["vr"] ** 2 + s["vt"] ** 2))
    W = -np.sum(m.astype(L) * (M - m) / r)
    lag = np.array([[r[int(np.searchsorted(M, f * M[-1]))] for f in FRACTIONS]])
    mass = m[1:-5] + m[2:-4] + m[3:-3] + m[4:-2] + m[5:-1]
    rho = (mass / (4.0 * math.pi / 3.0 * (r[6:] ** 3 - r[:-6] ** 3))).astype(L)
    core = [np.sum(rho * rho) / np.sum(rho), np.sum(rho * r[3:-3]) / np.sum(rho), len(rho)]
    return {"energy": np.array([[K, W, K + W]], dtype=float), "lagrange": lag,
            "core": np.array([core], dtype=float), "escaped": np.zeros((1, 2))}


def _philox(ids, step, tag, trial, seed):
    """Philox4x32-10 blocks (four uint32 arrays) of counters (id, step, tag, trial)."""
    u = np.uint64
    c = [ids.astype(u), np.full(len(ids), step, u), np.full(len(ids), tag, u),
         np.full(len(ids), trial, u)]
    k0, k1, low = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF, u(0xFFFFFFFF)
    for _ in range(10):
        p0, p1 = c[0] * u(0xD2511F53), c[2] * u(0xCD9E8D57)
        c = [(p1 >> u(32)) ^ c[1] ^ u(k0), p1 & low, (p0 >> u(32)) ^ c[3] ^ u(k1), p0 & low]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _uniform(lo, hi):
    """(2k + 1) 2^-53 from the top 52 bits k of (hi:lo)."""
    k = ((hi << np.uint64(32)) | lo) >> np.uint64(12)
    return (2 * k.astype(np.int64) + 1).astype(float) * 2.0 ** -53


def _angles(ids, step, tag, seed):
    """Random planar directions (cos, sin) by rejection in the unit disk."""
    c, s = np.ones(len(ids)), np.zeros(len(ids))
    todo = np.arange(len(ids))
    for t in range(64):
        if not len(todo):
            break
        w = _philox(ids[todo], step, tag, t, seed)
        u, v = 2.0 * _uniform(w[0], w[1]) - 1.0, 2.0 * _uniform(w[2], w[3]) - 1.0
        q = u * u + v * v
        ok = q <= 1.0
        at = todo[ok]
        c[at] = ((u * u - v * v) / q)[ok]
        s[at] = ((2.0 * u) * v / q)[ok]
        todo = todo[~ok]
    return c, s


def _orbits(r, phi, vr, vt, ids, seed, step, max_trials=1000, gone=False):
    """New orbits (Eqs. 12-15) of the bound stars; escapers (and the stars
    merged away, `gone`) get r_new = inf."""
    n = len(r)
    x = 1.0 / r
    xs, ps = np.append(x, 0.0), np.append(phi, 0.0)
    rs = np.append(r, np.inf)
    E, J = phi + 0.5 * (vr * vr + vt * vt), r * vt
    live = (E < 0.0) & ~np.asarray(gone)
    k = np.arange(n)

    def Q_at(j):
        return 2.0 * (E - ps[j]) - (J * xs[j]) ** 2

    # r_max: the last node in [k, n) before Q < 0; r_min: the last in [-1, k)
    lo, hi = k.copy(), np.full(n, n)
    while (hi - lo > 1).any():
        mid = (lo + hi) >> 1
        go = hi - lo > 1
        neg = Q_at(mid) < 0.0
        hi, lo = np.where(go & neg, mid, hi), np.where(go & ~neg, mid, lo)
    jmax = lo
    lo, hi = np.full(n, -1), k.copy()
    while (hi - lo > 1).any():
        mid = (lo + hi) >> 1
        go = hi - lo > 1
        neg = Q_at(np.maximum(mid, 0)) < 0.0
        lo, hi = np.where(go & neg, mid, lo), np.where(go & ~neg, mid, hi)
    jmin = lo

    def shell_root(j, outer):
        j = np.maximum(j, 0)
        flat = ~(xs[j] - xs[j + 1] > 0.0)
        B = (ps[j + 1] - ps[j]) / np.where(flat, 1.0, xs[j] - xs[j + 1])
        A = ps[j] + B * xs[j]
        sD = np.sqrt(np.maximum(B * B + 2.0 * (J * J) * (E - A), 0.0))
        root = (B + sD) / (2.0 * (A - E)) if outer else J * J / (B + sD)
        root = np.where(root >= rs[j], root, rs[j])
        return np.where(flat, rs[j], np.minimum(root, rs[j + 1]))

    def Phi_at(q):
        i = np.searchsorted(r, q, side="right") - 1
        j = np.maximum(i, 0)
        den = xs[j] - xs[j + 1]
        inside = ps[j] + (xs[j] - 1.0 / q) / np.where(den > 0.0, den, 1.0) * (ps[j + 1] - ps[j])
        return np.where(i < 0, ps[0], np.where(den > 0.0, inside, ps[j]))

    def g_at(a, s):
        q = c0[a] + c1[a] * (s * (3.0 - s * s))
        ph = Phi_at(q)
        Q = 2.0 * (E[a] - ph) - (J[a] / q) ** 2
        g = 3.0 * c1[a] * (1.0 - s * s) / np.sqrt(np.where(Q > 0.0, Q, 1.0))
        return q, ph, Q, np.where(Q > 0.0, g, 0.0)

    with np.errstate(all="ignore"):
        rmax = shell_root(jmax, True)
        central = np.minimum(np.nan_to_num(J / np.sqrt(2.0 * (E - phi[0])), nan=0.0), r[0])
        rmin = np.where(jmin < 0, central, shell_root(jmin, False))
        c0, c1 = 0.5 * (rmax + rmin), 0.25 * (rmax - rmin)
        F = np.zeros(n)
        at = k[live]
        for j in range(21):
            F[at] = np.maximum(F[at], g_at(at, -1.0 + (j + 0.5) / 10.5)[3])
        F = 1.2 * F
        out = {"r_new": np.where(live, r, np.inf), "vr": vr.copy(), "vt": vt.copy(),
               "phi_new": phi.copy(), "rmin": np.where(live, rmin, r),
               "rmax": np.where(live, rmax, r), "F": np.where(live, F, 0.0)}
        todo = k[live & (rmax > rmin) & (F > 0.0)]
        for t in range(max_trials):
            if not len(todo):
                break
            w = _philox(ids[todo], step, 2, t, seed)
            q, ph, Q, g = g_at(todo, 2.0 * _uniform(w[0], w[1]) - 1.0)
            ok = F[todo] * _uniform(w[2], w[3]) < g
            at = todo[ok]
            sign = np.where(_philox(ids[at], step, 3, 0, seed)[0] & np.uint64(1), -1.0, 1.0)
            out["r_new"][at], out["phi_new"][at] = q[ok], ph[ok]
            out["vr"][at], out["vt"][at] = sign * np.sqrt(Q[ok]), J[at] / q[ok]
            todo = todo[~ok]
    return out


def _relax(s, nb, nbin, dt, lnL, seed, step):
    """Two-body relaxation of the neighbour pairs (2j, 2j + 1)."""
    a = np.arange(0, nb - 1, 2)
    b = a + 1
    n = nbin[a // 20]
    use = n > 0.0
    a, b, n = a[use], b[use], n[use]
    m1, m2 = s["m"][a], s["m"][b]
    ms = m1 + m2
    cp, sp = _angles(s["id"][a], step, 0, seed)
    cf, sf = _angles(s["id"][a], step, 1, seed)
    v1 = np.stack([s["vr"][a], s["vt"][a], np.zeros(len(a))])
    v2 = np.stack([s["vr"][b], s["vt"][b] * cp, s["vt"][b] * sp])
    w = v1 - v2
    w2 = (w * w).sum(0)
    wl = np.sqrt(w2)
    merge = np.zeros(len(a), bool)
    if "R" in s:  # sticky spheres, with gravitational focusing
        R1, R2 = s["R"][a], s["R"][b]
        Rs = R1 + R2
        u = _philox(s["id"][a], step, 4, 0, seed)
        merge = _uniform(u[0], u[1]) < (math.pi * Rs * Rs * (1.0 + 2.0 * ms / (Rs * w2))) * n * wl * dt
    s2 = np.minimum(2.0 * math.pi * ms * ms * n * lnL * dt / (w2 * wl), 1.0)
    cosb, sinb = 1.0 - 2.0 * s2, 2.0 * np.sqrt(s2) * np.sqrt(1.0 - s2)
    wp = np.sqrt(w[1] ** 2 + w[2] ** 2)
    e1 = np.stack([np.zeros(len(a)), w[2] / wp, -w[1] / wp])
    dw = w * cosb + sinb * (wl * cf * e1 + sf * np.cross(w.T, e1.T).T) - w
    p1, p2 = v1 + m2 / ms * dw, v2 - m1 / ms * dw
    cm = (m1 * v1 + m2 * v2) / ms
    p1, p2 = np.where(merge, cm, p1), np.where(merge, v2, p2)
    s["vr"][a], s["vt"][a] = p1[0], np.hypot(p1[1], p1[2])
    s["vr"][b], s["vt"][b] = p2[0], np.where(merge, s["vt"][b], np.hypot(p2[1], p2[2]))
    if merge.any():
        a, b = a[merge], b[merge]
        s["m"][a], s["m"][b] = ms[merge], 0.0
        s["R"][a], s["R"][b] = np.cbrt(s["R"][a] ** 3 + s["R"][b] ** 3), -1.0


def _timestep(s, nb, lnL):
    """Eq. 7 on bins of 20 consecutive stars: the bins' densities, the step."""
    lo = np.arange(0, nb, 20)
    hi = np.minimum(lo + 20, nb)
    P = hi - lo
    vol = s["r"][hi - 1] ** 3 - s["r"][lo] ** 3
    with np.errstate(all="ignore"):
        n = np.where((P >= 2) & (vol > 0.0), 3.0 * (P - 1) / (4.0 * math.pi * vol), 0.0)
        q = nb // 2
        v2 = s["vr"][:nb] ** 2 + s["vt"][:nb] ** 2
        pv, pm = np.sqrt(v2[0:2 * q:2] + v2[1:2 * q:2]), s["m"][0:2 * q:2] + s["m"][1:2 * q:2]
        pad = np.zeros(len(lo) * 10 - q)
        sv = np.append(pv, pad).reshape(-1, 10).sum(1) / (P // 2)
        sm = np.append(pm * pm, pad).reshape(-1, 10).sum(1) / (P // 2)
        T = math.pi / 32.0 * sv ** 3 / (lnL * n * sm)
    ok = (n > 0.0) & (T > 0.0) & np.isfinite(T)
    dt = float(T[ok].min()) if ok.any() else math.inf
    return n, min(dt, _central(s, nb)) if "R" in s else dt


def _central(s, nb):
    """Eqs. 8-10: the collision and binary timesteps of the innermost 300 stars."""
    P = min(nb, 300)
    r, m, R, A = (s[k][:P] for k in ("r", "m", "R", "A"))
    n = 3.0 * (P - 1) / (4.0 * math.pi * (r[-1] ** 3 - r[0] ** 3))
    sig2 = float(np.sum(s["vr"][:P] ** 2 + s["vt"][:P] ** 2)) / P / 3.0
    c = math.sqrt(math.pi) * math.sqrt(sig2) * n
    R2, MR = np.mean(R * R), np.mean(m * R)
    T = 1.0 / (16.0 * c * R2 * (1.0 + MR / (2.0 * sig2 * R2)))
    bin = A > 0.0
    nbin = int(bin.sum())
    if nbin:
        a2, ma, am = (float(np.mean(v[bin])) for v in (A * A, m * A, A))
        T = min(T, 1.0 / (16.0 * c * (nbin / P) * a2 * (1.0 + ma / (2.0 * sig2 * a2))))
        if nbin < P:
            T = min(T, 1.0 / (4.0 * c * (1.0 - nbin / P) * a2 *
                              (1.0 + np.mean(m) * am / (sig2 * a2))))
    return float(T)


def _run_steps(s, seed, steps):
    n = len(s["r"])
    lnL = math.log(0.1 * n)
    order = np.lexsort((s["id"], s["r"]))
    s = {k: v[order] for k, v in s.items()}
    nb = n
    s["phi"] = _potential(s["r"], s["m"])[1]
    for step in range(steps):
        nbin, dt = _timestep(s, nb, lnL)
        if lnL > 0.0 and math.isfinite(dt):
            _relax(s, nb, nbin, dt, lnL, seed, step)
        gone = s["R"][:nb] < 0.0 if "R" in s else np.zeros(nb, bool)
        o = _orbits(s["r"][:nb], s["phi"][:nb], s["vr"][:nb], s["vt"][:nb], s["id"][:nb], seed,
                    step, gone=gone)
        r_old, phi_old = s["r"][:nb].copy(), s["phi"][:nb].copy()
        moved = o["r_new"] != r_old
        r_new = np.append(o["r_new"], s["r"][nb:])
        s["vr"][:nb], s["vt"][:nb] = o["vr"], o["vt"]
        c = np.where(moved, phi_old - o["phi_new"], 0.0)
        order = np.lexsort((s["id"], r_new))
        s = {k: v[order] for k, v in s.items()}
        s["r"] = r_new[order]
        nb = int(np.isfinite(s["r"]).sum())
        s["phi"] = np.zeros(n)
        s["phi"][:nb] = _potential(s["r"][:nb], s["m"][:nb])[1]
        # the energy correction: the work of the changing potential
        at = order[:nb]
        r, x = s["r"][:nb], np.append(1.0 / s["r"][:nb], 0.0)
        p = np.append(s["phi"][:nb], 0.0)
        i = np.searchsorted(r, r_old[at], side="right") - 1
        j = np.maximum(i, 0)
        with np.errstate(all="ignore"):
            den = x[j] - x[j + 1]
            there = p[j] + (x[j] - 1.0 / r_old[at]) / den * (p[j + 1] - p[j])
        there = np.where(i < 0, p[0], np.where(den > 0.0, there, p[j]))
        T = 0.5 * (s["vr"][:nb] ** 2 + s["vt"][:nb] ** 2)
        Tn = np.maximum(T + 0.5 * ((there - s["phi"][:nb]) - c[at]), 0.0)
        f = np.where(T > 0.0, np.sqrt(Tn / np.where(T > 0.0, T, 1.0)), 1.0)
        s["vr"][:nb] *= f
        s["vt"][:nb] *= f
    return s
