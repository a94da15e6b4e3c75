"""What is timed: the calls a user of the element volume term makes, over their range.

Each case is one pass through the package's public entry points (VolumeTerm.rhs and
rhs_host, Batch.advance, Engine.submit and run_until_idle) on the warped 10 km box with a
hydrostatic reference state, the setting of the package's own workloads.  Inputs are made
on the GPU from the seed; exact() evaluates the same operation in plain 64-bit torch.
"""
import math

import numpy as np
import torch

from paper_1604_08501_gb300.numa_vol import Batch, Engine, VolumeTerm

L, WARP = 10_000.0, 0.05
P0, R, CP, GRAV = 1.0e5, 287.17, 1004.67, 9.80616
GAMMA = CP / (CP - R)
DT = 0.01
DEVICE = "cuda:0"


def _rhs(name, precision, N, nx, ny, nz, tracers=0, kind="rhs"):
    return {"name": name, "kind": kind, "precision": precision, "N": N, "nx": nx, "ny": ny,
            "nz": nz, "tracers": tracers}


def _members(name, kind, precision, plan, count, ne_lo, ne_hi):
    return {"name": name, "kind": kind, "precision": precision, "plan": plan, "count": count,
            "ne_lo": ne_lo, "ne_hi": ne_hi}


def listed():
    return [
        # the smallest mesh a user steps interactively (and the package's parity
        # workload): one call is a launch and its latency
        _rhs("fp64 N4 512 elements", "fp64", 4, 8, 8, 8),
        # the headline evaluation, in the strict mode and the two faster modes
        _rhs("fp64 N7 32768 elements", "fp64", 7, 32, 32, 32),
        _rhs("mixed N7 32768 elements", "mixed", 7, 32, 32, 32),
        _rhs("df64 N7 13824 elements", "df64", 7, 24, 24, 24),
        # a regional mesh of ordinary size with ragged element counts and an odd
        # number of points per axis
        _rhs("mixed N4 23x19x17", "mixed", 4, 23, 19, 17),
        # the paper's study of Nq at 3.5 million points: its highest order, and its own
        # form with three tracers in both precisions
        _rhs("mixed N15 864 elements", "mixed", 15, 12, 12, 6),
        _rhs("mixed N11 3 tracers", "mixed", 11, 16, 16, 8, tracers=3),
        _rhs("fp64 N11 3 tracers", "fp64", 11, 16, 16, 8, tracers=3),
        # a solver whose state lives in host memory: copies included
        _rhs("host fp64 N7 4096 elements", "fp64", 7, 16, 16, 16, kind="host"),
        # ensembles of members of several orders and sizes, ten steps to a call
        _members("batch mixed 12 members", "batch", "mixed", 99, 12, 512, 16384),
        _members("batch fp64 6 members", "batch", "fp64", 7, 6, 512, 4096),
        # forecast requests of 1, 5 or 20 steps served from host memory
        _members("engine mixed 12 requests", "engine", "mixed", 99, 12, 512, 8192),
    ]


def draw(rng):
    kind = rng.choice(["rhs"] * 14 + ["host"] * 2 + ["batch"] * 3 + ["engine"])
    precision = rng.choice(["fp64", "mixed"])
    if kind in ("batch", "engine"):
        # at most as much as the listed fp64 batch and mixed ensembles
        count = rng.randint(1, 4 if precision == "fp64" else 12)
        hi = 4096 if precision == "fp64" else 8192
        return {"kind": kind, "precision": precision, "plan": rng.randrange(1000), "count": count,
                "ne_lo": 64, "ne_hi": rng.randint(128, hi)}
    precision = rng.choice([precision, precision, "df64"])
    N = rng.randint(1, 7 if precision == "df64" else 15)
    tracers = rng.choice([0, 0, 0, 1, 2, 3])
    # mesh points: from a few elements to the size of the headline mesh
    points = math.exp(rng.uniform(math.log(2 ** 12), math.log(2 ** 23)))
    if kind == "host":
        points = min(points, 2 ** 21)
    ne = max(1.0, points / (N + 1) ** 3)
    a, b = rng.uniform(0.7, 1.4), rng.uniform(0.7, 1.4)
    edge = ne ** (1 / 3)
    shape = [max(1, round(edge * a)), max(1, round(edge * b)), max(1, round(edge / (a * b)))]
    return {"kind": kind, "precision": precision, "N": N, "nx": shape[0], "ny": shape[1],
            "nz": shape[2], "tracers": tracers}


# ---------------------------------------------------------------- inputs


def _gll(N):
    """GLL points: -1, 1 and the roots of P_N', by Newton from the Chebyshev points."""
    x = -np.cos(np.pi * np.arange(N + 1) / N)
    for _ in range(50):
        p0, p1 = np.ones_like(x), x.copy()
        for m in range(2, N + 1):
            p0, p1 = p1, ((2 * m - 1) * x * p1 - (m - 1) * p0) / m
        inner = slice(1, N)
        xi = x[inner]
        dp = N * (p0[inner] - xi * p1[inner]) / (1 - xi * xi)
        d2p = (2 * xi * dp - N * (N + 1) * p1[inner]) / (1 - xi * xi)
        x[inner] = xi - dp / d2p
    x[0], x[-1] = -1.0, 1.0
    return x


def _mesh(N, shape):
    """Geometry and reference state of the sine-warped box, on the GPU: a dict of g (9, M),
    Jinv, rho_ref, theta_ref (M) and x (3, M)."""
    nx, ny, nz = shape
    r = (torch.from_numpy(_gll(N)).to(DEVICE) + 1.0) * 0.5
    n = N + 1

    def axis(count, view):
        h = L / count
        return ((torch.arange(count, device=DEVICE, dtype=torch.float64)[:, None] + r) * h).reshape(view), h

    xh, hx = axis(nx, (1, 1, nx, 1, 1, n))
    yh, hy = axis(ny, (1, ny, 1, 1, n, 1))
    zh, hz = axis(nz, (nz, 1, 1, n, 1, 1))
    full = (nz, ny, nx, n, n, n)
    A, k = WARP * L, math.pi / L
    sx, sy, sz = (torch.sin(k * v) for v in (xh, yh, zh))
    cx, cy, cz = (torch.cos(k * v) for v in (xh, yh, zh))
    x = [v.expand(full).reshape(-1) for v in (xh + A * sy * sz, yh + A * sz * sx, zh + A * sx * sy)]
    Ak = A * k
    a_r = (0.5 * hx + 0 * sx, 0.5 * hx * Ak * sz * cx, 0.5 * hx * Ak * cx * sy)
    a_s = (0.5 * hy * Ak * cy * sz, 0.5 * hy + 0 * sy, 0.5 * hy * Ak * sx * cy)
    a_t = (0.5 * hz * Ak * sy * cz, 0.5 * hz * Ak * cz * sx, 0.5 * hz + 0 * sz)

    def cross(u, v):
        return [u[1] * v[2] - u[2] * v[1], u[2] * v[0] - u[0] * v[2], u[0] * v[1] - u[1] * v[0]]

    g = [c.expand(full).reshape(-1) for p in (cross(a_s, a_t), cross(a_t, a_r), cross(a_r, a_s)) for c in p]
    J = sum((a_r[a].expand(full).reshape(-1) * g[a] for a in range(3)))
    T0 = 300.0
    p_h = P0 * torch.exp(-GRAV * x[2] / (R * T0))
    rho_ref = p_h / (R * T0)
    theta_ref = rho_ref * T0 * (P0 / p_h) ** (R / CP)
    return {"N": N, "Ne": nx * ny * nz, "M": J.numel(), "g": g, "Jinv": 1.0 / J, "x": x,
            "rho_ref": rho_ref, "theta_ref": theta_ref}


def _bumps(m, rng):
    """Sum of four Gaussian bumps at the mesh's points."""
    out = torch.zeros(m["M"], dtype=torch.float64, device=DEVICE)
    c, w, a = rng.uniform(0, L, (4, 3)), rng.uniform(0.1 * L, 0.3 * L, 4), rng.uniform(-1, 1, 4)
    for n in range(4):
        r2 = sum((m["x"][d] - float(c[n, d])) ** 2 for d in range(3))
        out += float(a[n]) * torch.exp(-r2 / float(w[n] * w[n]))
    return out


def _state(m, seed, tracers, smooth):
    """Perturbed hydrostatic state (5 + tracers, M): velocities up to 10 m/s, independent at
    each point for single evaluations and smooth for time integration, as the package's
    workloads have them; tracers are mixing ratios about 0.01."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEVICE).manual_seed(int(seed))
    q = torch.empty((5 + tracers, m["M"]), dtype=torch.float64, device=DEVICE)
    q[0] = m["rho_ref"] * (1 + 1e-3 * _bumps(m, rng))
    theta = m["theta_ref"] / m["rho_ref"] * (1 + 1e-3 * _bumps(m, rng))
    for a in range(3):
        if smooth:
            v = _bumps(m, rng)
            v *= 10.0 / v.abs().max()
        else:
            v = torch.rand(m["M"], generator=gen, dtype=torch.float64, device=DEVICE) * 20 - 10
        q[1 + a] = q[0] * v
    q[4] = q[0] * theta
    for t in range(tracers):
        q[5 + t] = q[0] * 0.01 * (1 + 0.5 * _bumps(m, rng))
    return q


def _given(m, q, precision):
    """The state as the entry points take it (mixed: FP32 perturbations)."""
    if precision != "mixed":
        return q
    q = q.clone()
    q[0] -= m["rho_ref"]
    q[4] -= m["theta_ref"]
    return q.float()


def _term(m, precision, tracers):
    return VolumeTerm(m["N"], m["Ne"], m["g"], m["Jinv"], m["rho_ref"], m["theta_ref"], P0, R, CP,
                      GRAV, precision=precision, tracers=tracers)


def _plan(case):
    """Orders, element counts per axis and steps of an ensemble's members: orders of the
    package's batched workload, sizes log-uniform, rounded to a cube."""
    rng = np.random.default_rng(case["plan"])
    out = []
    for i in range(case["count"]):
        N = int(rng.choice([3, 4, 5, 7]))
        ne = math.exp(rng.uniform(math.log(case["ne_lo"]), math.log(case["ne_hi"])))
        steps = 10 if case["kind"] == "batch" else int(rng.choice([1, 5, 20]))
        out.append((N, max(1, round(ne ** (1 / 3))), steps, i))
    return out


def _inputs(case, seed):
    """[(mesh, state in FP64 or in the mixed mode's form, steps)] of a case."""
    if "plan" in case:
        meshes = {}
        out = []
        for N, n, steps, i in _plan(case):
            if (N, n) not in meshes:
                meshes[N, n] = _mesh(N, (n, n, n))
            m = meshes[N, n]
            out.append((m, _given(m, _state(m, 1000 * seed + i, 0, True), case["precision"]), steps))
        return out
    m = _mesh(case["N"], (case["nx"], case["ny"], case["nz"]))
    return [(m, _given(m, _state(m, seed, case["tracers"], False), case["precision"]), 0)]


# ---------------------------------------------------------------- the passes


def prepare(case, seed):
    made = _inputs(case, seed)
    kind, precision = case["kind"], case["precision"]
    if kind in ("rhs", "host"):
        m, q, _ = made[0]
        s = {"kind": kind, "vt": _term(m, precision, case["tracers"])}
        if kind == "rhs":
            s["q"], s["out"] = q, torch.empty_like(q)
        else:   # pinned host memory, as a program that feeds a GPU keeps it
            s["q"] = q.cpu().pin_memory()
            s["out"] = torch.empty(q.shape, dtype=q.dtype, pin_memory=True)
        return s
    terms = {}
    for m, _, _ in made:
        if id(m) not in terms:
            terms[id(m)] = _term(m, precision, 0)
    if kind == "batch":
        # the members' initial states and their working copies, one buffer each; every
        # member's planes start on a 256-byte boundary
        sizes = [(q.numel() + 63) // 64 * 64 for _, q, _ in made]
        first = torch.zeros(sum(sizes), dtype=made[0][1].dtype, device=DEVICE)
        work, at, views = torch.empty_like(first), 0, []
        b = Batch(precision)
        for (m, q, _), size in zip(made, sizes):
            first[at:at + q.numel()] = q.reshape(-1)
            views.append(work[at:at + q.numel()].view(q.shape))
            b.add(terms[id(m)], views[-1])
            at += size
        return {"kind": kind, "batch": b, "first": first, "work": work, "views": views}
    members = []
    for m, q, steps in made:
        members.append((terms[id(m)], q.cpu().pin_memory(),
                        torch.empty(q.shape, dtype=q.dtype, pin_memory=True), steps))
    engine = Engine(precision, budget_bytes=1 << 31, max_members=64, round_steps=4,
                    round_policy="per_member")
    return {"kind": kind, "engine": engine, "members": members}


def run(state):
    if state["kind"] == "rhs":
        return state["vt"].rhs(state["q"], out=state["out"])
    if state["kind"] == "host":
        return state["vt"].rhs_host(state["q"], out=state["out"])
    if state["kind"] == "batch":
        # every forecast starts from the analysis
        state["work"].copy_(state["first"])
        state["batch"].advance(10, DT)
        return state["views"]
    e = state["engine"]
    for term, q, out, steps in state["members"]:
        e.submit(term, q, out, steps, DT)
    e.run_until_idle()
    return [out for _, _, out, _ in state["members"]]


def work(case):
    size = 4 if case["precision"] == "mixed" else 8
    if "plan" in case:
        b = f = 0
        seen = set()
        for N, n, steps, _ in _plan(case):
            M = n ** 3 * (N + 1) ** 3
            b += size * M * 10 + (0 if (N, n) in seen else size * M * 12)
            f += 5 * steps * M * _flops(N, 0)
            seen.add((N, n))
        return {"bytes": b, "flops": f}
    M = case["nx"] * case["ny"] * case["nz"] * (case["N"] + 1) ** 3
    nf = 5 + case["tracers"]
    return {"bytes": size * M * (2 * nf + 12), "flops": M * _flops(case["N"], case["tracers"])}


def _flops(N, tracers):
    """Per point: pressure 5, fluxes 17 (and a tracer's 1) per direction, the three sums of
    each field, scaling and gravity."""
    nf = 5 + tracers
    return 5 + 3 * (17 + tracers) + 6 * nf * (N + 1) + nf + 3


# ---------------------------------------------------------------- in 64 bits


def _diff(N):
    x = _gll(N)
    w = np.array([1 / np.prod(np.delete(x[i] - x, i)) for i in range(N + 1)])
    D = w[None, :] / w[:, None] / (x[:, None] - x[None, :] + np.eye(N + 1))
    np.fill_diagonal(D, 0.0)
    np.fill_diagonal(D, -D.sum(1))
    return torch.from_numpy(D).to(DEVICE)


def _volume(m, D, drho, U, dth, tracers):
    """The volume term of a state given as perturbations drho, dth from the reference."""
    n = D.shape[0]
    rho, th = m["rho_ref"] + drho, m["theta_ref"] + dth
    p_ref = P0 * (R * m["theta_ref"] / P0) ** GAMMA
    p = p_ref * torch.expm1(GAMMA * torch.log1p(dth / m["theta_ref"]))
    u = [sum(m["g"][3 * d + a] * U[a] for a in range(3)) / rho for d in range(3)]
    out = []
    for b in range(5 + len(tracers)):
        total = 0
        for d in range(3):
            if b == 0:
                F = rho * u[d]
            elif b < 4:
                F = U[b - 1] * u[d] + m["g"][3 * d + b - 1] * p
            else:
                F = (th if b == 4 else tracers[b - 5]) * u[d]
            if d == 0:
                S = F.view(-1, n) @ D.T
            elif d == 1:
                S = torch.matmul(D, F.view(-1, n, n))
            else:
                S = torch.matmul(D, F.view(-1, n, n * n))
            total = total + S.reshape(-1)
        out.append(-m["Jinv"] * total)
    out[3] = out[3] - drho * GRAV
    return out


#: Five-stage fourth-order low-storage Runge-Kutta scheme of Carpenter and Kennedy.
LSRK_A = (0.0, -567301805773 / 1357537059087, -2404267990393 / 2016746695238,
          -3550918686646 / 2091501179385, -1275806237668 / 842570457699)
LSRK_B = (1432997174477 / 9575080441755, 5161836677717 / 13612068292357,
          1720146321549 / 2090206949498, 3134564353537 / 4481467310338,
          2277821191437 / 14882151754819)


def exact(case, seed):
    outs = []
    for m, q, steps in _inputs(case, seed):
        D = _diff(m["N"])
        q = q.double()
        if case["precision"] != "mixed":
            q[0] -= m["rho_ref"]
            q[4] -= m["theta_ref"]
        if not steps:
            return torch.stack(_volume(m, D, q[0], q[1:4], q[4], q[5:]))
        dq = torch.zeros_like(q)
        for _ in range(steps):
            for a, b in zip(LSRK_A, LSRK_B):
                dq.mul_(a).add_(torch.stack(_volume(m, D, q[0], q[1:4], q[4], ())), alpha=DT)
                q.add_(dq, alpha=b)
        if case["precision"] != "mixed":
            q[0] += m["rho_ref"]
            q[4] += m["theta_ref"]
        outs.append(q)
    return outs
