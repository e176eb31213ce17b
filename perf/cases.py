"""Cases of the manufactured-solution PIC + DSMC framework to be measured.

Kinds of work, each through the framework's public calls:

  run       sample_mms, step, mms_error, get_state: one level of a refinement
            study, as the convergence studies and the README's example do it.
  advance   set_state, step, get_state: a caller's own state moved on, its
            arrays in device memory or in pinned host memory.
  collide   collide_avg on a held state: one K-averaged collision call.
  batch     sample_mms, step, mms_error, get_state of every replicate of a
            batch of uneven replicates (precision form, its own stream).
  gradient  adjoint_gradient: the objective and its pathwise gradient.
  solve     pic_poisson_solve_noalloc: the Poisson solve alone, from phi = 0.

``form`` is "fp64" (the plain form, the default of a configuration) or
"mixed" (the precision form, FP32 state). ``problem`` is "wave" (travelling
density wave, Gaussian velocities, hard spheres) or "paper" (the paper's
per-axis densities, non-Maxwellian velocities, odd-power cross section).
Sizes are the workload recipes' own (``workloads``) or a part of them.

``exact`` restates the method in plain torch FP64 (an FFT for the Poisson
solve, Algorithm 1 over all (cell, outcome) lanes at once); it shares no
code with the framework.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2602_15130_gb300 import Batch, Pic, load, workloads

F64 = torch.float64
TAU = 2.0 * math.pi
MASK = 0xFFFFFFFF


# ------------------------------------------------------------------ cases --
def _case(name, kind, p, steps, form="fp64", memory="device", aniso=False, problem="wave"):
    return dict(name=name, kind=kind, problem=problem, form=form, n=p["n"], particles=p["n_particles"], K=p["K"],
                dt=p["dt"], sigma0=p["sigma0"], max_ppc=p.get("max_ppc", 0), steps=steps, memory=memory, aniso=aniso)


def listed():
    w = workloads
    grad = w.scaled(w.differentiation(), 16)
    return [
        # the library's default configuration and the smallest workload, FP64:
        # ten steps; launches and the latency of a small Poisson solve count
        _case("smallest_fp64", "run", w.smallest(), 10),
        # the README's example: the same in the precision form
        _case("smallest_mixed", "run", w.smallest(), 10, "mixed"),
        # a whole level of Table 1's collisional study in FP64, its second
        # (odd mesh, 101.25 particles per cell, K = 243, anisotropic kernel)
        _case("table1_12_fp64", "run", w.table1_level(1), 12, aniso=True),
        # the paper's own problem on the same level in the precision form
        _case("paper_12_mixed", "run", w.paper_table1_level(1), 12, "mixed", problem="paper"),
        # one collision call of Table 1's third level: 320 particles per
        # cell and K = 1024, many outcomes on few, crowded cells
        _case("collide_16_k1024", "collide", w.table1_level(2), 0, "mixed"),
        # the fixed-32-per-cell sweep at 32^3 in FP64, host arrays in and out
        _case("refine_32_fp64_host", "advance", w.refinement_level(2), 2, memory="pinned"),
        # the same sweep at 64^3 without collisions: deposit, solve, push
        _case("refine_64_fp64_k0", "advance", w.refinement_level(3, collisions=False), 1),
        # the precision-form study at 64^3: 16.8M particles, K = 32
        _case("precision_64", "advance", w.scaled(w.precision_form(), 64), 4, "mixed"),
        # the benchmark's default workload: 128^3 cells, 134M particles, K = 32
        _case("precision_128", "advance", w.precision_form(), 4, "mixed"),
        # the batched study's recipe, 16 replicates of 8^3 to 32^3 cells
        dict(name="batch_16", kind="batch", replicates=16, largest=32, pick=42, steps=6),
        # pathwise gradient, 16^3 cells at 64 per cell, K = 8, FP64
        dict(_case("gradient_16", "gradient", grad, 8), every=4),
        # the allocation-free solve at its largest mesh
        dict(name="solve_48", kind="solve", n=48, tol=1e-10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["run", "run", "advance", "advance", "collide", "batch", "gradient", "solve"])
    if kind == "solve":
        return dict(kind=kind, n=rng.randint(6, 48), tol=10.0 ** -rng.randint(10, 12))
    if kind == "batch":
        return dict(kind=kind, replicates=_log(rng, 3, 20), largest=rng.choice([16, 32]), pick=rng.randrange(1 << 20),
                    steps=rng.randint(3, 8))
    form = rng.choice(["fp64", "mixed"])
    problem = "wave"
    aniso = False
    memory = "device"
    if kind == "gradient":
        n, ppc, K, form = rng.randint(8, 20), _log(rng, 8, 64), rng.choice([0, 4, 8]), "fp64"
        c = _case("", kind, workloads.base(n, ppc * n ** 3 + rng.randrange(n), 0.005, K,
                                           workloads.hard_sphere_sigma0(ppc, 0.005, 0.005)), rng.randint(4, 10))
        c["every"] = rng.randint(2, 5)
    elif kind == "collide":
        n, ppc, K = rng.randint(8, 32), _log(rng, 16, 256), _log(rng, 8, 512)
        dt = 0.1 / n
        p = workloads.base(n, ppc * n ** 3 + rng.randrange(n), dt, K, workloads.table1_sigma0(), max_ppc=_capacity(ppc))
        c = _case("", kind, p, 0, form)
    elif kind == "run":
        n, ppc, K, steps = rng.randint(8, 24), _log(rng, 8, 128), rng.choice([0, 8, 16, 32, 64, 200]), rng.randint(4, 12)
        problem = rng.choice(["wave", "wave", "paper"])
        np_ = ppc * n ** 3 + rng.randrange(n)
        if problem == "paper":
            p = workloads.paper_problem(n, np_, 1.0 / (2 * n), K)
        else:
            p = workloads.base(n, np_, 0.01, K, workloads.hard_sphere_sigma0(ppc, 0.01, 0.02), max_ppc=_capacity(ppc))
            aniso = rng.random() < 0.25
        c = _case("", kind, p, steps, form, aniso=aniso, problem=problem)
    else:
        n = _log(rng, 16, 96 if form == "mixed" else 40)
        if rng.random() < 0.4:
            n = 1 << max(4, round(math.log2(n)))
        ppc, K = _log(rng, 8, 64), rng.choice([0, 8, 16, 32])
        memory = rng.choice(["device", "device", "pinned"]) if n <= 48 else "device"
        p = workloads.base(n, ppc * n ** 3 + rng.randrange(n), 0.005, K,
                           workloads.hard_sphere_sigma0(ppc, 0.005, 0.01))
        c = _case("", kind, p, rng.randint(1, 4), form, memory)
    del c["name"]
    return c


def _capacity(ppc):
    return max(64, int(math.ceil((ppc * 1.3 ** 3 * 1.15 + 64) / 32.0)) * 32)


def _params(case, seed):
    """The configuration of a single-context case."""
    kw = dict(seed=seed, max_ppc=case["max_ppc"])
    if case["problem"] == "paper":
        p = workloads.paper_problem(case["n"], case["particles"], case["dt"], case["K"], **kw)
    else:
        p = workloads.base(case["n"], case["particles"], case["dt"], case["K"], case["sigma0"], **kw)
    if case["aniso"]:
        p["verify"] = 16  # PIC_VERIFY_ANISO
    return workloads.mixed(p) if case["form"] == "mixed" else p


def _replicates(case, seed):
    """The batched study's recipe with meshes up to ``largest``."""
    g = random.Random(case["pick"])
    meshes = [n for n in (8, 16, 32, 64) if n <= case["largest"]]
    out = []
    for r in range(case["replicates"]):
        n, ppc, K = g.choice(meshes), g.randint(8, 64), g.randint(4, 64)
        out.append(workloads.base(n, ppc * n ** 3, 0.005, K, workloads.hard_sphere_sigma0(ppc, 0.005),
                                  seed=1000 + r + 7919 * seed, precision=1, cg_tol=workloads.PRECISION_CG_TOL))
    return out


# --------------------------------------------------------- prepare and run --
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) + 1)


def _own_state(p, seed):
    """A caller's state [N, 3]: the manufactured one at t = 0, displaced as
    it is after some steps of the benchmark workload."""
    g = _generator(seed)
    x, v = [], []
    for lo in range(0, p["n_particles"], 1 << 24):
        pid = torch.arange(lo, min(p["n_particles"], lo + (1 << 24)), device="cuda")
        xi = _xi(p, pid)
        x.append(_xm(p, xi[:, :3], 0.0)[0])
        v.append(_vm(p, xi[:, 3:], 0.0))
    x, v = torch.cat(x), torch.cat(v)
    x.add_(torch.randn(x.shape, generator=g, device="cuda", dtype=F64), alpha=0.003)
    x.sub_(torch.floor(x))
    x[x >= 1.0] = 0.0
    v.add_(torch.randn(v.shape, generator=g, device="cuda", dtype=F64), alpha=0.05)
    return x, v


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        n = case["n"]
        b = torch.randn(n ** 3, generator=_generator(seed), device="cuda", dtype=F64)
        return dict(case=case, b=b, phi=torch.empty_like(b), E=torch.empty(3, n ** 3, device="cuda", dtype=F64))
    if kind == "batch":
        reps = _replicates(case, seed)
        out = [tuple(torch.empty(p["n_particles"], 3, device="cuda", dtype=F64) for _ in range(2)) for p in reps]
        return dict(case=case, sim=Batch(reps, stream=torch.cuda.Stream()), out=out)
    p = _params(case, seed)
    if kind == "gradient":
        return dict(case=case, sim=Pic(p), v0=_own_state(p, seed)[1])
    rows = (p["n_particles"], 3)
    if kind in ("advance", "collide"):
        x, v = _own_state(p, seed)
    s = dict(case=case, sim=Pic(p))
    if case["memory"] == "pinned":
        s["x"], s["v"] = x.cpu().pin_memory(), v.cpu().pin_memory()
        s["out"] = tuple(torch.empty(rows, dtype=F64, pin_memory=True) for _ in range(2))
    else:
        if kind == "advance":
            s["x"], s["v"] = x, v
        s["out"] = tuple(torch.empty(rows, device="cuda", dtype=F64) for _ in range(2))
    if kind == "collide":
        s["sim"].set_state(x, v, 0.0)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "solve":
        s["phi"].zero_()
        stream = torch.cuda.current_stream().cuda_stream
        status = load().pic_poisson_solve_noalloc(case["n"], s["b"].data_ptr(), s["phi"].data_ptr(), s["E"].data_ptr(),
                                                  case["tol"], 10000, stream, None, None)
        if status != 0:
            raise RuntimeError(f"pic_poisson_solve_noalloc: status {status}")
        return s["phi"], s["E"]
    sim = s["sim"]
    if kind == "batch":
        sim.sample_mms(0.0)
        sim.step(case["steps"])
        return dict(norms=sim.mms_error(), state=[sim.get_state(r, out=o) for r, o in enumerate(s["out"])])
    if kind == "gradient":
        return sim.adjoint_gradient(case["steps"], every=case["every"], E_app=(0.1, 0.1, 0.1), v0=s["v0"])
    if kind == "collide":
        return sim.collide_avg(0, out=s["out"])
    if kind == "run":
        sim.sample_mms(0.0)
        sim.step(case["steps"])
        norms = sim.mms_error()["array"]
        return dict(norms=norms, state=sim.get_state(out=s["out"]))
    sim.set_state(s["x"], s["v"], 0.0)
    sim.step(case["steps"])
    return sim.get_state(out=s["out"])


# ------------------------------------------------------------------- work --
def _work_single(p, steps, load_store, form):
    """Bytes: the caller's arrays once each way, and every step the particle
    state (positions, velocities, v^M, pid) read and written once and the
    mesh's rho, phi and E written once. Flops: per particle and step the
    deposit and gather weights, the gather and the push (about 150), per
    collision call the source (20) and per candidate pair the relative speed
    and accept test (12), with the scattering of the accepted ones (40 each,
    at about one in eight)."""
    np_, nc, K = p["n_particles"], p["n"] ** 3, p["K"]
    state, node = (56, 20) if form == "mixed" else (104, 40)
    sg = p["sigma0"] * p["g_max"] if not p.get("n_sigma") else 1.0 / (workloads.TABLE1_INV_PMAX_L1 * 512) * 10240 * 8
    pairs = 0.5 * np_ * max(0.0, np_ / nc - 1) * sg * p["dt"] / np_ * nc * K  # per call
    calls = 2 * steps if steps else 1
    if K == 0:
        calls = 0
    return {"bytes": load_store * 48.0 * np_ + steps * (2.0 * state * np_ + node * nc),
            "flops": steps * 150.0 * np_ + calls * (20.0 * np_ + 17.0 * pairs)}


def work(case):
    kind = case["kind"]
    if kind == "solve":
        m = case["n"] ** 3  # b read, phi and E written; the least a solve computes: three 1-D transforms each way
        return {"bytes": 40.0 * m, "flops": 2 * 3 * 5.0 * m * math.log2(case["n"])}
    if kind == "batch":
        each = [_work_single(p, case["steps"], 1, "mixed") for p in _replicates(case, 0)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    p = _params(case, 0)
    if kind == "collide":
        size = 12 if case["form"] == "mixed" else 24
        return {"bytes": (size + 48.0) * p["n_particles"], "flops": _work_single(p, 0, 0, case["form"])["flops"]}
    w = _work_single(p, case["steps"], {"run": 1, "advance": 2, "gradient": 1}[kind], case["form"])
    if kind == "gradient":  # forward, and a reverse sweep of at least the forward's work
        return {"bytes": 2 * w["bytes"], "flops": 2 * w["flops"]}
    return w


# ------------------------------------------------- the method in 64 bits --
def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al. 2011) on int64 tensors of 32-bit words."""
    k0, k1 = seed & MASK, (seed >> 32) & MASK
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & MASK) ^ c1 ^ k0, p1 & MASK, ((p0 >> 32) & MASK) ^ c3 ^ k1, p0 & MASK
        k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
    return c0, c1, c2, c3


def _u52(hi, lo):
    return (2 * ((hi << 20) | (lo >> 12)) + 1).to(F64) * 2.0 ** -53


def _u32(w):
    return (2 * w + 1).to(F64) * 2.0 ** -33


def _xi(p, pid):
    """xi [N, 6] of particles pid."""
    zero = torch.zeros_like(pid)
    out = []
    for j in range(3):
        w = _philox(pid & MASK, pid >> 32, zero, zero + (0xFFFFFF00 | j), p["seed"])
        out += [_u52(w[0], w[1]), _u52(w[2], w[3])]
    return torch.stack(out, 1)


def _wave(p, t, d):
    """Amplitude and phase of f_{x_d} = 1 + A sin 2 pi (x - s) and their rates."""
    if p.get("dist", 0):
        e = math.exp(t)
        return ((e / 5, 0.0, e / 5, 0.0), (0.2, 0.15 * e, 0.0, 0.15 * e), (-e / 6, -e / 15, -e / 6, -e / 15))[d]
    return p["fx_amp"], p["fx_speed"] * t, 0.0, p["fx_speed"]


def _vh(p, t):
    vb, pi = p["v_bar"], math.pi
    vh = [vb * (1 + math.sin(pi * t / 2) / 5), vb * (1 + math.cos(pi * t) / 5), vb * (1 + math.sin(1.5 * pi * t) / 5)]
    dvh = [vb * pi / 2 * math.cos(pi * t / 2) / 5, -vb * pi * math.sin(pi * t) / 5, vb * 1.5 * pi * math.cos(1.5 * pi * t) / 5]
    return torch.tensor(vh, dtype=F64, device="cuda"), torch.tensor(dvh, dtype=F64, device="cuda")


def _xm(p, xi, t):
    """x^M(t) and xdot^M(t) [N, 3]: F(x) = xi by Newton."""
    xs, ds = [], []
    for d in range(3):
        A, s, dA, sr = _wave(p, t, d)
        T = xi[:, d] - s - A / TAU * math.cos(TAU * s)
        y = T.clone()
        for _ in range(9 if abs(A) > 0.35 else 6):
            y = y - (y - A / TAU * torch.cos(TAU * y) - T) / (1 + A * torch.sin(TAU * y))
        sy, cy = torch.sin(TAU * y), torch.cos(TAU * y)
        xs.append(y + s)
        ds.append((A * sr * (sy + math.sin(TAU * s)) - dA / TAU * (math.cos(TAU * s) - cy)) / (1 + A * sy))
    x = torch.stack(xs, 1)
    return x - torch.floor(x), torch.stack(ds, 1)


def _tau(xi):
    """tau with (1 + erf tau)/2 - tau exp(-tau^2)/sqrt pi = xi, by bisection."""
    lo, hi = torch.full_like(xi, -7.0), torch.full_like(xi, 7.0)
    for _ in range(62):
        m = 0.5 * (lo + hi)
        below = 0.5 * torch.erfc(-m) - m * torch.exp(-m * m) / math.sqrt(math.pi) < xi
        lo, hi = torch.where(below, m, lo), torch.where(below, hi, m)
    return 0.5 * (lo + hi)


def _vm(p, xi, t):
    """v^M(t) [N, 3]."""
    if p.get("dist", 0):
        return _tau(xi) * _vh(p, t)[0]
    return torch.special.ndtri(xi) * p["v_sigma"] + torch.tensor(p["v_mean"], dtype=F64, device="cuda")


def _cells(p, x):
    n = p["n"]
    i = torch.clamp((x * n).floor().long(), 0, n - 1)
    return i, i[:, 0] + n * (i[:, 1] + n * i[:, 2])


def _corners(p, x):
    """The eight (node, weight) pairs of every particle."""
    n = p["n"]
    i, _ = _cells(p, x)
    f = x * n - i
    for c in (0, 1):
        for b in (0, 1):
            for a in (0, 1):
                j = (i + torch.tensor([a, b, c], device="cuda")) % n
                w = 1.0
                for d, up in enumerate((a, b, c)):
                    w = w * (f[:, d] if up else 1 - f[:, d])
                yield j[:, 0] + n * (j[:, 1] + n * j[:, 2]), w


def _solve(n, b):
    """phi and E [n^3, 3] of -Lap_h phi = b - mean b, E = -grad_h phi."""
    lam = 2 * n * n * (1 - torch.cos(TAU * torch.arange(n, device="cuda", dtype=F64) / n))
    lam = lam[:, None, None] + lam[None, :, None] + lam[None, None, :]
    bh = torch.fft.fftn(b.reshape(n, n, n).to(torch.complex128))
    keep = (lam > 0).to(F64)
    phi = torch.fft.ifftn(bh * keep / torch.where(lam > 0, lam, torch.ones_like(lam))).real
    E = [(torch.roll(phi, 1, k) - torch.roll(phi, -1, k)) * (0.5 * n) for k in (2, 1, 0)]
    return phi.reshape(-1), torch.stack(E, -1).reshape(-1, 3)


def _phi_m(p, t):
    """phi^M and prod_d f_{x_d} at the nodes."""
    n = p["n"]
    g = torch.arange(n, device="cuda", dtype=F64) / n
    s = [torch.sin(TAU * (g - sh)) for sh in p["phi_shift"]]
    f = [1 + A * torch.sin(TAU * (g - ph)) for A, ph, _, _ in (_wave(p, t, d) for d in range(3))]
    grid = lambda u: (u[0][None, None, :] * u[1][None, :, None] * u[2][:, None, None]).reshape(-1)  # noqa: E731
    return p["phi_amp"] * math.exp(t / (2 * p["phi_T"])) * grid(s), grid(f)


def _field(p, x, t):
    """phi and E at the nodes of the state's charge with the manufactured sources."""
    n = p["n"]
    q = 0.0 if p["couple_q_zero"] else p["q"]
    rho = torch.zeros(n ** 3, dtype=F64, device="cuda")
    for node, w in _corners(p, x):
        rho = rho.index_add(0, node, w)
    rho = rho * (q * p["n_phys"] / p["n_particles"] * n ** 3)
    phi_m, f = _phi_m(p, t)
    return _solve(n, rho / p["eps0"] + 3 * TAU ** 2 * phi_m - q * p["n_phys"] * f / p["eps0"])


def _lorentz(p, x, E, t, E_app):
    """dt q/m (E + E_app - E^M) at the particles."""
    e = 0.0
    for node, w in _corners(p, x):
        e = e + w[:, None] * E[node]
    a = TAU * (x - torch.tensor(p["phi_shift"], dtype=F64, device="cuda"))
    s, c = torch.sin(a), torch.cos(a)
    em = -TAU * p["phi_amp"] * math.exp(t / (2 * p["phi_T"])) * torch.stack(
        [c[:, 0] * s[:, 1] * s[:, 2], s[:, 0] * c[:, 1] * s[:, 2], s[:, 0] * s[:, 1] * c[:, 2]], 1)
    qm = 0.0 if p["couple_qm_zero"] else p["qm"]
    return p["dt"] * qm * (e + E_app - em)


def _sg(p, g2):
    """sigma(g) g."""
    if not p.get("n_sigma"):
        return p["sigma0"] * torch.sqrt(g2)
    s = p["sigma_n"]
    return s[0] + s[1] * g2 + s[2] * g2 * g2


def _sg_max(p):
    if not p.get("n_sigma"):
        return p["sigma0"] * p["g_max"]
    s, u1 = p["sigma_n"], p["g_max"] ** 2
    at = [0.0, u1] + ([-s[1] / (2 * s[2])] if s[2] and 0 < -s[1] / (2 * s[2]) < u1 else [])
    return max(s[0] + s[1] * u + s[2] * u * u for u in at)


def _source(p, v, count, t):
    """The analytic <Delta v^M> of every particle in a cell of ``count``."""
    pref = (p["n_phys"] / p["n_particles"] * p["dt"] / 2 * p["n"] ** 3) * (count - 1).to(F64)[:, None]
    if not p.get("n_sigma"):
        s = p["v_sigma"]
        m = torch.tensor(p["v_mean"], dtype=F64, device="cuda") - v
        a2 = (m * m).sum(1, keepdim=True) / s ** 2
        a = torch.sqrt(torch.clamp(a2, min=0.04))
        big = math.sqrt(2 / math.pi) * (1 + 1 / a ** 2) * torch.exp(-a * a / 2) + \
            (a + 2 / a - 1 / a ** 3) * torch.erf(a / math.sqrt(2))
        d = [(-1) ** k / (2.0 ** k * math.factorial(k)) for k in range(12)]
        e = [d[k] / (2 * k + 1) for k in range(12)]
        small = 0.0
        for j in range(9, -1, -1):
            small = small * a2 + math.sqrt(2 / math.pi) * (d[j] + d[j + 1] + (e[j - 1] if j else 0.0) + 2 * e[j] - e[j + 1])
        return pref * p["sigma0"] * s * torch.where(a2 > 0.04, big, small) * m
    s = p["sigma_n"]
    a2 = _vh(p, t)[0] ** 2
    h2, v2 = a2.sum(), (v * v).sum(1, keepdim=True)
    cross = (a2 * v * v).sum(1, keepdim=True)
    others = torch.stack([a2[1] * a2[2], a2[2] * a2[0], a2[0] * a2[1]])
    f1 = -0.5 * (3 * h2 + 6 * a2 + 2 * v2)
    f2 = -0.25 * (15 * h2 ** 2 + 36 * a2 ** 2 + 24 * v2 * a2 + 4 * v2 ** 2 + 24 * a2 * h2 + 12 * v2 * h2 + 24 * cross
                  - 12 * others)
    return pref * (-s[0] + s[1] * f1 + s[2] * f2) * v


def _chi(p, u):
    """sin^2(chi/2) of a uniform u."""
    if not p.get("verify", 0) & 16:
        return u
    lo, hi = torch.zeros_like(u), torch.ones_like(u)
    for _ in range(56):
        m = 0.5 * (lo + hi)
        below = m * (13 + m * (96 + m * (-160 + 80 * m))) / 29 < u
        lo, hi = torch.where(below, m, lo), torch.where(below, hi, m)
    return 0.5 * (lo + hi)


def _lanes(p, c0, cells, count, V):
    """Algorithm 1 for every (cell, outcome): the changes of V [cells, width, 3]
    summed over the K outcomes."""
    K, G, w = p["K"], len(cells), V.shape[1]
    dt_w = _sg_max(p) * (p["n_phys"] / p["n_particles"]) * p["dt"] * p["n"] ** 3
    cell, c = cells.repeat_interleave(K), count.repeat_interleave(K)
    o = torch.arange(K, device="cuda").repeat(G) << 8
    zero = torch.zeros_like(cell)
    first = _philox(zero + c0, cell, zero, o | 1, p["seed"])
    N = torch.where(c >= 2, torch.floor((c * (c - 1)).to(F64) * dt_w * 0.5 + _u32(first[0])), torch.zeros_like(c, dtype=F64))
    N = N.long()
    W = V.repeat_interleave(K, 0).reshape(-1, 3)
    for s in range(int(N.max()) if len(N) else 0):
        L = torch.nonzero(N > s)[:, 0]
        z = zero[L]
        u = _philox(z + c0, cell[L], z + s, o[L], p["seed"])
        i = (u[0] * c[L]) >> 32
        j = (u[1] * (c[L] - 1)) >> 32
        j = j + (j >= i).long()
        i, j = L * w + i, L * w + j
        vi, vj = W[i], W[j]
        g2 = ((vi - vj) ** 2).sum(1)
        hit = torch.nonzero(_u32(u[2]) < _sg(p, g2.detach()) / _sg_max(p))[:, 0]
        if len(hit) == 0:
            continue
        L, i, j, vi, vj = L[hit], i[hit], j[hit], vi[hit], vj[hit]
        k = s + 1
        uchi = _philox(zero[L] + c0, cell[L], zero[L] + (k >> 2), o[L] | 1, p["seed"])[k & 3]
        cchi = 1 - 2 * _chi(p, _u32(uchi))
        schi, eps = torch.sqrt(1 - cchi * cchi), TAU * _u32(u[3][hit])
        nv = torch.stack([torch.cos(eps) * schi, torch.sin(eps) * schi, cchi], 1)
        cm, hg = 0.5 * (vi + vj), 0.5 * torch.sqrt(g2[hit])[:, None] * nv
        if W.requires_grad:
            W = W.index_put((i,), cm + hg).index_put((j,), cm - hg)
        else:
            W[i], W[j] = cm + hg, cm - hg
    return (W.reshape(G, K, w, 3) - V[:, None]).sum(1)


def _collide(p, x, v, c0, t):
    """<dv> and <dv^M> [N, 3] of one collision call."""
    nc = p["n"] ** 3
    _, cell = _cells(p, x)
    count = torch.bincount(cell, minlength=nc)
    order = torch.argsort(cell, stable=True)
    start = torch.cumsum(count, 0) - count
    slot = torch.empty_like(order)
    slot[order] = torch.arange(len(order), device="cuda") - start[cell[order]]
    if p["K"] == 0:
        return torch.zeros_like(v), torch.zeros_like(v)
    width = int(count.max())
    per = max(1, int(2.5e8 // (24 * width * p["K"])))
    sums = []
    for lo in range(0, nc, per):
        cells = torch.arange(lo, min(nc, lo + per), device="cuda")
        ids = order[start[lo]:start[cells[-1]] + count[cells[-1]]]
        V = torch.zeros(len(cells) * width, 3, dtype=F64, device="cuda")
        at = (cell[ids] - lo) * width + slot[ids]
        V = V.index_put((at,), v[ids])
        d = _lanes(p, c0, cells, count[cells], V.reshape(len(cells), width, 3))
        sums.append(d.reshape(-1, 3)[at])
    dv = torch.zeros_like(v).index_put((order,), torch.cat(sums) / p["K"])
    return dv, _source(p, v, count[cell], t)


def _steps(p, x, v, steps, E_app=0.0):
    """The state after ``steps`` steps from t = 0, with phi and E there."""
    xi = _xi(p, torch.arange(p["n_particles"], device="cuda"))
    dt, paper = p["dt"], p.get("dist", 0)
    vm = _tau(xi[:, 3:]) if paper else _vm(p, xi[:, 3:], 0.0)
    zero = torch.zeros(3, dtype=F64, device="cuda")
    scale = lambda t: _vh(p, t)[0] if paper else zero + 1.0  # noqa: E731
    rate = lambda t: dt * vm * _vh(p, t)[1] if paper else zero  # noqa: E731

    def collided(c0, t):
        if p["K"] == 0:
            return 0.0
        a, m = _collide(p, x, v, c0, t)
        return a - m

    phi, E = _field(p, x, 0.0)
    L = _lorentz(p, x, E, 0.0, E_app)
    for k in range(steps):
        t0, th, t1 = k * dt, (k + 0.5) * dt, (k + 1) * dt
        v = v + 0.5 * (L + collided(2 * k, t0) + rate(t0))
        x = x + dt * (v + _xm(p, xi[:, :3], th)[1] - vm * scale(th))
        x = x - torch.floor(x.detach())
        phi, E = _field(p, x, t1)
        L = _lorentz(p, x, E, t1, E_app)
        v = v + 0.5 * (L + collided(2 * k + 1, th) + rate(t1))
    return x, v, phi, E, xi


def _norms(p, x, v, phi, xi, t):
    e = x - _xm(p, xi[:, :3], t)[0]
    e = e - torch.floor(e + 0.5)
    ev = v - _vm(p, xi[:, 3:], t)
    ep = phi - _phi_m(p, t)[0]
    rms = lambda u: torch.sqrt((u * u).mean(0))  # noqa: E731
    return torch.cat([rms(e), rms(ev), rms(ep)[None], e.abs().amax(0), ev.abs().amax(0), ep.abs().max()[None]])


def _sampled(p, steps):
    xi = _xi(p, torch.arange(p["n_particles"], device="cuda"))
    x, v, phi, _, xi = _steps(p, _xm(p, xi[:, :3], 0.0)[0], _vm(p, xi[:, 3:], 0.0), steps)
    return _norms(p, x, v, phi, xi, steps * p["dt"]), (x, v)


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        b = torch.randn(case["n"] ** 3, generator=_generator(seed), device="cuda", dtype=F64)
        phi, E = _solve(case["n"], b)
        return phi, E.T.contiguous()
    if kind == "batch":
        each = [_sampled(p, case["steps"]) for p in _replicates(case, seed)]
        return dict(norms=torch.stack([e[0] for e in each]), state=[e[1] for e in each])
    p = _params(case, seed)
    if kind == "gradient":
        v0 = _own_state(p, seed)[1].requires_grad_(True)
        E_app = torch.full((3,), 0.1, dtype=F64, device="cuda", requires_grad=True)
        xi = _xi(p, torch.arange(p["n_particles"], device="cuda"))
        x, v, _, E, xi = _steps(p, _xm(p, xi[:, :3], 0.0)[0], v0, case["steps"], E_app)
        field = 0.5 * p["eps0"] / p["n"] ** 3 * (E * E).sum()
        vel = ((v - _vm(p, xi[:, 3:], 0.0)) ** 2).sum() / p["n_particles"]
        dE, dv = torch.autograd.grad(field + vel, (E_app, v0))
        J, Jf, Jv = (float(u.detach()) for u in (field + vel, field, vel))
        return {"J": J, "J_field": Jf, "J_vel": Jv, "dJ_dEapp": dE, "dJ_dv0": dv}
    if p["n_particles"] > 3e7:
        return None  # the collisions of 134M particles in plain torch take minutes
    if kind == "run":
        norms, state = _sampled(p, case["steps"])
        return dict(norms=norms, state=state)
    x, v = _own_state(p, seed)
    if kind == "collide":
        return _collide(p, x, v, 0, 0.0)
    return _steps(p, x, v, case["steps"])[:2]
