"""The measured cases: what a user of the marching library has it do, through its public
entry points (Context, autograd.march), over the sizes and options that are used.

    listed()            the named cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) the inputs and the context that a user's program holds
    run(state)          one pass through the public calls
    work(case)          bytes and flops that a pass cannot do without
    exact(case, seed)   the outputs in 64 bits by plain numpy / torch (small cases)

Kinds of case:
  march     a march from rest over the pulse of a seeded plane wave, in chunks: the tested
            excitation of a chunk, its staging, the march.  `record` steps at the end are
            returned.  FP32-history currents are kept as float32, the accuracy they have.
  rhs       several plane waves on one scatterer, marched as right-hand sides
  gradient  one optimisation step: forward march, objective weights, checkpointed adjoint
  probes    the scattered field at probes around the grid and its transpose
  wave      the tested plane wave alone
  lanczos   extreme eigenvalues of the stability operator
"""
import math

import numpy as np
import torch

from paper_2407_03323_gb300 import Context, autograd

BF = 4.0 * math.pi


def listed():
    return [
        # the first thing a user tries, defaults throughout: a small cube, every lag direct
        _march("cube8_fp64", "cube", 8, 8, 8, 4.0, "fp64", "direct", 0, 96, 96),
        # a small scatterer in a parameter study: launch and barrier latency
        _march("sphere9_fp32", "sphere", 9, 9, 9, 12.0, "fp32_history", "blocked", 4, 128, 128),
        # the mid-size sphere of the precision studies, in the fast mode
        _march("sphere32_fp32", "sphere", 32, 32, 32, 12.0, "fp32_history", "blocked", 8, 192, 192),
        # the same in the reference precision
        _march("sphere32_fp64", "sphere", 32, 32, 32, 12.0, "fp64", "blocked", 8, 128, 128),
        # the large sphere, the framework's headline run
        _march("sphere104_fp32", "sphere", 104, 104, 104, 12.0, "fp32_history", "blocked", 8, 192, 64),
        # an elongated body with odd sides: ragged tiles, long lag windows, general FFT lengths
        _march("box133_fp32", "noise", 133, 27, 21, 12.0, "fp32_history", "blocked", 8, 128, 128),
        # an inhomogeneous block with numpy arrays in and out (the shortest program)
        dict(_march("block24_host", "noise", 24, 24, 24, 12.0, "fp64", "direct", 0, 64, 64), host=True),
        # the excitations of one scatterer of the batched study
        {"name": "rhs8_24_fp32", "kind": "rhs", "shape": "cube", "U": 24, "V": 24, "W": 24,
         "eps": 8.0, "precision": "fp32_history", "scheme": "blocked", "block": 8, "steps": 64,
         "n_rhs": 8},
        # a step of the inverse problem: gradient with respect to every permittivity
        {"name": "gradient20", "kind": "gradient", "shape": "noise", "U": 20, "V": 20, "W": 20,
         "eps": 12.0, "precision": "fp64", "scheme": "blocked", "block": 8, "steps": 96,
         "every": 48},
        # the objective of that problem and its source: the field at probes around the body
        {"name": "probes24", "kind": "probes", "shape": "noise", "U": 24, "V": 24, "W": 24,
         "eps": 12.0, "n_probes": 64, "steps": 128},
        # tested excitation of the headline run, one chunk
        {"name": "wave104", "kind": "wave", "shape": "sphere", "U": 104, "V": 104, "W": 104,
         "eps": 12.0, "steps": 32},
        # the stability analysis of a cube before a long march
        {"name": "lanczos20", "kind": "lanczos", "shape": "cube", "U": 20, "V": 20, "W": 20,
         "eps": 12.0, "k": 96},
    ]


def _march(name, shape, U, V, W, eps, precision, scheme, block, steps, record):
    return {"name": name, "kind": "march", "shape": shape, "U": U, "V": V, "W": W, "eps": eps,
            "precision": precision, "scheme": scheme, "block": block, "steps": steps,
            "record": record, "host": False}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["march", "march", "march", "march", "rhs", "gradient", "probes", "wave",
                       "lanczos"])
    shape = rng.choice(["cube", "sphere", "noise"])
    eps = round(rng.uniform(2.0, 30.0), 3)
    c = {"kind": kind, "shape": shape, "eps": eps}
    if kind == "march":
        precision = rng.choice(["fp32_history", "fp64"])
        scheme = rng.choice(["blocked", "blocked", "direct"])
        top = {("fp32_history", "blocked"): 90, ("fp32_history", "direct"): 48,
               ("fp64", "blocked"): 40, ("fp64", "direct"): 28}[precision, scheme]
        N = _log_int(rng, 6, top)
        sides = [max(3, int(round(N * rng.uniform(0.75, 1.2)))) for _ in range(3)]
        steps = _log_int(rng, 64, 192)
        c.update(U=sides[0], V=sides[1], W=sides[2], precision=precision, scheme=scheme,
                 block=rng.choice([4, 8]) if scheme == "blocked" else 0, steps=steps,
                 record=min(steps, 64), host=rng.random() < 0.25)
    elif kind == "rhs":
        N = rng.randint(12, 32)
        c.update(U=N, V=N, W=N, precision="fp32_history", scheme="blocked",
                 block=rng.choice([4, 8]), steps=rng.randint(32, 64), n_rhs=rng.randint(2, 8))
    elif kind == "gradient":
        N = rng.randint(8, 22)
        steps = rng.randint(48, 96)
        c.update(U=N, V=rng.randint(8, 22), W=N, precision="fp64",
                 scheme=rng.choice(["blocked", "direct"]), steps=steps, every=steps // 2)
        c["block"] = 4 if c["scheme"] == "blocked" else 0
    elif kind == "probes":
        N = rng.randint(9, 26)
        c.update(U=N, V=N, W=N, n_probes=rng.randint(8, 64), steps=rng.randint(32, 128))
    elif kind == "wave":
        N = _log_int(rng, 12, 104)
        c.update(U=N, V=N, W=max(3, N - rng.randint(0, 3)), steps=rng.randint(16, 32))
    else:
        N = rng.randint(8, 22)
        c.update(U=N, V=N, W=N, k=rng.randint(40, 96))
    return c


# ------------------------------------------------------------------ inputs

def _geometry(case, rng):
    """eps_r [W][V][U] of the case's shape."""
    U, V, W, eps = case["U"], case["V"], case["W"], case["eps"]
    if case["shape"] == "cube":
        return np.full((W, V, U), float(eps))
    if case["shape"] == "sphere":            # the ellipsoid that fills the box
        x, y, z = (((np.arange(n) + 0.5) / n * 2.0 - 1.0) ** 2 for n in (U, V, W))
        inside = z[:, None, None] + y[None, :, None] + x[None, None, :] < 1.0
        return np.where(inside, float(eps), 1.0)
    # smoothed noise up to eps; the thinnest material stays well above vacuum
    g = rng.uniform(size=(W, V, U))
    f = [np.fft.fftfreq(n) for n in (W, V, U)]
    k2 = f[0][:, None, None] ** 2 + f[1][None, :, None] ** 2 + f[2][None, None, :] ** 2
    g = np.real(np.fft.ifftn(np.fft.fftn(g) * np.exp(-2.0 * (2.0 * math.pi) ** 2 * k2)))
    return 1.0 + (eps - 1.0) * (0.1 + 0.9 * (g - g.min()) / (g.max() - g.min()))


def _wave(case, rng):
    """A plane wave from a random direction: ten voxels a wavelength inside the body, an
    amplitude spectrum of half the centre frequency, and the first of `steps` steps that
    cover the middle of its pulse."""
    k = rng.normal(size=3)
    k /= np.linalg.norm(k)
    p = rng.normal(size=3)
    p -= np.dot(p, k) * k
    p /= np.linalg.norm(p)
    f_c = 1.0 / (10.0 * math.sqrt(case["eps"]))
    sigma_t = 2.0 * math.sqrt(2.0 * math.log(2.0)) / (2.0 * math.pi * 0.5 * f_c)
    size = np.array([case["U"], case["V"], case["W"]], float)
    far = float(np.sum(np.maximum(size * k, 0.0)))
    t0 = 6.0 * sigma_t + far
    first = max(1, int(round(t0 + 0.5 * float(np.dot(size, k)) - 0.6 * case.get("steps", 1))))
    return {"k_hat": k, "p_hat": p, "f_c": f_c, "sigma_t": sigma_t, "t0": t0, "first": first}


def _taps(case):
    """The three-tap regularisation, 1e-7 per voxel; none for homogeneous cubes."""
    M = case["U"] * case["V"] * case["W"]
    return np.zeros(0) if case["shape"] == "cube" else 1e-7 * M * np.array([0.25, -0.5, 0.25])


def _inputs(case, seed):
    rng = np.random.default_rng([seed, 2407])
    eps_r = _geometry(case, rng)
    waves = [_wave(case, rng) for _ in range(case.get("n_rhs", 1))]
    return eps_r, _taps(case), waves, rng


def _options(case):
    return {"precision": case["precision"], "scheme": case["scheme"], "block": case["block"]}


def _chunks(case):
    """(first step, steps) of each chunk of a march: the unrecorded steps, then the recorded."""
    n, r = case["steps"], case["record"]
    if case["host"]:
        return [(0, n)]
    ends = list(range(0, n - r, 64)) + [n - r]
    return [(a, b - a) for a, b in zip(ends, ends[1:])] + [(n - r, r)]


def prepare(case, seed):
    eps_r, taps, waves, rng = _inputs(case, seed)
    kind, M = case["kind"], eps_r.size
    s = {"case": case, "kind": kind, "waves": waves}

    def device(*shape):
        return torch.empty(shape, dtype=torch.float64, device="cuda")

    if kind in ("march", "rhs"):
        s["ctx"] = Context(eps_r, taps, **_options(case))
    if kind == "march":
        s["chunks"] = _chunks(case)
        if case["host"]:
            w = waves[0]
            s["E"] = s["ctx"].plane_wave(w["k_hat"], w["p_hat"], w["f_c"], w["sigma_t"], w["t0"],
                                         w["first"], case["steps"])
        else:
            s["E"] = device(max(n for _, n in s["chunks"]), M, 3)
            s["J"] = device(case["record"], M, 3)
    elif kind == "rhs":
        s["E"] = device(case["n_rhs"], case["steps"], M, 3).zero_()
        s["J"] = device(case["n_rhs"], case["steps"], M, 3)
        torch.cuda.synchronize()
        s["ctx"].set_excitation_rhs(s["E"])      # makes the right-hand sides' states
    elif kind == "gradient":
        s["eps"] = torch.from_numpy(eps_r)
        s["taps"] = taps
        s["weight"] = torch.from_numpy(rng.normal(size=(case["steps"], M, 3))).cuda()
    elif kind == "probes":
        s["ctx"] = Context(eps_r, None, precision="fp32_history")
        N = case["U"]
        q = rng.normal(size=(case["n_probes"], 3))
        q *= 2.0 * N / np.linalg.norm(q, axis=1, keepdims=True)
        s["ctx"].probe_setup(np.floor(q + N / 2.0).astype(np.int32))
        s["J"] = torch.from_numpy(rng.normal(size=(case["steps"], M, 3))).cuda()
        s["W"] = torch.from_numpy(rng.normal(size=(case["steps"], case["n_probes"], 3))).cuda()
        s["E"] = device(case["steps"], case["n_probes"], 3)
        s["g"] = device(case["steps"], M, 3)
    elif kind == "wave":
        s["ctx"] = Context(eps_r, taps, precision="fp32_history", scheme="blocked", block=8)
        s["E"] = device(case["steps"], M, 3)
    else:
        s["ctx"] = Context(eps_r, taps)
        s["seed"] = int(seed)
    return s


# ------------------------------------------------------------------ one pass

def _plane_wave(ctx, w, at, out):
    ctx.plane_wave(w["k_hat"], w["p_hat"], w["f_c"], w["sigma_t"], w["t0"], w["first"] + at,
                   out.shape[0], out=out)


def run(s):
    case, kind = s["case"], s["kind"]
    if kind == "march":
        ctx = s["ctx"]
        ctx.restart(0, None)
        if case["host"]:
            ctx.set_excitation(s["E"])
            J = ctx.march(case["steps"])
        else:
            J = s["J"]
            for at, n in s["chunks"]:
                E = s["E"][:n]
                _plane_wave(ctx, s["waves"][0], at, E)
                ctx.set_excitation(E)
                ctx.march(n, out=J if at == case["steps"] - case["record"] else None)
        if case["precision"] == "fp64":
            return J
        return J.astype(np.float32) if case["host"] else J.float()
    if kind == "rhs":
        ctx = s["ctx"]
        for r, w in enumerate(s["waves"]):
            _plane_wave(ctx, w, 0, s["E"][r])
            ctx.rhs(r).restart(0, None)
        ctx.set_excitation_rhs(s["E"])
        ctx.march_rhs(case["steps"], out=s["J"])
        return s["J"].float()
    if kind == "gradient":
        eps = s["eps"].clone().requires_grad_(True)
        w = dict(s["waves"][0])
        w["t0"] = w["t0"] - (w["first"] - 1)
        J = autograd.march(eps, s["taps"], w, case["steps"], checkpoint_every=case["every"],
                           **_options(case))
        (J * s["weight"]).sum().backward()
        return {"J": J.detach(), "grad": eps.grad}
    if kind == "probes":
        ctx = s["ctx"]
        ctx.probe_field(s["J"], out=s["E"])
        ctx.probe_transpose(s["W"], out=s["g"])
        return {"E": s["E"], "g": s["g"]}
    if kind == "wave":
        _plane_wave(s["ctx"], s["waves"][0], 0, s["E"])
        return s["E"]
    ctx = s["ctx"]
    r = ctx.pdsa_lanczos(ctx.ell, case["k"], seed=s["seed"], reorth=True, n_out=4)
    return {"ritz": r["ritz"], "theta_max": r["theta_max"]}


# ------------------------------------------------------------------ what a pass needs

def _ell(case):
    return int(math.floor(math.sqrt(case["U"] ** 2 + case["V"] ** 2 + case["W"] ** 2))) + 2


def work(case):
    """Bytes: inputs and outputs once (for a march every step's excitation and its J where
    it is returned) and the interaction elements once.  Flops: for each step the two
    zero-padded transforms of three components (2.5 n log2 n each), the products of the
    lags (36 a bin and lag for the direct sum; log2(ell / B) levels of temporal transforms
    and products, 60 log2(2 S) + 144 a bin, for the blocked one) and ten products with the
    27-point operator."""
    kind = case["kind"]
    M = case["U"] * case["V"] * case["W"]
    ell = _ell(case)
    table = 6.0 * 8 * 8 * M
    if kind == "wave":
        return {"bytes": 24.0 * M * case["steps"], "flops": 60.0 * M * case["steps"]}
    if kind == "probes":
        pairs = float(case["n_probes"]) * M
        return {"bytes": 2.0 * 24 * (M + case["n_probes"]) * case["steps"] + 6 * 8 * 8 * pairs,
                "flops": 2.0 * 2 * 9 * 8 * pairs * case["steps"]}
    P = [2.0 * case[a] - 1 for a in "UVW"]
    n = P[0] * P[1] * P[2]
    bins = n / 2
    fft = 2.0 * 3 * 2.5 * n * math.log2(max(n, 2.0))
    if kind == "lanczos":
        k = case["k"]
        return {"bytes": 24.0 * M * (k + 1), "flops": k * (fft + 30 * bins) + 4.0 * 3 * M * k * k}
    if case["scheme"] == "direct":
        lags = 36.0 * ell * bins
    else:
        B = case["block"]
        levels = max(0, int(math.ceil(math.log2(ell / B))))
        lags = bins * (36.0 * (B - 1) + sum(60.0 * math.log2(2 * B * 2 ** i) + 144.0
                                            for i in range(levels)))
    step = fft + lags + 10 * 150.0 * M
    many = case["steps"] * (3.0 if kind == "gradient" else case.get("n_rhs", 1))
    out = case.get("record", case["steps"]) * case.get("n_rhs", 1)
    size = 4 if case["precision"] == "fp32_history" else 8
    return {"bytes": 24.0 * M * many + 3.0 * size * M * out + table, "flops": many * step}


# ------------------------------------------------------------------ the outputs in 64 bits

def exact(case, seed):
    M = case["U"] * case["V"] * case["W"]
    if case["kind"] == "wave":
        eps_r, _, waves, _ = _inputs(case, seed)
        return _tested(eps_r, waves[0], case["steps"])
    if case["kind"] == "march" and M <= 730 and not case["host"]:
        eps_r, taps, waves, _ = _inputs(case, seed)
        E = _tested(eps_r, waves[0], case["steps"]).cpu().numpy()
        return _direct_march(eps_r, taps, E)[case["steps"] - case["record"]:]
    return None


def _tested(eps_r, w, steps):
    """chi p times the pulse averaged over every voxel by a tensor Gauss rule: [n][M][3]."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    W, V, U = eps_r.shape
    x, g = np.polynomial.legendre.leggauss(7)
    x, g = 0.5 * x, 0.5 * g
    k = w["k_hat"]
    off = (x[:, None, None] * k[2] + x[None, :, None] * k[1] + x[None, None, :] * k[0]).ravel()
    wt = (g[:, None, None] * g[None, :, None] * g[None, None, :]).ravel()
    c = [torch.arange(n, dtype=torch.float64, device=dev) + 0.5 for n in (W, V, U)]
    r = (c[0][:, None, None] * k[2] + c[1][None, :, None] * k[1] + c[2][None, None, :] * k[0])
    r = r.reshape(-1)
    chi = torch.from_numpy((eps_r - 1.0) / eps_r).to(dev).reshape(-1)
    p = torch.from_numpy(w["p_hat"]).to(dev)
    out = torch.empty((steps, r.numel(), 3), dtype=torch.float64, device=dev)
    for i in range(steps):
        acc = torch.zeros_like(r)
        for o, t in zip(off, wt):
            tau = (w["first"] + i - w["t0"]) - (r + o)
            acc += t * torch.sin(2.0 * math.pi * w["f_c"] * tau) * torch.exp(
                -tau * tau / (2.0 * w["sigma_t"] ** 2))
        out[i] = (chi * acc)[:, None] * p[None, :]
    return out


def _hat(x, d, slope):
    """The unit hat about d, or its derivative."""
    y = x - d
    if slope:
        return np.where((y > -1) & (y < 0), 1.0, np.where((y > 0) & (y < 1), -1.0, 0.0))
    return np.maximum(0.0, 1.0 - np.abs(y))


def _pieces(a, b, rule):
    """Nodes and weights of a rule on [-1, 1] on the intervals [a, b] (last axis added)."""
    h = 0.5 * (b - a)[..., None]
    return 0.5 * (a + b)[..., None] + h * rule[0], h * rule[1]


_ARC = np.polynomial.legendre.leggauss(12)
_AXIAL = np.polynomial.legendre.leggauss(18)


def _end_rule(n=44, p=3):
    """Gauss nodes after u^p / (u^p + (1-u)^p), for square roots and logarithms at the ends."""
    x, g = np.polynomial.legendre.leggauss(n)
    u = 0.5 * (x + 1.0)
    a, b = u ** p, (1.0 - u) ** p
    return 2.0 * a / (a + b) - 1.0, g * p * (u * (1.0 - u)) ** (p - 1) / (a + b) ** 2


_RADIAL = _end_rule()


def _bins(r, w, second, shell, out):
    """Adds w f(l - r) / (4 pi) for the three lags l that a radius in `shell` reaches, f the
    quadratic B-spline of time or its second derivative."""
    q = r - shell
    vals = (1.0, -2.0, 1.0) if second else (0.5 * (1 - q) ** 2, 0.5 * (1 + 2 * q - 2 * q * q), 0.5 * q * q)
    for i, v in enumerate(vals):
        out += np.bincount(shell + i, weights=w * v / BF, minlength=out.size)[:out.size]


def _axis(dp, dq, dz, nlag):
    """Lag series of three integrals over the overlap of two voxels (p, q, z) apart, in
    cylinder coordinates about z: the hats' product against the second time derivative, its
    second z-derivative and its mixed p, q derivative against the spline itself."""
    kp, kq, kz = (d + np.array([-1.0, 0.0, 1.0]) for d in (dp, dq, dz))
    smax = math.hypot(np.abs(kp).max(), np.abs(kq).max())
    J = np.arange(1, int(math.hypot(smax, np.abs(kz).max())) + 2, dtype=float)
    cross = J[:, None] ** 2 - kz[None, :] ** 2
    cuts = np.concatenate([[0.0, smax], np.abs(kp), np.abs(kq), J,
                           np.hypot(kp[:, None], kq[None, :]).ravel(),
                           np.sqrt(np.maximum(cross, 0.0)).ravel()])
    cuts = np.unique(np.clip(cuts, 0.0, smax))
    cuts = cuts[np.concatenate([[True], np.diff(cuts) > 1e-13])]
    s, ws = _pieces(cuts[:-1], cuts[1:], _RADIAL)
    s, ws = s.ravel(), ws.ravel()
    # angular integrals of the hats over the circle of radius s, cut where it meets a knot
    ap = np.arccos(np.clip(kp[None, :] / s[:, None], -1, 1))
    aq = np.arcsin(np.clip(kq[None, :] / s[:, None], -1, 1))
    ang = np.concatenate([ap, -ap, aq, math.pi - aq, np.full((s.size, 1), -math.pi)], axis=1)
    ang = np.sort(np.mod(ang + math.pi, 2 * math.pi) - math.pi, axis=1)
    ang = np.concatenate([ang, np.full((s.size, 1), math.pi)], axis=1)
    phi, wp = _pieces(ang[:, :-1], ang[:, 1:], _ARC)
    x, y = s[:, None, None] * np.cos(phi), s[:, None, None] * np.sin(phi)
    oL = ws * s * np.sum(wp * _hat(x, dp, False) * _hat(y, dq, False), axis=(1, 2))
    oD = ws * s * np.sum(wp * _hat(x, dp, True) * _hat(y, dq, True), axis=(1, 2))
    vol, diag, off = np.zeros(nlag), np.zeros(nlag), np.zeros(nlag)
    for z, c in zip(kz, (1.0, -2.0, 1.0)):
        r = np.hypot(s, z)
        _bins(r, c * oL / r, False, np.floor(r).astype(int), diag)
    # axial integrals with z = s sinh u (dz / r = du), cut at the knots and the unit shells
    live = (np.abs(oL) > 0) | (np.abs(oD) > 0)
    s, oL, oD = s[live], oL[live], oD[live]
    zc = np.sqrt(np.maximum(J[None, :] ** 2 - s[:, None] ** 2, 0.0))
    z = np.clip(np.concatenate([np.broadcast_to(kz, (s.size, 3)), zc, -zc], axis=1), kz[0], kz[2])
    z.sort(axis=1)
    u = np.arcsinh(z / s[:, None])
    i, j = np.nonzero(z[:, 1:] - z[:, :-1] > 1e-15)
    un, wu = _pieces(u[i, j], u[i, j + 1], _AXIAL)
    zn = s[i][:, None] * np.sinh(un)
    rn = s[i][:, None] * np.cosh(un)
    shell = np.floor(np.hypot(s[i], 0.5 * (z[i, j] + z[i, j + 1]))).astype(int)
    shell = np.broadcast_to(shell[:, None], rn.shape).ravel()
    wu = wu * _hat(zn, dz, False)
    _bins(rn.ravel(), (wu * oL[i][:, None]).ravel(), True, shell, vol)
    _bins(rn.ravel(), (wu * oD[i][:, None]).ravel(), False, shell, off)
    return vol, diag, off


def _direct_march(eps_r, taps, E):
    """Z_0 J_n = E_n - sum_l Z_l J_{n-l} with dense matrices on the voxels that carry current."""
    W, V, U = eps_r.shape
    ell = int(math.floor(math.sqrt(U * U + V * V + W * W))) + 2
    L = ell + 1
    done = {}
    Goct = np.zeros((L, 3, 3, W, V, U))
    for dz in range(W):
        for dy in range(V):
            for dx in range(U):
                d = (dx, dy, dz)
                order = sorted(range(3), key=lambda a: -d[a])
                key = tuple(d[a] for a in order)
                if key not in done:
                    K = np.zeros((L, 3, 3))
                    for p, q, z in ((0, 1, 2), (1, 2, 0), (2, 0, 1)):
                        vol, diag, off = _axis(float(key[p]), float(key[q]), float(key[z]), L)
                        K[:, z, z] = diag - vol
                        K[:, p, q] = K[:, q, p] = off
                    done[key] = K
                at = np.argsort(order)
                Goct[:, :, :, dz, dy, dx] = done[key][:, at][:, :, at]
    chi = ((eps_r - 1.0) / eps_r).ravel()
    act = np.nonzero(chi > 0.0)[0]
    pos = np.stack([act % U, (act // U) % V, act // (U * V)], axis=1)
    dd = pos[:, None, :] - pos[None, :, :]
    ab, sg = np.abs(dd), np.sign(dd)
    n = act.size
    d0 = np.zeros(L)
    d0[:min(L, len(taps))] = taps[:L]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    Z = torch.empty((L, 3 * n, 3 * n), dtype=torch.float64, device=dev)
    for l in range(L):
        T = 0.5 if l < 2 else 0.0
        z = np.zeros((n, 3, n, 3))
        for a in range(3):
            for b in range(3):
                g = Goct[l, a, b][ab[..., 2], ab[..., 1], ab[..., 0]]
                if a != b:
                    g = g * sg[..., a] * sg[..., b]
                z[:, a, :, b] = -chi[act][:, None] * g
                if a == b:
                    z[np.arange(n), a, np.arange(n), b] += T * (1.0 - chi[act]) + d0[l]
        Z[l] = torch.from_numpy(z.reshape(3 * n, 3 * n))
    lu = torch.linalg.lu_factor(Z[0])
    Ea = torch.from_numpy(np.ascontiguousarray(E[:, act])).to(dev).reshape(len(E), 3 * n)
    J = torch.zeros_like(Ea)
    for i in range(len(E)):
        rhs = Ea[i].clone()
        for l in range(1, min(ell, i) + 1):
            rhs -= Z[l] @ J[i - l]
        J[i] = torch.linalg.lu_solve(*lu, rhs[:, None])[:, 0]
    out = np.zeros((len(E), chi.size, 3))
    out[:, act] = J.reshape(len(E), n, 3).cpu().numpy()
    return out
