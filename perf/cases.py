"""What a user of the framework runs, as measurable cases.

A program that uses this package holds a particle set on the GPU and a
``Context``, and calls ``Context.step`` in its time loop; or it
differentiates through steps (``autograd.step``), advances sync intervals of
hierarchical steps (``Context.step_hier``), or runs a single pass on frozen
inputs (``Context.gradients``, ``Context.hydro_fluxes``).  The cases are those
calls on the configured workloads (``inputs.py``: Sod, Sedov, turbulence,
Kelvin-Helmholtz, the many-box ensemble) at the sizes of the configurations
and tests, from the smallest box to 128^3, with odd lattices between them.

A time loop's step advances the state in place, so repeated passes of a step
case walk through the run, from the jittered lattice on.

Derivatives and the flux pass are taken in double precision: a gradient
through the slope limiter jumps wherever two neighbours tie to rounding, so
single-precision gradients say nothing to better than about 1e-3, and the
flux pass hands its rates out as float64 whatever the working precision.
"""
import math

import numpy as np
import torch

import paper_1712_01294_gb300 as gz
from paper_1712_01294_gb300 import autograd as gza

GAMMA = 5.0 / 3.0
NGB = 32.0
STATE = ("x", "y", "z", "vx", "vy", "vz", "m", "u", "h")
NMIN, NMAX = 8, 24  # lattice edges of the ensemble's boxes


# --------------------------------------------------------------- the cases
def _case(name, op, kind, n, **kw):
    c = {"op": op, "kind": kind, "n": n, "precision": "fp32", "scheme": "mfm", "riemann": "hllc"}
    c.update(kw)
    if name:
        c = {"name": name, **c}
    return c


def listed():
    return [
        # one small box on its own: a unit test, a parameter scan; launches count
        _case("step_sod_16", "step", "sod", 16),
        # the configured Sod tube
        _case("step_sod_32", "step", "sod", 32),
        # an odd lattice between the configured sizes, contact layers
        _case("step_kh_41", "step", "kh", 41),
        # the configured Sedov blast: strong contrasts, an emptying centre
        _case("step_sedov_64", "step", "sedov", 64),
        # the headline workload: one large turbulent box
        _case("step_turb_128", "step", "turb", 128),
        # the configured ensemble: 256 uneven boxes in the same launches
        _case("step_ensemble_256", "step", "ens", 256),
        # double precision, as reference runs and derivative checks use it
        _case("step_turb_48_fp64", "step", "turb", 48, precision="fp64"),
        # the MFV scheme (mass crosses the faces)
        _case("step_turb_80_mfv", "step", "turb", 80, scheme="mfv"),
        # the exact Riemann solver on every face
        _case("step_sod_50_exact", "step", "sod", 50, riemann="exact"),
        # one differentiable step, forward and backward (inversion, sensitivities)
        _case("grad_kh_40_fp64", "grad", "khs", 40, precision="fp64"),
        # the gradient pass on frozen inputs (a host code that owns the rest)
        _case("gradients_turb_75", "gradients", "turb", 75),
        # one sync interval of hierarchical steps on a blast
        _case("hier_sedov_64", "hier", "sedov", 64, K=4),
    ]


def _edge(rng, lo, hi):
    """A lattice edge, particle counts spread over their logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["step", "step", "step", "step", "grad", "fluxes", "gradients", "hier"])
    if op == "step":
        kind = rng.choice(["sod", "sedov", "turb", "kh", "ens"])
        if kind == "ens":
            return _case(None, op, kind, rng.randint(5, 256))
        option = rng.choice(["plain", "plain", "plain", "fp64", "mfv", "exact", "fallback"])
        if option == "fp64":
            return _case(None, op, kind, _edge(rng, 10, 48), precision="fp64")
        if option == "mfv":
            return _case(None, op, kind, _edge(rng, 12, 110), scheme="mfv")
        if option in ("exact", "fallback"):
            return _case(None, op, kind, _edge(rng, 12, 80), riemann=option)
        return _case(None, op, kind, _edge(rng, 10, 124))
    if op == "grad":
        return _case(None, op, rng.choice(["khs", "turbs"]), _edge(rng, 10, 42), precision="fp64")
    if op == "fluxes":
        return _case(None, op, rng.choice(["turb", "kh", "sod"]), _edge(rng, 10, 48), precision="fp64")
    if op == "hier":
        return _case(None, op, rng.choice(["sedov", "sod"]), _edge(rng, 16, 60), K=rng.randint(1, 4))
    return _case(None, op, rng.choice(["turb", "kh", "sod"]), _edge(rng, 12, 120))


# -------------------------------------------------------------- the inputs
def _counts(case):
    if case["kind"] != "ens":
        return [case["n"] ** 3]
    # edges NMIN..NMAX in a fixed uneven order: the sizes belong to the case
    return [(NMIN + (b * 7 + b // 5) % (NMAX - NMIN + 1)) ** 3 for b in range(case["n"])]


def _h0(N):
    return (3.0 * NGB / (4.0 * math.pi * N)) ** (1.0 / 3.0)


def _lattice(n, g):
    """Jittered cubic lattice, +-0.1 of the spacing per axis; x varies fastest."""
    k = torch.arange(n, device="cuda", dtype=torch.float64)
    kz, ky, kx = torch.meshgrid(k, k, k, indexing="ij")
    base = torch.stack([kx.reshape(-1), ky.reshape(-1), kz.reshape(-1)])
    jit = torch.rand(base.shape, generator=g, device="cuda", dtype=torch.float64) * 0.2 - 0.1
    return torch.remainder((base + 0.5 + jit) / n, 1.0)


def _random_fields(n, g, ncomp, solenoidal):
    """Gaussian fields of power k^-4 per mode on 2 <= |k| <= 16."""
    k1 = torch.fft.fftfreq(n, d=1.0 / n, device="cuda", dtype=torch.float64)
    kz, ky, kx = torch.meshgrid(k1, k1, k1, indexing="ij")
    k2 = kx * kx + ky * ky + kz * kz
    kk = torch.sqrt(k2)
    amp = torch.where((kk >= 2.0) & (kk <= 16.0), kk.clamp(min=1.0) ** -2.0, torch.zeros_like(kk))
    c = [torch.fft.fftn(torch.randn((n, n, n), generator=g, device="cuda", dtype=torch.float64)) * amp
         for _ in range(ncomp)]
    if solenoidal:
        kd = (kx * c[0] + ky * c[1] + kz * c[2]) / torch.where(k2 > 0, k2, torch.ones_like(k2))
        c = [c[0] - kx * kd, c[1] - ky * kd, c[2] - kz * kd]
    f = [torch.fft.ifftn(a).real.reshape(-1) for a in c]
    return [a - a.mean() for a in f]


def _box(kind, n, g, rng):
    """One box (FP64): positions [3, N], velocities [3, N], masses, energies."""
    x = _lattice(n, g)
    N = n ** 3
    v = torch.zeros_like(x)
    one = torch.ones(N, device="cuda", dtype=torch.float64)
    if kind in ("sod", "tube"):
        rr, pr = (0.125, 0.1) if kind == "sod" else (1.0 / rng.uniform(2, 10), 1.0 / rng.uniform(2, 20))
        left = x[0] < 0.5
        rho, P = torch.where(left, one, rr * one), torch.where(left, one, pr * one)
    elif kind in ("sedov", "blast"):
        E = 1.0 if kind == "sedov" else rng.uniform(0.1, 1.0)
        rho, P = one, 1e-6 * one
        r = (x - 0.5).square().sum(0).sqrt()
        d, near = torch.topk(r, 33, largest=False, sorted=True)
        q = d[:32] / d[32]
        w = torch.where(q <= 0.5, 1 - 6 * q ** 2 + 6 * q ** 3, 2 * (1 - q) ** 3)
        u = P / ((GAMMA - 1) * rho)
        u[near[:32]] += w / w.sum() * E * N
        return x, v, rho / N, u
    elif kind in ("turb", "turbs"):
        v = torch.stack(_random_fields(n, g, 3, True))
        v = v * (0.5 * math.sqrt(GAMMA) / v.square().sum(0).mean().sqrt())
        s = _random_fields(n, g, 1, False)[0]
        rho = torch.exp(0.3 * s / s.std() - 0.045)
        rho = rho / rho.mean()
        P = one
        if kind == "turbs":  # smooth pressure: no field exactly uniform (a kink of the limiter)
            P = one + 0.1 * torch.sin(2 * math.pi * x[0]) * torch.cos(2 * math.pi * x[1] + 0.3) \
                + 0.05 * torch.sin(2 * math.pi * (x[2] + x[0]))
    elif kind in ("kh", "khs"):
        phi = rng.random()
        if kind == "kh":
            inside = ((x[1] - 0.5).abs() < 0.25).double()
            P = 2.5 * one
        else:  # smooth interfaces, for derivatives
            inside = 0.5 * (torch.tanh((x[1] - 0.25) / 0.05) - torch.tanh((x[1] - 0.75) / 0.05))
            P = 2.5 * (1 + 0.01 * torch.sin(2 * math.pi * (x[0] + 2 * x[2])) * torch.cos(2 * math.pi * x[1]))
            v[2] = 0.01 * torch.sin(2 * math.pi * (x[1] - x[2] + phi))
        rho = 1.0 + inside
        v[0] = inside - 0.5
        v[1] = 0.01 * torch.sin(4 * math.pi * (x[0] + phi))
    else:
        raise ValueError(kind)
    return x, v, rho / N, P / ((GAMMA - 1) * rho)


def _particles(case, seed):
    """The particle set of a case: dict of CUDA tensors, as Context takes it."""
    g = torch.Generator(device="cuda").manual_seed(1712 + seed)
    rng = np.random.default_rng(1712 + seed)
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    counts = _counts(case)
    parts = []
    for c in counts:
        n = round(c ** (1.0 / 3.0))
        kind = case["kind"]
        if kind == "ens":
            kind = "tube" if rng.random() < 0.5 else "blast"
        parts.append(_box(kind, n, g, rng))
    x, v = (torch.cat([p[k] for p in parts], dim=1).to(dt) for k in (0, 1))
    m, u = (torch.cat([p[k] for p in parts]).to(dt) for k in (2, 3))
    x = torch.where(x >= 1.0, torch.zeros_like(x), x)  # (rounded up to 1)
    h = torch.cat([torch.full((c,), _h0(c), device="cuda", dtype=dt) for c in counts])
    out = {"x": x[0], "y": x[1], "z": x[2], "vx": v[0], "vy": v[1], "vz": v[2], "m": m, "u": u, "h": h}
    out = {k: t.contiguous().clone() for k, t in out.items()}
    out["id"] = torch.arange(x.shape[1], device="cuda", dtype=torch.int64)
    return out


def _context(case):
    prm = gz.default_params(
        precision=gz.GZ_FP64 if case["precision"] == "fp64" else gz.GZ_MIXED32,
        scheme=gz.GZ_MFV if case["scheme"] == "mfv" else gz.GZ_MFM,
        riemann={"hllc": gz.GZ_RIEMANN_HLLC, "exact": gz.GZ_RIEMANN_EXACT,
                 "fallback": gz.GZ_RIEMANN_FALLBACK}[case["riemann"]])
    return gz.Context(_counts(case), prm)


PASS_DT = 0.1  # the frozen flux pass's step, in sound crossings of a support radius


def _adjoint_weights(N, seed, dt):
    g = torch.Generator(device="cuda").manual_seed(99 + seed)
    return {k: torch.randn(N, generator=g, device="cuda", dtype=torch.float64).to(dt)
            for k in ("x", "y", "z", "vx", "vy", "vz", "u")}


def prepare(case, seed):
    p = _particles(case, seed)
    s = {"case": case, "ctx": _context(case), "p": p}
    N = p["x"].numel()
    if case["op"] == "grad":
        s["w"] = _adjoint_weights(N, seed, p["x"].dtype)
        for k in gza.GRADS:
            p[k].requires_grad_(True)
    if case["op"] in ("fluxes", "gradients"):
        # the frozen inputs of the pass, as a caller has them from its own (FP64)
        # passes before: converged H and n, limited gradients and E^-1
        q = {k: t if k == "id" else t.double() for k, t in p.items()}
        ref = _context({**case, "precision": "fp64"})
        n, _ = ref.density(q)
        dt = p["x"].dtype
        p["h"], s["n"] = q["h"].to(dt), n.to(dt)
        if case["op"] == "fluxes":
            s["grad"], s["B"] = (t.to(dt) for t in ref.gradients(q, n))
            s["pass_dt"] = PASS_DT * _h0(N)
        ref.close()
    return s


def run(s):
    ctx, p, op = s["ctx"], s["p"], s["case"]["op"]
    if op == "step":
        ctx.step(p)
        return {k: p[k] for k in STATE}
    if op == "hier":
        ctx.step_hier(p, s["case"]["K"])
        return {k: p[k] for k in STATE}
    if op == "grad":
        new = gza.step(ctx, p)
        outs = [new[k] for k in s["w"]]
        g = torch.autograd.grad(outs, [p[k] for k in gza.GRADS], [s["w"][k] for k in s["w"]])
        return {**{k: new[k] for k in gza.OUT}, "grads": dict(zip(gza.GRADS, g))}
    if op == "fluxes":
        dpdt, dEdt = ctx.hydro_fluxes(p, s["n"], s["grad"], s["B"], s["pass_dt"])
        return {"dpdt": dpdt, "dEdt": dEdt}
    grad, B = ctx.gradients(p, s["n"])
    return {"grad": grad, "B": B}


def work(case):
    """Each input read once, each output written once; the method's arithmetic
    per particle: 28 neighbours, 14.1 unordered flux pairs, 2.65 evaluations of
    the support-radius iteration."""
    N = sum(_counts(case))
    b = 8 if case["precision"] == "fp64" else 4
    density, gradients, fluxes = 2.65 * 28 * 24, 28 * 127 + 60, 14.1 * 276
    if case["scheme"] == "mfv":
        fluxes = 14.1 * 346
    if case["riemann"] == "exact":
        fluxes = 14.1 * (276 + 3 * 60)
    state = (9 * b + 8) + (8 + (case["scheme"] == "mfv")) * b
    step = density + gradients + fluxes
    if case["op"] == "step":
        return {"bytes": N * state, "flops": N * step}
    if case["op"] == "hier":  # the interval's start and its end; at least one step of every particle
        return {"bytes": N * state, "flops": N * step}
    if case["op"] == "grad":
        return {"bytes": N * (state + 15 * b), "flops": N * 3 * step}
    if case["op"] == "fluxes":
        return {"bytes": N * ((9 * b + 8) + 22 * b + 32), "flops": N * fluxes}
    return {"bytes": N * ((9 * b + 8) + b + 21 * b), "flops": N * gradients}


# ------------------------------------------- the same in plain torch, 64 bits
def _wrap_diff(d):
    d = torch.where(d >= 0.5, d - 1.0, d)
    return torch.where(d < -0.5, d + 1.0, d)


def _kern(q):
    inner = 1.0 - 6.0 * q * q + 6.0 * q ** 3
    outer = 2.0 * (1.0 - q) ** 3
    return torch.where(q <= 0.5, inner, torch.where(q < 1.0, outer, torch.zeros_like(q)))


def _kern_d(q):
    inner = -12.0 * q + 18.0 * q * q
    outer = -6.0 * (1.0 - q) ** 2
    return torch.where(q <= 0.5, inner, torch.where(q < 1.0, outer, torch.zeros_like(q)))


def _edges(X, R):
    """Ordered pairs (i, j), j != i, of points X [N, 3] closer than R."""
    N = X.shape[0]
    nc = int(1.0 / R)
    I, J = [], []
    if nc < 4:
        step = max(1, 50_000_000 // N)
        for a in range(0, N, step):
            d = _wrap_diff(X[None, :, :] - X[a:a + step, None, :])
            i, j = torch.nonzero(d.square().sum(2) < R * R, as_tuple=True)
            I.append(i + a)
            J.append(j)
    else:
        c = (X * nc).long().clamp(0, nc - 1)
        lin = (c[:, 0] * nc + c[:, 1]) * nc + c[:, 2]
        order = torch.argsort(lin, stable=True)
        cnt = torch.bincount(lin, minlength=nc ** 3)
        first = torch.cumsum(cnt, 0) - cnt
        width = int(cnt.max())
        table = torch.full((nc ** 3, width), -1, device=X.device, dtype=torch.long)
        sl = lin[order]
        table[sl, torch.arange(N, device=X.device) - first[sl]] = order
        o = torch.tensor([(a, b, e) for a in (-1, 0, 1) for b in (-1, 0, 1) for e in (-1, 0, 1)], device=X.device)
        step = max(1, 40_000_000 // (27 * width))
        for a in range(0, N, step):
            nb = torch.remainder(c[a:a + step, None, :] + o[None], nc)
            j = table[(nb[..., 0] * nc + nb[..., 1]) * nc + nb[..., 2]].reshape(nb.shape[0], -1)
            d = _wrap_diff(X[j.clamp(min=0)] - X[a:a + step, None, :])
            ok = (d.square().sum(2) < R * R) & (j >= 0)
            i, k = torch.nonzero(ok, as_tuple=True)
            I.append(i + a)
            J.append(j[i, k])
    i, j = torch.cat(I), torch.cat(J)
    keep = i != j
    return i[keep], j[keep]


def _sum(i, v, N):
    return torch.zeros(N, dtype=v.dtype, device=v.device).index_add(0, i, v)


def _support(i, r, N):
    """H with (4 pi / 3) H^3 n(H) = NGB: Newton kept inside a bracket."""
    H = torch.full((N,), _h0(N), device=r.device, dtype=torch.float64)
    lo, hi = torch.zeros_like(H), torch.full_like(H, 0.5)
    for _ in range(40):
        q = r / H[i]
        f = 32.0 / 3.0 * (1.0 + _sum(i, _kern(q), N)) - NGB
        fp = 32.0 / 3.0 * _sum(i, -_kern_d(q) * q, N) / H
        lo, hi = torch.where(f < 0, H, lo), torch.where(f < 0, hi, H)
        new = H - f / fp
        H2 = torch.where((new > lo) & (new < hi), new, 0.5 * (lo + hi))
        if bool(((H2 - H).abs() <= 1e-15 * H).all()):
            break
        H = H2
    return H


def _seg(i, v, init, how):
    return init.scatter_reduce(0, i, v, how, include_self=True)


def _clamp(v, lo, hi):
    return torch.where(v < lo, lo, torch.where(v > hi, hi, v))


def _gradients64(e, H, n, W):
    """E^-1 (6) and the limited gradients [5][3] of fields W."""
    i, j, d, r = e
    N = H.shape[0]
    psi = 8.0 / (math.pi * H[i] ** 3) * _kern(r / H[i]) / n[i]
    E = [_sum(i, psi * d[a] * d[b], N) for a, b in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))]
    a, b, c, dd, ee, ff = E
    co = [dd * ff - ee * ee, c * ee - b * ff, b * ee - c * dd, a * ff - c * c, b * c - a * ee, a * dd - b * b]
    det = a * co[0] + b * co[1] + c * co[2]
    B = [v / det for v in co]
    s = H[i] / (H[i] + H[j])
    out = []
    for f in W:
        df = f[j] - f[i]
        S = [_sum(i, df * psi * d[k], N) for k in range(3)]
        g = [B[0] * S[0] + B[1] * S[1] + B[2] * S[2], B[1] * S[0] + B[3] * S[1] + B[4] * S[2],
             B[2] * S[0] + B[4] * S[1] + B[5] * S[2]]
        top, bot = _seg(i, f[j], f, "amax"), _seg(i, f[j], f, "amin")
        D = s * (g[0][i] * d[0] + g[1][i] * d[1] + g[2][i] * d[2])
        Dn = torch.where(D == 0, torch.ones_like(D), D)
        al = torch.where(D > 0, (top - f)[i] / Dn, torch.where(D < 0, (bot - f)[i] / Dn, torch.ones_like(D)))
        al = _seg(i, al, torch.ones_like(f), "amin")
        out.append([al * g[k] for k in range(3)])
    return B, out


def _star(rL, uL, PL, rR, uR, PR):
    """Star pressure and contact speed of the exact Riemann problem; vacuum: 0, 0."""
    cL, cR = torch.sqrt(GAMMA * PL / rL), torch.sqrt(GAMMA * PR / rR)
    du = uR - uL
    ex = (GAMMA - 1) / (2 * GAMMA)

    def side(p, rho, P, c):
        A, b = 2 / ((GAMMA + 1) * rho), (GAMMA - 1) / (GAMMA + 1) * P
        q = torch.sqrt(A / (p + b))
        x = (p / P) ** ex
        f = torch.where(p > P, (p - P) * q, 2 * c / (GAMMA - 1) * (x - 1))
        g = torch.where(p > P, q * (1 - 0.5 * (p - P) / (p + b)), x / (p / P * rho * c))
        return f, g
    vac = 2 * (cL + cR) / (GAMMA - 1) <= du
    # the two-rarefaction estimate, then Newton in log p inside a bracket
    z = (cL + cR - 0.5 * (GAMMA - 1) * du).clamp(min=1e-12) / (cL / PL ** ex + cR / PR ** ex)
    p = z ** (1 / ex)
    lo, hi = torch.full_like(p, 0.0), torch.full_like(p, math.inf)
    for _ in range(80):
        fL, gL = side(p, rL, PL, cL)
        fR, gR = side(p, rR, PR, cR)
        F = fL + fR + du
        lo, hi = torch.where(F > 0, lo, p), torch.where(F > 0, p, hi)
        new = p - F / (gL + gR)
        half = torch.where(torch.isinf(hi), 2 * p, 0.5 * (lo + hi))
        new = torch.where((new > lo) & (new < hi), new, half)
        done = bool(((new - p).abs() <= 4e-16 * p)[~vac].all())
        p = new
        if done:
            break
    fL, _ = side(p, rL, PL, cL)
    fR, _ = side(p, rR, PR, cR)
    z = torch.zeros_like(p)
    return torch.where(vac, z, p), torch.where(vac, z, 0.5 * (uL + uR) + 0.5 * (fR - fL))


def _rates64(e, H, n, W, B, g, hdt, scheme, riemann):
    """d(momentum)/dt [3], dE/dt and dm/dt per particle, over ordered pairs."""
    i, j, d, r = e
    N = H.shape[0]

    def c(k):
        return 8.0 / (math.pi * H[k] ** 3) * torch.where(r < H[k], _kern(r / H[k]), torch.zeros_like(r)) / n[k] ** 2

    def Bd(k):
        return [B[0][k] * d[0] + B[1][k] * d[1] + B[2][k] * d[2], B[1][k] * d[0] + B[3][k] * d[1] + B[4][k] * d[2],
                B[2][k] * d[0] + B[4][k] * d[1] + B[5][k] * d[2]]
    ci, cj, Bi, Bj = c(i), c(j), Bd(i), Bd(j)
    A = [ci * Bi[k] + cj * Bj[k] for k in range(3)]
    q2 = A[0] ** 2 + A[1] ** 2 + A[2] ** 2
    ok = q2 > 0
    Am = torch.sqrt(torch.where(ok, q2, torch.ones_like(q2)))
    nh = [A[k] / Am for k in range(3)]
    si = H[i] / (H[i] + H[j])

    def face(k, s, sign):
        rho, P = W[0][k], W[4][k]
        div = g[1][0][k] + g[2][1][k] + g[3][2][k]
        inc = [-rho * div, -g[4][0][k] / rho, -g[4][1][k] / rho, -g[4][2][k] / rho, -GAMMA * P * div]
        return [W[f][k] + sign * s * (g[f][0][k] * d[0] + g[f][1][k] * d[1] + g[f][2][k] * d[2]) + hdt * inc[f]
                for f in range(5)]
    Fi, Fj = face(i, si, 1.0), face(j, 1.0 - si, -1.0)
    for f in range(5):
        lo, hi = torch.minimum(W[f][i], W[f][j]), torch.maximum(W[f][i], W[f][j])
        Fi[f], Fj[f] = _clamp(Fi[f], lo, hi), _clamp(Fj[f], lo, hi)
    vf = [W[1 + k][i] + si * (W[1 + k][j] - W[1 + k][i]) for k in range(3)]
    vfn = vf[0] * nh[0] + vf[1] * nh[1] + vf[2] * nh[2]
    ui = sum((Fi[1 + k] - vf[k]) * nh[k] for k in range(3))
    uj = sum((Fj[1 + k] - vf[k]) * nh[k] for k in range(3))
    ri, Pi, rj, Pj = Fi[0], Fi[4], Fj[0], Fj[4]
    ai, aj = torch.sqrt(GAMMA * Pi / ri), torch.sqrt(GAMMA * Pj / rj)
    SL, SR = torch.minimum(ui - ai, uj - aj), torch.maximum(ui + ai, uj + aj)
    ml, mr = ri * (SL - ui), rj * (SR - uj)
    ss = (Pj - Pi + ml * ui - mr * uj) / (ml - mr)
    ps = Pi + ml * (ss - ui)
    Aok = torch.where(ok, Am, torch.zeros_like(Am))
    if scheme == "mfv":
        left = (SL >= 0) | (ss >= 0)
        K = [torch.where(left, a, b) for a, b in zip(Fi, Fj)]
        uk, SK = torch.where(left, ui, uj), torch.where(left, SL, SR)
        star = torch.where(left, SL < 0, SR > 0)
        w = [K[1 + k] - vf[k] for k in range(3)]
        Et = K[4] / (GAMMA - 1) + 0.5 * K[0] * (w[0] ** 2 + w[1] ** 2 + w[2] ** 2)
        q = K[0] * (SK - uk) / (SK - ss)
        jump = torch.where(star, SK, torch.zeros_like(SK))
        Fm = K[0] * uk + jump * (q - K[0])
        Fw = [K[0] * uk * w[k] + K[4] * nh[k] + jump * (q * (w[k] + (ss - uk) * nh[k]) - K[0] * w[k]) for k in range(3)]
        Fe = uk * (Et + K[4]) + jump * (q * (Et / K[0] + (ss - uk) * (ss + K[4] / (K[0] * (SK - uk)))) - Et)
        v2 = vf[0] ** 2 + vf[1] ** 2 + vf[2] ** 2
        FE = Fe + vf[0] * Fw[0] + vf[1] * Fw[1] + vf[2] * Fw[2] + 0.5 * v2 * Fm
        return ([_sum(i, -(Fw[k] + vf[k] * Fm) * Aok, N) for k in range(3)], _sum(i, -FE * Aok, N),
                _sum(i, -Fm * Aok, N))
    if riemann != "hllc":
        pe, ue = _star(ri, ui, Pi, rj, uj, Pj)
        use = torch.ones_like(ok) if riemann == "exact" else ps < 0
        ps, ss = torch.where(use, pe, ps), torch.where(use, ue, ss)
    ps = ps.clamp(min=0.0)
    return ([_sum(i, torch.where(ok, -ps * A[k], torch.zeros_like(ps)), N) for k in range(3)],
            _sum(i, -ps * (ss + vfn) * Aok, N), None)


def _pairs(X, H, R):
    """Flux pairs r < max(H_i, H_j) and, among them, those with r < H_i."""
    i, j = _edges(X, R)
    d = [_wrap_diff(X[j, k] - X[i, k]) for k in range(3)]
    r = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
    if H is None:
        return i, j, d, r
    keep = r < torch.maximum(H[i], H[j])
    return i[keep], j[keep], [a[keep] for a in d], r[keep]


def _step64(p, case, grads_of=None):
    """One CFL step of one box in FP64; with grads_of, also its adjoint (lists,
    dt and branches frozen, H differentiated implicitly)."""
    q = {k: p[k].double() for k in STATE}
    if grads_of:
        for k in gza.GRADS:
            q[k] = q[k].detach().clone().requires_grad_(True)
    N = q["x"].shape[0]
    X = torch.stack([q["x"], q["y"], q["z"]], 1)
    with torch.no_grad():
        R = 1.3 * _h0(N)
        while True:
            i, j, d, r = _pairs(X.detach(), None, R)
            H = _support(i, r, N)
            if float(H.max()) < R or R >= 0.5:
                break
            R = min(0.5, 1.3 * R)
        keep = r < torch.maximum(H[i], H[j])
        i, j = i[keep], j[keep]
        own = r[keep] < H[i]
    d = [_wrap_diff(X[j, k] - X[i, k]) for k in range(3)]
    r = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
    io, jo, do, ro = i[own], j[own], [a[own] for a in d], r[own]
    if grads_of:
        f = 32.0 / 3.0 * (1.0 + _sum(io, _kern(ro / H[io]), N)) - NGB
        with torch.no_grad():
            fp = 32.0 / 3.0 * _sum(io, -_kern_d(ro / H[io]) * ro / H[io], N) / H
        H = H - f / fp
    n = 8.0 / (math.pi * H ** 3) * (1.0 + _sum(io, _kern(ro / H[io]), N))
    rho = q["m"] * n
    P = (GAMMA - 1) * rho * q["u"]
    W = [rho, q["vx"], q["vy"], q["vz"], P]
    B, g = _gradients64((io, jo, do, ro), H, n, W)
    with torch.no_grad():
        cs = torch.sqrt(GAMMA * P / rho)
        vd = sum((W[1 + k][j] - W[1 + k][i]) * d[k] for k in range(3)) / r
        vs = _seg(i, cs[i] + cs[j] - vd.clamp(max=0.0), torch.zeros_like(cs), "amax")
        dt = 0.2 * float((2 * n ** (-1.0 / 3.0) / vs)[vs > 0].min())
    dp, dE, dm = _rates64((i, j, d, r), H, n, W, B, g, 0.5 * dt, case["scheme"], case["riemann"])
    m2 = q["m"] + dt * dm if dm is not None else q["m"]
    v = [q[k] for k in ("vx", "vy", "vz")]
    E = q["m"] * (q["u"] + 0.5 * (v[0] ** 2 + v[1] ** 2 + v[2] ** 2)) + dt * dE
    v2 = [(q["m"] * v[k] + dt * dp[k]) / m2 for k in range(3)]
    u = E / m2 - 0.5 * (v2[0] ** 2 + v2[1] ** 2 + v2[2] ** 2)
    with torch.no_grad():
        floor = 1e-10 * torch.kthvalue(q["u"].detach(), (N - 1) // 2 + 1).values
    u = torch.where(u > 0, u, floor)
    new = {}
    for k, a in enumerate("xyz"):
        t = q[a] + dt * 0.5 * (v[k] + v2[k])
        t = torch.where(t < 0, t + 1.0, t)
        new[a] = torch.where(t >= 1.0, t - 1.0, t)
        new["v" + a] = v2[k]
    new.update({"u": u, "m": m2, "h": H})
    if grads_of:
        outs = [new[k] for k in grads_of]
        gr = torch.autograd.grad(outs, [q[k] for k in gza.GRADS], [grads_of[k].double() for k in grads_of])
        return {**{k: new[k].detach() for k in gza.OUT}, "grads": dict(zip(gza.GRADS, gr))}
    return new


def exact(case, seed):
    if case["op"] == "hier":
        return None  # many substeps of a state that each of them moves
    p = _particles(case, seed)
    if case["op"] == "grad":
        return _step64(p, case, _adjoint_weights(p["x"].numel(), seed, p["x"].dtype))
    if case["op"] == "step":
        parts, a = [], 0
        for c in _counts(case):
            parts.append(_step64({k: p[k][a:a + c] for k in STATE}, case))
            a += c
        return {k: torch.cat([b[k] for b in parts]) for k in STATE}
    # the frozen passes take H, n, gradients and B as the caller has them
    s = prepare(case, seed)
    q = {k: s["p"][k].double() for k in STATE}
    H, n = q["h"], s["n"].double()
    X = torch.stack([q["x"], q["y"], q["z"]], 1)
    rho = q["m"] * n
    W = [rho, q["vx"], q["vy"], q["vz"], (GAMMA - 1) * rho * q["u"]]
    i, j, d, r = _pairs(X, H, min(0.5, 1.0001 * float(H.max())))
    if case["op"] == "gradients":
        own = r < H[i]
        B, g = _gradients64((i[own], j[own], [a[own] for a in d], r[own]), H, n, W)
        return {"grad": torch.stack([a for f in g for a in f]), "B": torch.stack(B)}
    g = s["grad"].double()
    dp, dE, _ = _rates64((i, j, d, r), H, n, W, list(s["B"].double()), [[g[3 * f + k] for k in range(3)] for f in range(5)],
                         0.5 * s["pass_dt"], case["scheme"], case["riemann"])
    return {"dpdt": torch.stack(dp), "dEdt": dE}
