"""The equations do not know the unit of mass: masses multiplied by a power of
two at the same specific energies scale the densities, pressures and rates by
it, exactly in floating point while every intermediate stays in range, and
leave velocities, energies and positions alone.  Any intermediate of another
dimension (a square of an impedance, say) overflows or vanishes long before
the states do.  hydro_fluxes takes the gradients of the scaled state, scaled
likewise (rows 0-2 and 12-14: density and pressure)."""
import pytest

from gpu_common import cast_state, device
from paper_1712_01294_gb300 import inputs as I

pytestmark = pytest.mark.gpu

OUT = ("x", "y", "z", "vx", "vy", "vz", "u", "h")


def _state(prec):
    return cast_state(I.turbulence(12, seed=31), prec)


def _scaled(m, q, prec, k):
    d = device(q, prec)
    d["m"] = d["m"] * 2.0 ** k  # (exact)
    return d


def _rates(m, q, prec, k, kw, frozen):
    """hydro_fluxes of the state with masses times 2^k, times 2^-k; frozen: the
    density pass and gradients of the unscaled state."""
    import torch
    d = _scaled(m, q, prec, k)
    d["h"], n, g, B = frozen["h"].clone(), frozen["n"], frozen["grad"].clone(), frozen["B"]
    for r in (0, 1, 2, 12, 13, 14):
        g[r] *= 2.0 ** k
    ctx = m.Context([q.N], m.default_params(precision=prec, **kw))
    outs = ctx.hydro_fluxes(d, n, g, B, 0.01, with_mass="scheme" in kw)
    torch.cuda.synchronize()
    ctx.status(reset=True)
    ctx.close()
    return [t * 2.0 ** -k for t in outs]


def _frozen(m, q, prec):
    ctx = m.Context([q.N], m.default_params(precision=prec))
    d = device(q, prec)
    n, _ = ctx.density(d)
    g, B = ctx.gradients(d, n)
    ctx.close()
    return {"h": d["h"], "n": n, "grad": g, "B": B}


# FP32 rates are summed in FP64: at 2^-96 the terms of a lattice without tiny
# faces (about 2^-118) keep all their bits in FP32; what is left of their sums
# below the leading 24 bits does not fit in FP32 numbers any more
@pytest.mark.parametrize("prec,k", [(1, 96), (1, -96), (0, 600), (0, -600)])
def test_mfv_rates_scale_with_the_masses(prec, k):
    import torch
    import paper_1712_01294_gb300 as m
    q = cast_state(I.turbulence(12, seed=31, jitter=0.0), prec)
    f = _frozen(m, q, prec)
    for a, b in zip(_rates(m, q, prec, 0, {"scheme": m.GZ_MFV}, f), _rates(m, q, prec, k, {"scheme": m.GZ_MFV}, f)):
        assert float(a.abs().max()) > 0 and torch.equal(a, b)


FLUXES = [{}, {"riemann": 2}]
RANGE = [(1, 70), (1, -70), (0, 600), (0, -600)]


@pytest.mark.parametrize("prec,k", RANGE)
@pytest.mark.parametrize("kw", FLUXES)
def test_hllc_rates_scale_with_the_masses(kw, prec, k):
    import torch
    import paper_1712_01294_gb300 as m
    q = _state(prec)
    f = _frozen(m, q, prec)
    for a, b in zip(_rates(m, q, prec, 0, kw, f), _rates(m, q, prec, k, kw, f)):
        assert float(a.abs().max()) > 0 and torch.equal(a, b)


@pytest.mark.parametrize("prec,k", RANGE)
@pytest.mark.parametrize("K", [None, 2])
def test_steps_do_not_depend_on_the_mass_unit(K, prec, k):
    import torch
    import paper_1712_01294_gb300 as m
    q = _state(prec)
    outs = []
    for e in (0, k):
        d = _scaled(m, q, prec, e)
        ctx = m.Context([q.N], m.default_params(precision=prec))
        ctx.step(d) if K is None else ctx.step_hier(d, K)
        assert ctx.status(reset=True)["ok"]
        ctx.close()
        outs.append(d)
    for f in OUT:
        assert torch.equal(outs[0][f], outs[1][f]), f


# the adjoint's own sums mix dimensions (dJ/dm ~ 1/m): same values to rounding
@pytest.mark.parametrize("prec,k", RANGE)
def test_adjoint_scales_with_the_masses(prec, k):
    import torch
    import paper_1712_01294_gb300 as m
    q = cast_state(I.smooth_turbulence(12, seed=3), prec)
    outs = []
    for e in (0, k):
        d = _scaled(m, q, prec, e)
        ctx = m.Context([q.N], m.default_params(precision=prec))
        ctx.density(d)
        g = torch.Generator(device="cuda").manual_seed(5)
        gend = {f: torch.randn(q.N, generator=g, device="cuda", dtype=d["x"].dtype)
                for f in ("x", "y", "z", "vx", "vy", "vz", "u")}
        gs = {f: torch.zeros_like(d["x"]) for f in ("x", "y", "z", "vx", "vy", "vz", "u", "m")}
        ctx.step_backward(d, 0.01, gend, gs)
        torch.cuda.synchronize()
        ctx.close()
        gs["m"] *= 2.0 ** e
        outs.append({f: t.double() for f, t in gs.items()})
    for f in outs[0]:
        a, b = outs[0][f], outs[1][f]
        tol = 1e-12 if prec == 0 else 1e-5
        assert float((a - b).square().mean().sqrt()) <= tol * float(a.square().mean().sqrt()), f


# The exact solver's starting estimates take powers of the pressures, which do
# not scale exactly, so its star pressures agree to its stopping tolerance, 2e-6
# of them; a colliding stream's rates are sums of about 30 terms of one size,
# of which the net rate keeps at least a tenth: 30 * 10 * 2e-6 of the rms, and
# no more than 1e-3.
@pytest.mark.parametrize("k", [55, -55])
def test_exact_rates_scale_with_the_masses(k):
    import paper_1712_01294_gb300 as m
    q = cast_state(I.sod(12, rho_l=1.0, p_l=0.4, rho_r=1.0, p_r=0.4, u_l=4.0, u_r=-4.0), 1)
    f = _frozen(m, q, 1)
    for a, b in zip(_rates(m, q, 1, 0, {"riemann": 1}, f), _rates(m, q, 1, k, {"riemann": 1}, f)):
        assert float((a - b).abs().max()) <= 1e-3 * float(a.square().mean().sqrt())
