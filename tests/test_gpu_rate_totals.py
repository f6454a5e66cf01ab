"""The FP32 mode accumulates rates in FP64, as one number: a particle with one
partner whose energy flux overflows FP32 has an infinite rate, not NaN (a
two-word FP32 total forms inf - inf)."""
import pytest

from gpu_common import cast_state, device
from paper_1712_01294_gb300 import inputs as I


@pytest.mark.gpu
@pytest.mark.parametrize("n", [14, 33])  # four warps, one thread
def test_one_infinite_term_gives_an_infinite_rate(n):
    import torch
    import paper_1712_01294_gb300 as m
    q = cast_state(I.turbulence(n, seed=12), 1)
    hot = q.N // 2 + n // 2
    ctx = m.Context([q.N], m.default_params())
    d = device(q, 1)
    # rho c^2 = P and P c A with rho ~ 1e-9, P ~ 1e27, c ~ 1e18: the star
    # pressure (half of P) stays in range, its product with the contact speed
    # (4e17) and all but the smallest faces (2e-6) does not
    d["m"] *= 1e-9
    d["u"][hot] = 1.5e36
    h, _ = ctx.density(d)
    cnt, ids = ctx.neighbours(64)
    near = ids[: int(cnt[hot]), hot]  # (ids are caller indices)
    _, B = ctx.gradients(d, h)
    g = torch.zeros(15, q.N, device="cuda")
    dp, dE = ctx.hydro_fluxes(d, h, g, B, 0.0)
    ctx.status(reset=True)
    ctx.close()
    inf = torch.isinf(dE)
    assert inf[near].sum() > 20  # (a partner moving with the contact has a finite one)
    assert not torch.isnan(dE[near]).any()
    assert torch.isfinite(dp).all()
