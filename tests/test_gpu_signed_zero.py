"""-0 and +0 are one number: a component at rest may carry either sign (a
rotation, a product with a negative zero), and the clamps' tie rule and sides
must not see it."""
import numpy as np
import pytest

from gpu_common import cast_state, device
from paper_1712_01294_gb300 import inputs as I


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("share", [0.5, 1.0])
def test_flux_adjoint_with_negative_zeros(share, prec):
    import torch
    import paper_1712_01294_gb300 as m
    q = I.smooth_turbulence(10, seed=3)
    q.vz[:] = 0.0
    q = cast_state(q, prec)
    rng = np.random.default_rng(6)
    wp, wE = torch.as_tensor(rng.normal(size=(3, q.N))).cuda(), torch.as_tensor(rng.normal(size=q.N)).cuda()
    neg = torch.as_tensor(rng.uniform(size=q.N) < share).cuda()
    outs = []
    for signed in (False, True):
        d = device(q, prec)
        if signed:
            d["vz"] = torch.where(neg, -torch.zeros_like(d["vz"]), d["vz"])
            assert int(torch.signbit(d["vz"]).sum()) == int(neg.sum())
        ctx = m.Context([q.N], m.default_params(precision=prec))
        n, _ = ctx.density(d)
        g, B = ctx.gradients(d, n)
        outs.append(ctx.hydro_fluxes_backward(d, n, g, B, 0.01, wp, wE))
        torch.cuda.synchronize()
        ctx.close()
    for k in outs[0]:
        assert torch.equal(outs[0][k], outs[1][k]), k
