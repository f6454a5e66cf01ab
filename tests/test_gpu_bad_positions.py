"""A particle whose position is no number is flagged and is nobody's
neighbour: the others' supports and densities are those of the set without
it."""
import numpy as np
import pytest

from gpu_common import cast_state, device
from paper_1712_01294_gb300 import inputs as I


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("bits", [0x7ff8000000000000, 0xfff8000000000000])
@pytest.mark.parametrize("density_cache", [0, 40])
def test_nan_position_touches_no_one(density_cache, bits, prec):
    import torch
    import paper_1712_01294_gb300 as m
    q = cast_state(I.turbulence(12, seed=8), prec)
    bad = q.N // 2 + 77
    nan = np.array([bits], dtype=np.uint64).view(np.float64)
    keep = torch.arange(q.N, device="cuda") != bad
    outs = []
    for with_bad in (True, False):
        d = device(q, prec)
        if with_bad:
            v = torch.as_tensor(nan).cuda().to(d["x"].dtype)
            for k in ("x", "y", "z"):
                d[k][bad] = v[0]
        else:
            d = {k: t[keep].contiguous() for k, t in d.items()}
        N = d["x"].numel()
        ctx = m.Context([N], m.default_params(precision=prec, density_cache=density_cache))
        n, it = ctx.density(d)
        st = ctx.status(reset=True)
        assert st["ok"] == (not with_bad), st
        ctx.close()
        outs.append([t[keep] if with_bad else t for t in (d["h"], n)])
    tol = 1e-12 if prec == 0 else 1e-5  # (another cell grid: the same sums in another order)
    for a, b in zip(*outs):
        assert float((a / b - 1).abs().max()) <= tol
