"""The flux pass's two forms (one thread per particle, four warps per 32
particles) give the same bits: a step of one small box equals each copy's step
in a batch large enough for the other form.  Sizes leave partial blocks and
lists of every remainder of 8 slots; ngb = 80 makes long lists."""
import numpy as np
import pytest

from gpu_common import cast_state, device
from paper_1712_01294_gb300 import inputs as I


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("kw", [{}, {"scheme": 1}, {"riemann": 1}, {"riemann": 2}, {"hancock": 0},
                                {"ngb": 80.0, "max_ngb": 256}])
@pytest.mark.parametrize("make,copies", [(lambda: I.sedov(11, seed=4, p_bg=1e-3), 25),
                                         (lambda: I.turbulence(10, seed=5), 31)])
def test_one_box_equals_its_copies_in_a_batch(make, copies, kw, prec):
    import torch
    import paper_1712_01294_gb300 as m
    q = cast_state(make(), prec)
    assert q.N * copies >= 30000 > q.N
    out = []
    for c in (1, copies):
        ctx = m.Context([q.N] * c, m.default_params(precision=prec, **kw))
        d = {k: v.repeat(c).contiguous() for k, v in device(q, prec).items()}
        d["id"] = torch.arange(d["id"].numel(), device="cuda")
        for _ in range(4):
            ctx.step(d)
        assert ctx.status(reset=True)["ok"]
        ctx.close()
        out.append(d)
    for k in ("x", "y", "z", "vx", "vy", "vz", "m", "u", "h"):
        a, b = (d[k].cpu().numpy() for d in out)
        assert np.array_equal(np.tile(a, copies), b), k
