"""A kernel's set-up overlaps the end of the kernel before it.  The same boxes
stepped again, alone and beside others, give the same bits."""
import pytest

from gpu_common import cast_state, device
from paper_1712_01294_gb300 import inputs as I

OUT = ("x", "y", "z", "vx", "vy", "vz", "u", "h")


def _steps(m, q, prec, copies, steps=4):
    import torch
    ctx = m.Context([q.N] * copies, m.default_params(precision=prec))
    d = {k: v.repeat(copies).contiguous() for k, v in device(q, prec).items()}
    d["id"] = torch.arange(d["id"].numel(), device="cuda")
    for _ in range(steps):
        ctx.step(d)
    ctx.status(reset=True)
    ctx.close()
    return {k: d[k].reshape(copies, q.N) for k in OUT}


@pytest.mark.gpu
@pytest.mark.parametrize("prec,copies", [(1, 24), (1, 25), (0, 25)])
def test_chained_launches_give_the_same_bits(prec, copies):
    import torch
    import paper_1712_01294_gb300 as m
    q = cast_state(I.turbulence(20, seed=21), prec)
    alone = _steps(m, q, prec, 1)
    for _ in range(10):
        again = _steps(m, q, prec, 1)
        assert all(torch.equal(alone[k], again[k]) for k in OUT)
    many = _steps(m, q, prec, copies)
    for k in OUT:
        assert torch.equal(alone[k].expand(copies, q.N), many[k]), k
