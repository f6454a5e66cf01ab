"""An interval of hierarchical steps is refused on a capturing stream, whatever
its number of substeps, with nothing launched: the host reads the number of
active particles between substeps."""
import pytest

from gpu_common import cast_state, device
from paper_1712_01294_gb300 import inputs as I

OUT = ("x", "y", "z", "vx", "vy", "vz", "m", "u", "h")


@pytest.mark.gpu
@pytest.mark.parametrize("K", [0, 2])
def test_an_interval_refuses_stream_capture(K):
    import torch
    import paper_1712_01294_gb300 as m
    q = cast_state(I.turbulence(10, seed=5), 1)
    s = torch.cuda.Stream()
    ctx = m.Context([q.N], m.default_params(), stream=s)
    d = device(q, 1)
    torch.cuda.synchronize()
    ctx.step_hier(d, 1)
    s.synchronize()
    before = {k: d[k].clone() for k in OUT}
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        with pytest.raises(m.GZError):
            ctx.step_hier(d, K)
    torch.cuda.synchronize()
    assert all(torch.equal(before[k], d[k]) for k in OUT)
    ctx.step_hier(d, K)  # and the context goes on
    assert ctx.status()["ok"]
