"""FP64 supports do not depend on which form of the density pass iterates a
particle, also where a candidate lies just outside the candidate cache's
radius 1.05 H: the lane groups' FP32 prefilter lets such a candidate through,
the warp form does not see it, and the lanes' sums would round differently."""
import numpy as np
import pytest

from gpu_common import cast_state, device
from paper_1712_01294_gb300 import inputs as I


@pytest.mark.gpu
@pytest.mark.parametrize("gap", [1e-9, 1e-7, 3e-7])
def test_shell_candidates_do_not_show(gap):
    import paper_1712_01294_gb300 as m
    n = 24
    q = I.turbulence(n, seed=14)
    h0 = float(q.H[0])
    q.H[:] = h0
    R = h0 * 1.05
    # every fourth lattice site: one neighbour moved into the shell, on the side
    # the scan visits first (and held there by construction in FP64)
    ids = np.array([(k * n + j) * n + i for k in range(4, n, 4) for j in range(4, n, 4) for i in range(4, n, 4)])
    X = np.stack([q.x, q.y, q.z])
    u = np.array([-0.5, -0.6, -np.sqrt(1 - 0.61)])
    other = ids - (2 * n + 2) * n - 2  # two sites back on each axis: nobody else's centre
    X[:, other] = X[:, ids] + ((R + gap) * u)[:, None]
    q.x, q.y, q.z = X % 1.0
    q = cast_state(q, 0)
    outs = []
    for cache in (0, 40):  # ngb = 45: 52 candidates within 1.05 H, the group form's or the warp form's
        ctx = m.Context([q.N], m.default_params(precision=0, ngb=45.0, density_cache=cache))
        d = device(q, 0)
        nn, it = ctx.density(d)
        assert ctx.status(reset=True)["ok"]
        ctx.close()
        outs.append([t.cpu().numpy() for t in (d["h"], nn, it)])
    for a, b in zip(*outs):
        assert np.array_equal(a, b)
