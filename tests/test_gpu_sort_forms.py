"""The binning's two sorts: a counting sort on grids of about one support radius
a cell, the radix sort on grids much finer than the particles.  Both must find
the oracle's neighbours; a clumped cell keeps its particles in caller order
(lists come out in scan order, ascending id inside a cell)."""
import numpy as np
import pytest

import oracle as O
from gpu_common import cast_state, device, gpu_sets, ostate
from paper_1712_01294_gb300 import inputs as I


def _clumped(n, seed, share):
    p = I.turbulence(n, seed=seed)
    rng = np.random.default_rng(seed)
    X = rng.uniform(size=(3, p.N))
    k = int(share * p.N)
    X[:, :k] = 0.3 + 0.01 * rng.uniform(size=(3, k))
    p.x, p.y, p.z = X
    return p


@pytest.mark.gpu
@pytest.mark.parametrize("cell_factor", [1.0, 0.12])  # counting sort; radix sort
@pytest.mark.parametrize("make", [lambda: I.turbulence(10, seed=3), lambda: _clumped(11, 4, 0.4)])
def test_neighbours_under_either_sort(make, cell_factor):
    import paper_1712_01294_gb300 as m
    q = cast_state(make(), 0)
    s = ostate(q)
    Ho, no, it, _ = O.density(s, O.params())
    ctx = m.Context([q.N], m.default_params(precision=0, cell_factor=cell_factor, max_ngb=1400))
    d = device(q, 0)
    n, iters = ctx.density(d)
    keys = 8 ** int(np.ceil(np.log2(round(ctx.info()["cells"] ** (1 / 3)))))
    assert (keys > 8 * q.N + 65536) == (cell_factor < 1)
    assert np.array_equal(iters.cpu().numpy(), it)
    assert np.max(np.abs(d["h"].cpu().numpy() / Ho - 1)) < 1e-12
    off, nbr = O.neighbours(s, Ho, use_cells=0)
    cnt, sets = gpu_sets(ctx, 1400)
    for i in range(q.N):
        assert sets[i] == set(int(j) for j in nbr[off[i]:off[i + 1]]), i


@pytest.mark.gpu
def test_cell_keeps_caller_order():
    import torch
    import paper_1712_01294_gb300 as m
    rng = np.random.default_rng(5)
    q = _clumped(8, 6, 1.0)  # every particle in one small clump: one or a few cells
    ctx = m.Context([q.N], m.default_params(max_ngb=512, h_lim=0.4))
    perm = rng.permutation(q.N)
    d = {k: v[torch.as_tensor(perm, device="cuda")].contiguous() for k, v in device(cast_state(q, 1), 1).items()}
    d["id"] = torch.arange(q.N, device="cuda")
    d["h"].fill_(0.1)
    ctx.density(d)
    cnt, ids = ctx.neighbours(512)
    nc = round(ctx.info()["cells"] ** (1 / 3))
    cell = sum((d[k] * nc).floor().long() * w for k, w in (("x", 1), ("y", nc), ("z", nc * nc))).cpu().numpy()
    ids = ids.cpu().numpy()
    for i in (0, 17, q.N - 1):
        li = ids[: int(cnt[i]), i]
        for c in np.unique(cell[li]):
            mine = li[cell[li] == c]
            assert (np.diff(mine) > 0).all(), (i, c)
