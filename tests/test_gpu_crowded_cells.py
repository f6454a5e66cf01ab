"""Binning is linear in the particles also where many share one cell: a state
that went to NaN (all of them binned in the first cell) or a dense clump."""
import pytest

from gpu_common import cast_state, device
from paper_1712_01294_gb300 import inputs as I


def _time(m, n, bad=True):
    import torch
    q = cast_state(I.sod(n, seed=3), 1)
    d = device(q, 1)
    if bad:
        for k in ("x", "y", "z"):
            d[k].fill_(float("nan"))
    ctx = m.Context([q.N], m.default_params())
    best = 1e9
    for _ in range(4):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        ctx.density(d)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    ctx.status(reset=True)
    ctx.close()
    return best


@pytest.mark.gpu
def test_time_is_linear_in_the_crowd():
    # eight times the particles: linear work 8 times the time, quadratic 64
    import paper_1712_01294_gb300 as m
    _time(m, 32)
    small, large = _time(m, 32), _time(m, 64)
    print(f"all in one cell: 32^3 {small:.3f} ms, 64^3 {large:.3f} ms")
    assert large < 10 * small


@pytest.mark.gpu
@pytest.mark.parametrize("n", [30, 66])  # one block's window of caller indices, and more than one
def test_crowded_cells_keep_caller_order(n):
    # most particles in two cells (at NaN and beyond the far corner), in any order
    import numpy as np
    import torch
    import paper_1712_01294_gb300 as m
    q = cast_state(I.sod(n, seed=3), 1)
    rng = np.random.default_rng(n)
    what = rng.choice(3, size=q.N, p=[0.65, 0.25, 0.1] if n == 30 else [0.45, 0.45, 0.1])
    d = device(q, 1)
    for k in ("x", "y", "z"):
        v = d[k].cpu().numpy()
        v[what == 0], v[what == 1] = np.nan, 1.5
        d[k] = torch.as_tensor(v).cuda()
    x0 = [d[k].cpu().numpy() for k in ("x", "y", "z")]
    ctx = m.Context([q.N], m.default_params())
    nc = round(ctx.info()["cells"] ** (1 / 3))
    ck = ctx.new_checkpoint(2)
    ctx.step(d, 1e-4, None, ck, 2)
    ctx.status(reset=True)
    ctx.close()
    raw, at = ck.cpu().numpy(), 0
    for nbytes in (32 * q.N, 4 * q.N, 4 * q.N, 4 * q.N, 128 * q.N, 160 * q.N, 40 * q.N):  # (up to the keys)
        at += -(-nbytes // 256) * 256
    keys = raw[at:at + 4 * q.N].view(np.uint32)
    at += -(-4 * q.N // 256) * 256
    order = raw[at:at + 4 * q.N].view(np.uint32).astype(np.int64)
    assert np.array_equal(np.sort(order), np.arange(q.N))
    with np.errstate(invalid="ignore"):
        cell = [np.clip(np.nan_to_num(np.floor(c * np.float32(nc)), nan=0.0), 0, nc - 1).astype(np.int64)[order] for c in x0]
    assert (np.diff(keys.astype(np.int64)) >= 0).all()
    same = np.diff(keys.astype(np.int64)) == 0
    assert (np.diff(order)[same] > 0).all()  # caller order within a cell
    for c in cell:
        assert (np.diff(c)[same] == 0).all()  # one key, one cell
    assert np.bincount(keys).max() > 16384


@pytest.mark.gpu
def test_positions_that_are_no_numbers_keep_to_one_thread():
    # they see no candidates, so their supports grow to the limit; a warp for
    # each took the pass 4.6 ms at 64^3, where a lattice takes 0.15
    import paper_1712_01294_gb300 as m
    _time(m, 64)
    nan, lattice = _time(m, 64), _time(m, 64, bad=False)
    print(f"64^3: no positions {nan:.3f} ms, lattice {lattice:.3f} ms")
    assert nan < 8 * lattice
