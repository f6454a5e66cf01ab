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
@pytest.mark.parametrize("n", [30, 66])  # the cells sorted by a block of 256, of 1024
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


def _clump(n, share, size, seed=2):
    import numpy as np
    q = I.turbulence(n, seed=seed)
    rng = np.random.default_rng(seed)
    k = int(share * q.N)
    for c in ("x", "y", "z"):
        getattr(q, c)[:k] = 0.3 + size * rng.uniform(size=k)
    q.H[:k] *= 0.1
    return q


@pytest.mark.gpu
@pytest.mark.parametrize("n", [32, 40])  # a group of lanes, one thread a particle
def test_scans_of_a_dense_clump_are_shared(n):
    # an eighth of the particles in one cell: one lane walking it took the call
    # 60 ms at 32^3 (two walks a particle), 800 times a lattice's
    import torch
    import paper_1712_01294_gb300 as m

    def best(q):
        ctx = m.Context([q.N], m.default_params())
        d = device(q, 1)
        ctx.density(d)
        t = 1e9
        for _ in range(3):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            ctx.density(d)
            b.record()
            b.synchronize()
            t = min(t, a.elapsed_time(b))
        ctx.status(reset=True)
        ctx.close()
        return t

    lattice = best(cast_state(I.turbulence(n, seed=2), 1))
    clump = best(cast_state(_clump(n, 0.125, 0.002), 1))
    print(f"{n}^3 density call: lattice {lattice:.3f} ms, clump {clump:.3f} ms")
    assert clump < 150 * lattice


@pytest.mark.gpu
def test_interval_of_a_state_without_positions():
    # one thread walking the one cell for its smallest support took 12 ms at 64^3
    import torch
    import paper_1712_01294_gb300 as m
    q = cast_state(I.sod(64, seed=3), 1)
    t = {}
    for what in ("lattice", "nan"):
        d = device(q, 1)
        if what == "nan":
            for k in ("x", "y", "z"):
                d[k].fill_(float("nan"))
        ctx = m.Context([q.N], m.default_params())
        best = 1e9
        for _ in range(3):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            ctx.step_hier(d, 1, 1e-6)
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b))
        t[what] = best
        ctx.status(reset=True)
        ctx.close()
    print(t)
    assert t["nan"] < 8 * t["lattice"]


@pytest.mark.gpu
def test_interval_with_a_crowded_cell_follows_the_oracle():
    import numpy as np
    import torch
    import oracle as O
    import paper_1712_01294_gb300 as m
    from gpu_common import field_err, ostate
    q = cast_state(_clump(12, 0.2, 0.02), 0)
    s = ostate(q)
    o, D, bins_o, na = O.step_hier(s, O.params(), 3)
    ctx = m.Context([q.N], m.default_params(precision=0, max_ngb=512))
    d = device(q, 0)
    cell = np.floor(np.stack([q.x, q.y, q.z]) * round(ctx.info()["cells"] ** (1 / 3))).astype(int)
    assert np.unique(cell, axis=1, return_counts=True)[1].max() > 128
    bins = torch.zeros(q.N, dtype=torch.int32, device="cuda")
    assert ctx.step_hier(d, 3, 0.0, None, bins) == na
    assert ctx.status(reset=True)["ok"]
    ctx.close()
    assert np.array_equal(bins.cpu().numpy(), bins_o) and len(np.unique(bins_o)) > 1
    for k in ("vx", "vy", "vz", "u"):
        mx, _ = field_err(d[k].cpu().numpy() - getattr(s, k), getattr(o, k) - getattr(s, k))
        assert mx <= 1e-9, (k, mx)
