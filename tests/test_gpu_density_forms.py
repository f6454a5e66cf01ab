"""The density pass's forms (one thread, four or sixteen lanes, or a warp per
particle) give the same bits, so which one a launch or a particle takes never
shows; and the FP32 prefilter of the FP64 scan drops no neighbour."""
import numpy as np
import pytest

from gpu_common import cast_state, device
from paper_1712_01294_gb300 import inputs as I


def _random(n, seed, scale=1.0, clump=0.0):
    """Uniform random points, a share of them gathered in a small clump."""
    p = I.turbulence(n, seed=seed) if n > 3 else I.sod(n, seed=seed)
    rng = np.random.default_rng(seed)
    X = rng.uniform(size=(3, p.N))
    k = int(clump * p.N)
    X[:, :k] = (0.97 + 0.05 * rng.standard_normal((3, k))) % 1.0
    p.x, p.y, p.z = X
    p.H = p.H * scale
    return p


CASES = [("lattice 12", lambda: I.turbulence(12, seed=1)), ("lattice 33", lambda: I.turbulence(33, seed=2)),
         ("random 17", lambda: _random(17, 3)), ("wide start", lambda: _random(14, 4, scale=2.0)),
         ("narrow start", lambda: _random(14, 5, scale=0.3)), ("clump", lambda: _random(16, 6, clump=0.3)),
         ("8", lambda: I.turbulence(8, seed=7)), ("3", lambda: _random(3, 8))]


def _run(m, counts, q, prec, copies=1, **kw):
    import torch
    ctx = m.Context(counts * copies, m.default_params(precision=prec, **kw))
    d = {k: v.repeat(copies).contiguous() for k, v in device(q, prec).items()}
    d["id"] = torch.arange(d["id"].numel(), device="cuda")
    n, it = ctx.density(d)
    cnt, ids = ctx.neighbours(96)
    ctx.status(reset=True)
    ctx.close()
    return [t.cpu().numpy() for t in (d["h"], n, it, cnt, ids)]


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("name,make", CASES)
def test_forms_give_the_same_bits(name, make, prec):
    import paper_1712_01294_gb300 as m
    q = cast_state(make(), prec)
    ref = _run(m, [q.N], q, prec)
    for kw in ({"density_cache": 40}, {"density_cache": 48}):  # more particles left to the warp form
        for a, b in zip(ref, _run(m, [q.N], q, prec, **kw)):
            assert np.array_equal(a, b), (name, kw)
    # enough boxes for the four-lane and the one-thread form
    for copies in (-(-13000 // q.N), -(-100000 // q.N)):
        if prec == 0 or copies > 70:
            continue
        big = _run(m, [q.N], q, prec, copies)
        for a, b in zip(ref[:4], big[:4]):
            assert np.array_equal(np.tile(a, copies), b), name
        off = np.arange(copies)[None, :, None] * q.N
        ids = big[4].reshape(96, copies, q.N)
        assert np.array_equal(np.where(ids >= 0, ids - off, -1),
                              np.broadcast_to(ref[4][:, None, :], ids.shape)), name


def test_prefilter_bound_covers_every_pair_inside():
    # chop() and r2_chop() restated: leading 24 bits of each coordinate, FP32
    # differences folded to the nearest image, against the bound for radius R
    rng = np.random.default_rng(11)
    f = np.float32

    def chop(x):
        b = x.view(np.int64)
        h = np.maximum(b >> 32, 0x38000000)
        return (((h - 0x38000000) << 3) | ((b & 0xffffffff) >> 29)).astype(np.int32).view(f)

    for R in (1e-4, 0.003, 0.0154, 0.07, 0.25, 0.4999):
        n = 200000
        xi = rng.uniform(size=(3, n)) * np.where(rng.uniform(size=n) < 0.2, 1e-5, 1.0)
        d = rng.standard_normal((3, n))
        d *= R * (1 - 10.0 ** rng.uniform(-17, -1, n)) / np.sqrt((d * d).sum(0))
        xj = (xi + d) % 1.0
        dd = xj - xi
        dd = np.where(dd >= 0.5, dd - 1, np.where(dd < -0.5, dd + 1, dd))
        inside = (dd * dd).sum(0) < R * R
        e = chop(xj) - chop(xi)
        e = e - np.rint(e)
        r2 = (e * e).sum(0, dtype=f)
        b = (f(R) + f(4e-7)) * f(1 + 1e-6)
        assert (r2[inside] < b * b).all(), R


@pytest.mark.gpu
@pytest.mark.parametrize("make", [lambda: I.turbulence(49, seed=9), lambda: _random(49, 10), lambda: _random(50, 11, clump=0.1)])
def test_windows_inside_the_box_give_the_same_bits(make):
    # alone, a large box's inner warps scan without periodic shifts; beside a
    # small box the launch keeps the general scan
    import paper_1712_01294_gb300 as m
    q, tiny = cast_state(make(), 1), cast_state(I.turbulence(8, seed=1), 1)
    alone = _run(m, [q.N], q, 1)
    both = q.copy()
    for k in I.FIELDS + ("id",):
        setattr(both, k, np.concatenate([getattr(q, k), getattr(tiny, k)]))
    mixed = _run(m, [q.N, tiny.N], both, 1)
    for a, b in zip(alone, mixed):
        assert np.array_equal(a, b[..., :q.N])


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("name,make,copies", [(n, mk, 1) for n, mk in CASES] + [
    ("lattice 12, many", CASES[0][1], 30), ("clump, many", CASES[5][1], 12), ("wide start, many", CASES[3][1], 18),
    ("large box", lambda: _random(38, 12, clump=0.05), 1), ("large lattice", lambda: I.turbulence(49, seed=9), 1)])
def test_lists_of_a_given_support_are_the_density_pass_s(name, make, copies, prec):
    # the lists of the frozen-input calls (four lanes, one thread, inner
    # windows of a large box) against those the density pass left, in order
    import torch
    import paper_1712_01294_gb300 as m
    q = cast_state(make(), prec)
    ctx = m.Context([q.N] * copies, m.default_params(precision=prec))
    d = {k: v.repeat(copies).contiguous() for k, v in device(q, prec).items()}
    d["id"] = torch.arange(d["id"].numel(), device="cuda")
    n, _ = ctx.density(d)
    ref = [t.cpu().numpy() for t in ctx.neighbours(96)]
    ctx.gradients(d, n)
    got = [t.cpu().numpy() for t in ctx.neighbours(96)]
    ctx.status(reset=True)
    ctx.close()
    for a, b in zip(ref, got):
        assert np.array_equal(a, b), name
