"""Intervals of hierarchical steps in every form their launches take: one small
box (lanes sharing a particle, four warps an exchange, lists compacted
directly) against the same box among enough copies for the one-thread forms
over an index list, which the first substep of a large box runs.  The same
bits, bins and counts."""
import pytest

from gpu_common import cast_state, device
from paper_1712_01294_gb300 import inputs as I

OUT = ("x", "y", "z", "vx", "vy", "vz", "m", "u", "h")


def _interval(m, q, prec, copies, K, kw):
    import torch
    ctx = m.Context([q.N] * copies, m.default_params(precision=prec, **kw))
    d = {k: v.repeat(copies).contiguous() for k, v in device(q, prec).items()}
    d["id"] = torch.arange(d["id"].numel(), device="cuda")
    bins = torch.full((q.N * copies,), -1, dtype=torch.int32, device="cuda")
    na = ctx.step_hier(d, K, 0.0, None, bins)
    ctx.status(reset=True)
    ctx.close()
    return [d[k].reshape(copies, q.N) for k in OUT] + [bins.reshape(copies, q.N)], na


def _compare(q, prec, copies, K, kw):
    import torch
    import paper_1712_01294_gb300 as m
    ref, na = _interval(m, q, prec, 1, K, kw)
    assert len(torch.unique(ref[-1])) > 1  # (substeps of few active particles beside the first of all)
    many, nb = _interval(m, q, prec, copies, K, kw)
    assert nb == na * copies
    for k, a, b in zip(OUT + ("bins",), ref, many):
        assert torch.equal(a.expand(copies, q.N), b), k


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("kw", [{}, {"scheme": 1}, {"riemann": 1}, {"riemann": 2}, {"hancock": 0}])
def test_one_box_equals_its_copies_in_a_batch(kw, prec):
    q = cast_state(I.sedov(13, seed=4, p_bg=1e-3), prec)
    assert q.N * 24 >= 45000 > 12000 > q.N
    _compare(q, prec, 24, 3, kw)


@pytest.mark.gpu
def test_lists_of_more_blocks_than_the_direct_compaction_takes():
    q = cast_state(I.sedov(129, seed=4, p_bg=1e-2), 1)
    assert q.N < 4096 * 1024 < 2 * q.N
    _compare(q, 1, 2, 2, {})
