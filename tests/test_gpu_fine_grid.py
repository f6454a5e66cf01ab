"""Grids finer than one support radius a cell (an autotuner's candidates) keep
the density pass's one-thread form: a support of many cells there holds no
more particles than on the usual grid, and with a warp for each the pass took
six times as long (64^3: 946 us at half the cell length, 158 at one)."""
import pytest

from gpu_common import cast_state, device
from paper_1712_01294_gb300 import inputs as I


def _time(m, q, cell_factor):
    import torch
    ctx = m.Context([q.N], m.default_params(cell_factor=cell_factor))
    d = device(q, 1)
    best = 1e9
    for _ in range(8):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        ctx.density(d)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    assert ctx.status()["ok"]
    ctx.close()
    return best


@pytest.mark.gpu
def test_half_the_cell_length_keeps_the_form():
    # eight times the cells, 1.7 to 2 times the candidates and cells tested
    import paper_1712_01294_gb300 as m
    q = cast_state(I.turbulence(64, seed=3), 1)
    one, half = _time(m, q, 1.0), _time(m, q, 0.5)
    print(f"density call: cell_factor 1 {one:.3f} ms, 0.5 {half:.3f} ms")
    assert half < 3 * one
