"""FP32: the sum over N_i of -w'(q) q that the adjoint divides by (kept in every
step checkpoint, sorted order) for long neighbour lists, which a warp sums.
Lane sums of a dozen terms added up in FP64 leave about 3e-8 of it, one FP32
chain of 400 terms 2.6e-7 (both simulated on the same FP32 terms); the terms'
own rounding averages to under 3e-8.  45 terms (more than the cache of 40 holds
within 1.05 H, so a warp's too): a compensated sum 4.5e-8 with its storing, one
chain 1.1e-7.  1/H is taken rounded, as the pass forms
it: its rounding shifts every q alike."""
import numpy as np
import pytest

from gpu_common import cast_state, device, min_image
from paper_1712_01294_gb300 import inputs as I


def _slices(ctx, ck, N):
    """sd [N] and the order [N] from a GZ_CKPT_LISTS checkpoint: FP64 rates, then
    H, n, sd, flux records, adjoint info, limiter indices, keys, order."""
    raw, at, out = ck.cpu().numpy(), 0, []
    for nbytes in (32 * N, 4 * N, 4 * N, 4 * N, 128 * N, 160 * N, 40 * N, 4 * N, 4 * N):
        out.append(raw[at:at + nbytes])
        at += -(-nbytes // 256) * 256
    return out[3].view(np.float32), out[8].view(np.uint32)


@pytest.mark.gpu
@pytest.mark.parametrize("ngb,tol", [(400.0, 1e-7), (45.0, 7e-8)])
def test_sum_of_long_lists(ngb, tol):
    import torch
    import paper_1712_01294_gb300 as m
    q = cast_state(I.turbulence(14, seed=9), 1)
    ctx = m.Context([q.N], m.default_params(ngb=ngb, max_ngb=640, density_cache=40))
    d = device(q, 1)
    d["h"] *= (ngb / 32.0) ** (1.0 / 3.0)
    ck = ctx.new_checkpoint(2)
    ctx.step(d, 1e-4, None, ck, 2)
    assert ctx.status(reset=True)["ok"]
    sd, order = _slices(ctx, ck, q.N)
    H = d["h"].cpu().numpy()
    ctx.close()
    X = np.stack([q.x, q.y, q.z])
    err = []
    for k in range(0, q.N, 7):
        i = int(order[k])
        dd = min_image(X - X[:, i:i + 1])
        r2 = (dd * dd).sum(0)
        r2[i] = 9.0
        qq = np.sqrt(r2[r2 < float(H[i]) ** 2]) * float(np.float32(1) / H[i])
        assert (qq.size > 64) == (ngb > 100)
        ref = np.where(qq <= 0.5, 12 * qq ** 2 - 18 * qq ** 3, 6 * (1 - qq) ** 2 * qq).sum()
        err.append(sd[k] / ref - 1)
    assert np.sqrt(np.mean(np.square(err))) < tol
