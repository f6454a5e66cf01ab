"""The FP32 path's support update is the FP64 one: H - f/f' of FP32 numbers,
its place in the bracket and its FP32 rounding, formed by FP32 operations
(h_step, restated here) and in FP64, give one result, also where the FP32
difference falls on an end of the bracket."""
import numpy as np

f = np.float32


def _fp32(H, q, lo, hi):
    Hn = H - q
    ok = (Hn > lo) & (Hn < hi)
    t = Hn - H
    err = (H - (Hn - t)) - (q + t)
    return Hn, np.where(Hn == lo, err > 0, np.where(Hn == hi, err < 0, ok))


def _fp64(H, q, lo, hi):
    Hn = H.astype(np.float64) - q.astype(np.float64)
    return Hn.astype(f), (Hn > lo) & (Hn < hi)


def test_update_and_bracket():
    rng = np.random.default_rng(3)
    n = 400000
    H = (0.5 * 10.0 ** rng.uniform(-3, 0, n)).astype(f)
    q = (H * 10.0 ** rng.uniform(-7.2, 0.5, n) * rng.choice([-1, 1], n)).astype(f)
    lo, hi = f(0.5) * H, f(2) * H
    # set ends: anywhere, at H itself, and at or one place from the difference
    kind = rng.integers(0, 5, n)
    near = H - q
    end = np.where(kind == 0, (H * rng.uniform(0.3, 1, n)).astype(f),
                   np.where(kind == 1, H, np.where(kind == 2, near, np.nextafter(near, f(0)))))
    lo = np.where((kind < 4) & (q > 0) & (end <= H), end, lo)
    hi = np.where((kind < 4) & (q < 0) & (end >= H), end, hi)
    a, b = _fp32(H, q, lo, hi), _fp64(H, q, lo, hi)
    assert ((a[0] == lo) | (a[0] == hi)).sum() > 10000
    assert np.array_equal(a[0], b[0])
    assert np.array_equal(a[1], b[1])
