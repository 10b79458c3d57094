"""Bounds that the contraction's operand splits state (half-precision parts of a
scaled FP32 value), by the arithmetic itself: IEEE half and single on the CPU."""
import numpy as np

F, H = np.float32, np.float16


def _values(n, seed):
    """FP32 values as a cell's, scaled: the largest in [2^14, 2^15), the others spread below it."""
    rng = np.random.default_rng(seed)
    x = (rng.uniform(1, 2, n) * 2.0 ** rng.integers(-6, 14, n) * rng.choice([-1, 1], n)).astype(F)
    x[0] = F(2.0 ** 15 - 2.0 ** -9)  # the largest there is
    return x


def test_two_parts():
    x = np.concatenate([_values(200000, 1), np.array([F(2.0 ** 14) * (1 + F(2049) * F(2.0 ** -23))])])
    hi = x.astype(H)
    lo = (x - hi.astype(F)).astype(H)
    err, ax = np.abs(hi.astype(float) + lo.astype(float) - x.astype(float)), np.abs(x.astype(float))
    assert (err <= np.maximum(2.0 ** -23 * ax, 2.0 ** -25)).all()
    assert err[-1] > 2.0 ** -23.1 * ax[-1]  # a whole unit in the last place of FP32, at worst
    # the product of the low parts, which is left out
    assert (np.abs(lo.astype(float)) <= 2.0 ** -11 * ax).all()


def test_three_parts():
    x = _values(200000, 2)
    x0 = np.rint(x * F(2.0 ** -7)) * F(2.0 ** 7)
    assert (np.abs(x0) <= 2.0 ** 15).all() and (x0.astype(H).astype(F) == x0).all()
    x1 = (x - x0).astype(H)
    x2 = ((x - x0) - x1.astype(F)).astype(H)
    err, ax = np.abs(x0.astype(float) + x1.astype(float) + x2.astype(float) - x.astype(float)), np.abs(x.astype(float))
    assert (err[ax >= 64] == 0).all()  # down to 2^-9 of the largest: all bits
    assert (err <= np.maximum(2.0 ** -23 * ax, 2.0 ** -25)).all()  # below: two halves, 2^-32 of the largest
    # leading products of the largest order (216 values): integers of one unit below 2^24
    assert 216 * 256 * 256 < 2 ** 24
