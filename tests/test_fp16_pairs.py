"""FP16 pairs of the tensor-core Step II (split2 of csrc/step2_tc.cu), emulated with
numpy: hi = x rounded to FP16, lo = the remainder rounded to FP16.  FP16 has 11
significant bits and no spacing below 2^-24, so

    |x - hi - lo| <= max(2^-23 |x|, 2^-25),    |lo| <= max(2^-11 |x|, 2^-25)

over the scaled range (fields up to 250, their products up to 62500)."""
import numpy as np


def _split(x):
    hi = x.astype(np.float16)
    r = hi.astype(np.float32) - x                     # exact: the kernel's remainder, negated
    lo = -(r.astype(np.float16).astype(np.float32))
    return hi.astype(np.float32), lo


def test_pairs_hold_their_values():
    rng = np.random.default_rng(3)
    x = np.concatenate([
        (rng.uniform(1.0, 2.0, 400000) * 2.0 ** rng.integers(-30, 15, 400000)),
        2.0 ** np.arange(-30, 16), np.float64(62500.0) * rng.uniform(0.9, 1.0, 1000),
        # the worst of a binade: half a spacing of hi away from it, and next to that
        (1 + 2.0 ** -11 + 2.0 ** -23 * np.arange(-4, 5))[None, :].repeat(40, 0).ravel() * 2.0 ** np.repeat(np.arange(-25, 15), 9),
    ]).astype(np.float32)
    x = np.concatenate([x, -x])
    x = x[np.abs(x) <= 62500.0]
    hi, lo = _split(x)
    assert np.isfinite(hi).all()
    d = x.astype(np.float64)
    a = np.abs(d)
    err = np.abs(d - hi.astype(np.float64) - lo.astype(np.float64))
    assert (err <= np.maximum(2.0 ** -23 * a, 2.0 ** -25)).all()
    assert (np.abs(lo) <= np.maximum(2.0 ** -11 * a, 2.0 ** -25)).all()
    # the bounds are reached, so no smaller power of two would do
    big = a >= 0.25
    assert (err[big] / a[big]).max() > 2.0 ** -24 and err[~big].max() > 2.0 ** -26


def test_low_parts_product():
    """lo lo', which the kernel leaves out, is at most 2^-22 |x x'| for |x|, |x'| >= 2^-14."""
    rng = np.random.default_rng(4)
    x, y = (rng.uniform(1, 2, 200000).astype(np.float32) * np.float32(2.0) ** rng.integers(-14, 8, 200000) for _ in "xy")
    (_, lx), (_, ly) = _split(x.astype(np.float32)), _split(y.astype(np.float32))
    assert (np.abs(lx.astype(np.float64) * ly) <= 2.0 ** -22 * np.abs(x.astype(np.float64) * y)).all()
