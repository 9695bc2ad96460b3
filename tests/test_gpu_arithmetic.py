"""The FP64 arithmetic done on the FP32 and integer pipes, directly.

1 / x and 1 / sqrt(x) start from an FP32 estimate and take one cubic correction
that leaves less than 2^-60; the last multiply-add rounds by 2^-53, and for the
square root the rounding of y^2 adds 2^-54 and that of y h less than 2^-70: both
within 2^-52 of the value, against the correctly rounded one within 2^-52 + 2^-53.
The scatter's accumulator returns one term as it is, and two terms as their
correctly rounded sum where their exponents are at most 5 apart (no bit is cut
off), else within 2^-57 of the larger before the rounding. The read-out of an
integer is its nearest double, ties away from zero."""
import fractions

import numpy as np
import pytest
import torch

from paper_1708_01773_gb300 import build, feasm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    feasm.lib()


def values():
    rng = np.random.default_rng(7)
    m = rng.uniform(1, 2, 40000)
    x = np.ldexp(m, rng.integers(-1021, 1023, m.size)) * rng.choice([-1, 1], m.size)
    near = np.ldexp(rng.uniform(1, 2, 40000), rng.integers(-8, 9, 40000)) * rng.choice([-1, 1], 40000)
    one = np.concatenate([np.nextafter(1.0, [0, 2]), 1 + np.arange(1, 200) * 2.0**-52, 2 - np.arange(1, 200) * 2.0**-52,
                          1 - np.arange(1, 200) * 2.0**-53, 4 - np.arange(1, 200) * 2.0**-51])
    powers = 2.0 ** np.arange(-1022, 1024)
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -2.0**-1074, 2.0**-1022, np.finfo(float).max])
    cancel = np.repeat(near[:500], 2)
    cancel[1::2] *= -1
    cancel[1::4] = np.nextafter(cancel[1::4], 0)
    return np.concatenate([x, near, one, -one, powers, -powers, special, cancel])


def integers(n):
    rng = np.random.default_rng(8)
    bits = rng.integers(0, 63, n)
    v = rng.integers(0, 2**62, n) >> (62 - bits)
    v[:64] = [1 << k for k in range(63)] + [0]
    k = np.arange(64, 2064)
    v[k] = (rng.integers(2**52, 2**53, k.size) << 9) + (1 << 8)   # ties
    v[2064:2100] = 2**62 - 1 - np.arange(36)
    return v * rng.choice([-1, 1], n)


def test_arithmetic_on_other_pipes():
    x = values()
    v = integers(x.size)
    out = torch.empty(x.size * 5, dtype=torch.float64, device="cuda")
    feasm.fe_selftest_arithmetic(torch.tensor(x, device="cuda"), torch.tensor(v, device="cuda"), out)
    o = out.cpu().numpy().reshape(-1, 5)
    y = np.roll(x, -1)
    with np.errstate(all="ignore"):
        want = 1.0 / x
        normal = np.isfinite(want) & (np.abs(want) >= 2.0**-1022) & (np.abs(x) >= 2.0**-1022)
        assert (np.abs(o[normal, 0] - want[normal]) <= (2.0**-52 + 2.0**-53) * np.abs(want[normal])).all()
        assert np.array_equal(o[~normal, 0], want[~normal], equal_nan=True)
        positive = (x >= 2.0**-1022) & np.isfinite(x)
        ref = 1 / np.sqrt(x[positive].astype(np.longdouble))
        assert (np.abs(o[positive, 1] - ref) <= 2.0**-52 * ref).all()
        assert np.isnan(o[~positive, 1]).all()
        assert np.array_equal(o[:, 2], x, equal_nan=True)
        total = x + y
    ok = np.isfinite(x) & np.isfinite(y) & np.isfinite(total)
    ex, ey = np.frexp(x)[1], np.frexp(y)[1]
    close = ok & ((np.abs(ex - ey) <= 5) | (x == 0) | (y == 0))
    assert close.sum() > 20000 and np.array_equal(o[close, 3], total[close])
    far = ok & ~close
    big = np.maximum(np.abs(x[far]), np.abs(y[far]))
    with np.errstate(over="ignore"):  # the spacing at the largest double
        assert (np.abs(o[far, 3] - total[far]) <= np.spacing(np.abs(total[far])) + 2.0**-56 * big).all()


def test_read_out_of_integers():
    v = integers(20000)
    x = torch.ones(v.size, dtype=torch.float64, device="cuda")
    out = torch.empty(v.size * 5, dtype=torch.float64, device="cuda")
    feasm.fe_selftest_arithmetic(x, torch.tensor(v, device="cuda"), out)
    got = out.cpu().numpy().reshape(-1, 5)[:, 4]
    for i, g in zip(v.tolist(), got):
        m = abs(i)
        sh = max(m.bit_length() - 53, 0)
        r = ((m >> (sh - 1)) + 1) >> 1 if sh else m   # half away from zero
        assert fractions.Fraction(float(g)) == fractions.Fraction((r << sh) * (1 if i >= 0 else -1), 2**60), i
