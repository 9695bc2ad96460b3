"""The body force of every entry point: whatever np.resize(np.asarray(f, float64), 3)
takes, with its values, and what that refuses is refused."""
import warnings
from decimal import Decimal

import numpy as np
import pytest

from paper_1708_01773_gb300 import feasm

FORCES = [
    np.array([1.0, -2.5, 3e-300]), np.array([1.5, 2.5]), np.array([4.0]), np.arange(7.0), np.array([np.nan, np.inf, -0.0]),
    np.array([1, 2, 3]), np.array([2**63 - 1, -2**63 + 513, 2**53 + 1]), np.array([2**64 - 1, 0, 1], dtype=np.uint64),
    np.array([True, False, True]), np.array([0.1, 0.2, 0.3], dtype=np.float32), np.array([0.1, 6e4, 1], dtype=np.float16),
    np.array([1, 3, 5], dtype=np.longdouble) / 3, np.array([1.0, 2.0, 3.0], dtype=">f8"), np.arange(12.0)[::4], np.zeros(0),
    np.array([[1.0, 2.0], [3.0, 4.0]]), np.array(7.0), np.array(["1.5", "2", "-3e4"]), np.array([b"1.5", b"2"]),
    np.array([1 + 0j, 2, 3]), np.array([1, 2.5, True], dtype=object), np.array([None, 1.0, 2.0], dtype=object),
    np.array([Decimal("0.1"), Decimal(2)], dtype=object), np.array(["0.25", 1, 2], dtype=object),
    np.array([1, 2, 3], dtype="m8[s]"), np.ma.array([1.0, 2.0, 3.0], mask=[0, 1, 0]),
    [1, 2, 3], (0.5,), 2, 2.5, range(4), ["1", "2", "3"],
]


@pytest.mark.parametrize("force", FORCES, ids=lambda f: f"{type(f).__name__}-{getattr(f, 'dtype', '')}-{f!r}"[:40])
def test_force_as_numpy_converts_it(force):
    with warnings.catch_warnings():
        warnings.simplefilter("ignore")  # complex values lose their imaginary part
        want = np.ascontiguousarray(np.resize(np.asarray(force, dtype=np.float64), 3))
        got = np.array(list(feasm._force(force)))
    assert got.tobytes() == want.tobytes() or (np.isnan(want).any() and np.array_equal(got, want, equal_nan=True))


@pytest.mark.parametrize("force", [np.array(["x", "y", "z"]), np.array([object()], dtype=object), "abc", [[1, 2], [3]]])
def test_force_that_numpy_refuses(force):
    with pytest.raises((TypeError, ValueError)):
        np.asarray(force, dtype=np.float64)
    with pytest.raises((TypeError, ValueError)):
        feasm._force(force)
