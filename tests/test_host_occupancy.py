"""Occupancy arrays reach the library as contiguous bytes, nonzero = occupied: byte and truth arrays as they
are, every other type through a comparison."""
import numpy as np
import pytest

from paper_2503_06757_gb300 import prrtc as P


@pytest.mark.parametrize("make", [
    lambda a: a.astype(np.uint8), lambda a: a.astype(np.uint8) * 255, lambda a: a.astype(bool),
    lambda a: a.astype(np.int64) * 256, lambda a: a.astype(np.float32) * 0.25, lambda a: a.astype(np.int8) * -1,
    lambda a: a.tolist(), lambda a: np.asfortranarray(a.astype(np.uint8)),
    lambda a: np.repeat(a.astype(bool), 2, axis=2)[:, :, ::2],
    lambda a: np.where(a, np.nan, 0.0),
])
def test_occupancy_bytes(make):
    a = np.random.default_rng(0).random((3, 4, 5)) < 0.4
    got = P._occ(make(a))
    assert got.dtype == np.uint8 and got.flags.c_contiguous and got.shape == a.shape
    np.testing.assert_array_equal(got != 0, a)
