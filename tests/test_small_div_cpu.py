"""The force kernel's division of small integers (a + 1/2 over b in FP32): the quotient truncates to a / b for every
a < 2^14 and b <= 2^8, whatever the two units that an approximate FP32 quotient may be off."""
import numpy as np


def test_every_small_quotient():
    a = np.arange(1 << 14, dtype=np.int64)
    for b in range(1, 257):
        q = ((a + np.float32(0.5)).astype(np.float32) / np.float32(b)).astype(np.float32)  # to nearest: half a unit
        for units in (-3, 0, 3):
            off = (q.view(np.int32) + units).view(np.float32)
            assert np.array_equal(off.astype(np.int64), a // b), (b, units)
