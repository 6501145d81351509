"""The pair kernels' arithmetic that splits a list entry's stencil number into
its coordinates: every operation rounded to float32, for all 27 numbers and
index bits at both ends.  Each quotient is at least 1/18 from a rounding tie,
so float64 products rounded once stand for the multiply-adds."""
import numpy as np
import pytest


def fma32(a, b, c):
    return np.float32(np.float64(a) * np.float64(b) + np.float64(c))


@pytest.mark.parametrize("index", [0, 1, (1 << 26) + 12345, (1 << 27) - 1])
def test_every_stencil_number(index):
    r32 = np.float32(12582912.0)
    for st in range(27):
        ent = (st << 27) | index
        word = ((0x02580000 << 32 | ent) << 5 >> 32) & 0xFFFFFFFF
        c = np.float32(np.array(word, np.uint32).view(np.float32) - np.float32(8388621.0))
        z = np.float32(fma32(c, np.float32(1) / np.float32(9), r32) - r32)
        r = fma32(z, np.float32(-9), c)
        y = np.float32(fma32(r, np.float32(1) / np.float32(3), r32) - r32)
        x = fma32(y, np.float32(-3), r)
        assert (x, y, z) == (st % 3 - 1, st // 3 % 3 - 1, st // 9 - 1)
