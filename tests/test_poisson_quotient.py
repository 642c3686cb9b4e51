"""The quotient g / m of the rough surface's term probabilities (gr_render.cu
forms it from a table of reciprocals in two parts): the product with both parts
is the correctly rounded quotient for every term count of the table; the product
with the rounded reciprocal alone is not."""
import ctypes
import ctypes.util

import numpy as np


def test_product_with_both_parts_is_the_quotient():
    fma = ctypes.CDLL(ctypes.util.find_library("m")).fma
    fma.restype, fma.argtypes = ctypes.c_double, [ctypes.c_double] * 3
    rng = np.random.default_rng(1)
    g = np.concatenate([rng.uniform(0, 50, 400), 10.0 ** rng.uniform(-12, 1.7, 400), [50.0, np.nextafter(50.0, 0), 0.0]])
    plain = 0
    for m in range(1, 128):
        hi = 1.0 / m
        lead = float(np.float32(hi))
        lo = ((1.0 - m * lead) - m * (hi - lead)) / m
        assert lo == fma(-float(m), hi, 1.0) / m
        # near the middle between two quotients too
        q = g / m
        near = np.concatenate([g, (q + 0.5 * np.spacing(q)) * m, np.nextafter(q, np.inf) * m])
        for x in map(float, near):
            plain += x * hi != x / m
            assert fma(x, hi, x * lo) == x / m
    assert plain > 0
