"""The quotient g / m of the rough surface's term probabilities (gr_render.cu
forms it from a table of reciprocals): the corrected product is the correctly
rounded quotient for every term count of the table; the plain product is not."""
import ctypes
import ctypes.util

import numpy as np


def test_corrected_product_is_the_quotient():
    fma = ctypes.CDLL(ctypes.util.find_library("m")).fma
    fma.restype, fma.argtypes = ctypes.c_double, [ctypes.c_double] * 3
    rng = np.random.default_rng(1)
    g = np.concatenate([rng.uniform(0, 50, 400), 10.0 ** rng.uniform(-12, 1.7, 400), [50.0, np.nextafter(50.0, 0), 0.0]])
    plain = 0
    for m in range(1, 128):
        r = 1.0 / m
        for x in map(float, g):
            q = x * r
            plain += q != x / m
            assert fma(fma(-q, float(m), x), r, q) == x / m
    assert plain > 0
