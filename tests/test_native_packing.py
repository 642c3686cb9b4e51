"""Materials and lights as the C structs: kinds are whole numbers modulo 2^32,
as ctypes stores them, and one that is no number is refused."""
import numpy as np
import pytest

from paper_2303_15762_gb300 import _native as nat


def _material(**words):
    r = np.zeros(16, np.float32)
    r[[0, 1]] = 2.0, 1.0
    r[2:] = np.arange(2, 16) / 7
    for k, v in words.items():
        r[int(k[1:])] = v
    return r


@pytest.mark.parametrize("words", [{}, dict(w0=3.9), dict(w1=-0.9), dict(w0=-2.0), dict(w0=3e9), dict(w1=2.0 ** 40), dict(w0=-1e38)])
@pytest.mark.parametrize("rows", [2, 70])
def test_struct_fields(words, rows):
    out, n = nat._pack_rows([_material()] * (rows - 1) + [_material(**words)], 16, 2)
    r = _material(**words)
    m = nat.gr_material.from_buffer_copy(out[-1].tobytes())
    want = nat.gr_material()
    want.type, want.fresnel = int(r[0]), int(r[1])
    assert n == rows and (m.type, m.fresnel) == (want.type, want.fresnel)
    assert [m.n_re, m.n_im, m.period_um, m.height_um, *m.gdir] == [float(x) for x in r[2:9]]
    assert [m.sigma_h_um, m.corr_len_um, m.Le, m.coh_len_um, m.cauchy_b_um2] == [float(x) for x in r[9:14]]
    assert not np.any(out[:, 14:])


@pytest.mark.parametrize("word", [0, 1])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("rows", [1, 70])
def test_kind_that_is_no_number(word, value, rows):
    with pytest.raises((ValueError, OverflowError)):
        nat._pack_rows([_material()] * (rows - 1) + [_material(**{"w%d" % word: value})], 16, 2)


def test_lights():
    out, n = nat._pack_rows(np.zeros((0, 8)), 8, 1)
    assert n == 0 and out.shape == (1, 8)
    with pytest.raises(ValueError):
        nat._pack_rows([[np.nan] + [0.0] * 7], 8, 1)
