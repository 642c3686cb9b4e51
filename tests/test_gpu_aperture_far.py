"""Aperture samples outside every truncation radius contribute nothing, however
far away: at infinity, or where the squared distance overflows FP32 and the
phase is not a number.  The elements equal, bit for bit, those without the
sample; a sample that is not a number still makes them so.  And fields too weak for a
normal FP32 number count when nothing is truncated."""
import numpy as np
import pytest

from paper_2303_15762_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("x", [np.inf, -np.inf, 1e300, -3e19, 2e17])
@pytest.mark.parametrize("at", [0, 70, 200])
def test_far_sample_of_a_slit(gr, x, at):
    s = sg.double_slit_setup(d=200.0, n_per_slit=100, x0=np.array([0.0, -333.0, 500.0]), dkappa=1e-3)
    tail = (s["beta"], s["z"], s["k"], s["reach"], s["dtheta"], s["rho_cut"])
    want, _ = gr.aperture_backward_2d(s["x0"], s["x_ap"], s["w_ap"], *tail)
    got, _ = gr.aperture_backward_2d(s["x0"], np.insert(s["x_ap"], at, x), np.insert(s["w_ap"], at, 0.3), *tail)
    assert np.min(want) > 0 and np.array_equal(got, want)


@pytest.mark.parametrize("x", [(3e19, 0.0), (5.0, -4e19), (1e17, 1e17)])
@pytest.mark.parametrize("at", [0, 70, 450])
def test_far_sample_of_an_aperture(gr, x, at):
    s = sg.aperture3d_setup("disk", n_nodes=15, dt=2e-3, x0=[[0.0, 0.0], [60.0, -20.0]])
    tail = (s["beta"], s["z"], s["k"], s["reach"], s["dt"], s["rho_cut"])
    want, _ = gr.aperture_backward_3d(s["x0"], s["x_ap"], s["w_ap"], *tail)
    got, _ = gr.aperture_backward_3d(s["x0"], np.insert(s["x_ap"], at, x, 0), np.insert(s["w_ap"], at, 0.3), *tail)
    assert np.min(want) > 0 and np.array_equal(got, want)


def test_sample_that_is_not_a_number(gr):
    s = sg.double_slit_setup(d=200.0, n_per_slit=40, x0=np.array([0.0, 90.0]), dkappa=1e-3)
    x = s["x_ap"].copy()
    x[33] = np.nan
    got, _ = gr.aperture_backward_2d(s["x0"], x, s["w_ap"], s["beta"], s["z"], s["k"], s["reach"], s["dtheta"], s["rho_cut"])
    assert np.all(np.isnan(got))


@pytest.mark.parametrize("u2", [60.0, 90.0, 95.0])
def test_field_far_below_the_axis(gr, u2):
    """Without truncation a field of e^-u2 below 2^-126 still counts: one sample
    of a large weight, as seen from its own tail.  FP32 knows the exponent to
    ~2^-17 and such a field (2^-137 at u2 = 95) to 2^-13, the square to twice that."""
    from oracle import aperture3d as a3
    s = sg.aperture3d_setup("rect", size=24.0, n_nodes=9, x0=[[0.0, 0.0], [0.4, -0.3]])
    x, w = np.array([[np.sqrt(2 * u2) * s["beta_ap"], 0.0]]), np.array([1e30])
    reach, dt = 2.0, 1.0 / s["z"]
    got, _ = gr.aperture_backward_3d(s["x0"], x, w, s["beta"], s["z"], s["k"], reach, dt, 50.0)
    ref = a3.backward_generalized_rays(s["x0"], s["z"], s["k"], x, w, s["beta"], reach, dt, 50.0)
    assert np.min(ref) > 0 and np.max(np.abs(got / ref - 1)) < 2 ** -11
    # the 2D form: sum of |w e^-u2|^2 k cos^2(theta) / (sqrt(pi) beta') dtheta / (2 pi)
    th = np.arctan((0.0 - reach) / s["z"])
    dth = 0.7 / s["z"]
    n = int(np.ceil(2 * np.arctan(reach / s["z"]) / dth))
    c = np.cos(th + dth * np.arange(n))
    b2 = s["beta"] ** 2 + (s["z"] / c / s["k"]) ** 2 / s["beta"] ** 2
    u = (x[0, 0] + s["z"] * np.tan(th + dth * np.arange(n))) * c
    want = np.sum(w[0] ** 2 * np.exp(-u * u / b2) * s["k"] * c * c / np.sqrt(np.pi * b2)) * dth / (2 * np.pi)
    got, _ = gr.aperture_backward_2d(np.zeros(1), x[:, 0], w, s["beta"], s["z"], s["k"], reach, dth, 50.0)
    assert abs(got[0] / want - 1) < 2 ** -11
