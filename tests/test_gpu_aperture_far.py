"""Aperture samples outside every truncation radius contribute nothing, however
far away: at infinity, or where the squared distance overflows FP32 and the
phase is not a number.  The elements equal, bit for bit, those without the
sample; a sample that is not a number still makes them so."""
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
