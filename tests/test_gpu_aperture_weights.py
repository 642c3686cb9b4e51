"""The FP64 terms of a direction at FP64's accuracy: a single direction whose ray
lands on the only sample (phase and footprint terms vanish, the amplitude is
exactly 1) leaves its weight, a product of FP64 terms of a few roundings each:
16 in all at most."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 16 * 2.0 ** -53


@pytest.mark.parametrize("z", [40.0, 9000.0])
def test_weight_of_a_direction(gr, z):
    k, reach, worst = 2 * np.pi / 0.7, 16.0, 0.0
    for beta in np.geomspace(0.3, 30.0, 64):
        dth = 3 * np.arctan(reach / z)
        got, _ = gr.aperture_backward_2d([0.0], [reach], [1.0], beta, z, k, reach, dth, 2.5)
        c = np.cos(np.arctan(-reach / z))
        b2 = beta ** 2 + (z / k / c) ** 2 / beta ** 2
        worst = max(worst, abs(got[0] / (k * c * c * dth / np.sqrt(np.pi * b2) / (2 * np.pi)) - 1))
    assert worst <= TOL


@pytest.mark.parametrize("z", [40.0, 9000.0])
def test_weight_of_a_direction_3d(gr, z):
    k, reach, worst = 2 * np.pi / 0.7, 16.0, 0.0
    for beta in np.geomspace(0.3, 30.0, 64):
        dt = 33.0 / z
        got, _ = gr.aperture_backward_3d([[0.0, 0.0]], [[reach, reach]], [1.0], beta, z, k, reach, dt, 2.5)
        s2 = 1 / (1 + 2 * (reach / z) ** 2)
        b2 = beta ** 2 + (z / k) ** 2 / s2 / beta ** 2
        worst = max(worst, abs(got[0] / (s2 ** 2.5 / (np.pi * b2) * (k * dt) ** 2 / (4 * np.pi ** 2)) - 1))
    assert worst <= TOL
