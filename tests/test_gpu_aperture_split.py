"""Apertures and screens at the edges of the aperture kernels' split: sample
counts around the 64-sample chunks that are skipped together, samples in any
order, one detector element and a few, one direction and a ragged number of
them, and sample sets beyond 48 KB of shared memory, against the oracle's FP64
sums to the tolerance of the other aperture tests."""
import numpy as np
import pytest

from paper_2303_15762_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dkappa,x0", [(1, 3e-4, [0.0]), (31, 2e-4, [50.0, -333.0]), (32, 7e-4, [0.0, 500.0, 90.0]),
                                         (33, 2e-4, [-900.0]), (129, 9e-4, [10.0, 1500.0]), (3100, 4e-3, [120.0])])
@pytest.mark.parametrize("shuffled", [False, True])
def test_slit_sizes(gr, n, dkappa, x0, shuffled):
    from oracle import doubleslit as ds
    s = sg.double_slit_setup(d=200.0, n_per_slit=n, x0=np.array(x0), dkappa=dkappa)
    o = np.random.default_rng(n).permutation(2 * n) if shuffled else np.arange(2 * n)
    got, _ = gr.aperture_backward_2d(s["x0"], s["x_ap"][o], s["w_ap"][o], s["beta"], s["z"], s["k"], s["reach"],
                                     s["dtheta"], s["rho_cut"])
    ref = ds.backward_generalized_rays(s["x0"], 200.0, s["beta"], n=n, dkappa=dkappa)
    assert np.max(np.abs(got - ref)) / np.max(ref) < 2e-5


@pytest.mark.parametrize("n_ap", [1, 2, 63, 64, 65, 129, 450])
@pytest.mark.parametrize("dt,n_det", [(9e-4, 1), (3.3e-3, 5)])
def test_aperture_sizes(gr, n_ap, dt, n_det):
    from oracle import aperture3d as a3
    rng = np.random.default_rng(n_ap)
    s = sg.aperture3d_setup("disk", n_nodes=15, dt=dt)
    o = rng.permutation(len(s["w_ap"]))[:n_ap]
    x0 = rng.uniform(-80.0, 80.0, (n_det, 2))
    got, _ = gr.aperture_backward_3d(x0, s["x_ap"][o], s["w_ap"][o], s["beta"], s["z"], s["k"], s["reach"], dt,
                                     s["rho_cut"])
    ref = a3.backward_generalized_rays(x0, s["z"], s["k"], s["x_ap"][o], s["w_ap"][o], s["beta"], s["reach"], dt,
                                       s["rho_cut"])
    assert np.max(np.abs(got - ref)) / np.max(ref) < 2e-5


def test_one_direction(gr):
    """A grid of one direction per element: the rest of the block only votes."""
    from oracle import aperture3d as a3
    s = sg.aperture3d_setup("rect", size=24.0, n_nodes=9)
    reach, dt = 20.0, 41.0 / s["z"]     # the one ray of each element lands at (20, 20)
    x0 = np.array([[0.0, 0.0], [35.0, -60.0]])
    assert len(a3.direction_grid(x0[0], s["z"], reach, dt)[0]) == 1
    got, _ = gr.aperture_backward_3d(x0, s["x_ap"], s["w_ap"], s["beta"], s["z"], s["k"], reach, dt, s["rho_cut"])
    ref = a3.backward_generalized_rays(x0, s["z"], s["k"], s["x_ap"], s["w_ap"], s["beta"], reach, dt, s["rho_cut"])
    assert np.min(ref) > 0
    assert np.max(np.abs(got - ref)) / np.max(ref) < 2e-5
