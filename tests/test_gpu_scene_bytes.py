"""The 4-wide nodes' arrays hold what the collapse can make and no more: pairs of
triangles on a grid of 2^k squares a side make (2 n - 1) / 3 nodes for n = 8, 32
and 128, the most there can be, and the arrays behind them stay intact."""
import numpy as np
import pytest

from paper_2303_15762_gb300 import scenegen as sg
from paper_2303_15762_gb300.serving import Request

pytestmark = pytest.mark.gpu


def _pairs(side):
    t = []
    for x in range(side):
        for y in range(side):
            a = 0.3
            t += [[(x, y, 0), (x + a, y, 0), (x, y + a, 0)], [(x + a, y + a, 0), (x, y + a, 0), (x + a, y, 0)]]
    return np.asarray(t, np.float32) / side


@pytest.mark.parametrize("side", [1, 2, 4, 8, 40])
def test_most_wide_nodes(gr, side):
    t = _pairs(side)
    n = len(t)
    mats = [sg.material(sg.MAT_MIRROR, fresnel=1, n_re=0.4, n_im=3.0),
            sg.material(sg.MAT_ROUGH, fresnel=1, n_re=0.3, n_im=3.5, sigma_h_um=0.2, corr_len_um=3.0)]
    scene = sg._scene(t, np.arange(n) % 2, mats, [sg.light(sg.LIGHT_ENV, E=0.3)])
    v = sg.view(eye=(0.5, 0.45, 2.0), look_at=(0.5, 0.5, 0.0), up=(0, 1, 0), vfov_deg=30.0, width=33, height=31, n_bins=2,
                spp=4, max_depth=3)
    a = gr.render_image(scene, v, seed=5, flags=gr.FLAG_NEE)
    for flag in (gr.FLAG_FP32_NODES, gr.FLAG_WIDE_BVH):
        assert np.array_equal(a, gr.render_image(scene, v, seed=5, flags=gr.FLAG_NEE | flag))
    # vertices, material, binary node, key; two sets of 4-wide nodes (96 B, as
    # much as a binary node in FP16 and a 4-wide one per triangle); the rest
    held = gr.Scene(scene).device_bytes()
    assert held <= n * (48 + 4 + 64 + 8 + 96) + 13 * 256 + 4096
    assert held <= Request(0, scene, v, 1).scene_bytes_bound()
