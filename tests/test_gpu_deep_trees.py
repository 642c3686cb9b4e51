"""Scenes whose trees are chains: triangles on one another merge one pair per
round of the clustering, so n of them make n - 1 binary levels and a third as
many 4-wide ones (256 at 769 triangles, 257 at 770).  They are created and
render as any other scene, alone and inside one, whichever nodes are asked for.
And scenes of nested shells, whose walk leaves three subtrees waiting at every
level: 121 entries, where the binary tree's walk leaves 42."""
import numpy as np
import pytest

from paper_2303_15762_gb300 import scenegen as sg
from _parity import assert_parity

pytestmark = pytest.mark.gpu


def _stack(n):
    """n equal mirror triangles above a rough floor's centre."""
    t = np.array([[-0.3, 0.2, -0.2], [0.3, 0.2, -0.2], [0.0, 0.2, 0.4]], np.float32)[[0, 2, 1]]
    return np.repeat(t[None], n, 0)


def _scene(n, inside):
    mats = [sg.material(sg.MAT_MIRROR, fresnel=1, n_re=0.4, n_im=3.0)]
    env = sg.light(sg.LIGHT_ENV, E=0.3)
    if not inside:
        return sg._scene(_stack(n), [0] * n, mats, [env])
    s = sg.procedural_scene(seed=3, n_objects=4, target_tris=2000, n_emitters=1)
    tri_mat = np.concatenate([s["tri_mat"], np.full(n, len(s["mats"]))]).astype(np.int32)
    return sg._scene(np.concatenate([np.asarray(s["verts"], np.float32).reshape(-1, 3, 3), _stack(n)]), tri_mat,
                     np.concatenate([s["mats"], mats]), [env])


@pytest.mark.parametrize("n,inside", [(769, False), (770, False), (800, True), (5000, False), (5000, True)])
def test_equal_triangles(gr, oracle, n, inside):
    scene = _scene(n, inside)
    v = sg.view(eye=(0.1, 1.3, 2.0), look_at=(0.0, 0.1, 0.0), up=(0, 1, 0), vfov_deg=40.0, width=19, height=17, n_bins=4,
                spp=8, max_depth=3)
    a = gr.render_image(scene, v, seed=5, flags=gr.FLAG_NEE)
    for flag in (gr.FLAG_FP32_NODES, gr.FLAG_WIDE_BVH):
        assert np.array_equal(a, gr.render_image(scene, v, seed=5, flags=gr.FLAG_NEE | flag))
    ref = oracle.Scene(scene).render(v, 5, gr.FLAG_NEE)
    assert_parity(a, ref)


def test_nested_shells(gr):
    """Seen from their common centre: 40 shells of 8 triangles, each 0.35 of the
    last, whose boxes a ray along the axis enters and whose triangles it passes
    (the smallest first: of boxes entered at once the walk takes the first)."""
    t = []
    for i in reversed(range(40)):
        for j in range(8):
            z = 0.35 ** i * (1 + 0.02 * j)
            t.append([(-0.08 * z, 0.4 * z, z), (0.4 * z, -0.08 * z, z), (0.4 * z, 0.4 * z, z)])
    ground = sg._tile_tris(np.array([0.0, -3.0, 0.0]), 4.0, 60, 0.1, np.random.default_rng(0), 0.0)
    mats = [sg.material(sg.MAT_MIRROR, fresnel=1, n_re=0.4, n_im=3.0),
            sg.material(sg.MAT_ROUGH, fresnel=1, n_re=0.3, n_im=3.5, sigma_h_um=0.2, corr_len_um=3.0)]
    scene = sg._scene(np.concatenate([np.asarray(t), ground]), [0] * len(t) + [1] * len(ground), mats,
                      [sg.light(sg.LIGHT_ENV, E=0.3)])
    v = sg.view(eye=(0, 0, 0), look_at=(0, 0, 1.0), up=(0, 1, 0), vfov_deg=50.0, width=33, height=31, n_bins=2, spp=4,
                max_depth=3)
    a = gr.render_image(scene, v, seed=5, flags=gr.FLAG_NEE)
    assert len(np.unique(a)) > 1
    assert np.array_equal(a, gr.render_image(scene, v, seed=5, flags=gr.FLAG_NEE | gr.FLAG_FP32_NODES))
