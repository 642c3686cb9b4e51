"""The default 4-wide nodes on a 16-bit grid give the images of the FP32 binary
nodes bit for bit, where the grid can go wrong: planes that lie on grid lines,
axes without extent, rays along the axes (zero direction components), scenes
far from the origin, a whole scene in one plane, and scenes whose triangles are
too small for the grid (those walk the FP32 nodes)."""
import numpy as np
import pytest

from paper_2303_15762_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu


def _boxes(offset=0.0, scale=1.0):
    """Axis-aligned mirror boxes on a rough floor, an emitter above."""
    rng = np.random.default_rng(3)
    tris, mat = [], []
    mats = [sg.material(sg.MAT_ROUGH, fresnel=1, n_re=0.3, n_im=3.5, sigma_h_um=0.2, corr_len_um=3.0),
            sg.material(sg.MAT_MIRROR, fresnel=1, n_re=0.4, n_im=3.0),
            sg.material(sg.MAT_EMITTER, Le=1.0, coh_len_um=20.0)]
    for i in range(6):
        for j in range(6):
            tris.append(sg._quad((i - 2.5, 0.0, j - 2.5), (0, 0, 0.5), (0.5, 0, 0)))
            mat += [0, 0]
    for _ in range(12):
        t = sg._box(rng.integers(-8, 8, 3) * 0.25 * (1, 0, 1) + (0, 0.25, 0), (0.125, 0.25, 0.125))
        tris.append(t)
        mat += [1] * len(t)
    tris.append(sg._quad((0.0, 2.0, 0.0), (1.5, 0, 0), (0, 0, 1.5)))
    mat += [2, 2]
    return sg._scene(np.concatenate(tris) * scale + offset, mat, mats, [sg.light(sg.LIGHT_ENV, E=0.1)])


def _view(offset=0.0, ortho=0, eye=(0.0, 1.5, 4.0), **kw):
    e = np.array(eye) + offset
    return sg.view(eye=e, look_at=np.array((0.0, 0.0, 0.0)) + offset, up=(0, 0, -1) if ortho else (0, 1, 0),
                   vfov_deg=50.0, width=41, height=37, n_bins=4, spp=16, max_depth=5, n_stokes=4, ortho=ortho,
                   ortho_half_m=2.0, **kw)


def _same(gr, scene, view):
    a = gr.render_image(scene, view, seed=8, flags=gr.FLAG_NEE)
    b = gr.render_image(scene, view, seed=8, flags=gr.FLAG_NEE | gr.FLAG_FP32_NODES)
    assert np.linalg.norm(a) > 0
    assert np.array_equal(a, b)


@pytest.mark.parametrize("offset", [0.0, 1000.0, -3.0e4])
def test_planes_on_grid_lines(gr, offset):
    _same(gr, _boxes(offset), _view(offset))


def test_rays_along_an_axis(gr):
    _same(gr, _boxes(), _view(ortho=1, eye=(0.0, 1.9, 0.0)))


def test_scene_in_one_plane(gr):
    q = np.concatenate([sg._quad((x, y, 0.0), (0.25, 0, 0), (0, 0.25, 0)) for x in (-0.5, 0, 0.5) for y in (-0.5, 0.5)])
    scene = sg._scene(q, [0] * len(q), [sg.material(sg.MAT_MIRROR)], [sg.light(sg.LIGHT_ENV)])
    for eye in ((0.0, 0.0, 2.0), (0.3, -0.2, 1.0)):
        v = sg.view(eye=eye, look_at=(0, 0, 0), width=33, height=31, n_bins=2, spp=4, max_depth=2, vfov_deg=70.0)
        _same(gr, scene, v)


def test_all_triangles_at_one_point(gr):
    """Every vertex the same: a grid without extent, no hit anywhere."""
    v = np.full((5, 3, 3), 0.25, np.float32)
    scene = sg._scene(v, [0] * 5, [sg.material(sg.MAT_MIRROR)], [sg.light(sg.LIGHT_ENV)])
    _same(gr, scene, sg.view(eye=(0.25, 0.25, 2.0), look_at=(0.25, 0.25, 0.0), width=9, height=9, n_bins=1, spp=4))


@pytest.mark.parametrize("far", [40.0, 4.0e5])
def test_small_triangles_in_a_wide_scene(gr, far):
    """A distant triangle stretches the grid; at 4e5 m its step (6 m) exceeds
    the boxes and the FP32 nodes are walked."""
    s = _boxes()
    extra = np.array([[[far, 0, 0], [far + 1, 0, 0], [far, 1, 0]]], np.float32)
    scene = dict(s, verts=np.concatenate([s["verts"], extra]), tri_mat=np.concatenate([s["tri_mat"], [1]]).astype(np.int32))
    _same(gr, scene, _view())
