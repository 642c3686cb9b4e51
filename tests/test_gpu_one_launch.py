"""Renders of scenes of a few triangles as one launch give the wavefront's images
bit for bit (an iteration bound, however large, asks for the wavefront), over
what the rule accepts: 0 to 16 triangles, every material, 1 and 4 Stokes
components, the table types, Russian roulette, raw order weights, each tree
flag, uneven sample counts and offsets, an orthographic camera, several views
and scenes, block and pool options; 17 triangles and next-event estimation take
the wavefront anyway."""
import numpy as np
import pytest

from paper_2303_15762_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu


def _scene(kind):
    """Quads around the origin, open to a distant source and an environment."""
    mats = {"grating": sg.material(sg.MAT_GRATING, fresnel=1, n_re=0.3, n_im=3.0, period_um=1.7, height_um=0.25),
            "rough": sg.material(sg.MAT_ROUGH, fresnel=1, n_re=0.3, n_im=3.5, sigma_h_um=0.15, corr_len_um=3.0),
            "mirror": sg.material(sg.MAT_MIRROR, fresnel=1, n_re=0.4, n_im=2.5),
            "emitter": sg.material(sg.MAT_EMITTER, Le=1.0, coh_len_um=15.0),
            "absorber": sg.material(sg.MAT_ABSORBER)}
    lights = [sg.light(sg.LIGHT_DISTANT, (0.3, 0.2, 0.9), 1.0, 10.0), sg.light(sg.LIGHT_ENV, E=0.2)]
    if kind == "empty":
        return sg._scene(np.zeros((0, 3, 3)), [], [mats["mirror"]], lights)
    if kind == "triangle":
        return sg._scene(np.array([[[-1, -1, 0], [1, -1, 0], [0, 1, 0]]]), [0], [mats["rough"]], lights)
    if kind == "glass":      # a closed slab (12 triangles) above a rough floor
        s = sg.dielectric_scene(env=0.3)
        return s if len(s["tri_mat"]) <= 16 else None
    if kind == "grating":
        return sg.grating_scene(fresnel=1)
    # "mixed": 16 triangles, "seventeen": one more
    at = [("grating", (0, 0, 0)), ("rough", (0.9, 0, 0.1)), ("mirror", (-0.9, 0, 0.1)), ("emitter", (0, 0.9, 0.6)),
          ("absorber", (0, -0.9, 0.1)), ("mirror", (0.9, 0.9, 0.3)), ("rough", (-0.9, 0.9, 0.2)), ("grating", (0.9, -0.9, 0.1))]
    names = ["grating", "rough", "mirror", "emitter", "absorber"]
    tris = [sg._quad(c, (0.45, 0, 0.1), (0, 0.45, 0.05)) for _, c in at]
    mat = [names.index(n) for n, _ in at for _ in (0, 1)]
    if kind == "seventeen":
        tris.append(np.array([[[-0.9, -0.9, 0.2], [-0.5, -0.9, 0.2], [-0.9, -0.5, 0.3]]]))
        mat.append(2)
    return sg._scene(np.concatenate(tris), mat, [mats[n] for n in names], lights)


def _view(kind, **kw):
    a = dict(eye=(0.3, -0.2, 3.0), look_at=(0, 0, 0), vfov_deg=50.0, width=37, height=23, n_bins=5, spp=12, max_depth=6)
    if kind == "glass":
        a.update(eye=(0.0, 0.22, 0.6), look_at=(0.0, 0.08, 0.0), vfov_deg=40.0)
    if kind == "grating":
        a.update(eye=(0, 0, 0.2), look_at=(0, 0, 0), vfov_deg=28.0)
    return sg.view(**dict(a, **kw))


def _both(gr, scenes, views, **opts):
    images = []
    for extra in ({}, dict(max_iterations=100_000)):
        f = gr.Frame(views)
        gr.render([gr.Scene(s) for s in scenes], views, f, seed=9, **opts, **extra)
        images.append([f.readback(i) for i in range(len(views))])
        st = f.stats()
        assert st["samples"] == sum(v["width"] * v["height"] * v["spp"] for v in views)
        images[-1].append(st["iterations"])
        f.close()
    assert any(np.any(x) for x in images[0][:-1])
    for a, b in zip(images[0][:-1], images[1][:-1]):
        assert np.array_equal(a, b)
    return images[0][-1], images[1][-1]


@pytest.mark.parametrize("kind", ["empty", "triangle", "grating", "mixed", "seventeen", "glass"])
@pytest.mark.parametrize("stokes", [1, 4])
@pytest.mark.parametrize("table", ["f32", "f16", "bf16"])
def test_scenes_and_tables(gr, kind, stokes, table):
    s = _scene(kind)
    assert s is not None
    one, wave = _both(gr, [s], [_view(kind, n_stokes=stokes)], table_dtype=table, flags=gr.FLAG_RR)
    assert (one == 1) == (kind != "seventeen") and wave > 1


@pytest.mark.parametrize("flags", ["FLAG_NO_RENORM", "FLAG_WIDE_BVH", "FLAG_FP32_NODES", "FLAG_NEE"])
def test_flags(gr, flags):
    one, _ = _both(gr, [_scene("mixed")], [_view("mixed", n_stokes=4)], flags=getattr(gr, flags))
    assert (one == 1) == (flags != "FLAG_NEE")


@pytest.mark.parametrize("kw", [dict(spp=3, n_bins=7, first_sample=11), dict(spp=1, n_bins=1), dict(max_depth=0),
                                dict(ortho=1, ortho_half_m=1.2), dict(width=1, height=1, spp=700, n_bins=3)])
def test_views(gr, kw):
    for opts in (dict(), dict(block=32), dict(pool_size=300, regen_threshold_pct=40, use_graph=True)):
        _both(gr, [_scene("mixed")], [_view("mixed", n_stokes=4, **kw)], **opts)


def test_several_views_and_scenes(gr):
    kinds = ["mixed", "empty", "grating", "triangle"]
    views = [_view(k, scene_index=i, view_index=5 + i, max_depth=1 + 2 * i, width=9 + 8 * i) for i, k in enumerate(kinds)]
    _both(gr, [_scene(k) for k in kinds], views)
