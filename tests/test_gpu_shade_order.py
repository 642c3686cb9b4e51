"""Shading in the order of what each ray met: chunks of the queue with one kind
of entry, with all kinds, ragged ends and block sizes down to one warp give the
images of a pool of one warp-sized chunk at a time, bit for bit."""
import numpy as np
import pytest

from paper_2303_15762_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu


def _scene(kind):
    if kind == "escapes":    # every ray misses
        s = sg.grating_scene()
        return dict(s, verts=s["verts"] + np.float32(50.0))
    if kind == "one":        # every entry a rough surface or an escape
        return sg.procedural_scene(seed=4, n_objects=1, target_tris=700, n_emitters=1)
    s = sg.procedural_scene(seed=31, n_objects=8, target_tris=6000, n_emitters=2)
    return sg.add_glass(s, n_glass=6, seed=2, env_radiance=0.1)


@pytest.mark.parametrize("kind", ["escapes", "one", "all"])
@pytest.mark.parametrize("mode", ["plain", "hero", "aniso"])
@pytest.mark.parametrize("stokes", [1, 4])
def test_shading_order_leaves_images_unchanged(gr, kind, mode, stokes):
    S = [gr.Scene(_scene(kind))]
    flags = gr.FLAG_NEE | gr.FLAG_RR | {"plain": 0, "hero": gr.FLAG_HERO, "aniso": gr.FLAG_ANISO}[mode]
    v = sg.procedural_view(width=67, height=41, spp=16, n_bins=8, n_stokes=stokes, max_depth=5)
    images = []
    for opts in (dict(block=32, pool_size=256), dict(), dict(block=96), dict(block=256, pool_size=5000, use_graph=True)):
        f = gr.Frame([v])
        gr.render(S, [v], f, seed=3, flags=flags, **opts)
        images.append(f.readback(0))
        f.close()
    assert kind == "escapes" or np.linalg.norm(images[0]) > 0
    for k in (1, 2, 3):
        assert np.array_equal(images[0], images[k]), k
