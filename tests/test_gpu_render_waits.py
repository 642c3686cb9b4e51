"""What a render leaves running: nothing when it is one launch or one graph or
when it fails; else launches that find nothing to do, which the frame's next
use, on any stream, comes after (they read the counters and slots that a render
resets)."""
import ctypes

import numpy as np
import pytest

from paper_2303_15762_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu


def _handle(stream):
    return ctypes.c_void_p(stream.cuda_stream)


@pytest.mark.parametrize("opts", [dict(use_graph=True), dict(), dict(profile=True), dict(max_iterations=4)])
def test_stream_is_idle(gr, opts):
    import torch
    if not opts or "profile" in opts:
        s, v = gr.Scene(sg.grating_scene()), sg.grating_view(width=320, height=240, n_bins=8, spp=64)
    else:
        s = gr.Scene(sg.procedural_scene(seed=4, n_objects=4, target_tris=3000))
        v = sg.procedural_view(width=320, height=240, n_bins=8, n_stokes=1, spp=64, max_depth=6)
    f = gr.Frame([v])
    torch.cuda.synchronize()
    x = torch.cuda.Stream()
    for _ in range(10):
        if "max_iterations" in opts:
            with pytest.raises(gr.GrError):
                gr.render([s], [v], f, stream=_handle(x), seed=2, **opts)
        else:
            gr.render([s], [v], f, stream=_handle(x), seed=2, **opts)
        assert x.query()


@pytest.mark.parametrize("pool", [0, 4096])
def test_next_use_comes_after(gr, pool):
    import torch
    s = gr.Scene(sg.procedural_scene(seed=4, n_objects=4, target_tris=3000))
    v = sg.procedural_view(width=640, height=480, n_bins=8, n_stokes=1, spp=8)
    opts = dict(seed=2, flags=gr.FLAG_NEE, pool_size=pool)
    f = gr.Frame([v])
    torch.cuda.synchronize()
    x, y = torch.cuda.Stream(), torch.cuda.Stream()
    gr.render([s], [v], f, stream=_handle(x), **opts)
    torch.cuda.synchronize()
    image = f.readback(0)
    for k in range(2, 12):
        gr.render([s], [v], f, stream=_handle(x if k % 2 else y), **opts)
        seen = f.stats(stream=_handle(y if k % 2 else x))["iterations"]
        torch.cuda.synchronize()
        assert f.stats()["iterations"] == seen
        f.reset(stream=_handle(x))
        gr.render([s], [v], f, stream=_handle(x), **opts)
        assert np.array_equal(f.readback(0, stream=_handle(y)), image)


def test_failed_allocation_leaves_nothing_running(gr):
    import torch
    s = gr.Scene(sg.procedural_scene(seed=4, n_objects=4, target_tris=3000))
    v = sg.procedural_view(width=640, height=480, n_bins=8, n_stokes=1, spp=8)
    many = dict(sg.procedural_view(width=8192, height=8192, n_bins=16, n_stokes=1, spp=16), view_index=0)
    f, g = gr.Frame([v]), gr.Frame([many])
    torch.cuda.synchronize()
    x, y = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(3):
        gr.render([s], [v], f, stream=_handle(x), seed=2, flags=gr.FLAG_NEE)
        want = f.readback(0, stream=_handle(x))
        # frames[0]'s scratch serves the call: 2^30 slots of 429 bytes, more than any device has
        with pytest.raises(gr.GrError, match="scratch allocation failed"):
            gr.render_multi([s], [v, many], [f, g], [0, 0], stream=_handle(y), seed=2, flags=gr.FLAG_NEE | gr.FLAG_HERO,
                            pool_size=(1 << 30) - 256)
        assert x.query() and y.query()
        assert np.array_equal(f.readback(0), want)
