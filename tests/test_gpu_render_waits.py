"""A render returns when nothing of it runs any more, on every exit: the host
loop enqueues a batch beyond the one that ends the render, and the next call on
the frame, on another stream, would reset the counters and slots it reads."""
import ctypes

import pytest

from paper_2303_15762_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts", [dict(flags="nee"), dict(flags="nee", profile=True), dict(flags="nee", use_graph=True),
                                  dict(flags="nee", pool_size=4096), dict(), dict(profile=True)])
def test_stream_is_idle_after_a_render(gr, opts):
    import torch
    nee = opts.get("flags") == "nee"
    opts = dict(opts, flags=gr.FLAG_NEE if nee else 0)
    s = gr.Scene(sg.procedural_scene(seed=4, n_objects=4, target_tris=3000) if nee else sg.grating_scene())
    v = (sg.procedural_view if nee else sg.grating_view)(width=320, height=240, n_bins=8, n_stokes=1, spp=8)
    f = gr.Frame([v])
    torch.cuda.synchronize()
    x = torch.cuda.Stream()
    for _ in range(10):
        gr.render([s], [v], f, stream=ctypes.c_void_p(x.cuda_stream), seed=2, **opts)
        assert x.query()


def test_stream_is_idle_after_the_iteration_bound(gr):
    import torch
    s = gr.Scene(sg.procedural_scene(seed=4, n_objects=4, target_tris=3000))
    v = sg.procedural_view(width=320, height=240, n_bins=8, n_stokes=1, spp=64, max_depth=6)
    f = gr.Frame([v])
    torch.cuda.synchronize()
    x = torch.cuda.Stream()
    for _ in range(10):
        with pytest.raises(gr.GrError):
            gr.render([s], [v], f, stream=ctypes.c_void_p(x.cuda_stream), seed=2, max_iterations=4)
        assert x.query()
