"""Renders return with their samples in the accumulators, so what follows on
another stream (a render into the same scratch, the statistics, the read-back,
a tensor the frame wraps) needs no wait; small scenes take one launch and
larger ones the wavefront, and both keep this."""
import ctypes

import numpy as np
import pytest

from paper_2303_15762_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("big", [False, True])
def test_calls_on_several_streams_follow_each_other(gr, big):
    import torch
    scene = sg.procedural_scene(seed=4, n_objects=4, target_tris=3000) if big else sg.grating_scene()
    s = gr.Scene(scene)
    make = sg.procedural_view if big else sg.grating_view
    shape = dict(width=640, height=480, n_bins=8, n_stokes=1)
    a, b = make(spp=32, **shape), make(spp=16, first_sample=32, **shape)
    flags = gr.FLAG_NEE if big else 0
    one = gr.Frame([a])
    for v in (a, b):
        gr.render([s], [v], one, seed=2, flags=flags)
    want = one.readback(0)
    streams = [torch.cuda.Stream() for _ in range(3)]
    h = [ctypes.c_void_p(x.cuda_stream) for x in streams]
    for _ in range(3):
        f = gr.Frame([a], stream=h[0])
        gr.render([s], [a], f, stream=h[0], seed=2, flags=flags)
        gr.render([s], [b], f, stream=h[1], seed=2, flags=flags)
        assert f.stats(stream=h[2])["samples"] == 640 * 480 * 16
        assert np.array_equal(f.readback(0, stream=h[2]), want)
