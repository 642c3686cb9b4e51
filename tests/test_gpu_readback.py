"""The read-back's transposition at the edges of its 32 x 32 tiles, for 1 and 4
Stokes components, and for accumulators and images that are only 4-byte
aligned: exactly (sum - compensation) * (1 / count) of the wrapped buffer."""
import numpy as np
import pytest

from paper_2303_15762_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,height,bins", [(1, 1, 1), (31, 1, 33), (8, 4, 32), (33, 3, 31), (65, 17, 70)])
@pytest.mark.parametrize("stokes", [1, 4])
@pytest.mark.parametrize("shift", [0, 1])
def test_readback_transposes(gr, width, height, bins, stokes, shift):
    import torch
    v = sg.grating_view(width=width, height=height, spp=2 * bins + 1, n_bins=bins, n_stokes=stokes)
    n = gr.accum_floats([v])
    acc = torch.zeros(n + 4, dtype=torch.float32, device="cuda")[shift:shift + n]
    f = gr.Frame([v], accum=acc)
    s = gr.Scene(sg.grating_scene(fresnel=1))
    gr.render([s], [v], f, seed=3)
    out = torch.empty(width * height * bins * stokes + 4, dtype=torch.float32, device="cuda")[shift:]
    got = f.readback(0, out=out)[:n // 2].cpu().numpy().reshape(height, width, bins, stokes)
    host = f.readback(0)
    a = acc.cpu().numpy().reshape(2, bins, height, width, stokes)
    inv = np.float32(1) / np.array([3.0] + [2.0] * (bins - 1), np.float32)
    want = np.transpose((a[0] - a[1]) * inv[:, None, None, None], (1, 2, 0, 3))
    assert np.any(want)
    assert np.array_equal(got, want) and np.array_equal(host, want)
