"""The read-back of few bins, whose blocks take runs of pixels: bins around the
powers of two and the line to the tiles, images that end inside a run (4096
elements of one component, 1024 of four) and within its first row of 32, for
accumulators and images that are only 4-byte aligned too: exactly
(sum - compensation) * (1 / count) of the wrapped buffer."""
import numpy as np
import pytest

from paper_2303_15762_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,height,bins", [(1, 1, 1), (31, 1, 1), (64, 64, 1), (4097, 1, 1), (683, 3, 2), (1365, 1, 3),
                                               (37, 29, 4), (61, 47, 5), (73, 7, 8), (241, 1, 17), (151, 1, 27), (133, 1, 28)])
@pytest.mark.parametrize("stokes", [1, 4])
@pytest.mark.parametrize("shift", [0, 1])
def test_few_bins(gr, width, height, bins, stokes, shift):
    import torch
    v = sg.grating_view(width=width, height=height, spp=bins + 1, n_bins=bins, n_stokes=stokes)
    n = gr.accum_floats([v])
    acc = torch.zeros(n + 4, dtype=torch.float32, device="cuda")[shift:shift + n]
    f = gr.Frame([v], accum=acc)
    gr.render([gr.Scene(sg.grating_scene(fresnel=1))], [v], f, seed=3)
    acc.copy_(torch.as_tensor(np.random.default_rng(bins).standard_normal(n).astype(np.float32)))
    out = torch.full((n // 2 + 8,), 7.0, dtype=torch.float32, device="cuda")[shift:]
    got = f.readback(0, out=out)[:n // 2 + 4].cpu().numpy()
    assert np.all(got[n // 2:] == 7.0)
    a = acc.cpu().numpy().reshape(2, bins, height, width, stokes)
    counts = np.array([2.0] + [1.0] * (bins - 1), np.float32)
    want = np.transpose((a[0] - a[1]) * (np.float32(1) / counts)[:, None, None, None], (1, 2, 0, 3))
    assert np.array_equal(got[:n // 2].reshape(want.shape), want)
    assert np.array_equal(f.readback(0), want)
