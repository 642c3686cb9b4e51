"""Where the scene's 16-bit grid is coarse against its triangles: down to 2 steps
per triangle the default walk is that of the 4-wide grid nodes (fewer visits than
the FP32 nodes' binary walk), below it is the FP32 nodes', and the images are the
FP32 nodes' bit for bit on both sides of the line."""
import numpy as np
import pytest

from test_gpu_grid_nodes import _boxes, _view

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("far,grid", [(3000.0, True), (5000.0, True), (7800.0, True), (20000.0, False)])
def test_line_to_the_fp32_nodes(gr, far, grid):
    s = _boxes()  # most boxes' sides are 0.25 to 0.5 m
    extra = np.array([[[far, 0, 0], [far + 1, 0, 0], [far, 1, 0]]], np.float32)
    s = gr.Scene(dict(s, verts=np.concatenate([s["verts"], extra]), tri_mat=np.concatenate([s["tri_mat"], [1]]).astype(np.int32)))
    v = _view()
    images, visits = [], []
    for flag in (0, gr.FLAG_FP32_NODES):
        f = gr.Frame([v])
        gr.render([s], [v], f, seed=8, flags=gr.FLAG_NEE | flag)
        images.append(f.readback(0))
        visits.append(f.stats()["node_visits"])
    assert np.any(images[0]) and np.array_equal(*images)
    # (which leaves are tested before a visit, and so which visits are made, varies from run to run)
    assert (visits[0] < 0.8 * visits[1]) == grid
