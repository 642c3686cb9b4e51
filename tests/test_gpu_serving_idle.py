"""A server is not idle while a request's scene is being built: the replay of
arrivals must serve it, however long that takes."""
import time

import numpy as np
import pytest

from paper_2303_15762_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu


def test_request_being_built(gr):
    from paper_2303_15762_gb300 import serving

    class Slow:
        def __getattr__(self, name):
            return getattr(gr, name)

        def Scene(self, *args, **kw):
            time.sleep(0.3)
            return gr.Scene(*args, **kw)

    scene, view = sg.serving_request(np.random.default_rng(1), 1)
    slow = Slow()
    srv = serving.ProgressiveServer(slow, memory_budget_bytes=1 << 33)
    stats = serving.run_poisson(slow, [serving.Request(1, scene, dict(view, width=24, height=16), 2)], 500.0, srv, seed=2)
    srv.close()
    assert stats["requests"] == 1
