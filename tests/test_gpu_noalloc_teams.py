"""gf_fill_noalloc with steps of more tiles than a cluster has warps (several clusters on the
frame), twice in a row on the same scratch, bit for bit against gf_fill on one cluster."""
import numpy as np
import pytest

from synth import labels_from, polygon_image, random_guide

import _gpu
from test_zz_no_alloc import _run

pytestmark = pytest.mark.gpu

H, W = 600, 840


@pytest.mark.parametrize("eps", [3.0, 4.0, 6.0])
@pytest.mark.parametrize("data_term", [False, True])
def test_wide_fronts(cuda_device, monkeypatch, eps, data_term):
    import paper_1611_05319_gb300 as gf
    from paper_1611_05319_gb300 import _lib
    make = _lib.make_params
    monkeypatch.setattr(_lib, "make_params", lambda **kw: make(**dict(kw, eps=eps)))
    ctx = gf.Context(0)
    img, g = _gpu.rgba(polygon_image(H, W, 9, 2)), random_guide(H, W, 4)
    hole = np.zeros((H, W), bool)
    hole[3:-3, 3:-3] = (np.add.outer(np.arange(H - 6) // 12, np.arange(W - 6) // 12) % 2) == 0  # a chequerboard
    lab = labels_from(hole)
    ctx.set_launch_config(16, 1)
    want = _run("gf_fill", img, lab, g, ctx, data_term=data_term)
    for _ in range(2):
        got = _run("gf_fill_noalloc", img, lab, g, data_term=data_term)
        for k in ("u", "shell", "enter"):
            assert np.array_equal(want[k], got[k])
        assert want["stats"] == got["stats"]
    ctx.close()
