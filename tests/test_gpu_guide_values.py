"""The guide field's values bit for bit against the oracle's FP64 evaluation over what the
pair arithmetic has to hold: segments from a hundredth of a pixel to the frame's
diagonal, axis-parallel ones, weights, radii, ends inside and outside the frame, strips
and bins cut by the border, bins with more segments than their list holds."""
import numpy as np
import pytest

import oracle

import _gpu

pytestmark = pytest.mark.gpu


def _lines(rng, n, H, W, length):
    a = rng.uniform([-20, -20], [W + 20, H + 20], (n, 2))
    ang = rng.uniform(0, 2 * np.pi, n)
    ang[::5] = np.round(ang[::5] / (np.pi / 2)) * (np.pi / 2)  # axis-parallel, nearly or exactly
    b = a + length * np.stack([np.cos(ang), np.sin(ang)], 1)
    pts = np.stack([a, b], 1).reshape(-1, 2).astype(np.float32)
    pts[1::20, 1] = pts[0::20, 1]  # exactly
    return np.arange(0, 2 * n + 1, 2, dtype=np.int32), pts


@pytest.mark.parametrize("eta", [0.4, 3.0, 11.0])
@pytest.mark.parametrize("length,n,weighted", [(0.01, 300, False), (3.0, 400, True), (40.0, 150, False),
                                               (900.0, 60, True), (5000.0, 30, False), (2.0, 6000, False)])
def test_values(cuda_device, eta, length, n, weighted):
    import torch

    import paper_1611_05319_gb300 as gf
    H, W = 203, 331
    rng = np.random.default_rng(int(length * 10) + n)
    off, pts = _lines(rng, n, H, W, length)
    w = rng.uniform(0.0, 1.0, n).astype(np.float32) if weighted else None
    labels = (rng.uniform(size=(H, W)) < 0.7).astype(np.uint8)
    labels[:40] = 0
    ties = oracle.guidance_ties(labels, off, pts, eta=eta, **({} if w is None else {"weight": w}))
    g = gf.context(0).guidance(torch.from_numpy(labels).cuda(), off, pts, eta=eta, weight=w)
    torch.cuda.synchronize()
    got = g.cpu().numpy()
    assert (got != 0).any()
    assert _gpu.assert_guide_parity(ties, got, labels) < (labels == 1).sum()
