"""Bins with more segments than their list holds scan every point of their frame: polylines of
any length with repeated points, points before the first spline and after the last, splines
of one point and of none, whole frames and single strips of hole pixels."""
import numpy as np
import pytest

import oracle

import _gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,n,eta", [(70, 100, 900, 11.0), (33, 31, 600, 3.0), (8, 200, 1500, 20.0)])
@pytest.mark.parametrize("frac", [1.0, 0.02])
def test_every_point_scanned(cuda_device, H, W, n, eta, frac):
    import torch

    import paper_1611_05319_gb300 as gf
    rng = np.random.default_rng(n)
    lens = rng.choice([0, 1, 2, 3, 9], n)
    off = 5 + np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)  # five points belong to no spline
    start = rng.uniform([0, 0], [W, H], (n + 1, 2))
    pts = np.concatenate([start[-1] + rng.normal(size=(5, 2))] +
                         [s + np.cumsum(rng.normal(scale=3.0, size=(k, 2)), 0) for s, k in zip(start, lens)] +
                         [rng.uniform(0, 30, (40, 2))]).astype(np.float32)
    pts[7::6] = pts[6:-1:6][:len(pts[7::6])]  # segments of no length
    w = rng.uniform(0.1, 1.0, n).astype(np.float32)
    labels = (rng.uniform(size=(H, W)) < frac).astype(np.uint8)
    ties = oracle.guidance_ties(labels, off, pts, eta=eta, weight=w)
    got = gf.context(0).guidance(torch.from_numpy(labels).cuda(), off, pts, eta=eta, weight=w).cpu().numpy()
    assert (got != 0).any()
    _gpu.assert_guide_parity(ties, got, labels)
