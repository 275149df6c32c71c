"""Segments whose far end lies 1e4 to 1e9 px away, where FP32 coordinates are rounded by up to
tens of pixels: in a frame of one bin, whose list holds every segment that ends in it, the
nearest segment within 3 eta is the one of the fixed FP32 expression over all segments."""
import numpy as np
import pytest

import oracle

import _gpu

H = W = 32


def scene(length, seed):
    rng = np.random.default_rng([seed, int(np.log10(length))])
    n = 3
    b = rng.uniform(0, H, (n, 2))
    ang = rng.uniform(0, 2 * np.pi, n)
    ang[0] = np.round(ang[0] / (np.pi / 2)) * (np.pi / 2)
    a = b - length * np.stack([np.cos(ang), np.sin(ang)], 1)
    pts = np.stack([a, b], 1)
    pts[1::2] = pts[1::2, ::-1]  # the near end first
    labels = (rng.uniform(size=(H, W)) < (0.05 if seed % 2 else 1.0)).astype(np.uint8)
    return np.arange(0, 2 * n + 1, 2, dtype=np.int32), pts.reshape(-1, 2).astype(np.float32), labels


@pytest.mark.gpu
@pytest.mark.parametrize("length", [1e4, 1e6, 1e8, 1e9])
def test_far_ends(cuda_device, length):
    import torch

    import paper_1611_05319_gb300 as gf
    for seed in range(12):
        off, pts, labels = scene(length, seed)
        ties = oracle.guidance_ties(labels, off, pts, eta=3.0)
        got = gf.context(0).guidance(torch.from_numpy(labels).cuda(), off, pts).cpu().numpy()
        _gpu.assert_guide_parity(ties, got, labels)
