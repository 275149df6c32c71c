"""The autograd layer against the frame calls it is made of: batches, inputs that are not
contiguous, an output that the caller overwrites before the backward pass."""
import numpy as np
import pytest

from synth import labels_from, polygon_image, random_guide

import _gpu

pytestmark = pytest.mark.gpu

H, W = 40, 52


@pytest.mark.parametrize("B", [1, 3])
@pytest.mark.parametrize("strided", [False, True])
def test_layer_equals_frame_calls(cuda_device, B, strided):
    import torch

    import paper_1611_05319_gb300 as gf
    from paper_1611_05319_gb300.autograd import guidefill_fill
    ctx = gf.context(0)
    rng = np.random.default_rng(B)
    rgba = torch.from_numpy(np.stack([_gpu.rgba(polygon_image(H, W, 5, i)) for i in range(B)])).cuda()
    labels = torch.from_numpy(np.stack([labels_from(_gpu.hole_blobs(H, W, i, n=5, rmin=2, rmax=6))
                                        for i in range(B)])).cuda()
    g = np.stack([random_guide(H, W, i) for i in range(B)])
    mag, phi = (torch.from_numpy(v).cuda() for v in (np.hypot(g[..., 0], g[..., 1]), np.arctan2(g[..., 1], g[..., 0])))
    up = torch.from_numpy(rng.normal(size=(B, H, W, 4)).astype(np.float32)).cuda()
    guides = [ctx.guide_from_angle(labels[i], mag[i], phi[i]) for i in range(B)]
    rs = ctx.fill_batched(list(rgba), list(labels), guides, mu=10.0, stall=True)
    gi, gp, gmu = ctx.fill_backward(rs, guides, list(up), mu=10.0)
    if strided:  # every second column of wider tensors, the same values
        def wide(t):
            w = torch.zeros(t.shape[:2] + (2 * W,) + t.shape[3:], dtype=t.dtype, device=t.device)
            w[:, :, ::2] = t
            return w[:, :, ::2]
        rgba, labels, mag, phi, up = (wide(t) for t in (rgba, labels, mag, phi, up))
    rgba.requires_grad_()
    phi.requires_grad_()
    mu = torch.tensor(10.0, requires_grad=True)
    out = guidefill_fill(rgba, labels, mag, phi, mu)
    assert torch.equal(out.detach(), torch.stack([r.rgba for r in rs]))
    with torch.no_grad():
        out.zero_()
    d = torch.autograd.grad(out, [rgba, phi, mu], grad_outputs=up)
    # the scatter's atomics add a pixel's up to 28 terms of one step in any order
    scale = float(torch.stack(gi).abs().max())
    assert float((d[0] - torch.stack(gi)).abs().max()) <= 64 * 2.0 ** -24 * scale
    top = float(torch.stack(gp).abs().max())
    assert float((d[1] - torch.stack(gp)).abs().max()) <= 1e-4 * top
    assert abs(float(d[2]) - float(gmu.sum())) <= 1e-4 * float(gmu.abs().sum())
