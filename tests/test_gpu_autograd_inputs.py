"""The autograd layer on the inputs that its frame calls take, against contiguous batches of
the same values on the device."""
import numpy as np
import pytest

from synth import labels_from, polygon_image, random_guide

import _gpu

pytestmark = pytest.mark.gpu

B, H, W = 2, 40, 52


def _inputs():
    import torch
    rgba = torch.from_numpy(np.stack([_gpu.rgba(polygon_image(H, W, 5, i)) for i in range(B)])).cuda()
    labels = torch.from_numpy(np.stack([labels_from(_gpu.hole_blobs(H, W, i, n=5, rmin=2, rmax=6))
                                        for i in range(B)])).cuda()
    g = np.stack([random_guide(H, W, i) for i in range(B)])
    mag, phi = (torch.from_numpy(v).cuda() for v in (np.hypot(g[..., 0], g[..., 1]), np.arctan2(g[..., 1], g[..., 0])))
    up = torch.from_numpy(np.random.default_rng(3).normal(size=(B, H, W, 4)).astype(np.float32)).cuda()
    return rgba, labels, mag, phi.requires_grad_(), up


def _run(rgba, labels, mag, phi, wrt, up):
    import torch

    from paper_1611_05319_gb300.autograd import guidefill_fill
    mu = torch.tensor(10.0, requires_grad=True)
    out = guidefill_fill(rgba, labels, mag, phi, mu)
    return out.detach(), torch.autograd.grad(out, [wrt, mu], grad_outputs=up)


def _assert_same(a, b):
    """Outputs bit for bit; the gradients but for the order of the scatter's atomics (as in
    test_gpu_autograd_batch.py)."""
    import torch
    assert a[0].device == b[0].device and torch.equal(a[0], b[0])
    (pa, ma), (pb, mb) = a[1], b[1]
    assert float((pa - pb).abs().max()) <= 1e-4 * float(pb.abs().max())
    assert abs(float(ma) - float(mb)) <= 1e-4 * abs(float(mb))


def test_colours_on_the_cpu(cuda_device):
    """They are copied to the device; the output and the gradients are there."""
    rgba, labels, mag, phi, up = _inputs()
    want = _run(rgba, labels, mag, phi, phi, up)
    _assert_same(_run(rgba.cpu(), labels, mag, phi, phi, up), want)


@pytest.mark.parametrize("form", ["lists", "longer", "mixed"])
def test_labels_and_angles_by_frame(cuda_device, form):
    """They are taken frame by frame: lists of frames and batches longer than rgba's."""
    import torch
    rgba, labels, mag, phi, up = _inputs()
    rgba.requires_grad_()
    want = _run(rgba, labels, mag, phi, rgba, up)
    if form == "lists":
        labels, mag, phi = list(labels), list(mag), list(phi.detach())
    elif form == "longer":
        labels, mag, phi = (torch.cat([t, t[:1]]) for t in (labels, mag, phi.detach()))
    else:
        labels, mag = list(labels), torch.cat([mag, mag[:1]])
    _assert_same(_run(rgba, labels, mag, phi, rgba, up), want)
