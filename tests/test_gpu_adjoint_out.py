"""``Context.fill_backward(out=...)`` writes through the pointers of the tensors it is given, so
it takes only those that the kernel's writes fit."""
import numpy as np
import pytest

from synth import labels_from, polygon_image, random_guide

import _gpu

H, W = 24, 37


def test_outputs_on_the_cpu_are_refused():
    """Before any call of CUDA."""
    import torch

    import paper_1611_05319_gb300 as gf
    ctx = gf.Context.__new__(gf.Context)
    ctx.device = 0
    r = gf.FillResult(None, torch.empty((H, W), dtype=torch.int32), None, None, None)
    with pytest.raises(ValueError):
        ctx.fill_backward([r], [None], [None], out=([torch.empty(H, W, 4)], [torch.empty(H, W)]))
    with pytest.raises(ValueError):
        ctx.fill_backward([r, r], [None] * 2, [None] * 2, out=([torch.empty(H, W, 4)], [torch.empty(H, W)]))


@pytest.mark.gpu
def test_outputs_given(cuda_device):
    import torch

    import paper_1611_05319_gb300 as gf
    ctx = gf.context(0)
    rgba = torch.from_numpy(_gpu.rgba(polygon_image(H, W, 5, 1))).cuda()
    labels = torch.from_numpy(labels_from(_gpu.hole_blobs(H, W, 1, n=5, rmin=2, rmax=6))).cuda()
    guide = torch.from_numpy(random_guide(H, W, 1)).cuda()
    rs = ctx.fill_batched([rgba], [labels], [guide], mu=10.0, stall=True)
    up = torch.from_numpy(np.random.default_rng(0).normal(size=(H, W, 4)).astype(np.float32)).cuda()
    gi, gp, _ = ctx.fill_backward(rs, [guide], [up], mu=10.0)

    def new(*shape, **kw):
        return torch.empty(shape, device="cuda", **kw)
    a, b = new(H, W, 4), new(H, W)
    for bad in [(new(H, W, 3), b), (new(H - 1, W, 4), b), (new(W, H, 4).transpose(0, 1), b),
                (new(H, W, 4, dtype=torch.float64), b), (new(H, W, 4, dtype=torch.float16), b), (a, new(H, W - 1)),
                (a, new(H, 2 * W)[:, ::2]), (a, new(H, W, dtype=torch.int32)), (a.cpu(), b), (a, b.cpu()), (None, b)]:
        with pytest.raises(ValueError):
            ctx.fill_backward(rs, [guide], [up], mu=10.0, out=([bad[0]], [bad[1]]))
    o = ctx.fill_backward(rs, [guide], [up], mu=10.0, out=([a], [b]))
    assert o[0][0] is a and o[1][0] is b
    # but for the order of the scatter's atomics, as in test_gpu_autograd_batch.py
    assert float((a - gi[0]).abs().max()) <= 64 * 2.0 ** -24 * float(gi[0].abs().max())
    assert float((b - gp[0]).abs().max()) <= 1e-4 * float(gp[0].abs().max())
