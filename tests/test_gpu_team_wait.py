"""Clusters that fill a frame together give up waiting for each other after a set number of
polls: with a limit of one poll nearly every wait between them gives up.  The call returns,
every frame has either its complete result or GF_ERR_TIMEOUT (frames that no cluster has
taken any more included), and the context fills the same frames afterwards."""
import numpy as np
import pytest

from synth import labels_from, polygon_image, random_guide, rect_mask

import _gpu

pytestmark = pytest.mark.gpu

H, W = 137, 211
TIMEOUT = -3


def _batch(n):
    import torch
    labels, rgbas, guides = [], [], []
    for i in range(n):
        hole = rect_mask(H, W, 9, 7, 190, 120) if i % 2 == 0 else _gpu.hole_blobs(H, W, 5 + i, n=24, rmin=3, rmax=11)
        labels.append(torch.from_numpy(labels_from(hole)).cuda())
        rgbas.append(torch.from_numpy(_gpu.rgba(polygon_image(H, W, 9, i))).cuda())
        guides.append(torch.from_numpy(random_guide(H, W, i)).cuda())
    return rgbas, labels, guides


def _run(ctx, batch, **kw):
    import torch
    rs = ctx.fill_batched(*batch, **kw)
    torch.cuda.synchronize()
    return [(r.stats(), r.rgba.cpu().numpy(), r.shell.cpu().numpy()) for r in rs]


def _same(a, b):
    return a[0] == b[0] and np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])


@pytest.mark.parametrize("n,cs,nc", [(1, 1, 0), (1, 4, 0), (5, 1, 0), (5, 2, 0), (9, 1, 4), (9, 4, 3)])
@pytest.mark.parametrize("kw", [dict(), dict(rescan=True)], ids=["tracked", "rescan"])
def test_short_wait(cuda_device, n, cs, nc, kw):
    import paper_1611_05319_gb300 as gf
    ctx = gf.context(0)
    batch = _batch(n)
    try:
        ctx.set_launch_config(16, 1)  # no team
        want = _run(ctx, batch, **kw)
        ctx.set_launch_config(cs, nc)
        ctx.set_wait_limit(1)
        late = 0
        for _ in range(3):
            for a, b in zip(_run(ctx, batch, **kw), want):
                assert a[0]["status"] == TIMEOUT or _same(a, b)
                late += a[0]["status"] == TIMEOUT
        if nc == 0:  # more clusters than frames: there were teams
            assert late > 0
        ctx.set_wait_limit(0)
        assert all(_same(a, b) for a, b in zip(_run(ctx, batch, **kw), want))
    finally:
        ctx.set_wait_limit(0)
        ctx.set_launch_config(0, 0)


def test_a_cluster_joins_a_running_frame(cuda_device):
    """Two clusters, two frames: the cluster whose frame ends first joins the other frame in
    the middle.  With one poll the wait at that team's barrier gives up, so the timeout of the
    large frame shows that the team was formed."""
    import torch

    import paper_1611_05319_gb300 as gf
    ctx = gf.context(0)
    batch = _batch(1)
    small = np.zeros((H, W), bool)
    small[60, 100] = True
    batch = (batch[0] * 2, batch[1] + [torch.from_numpy(labels_from(small)).cuda()], batch[2] * 2)
    try:
        ctx.set_launch_config(16, 1)
        want = _run(ctx, batch)
        ctx.set_launch_config(1, 2)
        assert all(_same(a, b) for a, b in zip(_run(ctx, batch), want))
        ctx.set_wait_limit(1)
        got = [_run(ctx, batch) for _ in range(3)]
        assert any(g[0][0]["status"] == TIMEOUT for g in got)
        assert all(_same(g[1], want[1]) for g in got)
    finally:
        ctx.set_wait_limit(0)
        ctx.set_launch_config(0, 0)
