"""Several clusters on one frame: clusters of 1 CTA (16 or 12 warps) make teams on
small frames, growing at the start, shrinking as the front does and leaving one
cluster at the end.  Which warp processes a tile changes no value, so every output
has to equal, bit for bit, that of one cluster of 16 CTAs (no team)."""
import numpy as np
import pytest

from synth import annulus_mask, const_guide, labels_from, polygon_image, random_guide, rect_mask
import _gpu

pytestmark = pytest.mark.gpu

H, W = 137, 211


def _frames():
    big = rect_mask(H, W, 9, 7, 190, 120)
    blobs = _gpu.hole_blobs(H, W, 5, n=24, rmin=3, rmax=11)
    ring = annulus_mask(H, W, 20.0, 60.0)
    walls = np.zeros((H, W), bool)
    walls[40:60, 30:180] = True
    shut = walls.copy()
    shut[42:58, 32:178] = False  # a region that the front never reaches: hole inside a wall of bystanders
    band = rect_mask(H, W, 0, 50, W, 24)  # across the image: the stall rule
    return dict(big=labels_from(big), blobs=labels_from(blobs), ring=labels_from(ring),
                shut=labels_from((blobs | walls) & ~shut, shut), band=labels_from(band))


def _run(ctx, frames, guides, rgbas, **kw):
    import torch
    rs = ctx.fill_batched(rgbas, frames, guides, enter=True, stall=True, **kw)
    torch.cuda.synchronize()
    out = []
    for r in rs:
        st = r.stats()
        words = (st["shells"] + 31) // 32
        out.append((r.rgba.cpu().numpy(), r.shell.cpu().numpy(), r.enter.cpu().numpy(),
                    r.stall.cpu().numpy()[:words], st))
    return out


@pytest.mark.parametrize("cs", [1, 2, 4, 16])
@pytest.mark.parametrize("kw", [dict(), dict(eps=4.0), dict(eps=5.5), dict(ghost=False), dict(smart=False),
                                dict(rescan=True), dict(data_term=True), dict(max_shells=3)],
                         ids=["eps3", "eps4", "eps5.5", "lattice", "onion", "rescan", "data", "max_shells"])
def test_teams_change_no_result(cuda_device, cs, kw):
    import torch

    import paper_1611_05319_gb300 as gf
    ctx = gf.context(0)
    fr = _frames()
    labels = [torch.from_numpy(v).cuda() for v in fr.values()]
    rgbas = [torch.from_numpy(_gpu.rgba(polygon_image(H, W, 9, 3 + i))).cuda() for i in range(len(labels))]
    guides = [torch.from_numpy(random_guide(H, W, 7 + i) if i % 2 else const_guide(H, W, 0.0 if i == 4 else 31.0)).cuda()
              for i in range(len(labels))]
    try:
        for n in (1, 2, 5):
            pick = [(i * 3 + 4) % 5 for i in range(n)]
            args = ([labels[i] for i in pick], [guides[i] for i in pick], [rgbas[i] for i in pick])
            ctx.set_launch_config(16, 1)
            want = _run(ctx, *args, **kw)
            ctx.set_launch_config(cs, 0)
            got = _run(ctx, *args, **kw)
            if cs == 1:
                assert ctx.last_launch()[1] > n
            for a, b in zip(want, got):
                for x, y in zip(a[:4], b[:4]):
                    assert np.array_equal(x, y, equal_nan=x.dtype.kind == "f")
                assert a[4] == b[4]
    finally:
        ctx.set_launch_config(0, 0)


def test_more_frames_than_clusters_help_at_the_end(cuda_device):
    """The queue runs dry while frames are still being filled: the clusters without a
    frame join them."""
    import torch

    import paper_1611_05319_gb300 as gf
    ctx = gf.context(0)
    fr = list(_frames().values())
    rng = np.random.default_rng(2)
    labels, rgbas, guides = [], [], []
    for i in range(9):
        labels.append(torch.from_numpy(fr[i % 5]).cuda())
        rgbas.append(torch.from_numpy(_gpu.rgba(polygon_image(H, W, 9, int(rng.integers(99))))).cuda())
        guides.append(torch.from_numpy(random_guide(H, W, i)).cuda())
    try:
        ctx.set_launch_config(16, 1)
        want = _run(ctx, labels, guides, rgbas)
        ctx.set_launch_config(1, 4)
        got = _run(ctx, labels, guides, rgbas)
    finally:
        ctx.set_launch_config(0, 0)
    for a, b in zip(want, got):
        for x, y in zip(a[:4], b[:4]):
            assert np.array_equal(x, y, equal_nan=x.dtype.kind == "f")
        assert a[4] == b[4]
