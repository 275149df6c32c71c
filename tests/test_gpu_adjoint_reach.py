"""The reverse sweep against the oracle's where its forms change: the reach of the row
words (eps, a snap too narrow for it), weights that underflow, rotations that are not
one, steps of every size, more frames than clusters, stall steps, frame borders."""
import numpy as np
import pytest

import oracle
from synth import const_guide, labels_from, polygon_image, random_guide

import _gpu

pytestmark = pytest.mark.gpu


def _check(img, labels, guide, seed, eps=3.0, mu=10.0, tau=1e-5, smart=True, n=1):
    import torch

    import paper_1611_05319_gb300 as gf
    ctx = gf.context(0)
    rgba = _gpu.rgba(img)
    o = oracle.fill(rgba, labels, guide, eps=eps, mu=mu, tau=tau, smart=smart)
    up = np.random.default_rng(seed).normal(size=rgba.shape).astype(np.float32)
    gi, gphi, gmu = oracle.fill_backward(o["u"], labels, guide, o["shell"], o["stall_steps"], up, eps=eps, mu=mu, tau=tau)
    args = [[torch.from_numpy(v).cuda() for _ in range(n)] for v in (rgba, labels, guide)]
    rs = ctx.fill_batched(*args, eps=eps, mu=mu, snap_tau=tau, smart=smart, stall=True)
    bi, bphi, bmu = ctx.fill_backward(rs, args[2], [torch.from_numpy(up).cuda()] * n, eps=eps, mu=mu, smart=smart,
                                      snap_tau=tau)
    torch.cuda.synchronize()
    # every term is a product of weights of at most 1 with |up| of a few units, summed over
    # a chain of steps in FP32; the same bounds as the adjoint's other tests
    top = np.abs(gphi).max()
    for i in range(n):
        assert np.array_equal(rs[i].shell.cpu().numpy(), o["shell"])
        assert np.abs(bi[i].cpu().numpy() - gi).max() <= 1e-4 * max(1.0, np.abs(gi).max())
        err = np.abs(bphi[i].cpu().numpy() - gphi)
        assert (err <= 1e-3 * np.maximum(np.abs(gphi), 1e-2 * top)).all() or top == 0.0
        assert abs(float(bmu[i]) - gmu) <= 1e-3 * max(abs(gmu), 1e-6) + 1e-6


H, W = 47, 66


@pytest.mark.parametrize("eps,tau", [(1.0, 1e-5), (2.0, 1e-5), (3.0, 1e-5), (3.0, 0.0), (3.5, 1e-5), (4.0, 0.0),
                                     (5.0, 1e-5), (7.0, 1e-5), (7.0, 0.0)])
def test_reach(cuda_device, eps, tau):
    hole = _gpu.hole_blobs(H, W, int(eps * 3), n=8, rmin=1, rmax=6, margin=3)  # some cross the border
    byst = np.zeros((H, W), bool)
    byst[:, W - 5:] = True
    img = polygon_image(H, W, 6, 5)
    for i, g in enumerate((random_guide(H, W, 4), const_guide(H, W, 90.0))):
        _check(img, labels_from(hole, byst & ~hole), g, i, eps=eps, tau=tau)


def test_stall_steps_and_small_steps(cuda_device):
    hole = np.zeros((H, W), bool)
    hole[10:31, :] = True  # a band across the image, guidance along it
    _check(polygon_image(H, W, 6, 2), labels_from(hole), const_guide(H, W, 0.0), 1)
    hole[:] = False
    hole[20, 5:60] = True
    hole[20:27, 30] = True
    _check(polygon_image(H, W, 6, 3), labels_from(hole), random_guide(H, W, 8), 2)


def test_weights_that_underflow(cuda_device):
    # without the ready test every front pixel is filled, readable m = 0 samples or not
    hole = _gpu.hole_blobs(H, W, 3, n=6, rmin=2, rmax=7)
    _check(polygon_image(H, W, 6, 4), labels_from(hole), const_guide(H, W, 37.0), 5, mu=400.0, smart=False)


@pytest.mark.parametrize("units", [0.6, 1.49])
def test_guides_of_a_few_denormals(cuda_device, units):
    """g^2 of about one unit of the smallest denormal: g/|g| is no rotation (its length is
    off by tens of per cent), which the reverse sweep has to share with the fill.  With the
    schedule fixed the fill is linear in the known colours: <up, fill(u + v) - fill(u)> =
    <grad, v>.  Both sides are FP32 averages of O(1) values over a chain of under 16 steps,
    a few units of 2^-24 each."""
    import torch

    import paper_1611_05319_gb300 as gf
    ctx = gf.context(0)
    hole = _gpu.hole_blobs(H, W, 6, n=6, rmin=2, rmax=7)
    rng = np.random.default_rng(5)
    g = (rng.choice([-1.0, 1.0], (H, W, 2)) * np.float32(np.sqrt(units * 2.0 ** -149))).astype(np.float32)
    u, v = (rng.uniform(0.0, 1.0, (H, W, 4)).astype(np.float32) for _ in "uv")
    up = rng.normal(size=(H, W, 4)).astype(np.float32)
    lab, gd = torch.from_numpy(labels_from(hole)).cuda(), torch.from_numpy(g).cuda()
    out = []
    for w in (u, u + v):
        rs = ctx.fill_batched([torch.from_numpy(w).cuda()], [lab], [gd], mu=10.0, stall=True)
        out.append(rs[0].rgba.cpu().numpy().astype(np.float64))
        assert rs[0].stats()["shells"] < 16
    grad = ctx.fill_backward(rs, [gd], [torch.from_numpy(up).cuda()], mu=10.0)[0][0].cpu().numpy().astype(np.float64)
    step = (u + v).astype(np.float64) - u
    lhs, rhs = float((up * (out[1] - out[0])).sum()), float((grad * step).sum())
    assert abs(lhs - rhs) <= 16 * 8 * 2.0 ** -24 * float(np.abs(up).sum())


@pytest.mark.parametrize("n", [2, 20])
def test_batches(cuda_device, n):
    hole = _gpu.hole_blobs(H, W, 9, n=7, rmin=2, rmax=8)
    _check(polygon_image(H, W, 6, 4), labels_from(hole), random_guide(H, W, 7), 6, n=n)
