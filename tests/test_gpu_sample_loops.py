"""The sample loops of the fill against the oracle where their forms change: every ball
radius and window, a snap too narrow for the one-word readability test, every number of
front pixels per tile (lanes per pixel), weights that underflow, rotations that are not
one, colours that are not finite."""
import numpy as np
import pytest

from synth import const_guide, labels_from, polygon_image, random_guide

import _gpu

pytestmark = pytest.mark.gpu

H, W = 61, 83


def _scene(seed, byst=True):
    hole = _gpu.hole_blobs(H, W, seed, n=10, rmin=1, rmax=8)
    known = np.zeros((H, W), bool)
    if byst:
        known[:, W - 9:] = True
    return polygon_image(H, W, 7, seed), labels_from(hole, known & ~hole)


@pytest.mark.parametrize("eps", [1.0, 1.5, 2.9, 3.0, 3.7, 4.0, 5.0, 6.3, 7.0])
@pytest.mark.parametrize("kw", [dict(), dict(smart=False), dict(ghost=False), dict(ghost=False, smart=False),
                                dict(tau=0.0), dict(tau=0.0, smart=False)],
                         ids=["rotated", "rotated-onion", "lattice", "lattice-onion", "no-snap", "no-snap-onion"])
def test_every_ball(cuda_device, eps, kw):
    img, labels = _scene(int(eps * 10))
    for g in (random_guide(H, W, 3), const_guide(H, W, 90.0), const_guide(H, W, 30.0, 0.3)):
        kg = dict(kw)
        if "tau" in kg:
            kg["snap_tau"] = kg.pop("tau")
        o = _gpu.oracle_fill(img, labels, g, eps=eps, **kw)
        _gpu.assert_parity(o, _gpu.gpu_fill(img, labels, g, eps=eps, **kg), labels)


@pytest.mark.parametrize("width", [80, 84, 85, 96])
@pytest.mark.parametrize("eps", [3.0, 4.0, 5.0, 7.0])
def test_windows_at_every_width(cuda_device, width, eps):
    """16-byte and plain loads of the state window, tiles cut by the right border."""
    hole = _gpu.hole_blobs(H, width, 12, n=14, rmin=1, rmax=7, margin=4)
    img, g = polygon_image(H, width, 7, 2), random_guide(H, width, 6)
    for kw in (dict(), dict(ghost=False)):
        o = _gpu.oracle_fill(img, labels_from(hole), g, eps=eps, **kw)
        _gpu.assert_parity(o, _gpu.gpu_fill(img, labels_from(hole), g, eps=eps, **kw), labels_from(hole))


@pytest.mark.parametrize("n", list(range(1, 18)) + [23, 32, 33, 48, 64])
def test_front_pixels_per_tile(cuda_device, n):
    """n isolated hole pixels or short rows of them in one 8x8 tile."""
    rng = np.random.default_rng(n)
    hole = np.zeros((24, 24), bool)
    hole[8:16, 8:16].flat[rng.permutation(64)[:n]] = True
    img = polygon_image(24, 24, 4, n)
    g = random_guide(24, 24, n)
    for kw in (dict(), dict(eps=5.0), dict(ghost=False)):
        o = _gpu.oracle_fill(img, labels_from(hole), g, **kw)
        _gpu.assert_parity(o, _gpu.gpu_fill(img, labels_from(hole), g, **kw), labels_from(hole))


@pytest.mark.parametrize("kw", [dict(smart=False), dict(ghost=False, smart=False), dict(ghost=False), dict()],
                         ids=["rotated-onion", "lattice-onion", "lattice", "rotated"])
@pytest.mark.parametrize("mu,eps", [(400.0, 3.0), (3000.0, 1.5)])
def test_weights_that_underflow(cuda_device, kw, mu, eps):
    img, labels = _scene(4)
    for g in (const_guide(H, W, 37.0), random_guide(H, W, 8)):
        o = _gpu.oracle_fill(img, labels, g, eps=eps, mu=mu, **kw)
        _gpu.assert_parity(o, _gpu.gpu_fill(img, labels, g, eps=eps, mu=mu, **kw), labels)


def test_guides_of_a_few_denormals(cuda_device):
    """g^2 rounds to a few units of the smallest denormal: g/|g| is off by tens of per
    cent and the rotated offsets may leave the ball's square."""
    img, labels = _scene(6)
    g = random_guide(H, W, 5, zero_fraction=0.0)
    g = (g / np.linalg.norm(g, axis=-1, keepdims=True) * 2.9e-23).astype(np.float32)
    for kw in (dict(), dict(smart=False), dict(eps=4.0), dict(eps=5.0)):
        o = _gpu.oracle_fill(img, labels, g, **kw)
        _gpu.assert_parity(o, _gpu.gpu_fill(img, labels, g, **kw), labels)


def test_rotations_longer_than_one(cuda_device):
    """Both components of g square to 1.49 units of the smallest denormal, which rounds to
    one: (g/|g|)^2 sums to 1.49, and the sample (2, -2) lands 3.45 px away."""
    img, labels = _scene(6)
    v = np.float32(np.sqrt(1.49 * 2.0 ** -149))
    rng = np.random.default_rng(3)
    g = (rng.choice([-1.0, 1.0], (H, W, 2)) * v).astype(np.float32)
    for kw in (dict(), dict(smart=False), dict(eps=2.9), dict(eps=4.0), dict(eps=5.0)):
        o = _gpu.oracle_fill(img, labels, g, **kw)
        _gpu.assert_parity(o, _gpu.gpu_fill(img, labels, g, **kw), labels)


def test_colours_that_are_not_finite(cuda_device):
    """A tap of zero weight is not read: an infinite known colour spreads to the pixels
    whose samples use it, with its sign, and to no other."""
    img, labels = _scene(9, byst=False)
    rng = np.random.default_rng(1)
    rgba = _gpu.rgba(img)
    known = np.argwhere(labels == 0)
    for y, x in known[rng.permutation(len(known))[:40]]:
        rgba[y, x, 1] = np.inf
    for g in (const_guide(H, W, 0.0), random_guide(H, W, 2)):
        o = _gpu.oracle_fill(rgba, labels, g, mu=1.0)  # no weight underflows to 0 in FP32
        r = _gpu.gpu_fill(rgba, labels, g, mu=1.0)
        assert np.array_equal(o["shell"], r["shell"])
        filled = o["shell"] >= 0
        a, b = o["u"][filled], r["u"][filled]
        assert np.isinf(a).any() and np.array_equal(np.isposinf(a), np.isposinf(b))
        fine = np.isfinite(a)
        assert np.abs(a[fine] - b[fine]).max() <= _gpu.COLOUR_ATOL
