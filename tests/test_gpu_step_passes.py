"""Steps of more than one pass (the data term switched off inside a step, the stall rule,
both in one step) and the count of guided pixels that switches the data term off, on
clusters of every kind: every thread of every cluster has to take the same way, so
repeated runs equal the oracle on each."""
import numpy as np
import pytest

from synth import labels_from, polygon_image, random_guide

import _gpu

pytestmark = pytest.mark.gpu

H, W = 61, 83


def _scene(seed, guided):
    hole = _gpu.hole_blobs(H, W, seed, n=10, rmin=1, rmax=8)
    known = np.zeros((H, W), bool)
    known[:, W - 9:] = True
    labels = labels_from(hole, known & ~hole)
    g = random_guide(H, W, seed)
    if guided == "patches":  # guided pixels are left when none of them is ready
        m = np.kron(np.random.default_rng(seed + 100).uniform(size=(H // 8 + 1, W // 8 + 1)) < 0.5, np.ones((8, 8)))
        g = g * m[:H, :W, None].astype(np.float32)
    else:  # within 3 px of the known pixels only: in onion order they run out after some steps
        k = np.pad(labels == 0, 3)
        near = sum(k[3 + dy:H + 3 + dy, 3 + dx:W + 3 + dx] for dy in range(-3, 4) for dx in range(-3, 4)) > 0
        g = random_guide(H, W, seed, zero_fraction=0.0) * near[..., None].astype(np.float32)
    return polygon_image(H, W, 7, seed), labels, g


SCENES = [(0, "patches", dict(c=0.6), 0), (4, "patches", dict(c=0.6), 0), (11, "patches", dict(c=0.3, mu=10.0), 4),
          (2, "rim", dict(smart=False), 6), (10, "rim", dict(smart=False), 4)]


@pytest.fixture(scope="module")
def cases():
    out = []
    for seed, guided, kw, switch in SCENES:
        img, labels, g = _scene(seed, guided)
        out.append((img, labels, g, kw, _gpu.oracle_fill(img, labels, g, data_term=True, **kw)))
        guided_left = (labels == 1) & (g != 0).any(-1) & ((out[-1][4]["shell"] >= switch) | (out[-1][4]["shell"] < 0))
        assert out[-1][4]["stats"]["data_switch"] == switch and guided_left.any() == (guided == "patches")
    assert all(o[4]["stall_steps"][0] for o in out[:2])  # three passes in step 0
    return out


@pytest.mark.parametrize("cs", [1, 2, 8, 16])
@pytest.mark.parametrize("rescan", [False, True])
def test_every_thread_goes_the_same_way(cuda_device, cases, cs, rescan):
    import paper_1611_05319_gb300 as gf
    ctx = gf.context(0)
    try:
        ctx.set_launch_config(cs, 0)
        for img, labels, g, kw, o in cases:
            for _ in range(6):
                _gpu.assert_parity(o, _gpu.gpu_fill(img, labels, g, data_term=True, rescan=rescan, **kw), labels)
    finally:
        ctx.set_launch_config(0, 0)
