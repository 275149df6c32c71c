"""The preparation's ranges on the host: the words of the stall bitmap that the strips
of a frame clear are every word once and no other, up to the largest frames accepted.  On the GPU the bitmap of ordinary frames, narrow ones among them."""
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include "%s/paper_1611_05319_gb300/csrc/gf_internal.cuh"
int main()
{
    const long long most = (1ll << 31) - 64;
    const long long sizes[][2] = {{1, 1}, {8, 256}, {8, 257}, {9, 256}, {16, 512}, {1080, 1920}, {4097, 4097}, {1, most},
                                  {most, 1}, {most / 2, 2}, {most / 3, 3}, {most / 7, 7}, {most / 9, 9}, {1ll << 28, 7},
                                  {(1ll << 28) + 8, 5}, {46340, 46340}};
    for (auto &s : sizes) {
        const long long H = s[0], W = s[1], px = H * W, words = (px + 1 + 31) / 32;
        const int TH = (int)((H + 7) / 8), units = TH * (int)(((W + 7) / 8 + 31) / 32);
        long long next = 0;
        for (int u = 0; u < units; u++) {
            const gf::WordRange r = gf::stall_words(px, u, units);
            // empty, or the words that follow the strips before
            if (r.begin < 0 || r.end > words || r.end < r.begin || (r.begin < r.end && r.begin != next)) {
                printf("%%lld x %%lld: strip %%d clears %%d .. %%d\n", H, W, u, r.begin, r.end);
                return 1;
            }
            if (r.begin < r.end) next = r.end;
        }
        if (next != words) {
            printf("%%lld x %%lld: %%lld of %%lld words\n", H, W, next, words);
            return 1;
        }
    }
    return 0;
}
"""


def test_stall_words_once_each(tmp_path):
    from paper_1611_05319_gb300 import build
    src, exe = tmp_path / "ranges.cu", tmp_path / "ranges"
    src.write_text(SRC % ROOT)
    subprocess.run([build._nvcc(), "-O2", "-std=c++17", str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.gpu
@pytest.mark.parametrize("h,w", [(4099, 1), (2050, 3), (1031, 7), (4096, 8), (64, 2048), (3, 1)])
def test_stall_bitmap_cleared(cuda_device, h, w):
    """Every word of the caller's bitmap, whatever it held, on narrow frames too."""
    import torch

    import _gpu
    import paper_1611_05319_gb300 as gf
    from paper_1611_05319_gb300 import _lib
    from synth import const_guide, labels_from, polygon_image
    hole = np.zeros((h, w), bool)
    hole[h // 3:max(h // 3 + 1, h - h // 3)] = True
    img, g = polygon_image(h, w, 3, 1), const_guide(h, w, 90.0)
    o = _gpu.oracle_fill(img, labels_from(hole), g, c=0.6)
    ctx = gf.context(0)
    # the frame's descriptor with a bitmap that is all ones, between two guard words
    room = torch.full(((h * w + 32) // 32 + 2,), -1, dtype=torch.int32, device="cuda")
    fr, out, shell, _, _, keep = ctx._frame(torch.from_numpy(_gpu.rgba(img)).cuda(), torch.from_numpy(labels_from(hole)).cuda(),
                                            torch.from_numpy(g).cuda(), None, False, False)
    fr.out_stall = room.data_ptr() + 4
    stats = torch.empty((_lib.STATS_BYTES,), dtype=torch.uint8, device="cuda")
    ctx.fill_frames((_lib.Frame * 1)(fr), stats, _lib.make_params(c=0.6))
    room = room.cpu().numpy()
    assert room[0] == -1 and room[-1] == -1
    assert np.array_equal(shell.cpu().numpy(), o["shell"])
    bits = np.unpackbits(room[1:-1].view(np.uint8), bitorder="little")
    want = np.zeros_like(bits)
    want[:len(o["stall_steps"])] = o["stall_steps"][:len(bits)]
    assert np.array_equal(bits, want)
