"""Polylines given as Python numbers that their types cannot hold are refused (no GPU: before
anything is sent to the device)."""
import pytest


@pytest.mark.parametrize("last", [2 ** 31, 2 ** 32 + 2, -2 ** 31 - 1])
def test_offsets_beyond_32_bits(last):
    import torch

    import paper_1611_05319_gb300 as gf
    ctx = gf.Context.__new__(gf.Context)
    ctx.device = 0
    with pytest.raises(RuntimeError, match="overflow"):
        ctx.guidance(torch.zeros((4, 4), dtype=torch.uint8), [0, last], [[0.0, 0.0], [1.0, 1.0]])
