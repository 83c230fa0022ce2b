"""An allocation of TMEM columns waits without a limit: CTAs that one SM's shared memory (228 KB, 1 KB of it beside each CTA's own)
admits may not want more than its 512 columns together, whatever launches and streams they are of."""
import pytest
import torch

from paper_2405_13053_b200 import binding as mb


def check(T, d_in, d_out, N, r):
    text = mb.meteora_describe_plan(mb.make_shape(T, d_in, d_out, N, r, 2, torch.bfloat16))
    fields = dict(f.split("=") for f in text.split() if "=" in f)
    cols = 512                                               # the persistent walk: two accumulators of 256
    if "persistent_pairs" not in fields:
        tokens = int(fields["tile_tokens"]) if "tile_tokens" in fields else int(fields["tile"].split("x")[1])
        cols = max(32, 1 << (tokens - 1).bit_length())
    assert (int(fields["smem"]) + 1024) * (512 + 32) > 228 * 1024 * cols, text


@pytest.mark.parametrize("shape", [(1, 64, 128, 28, 8), (120, 64, 128, 4, 8), (250, 64, 64, 2, 8), (300, 64, 256, 28, 8), (300, 40, 256, 28, 24),
                                   (700, 128, 512, 4, 8), (128, 4096, 4096, 28, 8), (2048, 4096, 14336, 28, 8)])
def test_plans_without_a_device(shape):
    check(*shape)


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(64, 4096, 14336, 28, 8), (512, 4096, 1024, 28, 8), (300, 64, 256, 28, 8), (2048, 4096, 4096, 28, 8), (2048, 4096, 4096, 28, 32),
                                   (1, 64, 128, 28, 8), (200, 64, 64, 2, 8), (300, 40, 256, 28, 24)])
def test_plans_on_the_device(shape):
    check(*shape)
