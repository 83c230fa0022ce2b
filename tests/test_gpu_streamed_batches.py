"""Decode batches on the streamed kernel where its tiling has edges: several modules in one launch (each with its own aux
CTAs and row tiles, a last row tile that is not full, more CTAs than tokens), and batches of 129 to 256 tokens, against the CPU oracle."""
import pytest
import torch

from paper_2405_13053_b200 import binding as mb
from paper_2405_13053_b200 import workloads
from .test_gpu_group import check_group, make_group

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d_in,d_outs,k", [(1, 512, (384, 128, 128), 2),        # fewer tokens than aux CTAs
                                             (3, 2048, (1032, 264), 4),           # ragged last row tiles
                                             (64, 1024, (512, 512, 512, 512), 1),
                                             (65, 1024, (136, 2048), 2),
                                             (128, 512, (1536, 256, 256), 2),
                                             (129, 2048, (1024, 256), 2),         # one token above 128
                                             (256, 2048, (1024, 264), 2),
                                             (129, 2048, (1032,), 4),
                                             (200, 2048, (2048,), 2),
                                             (256, 1088, (1288,), 1)])
def test_streamed_batches(T, d_in, d_outs, k):
    if len(d_outs) > 1:
        assert mb.meteora_group_plan(T, d_in, list(d_outs), 28, 8, k, torch.bfloat16) == 1
    else:
        assert "path=stream_decode" in mb.meteora_describe_plan(mb.make_shape(T, d_in, d_outs[0], 28, 8, k, torch.bfloat16))
    check_group(make_group(T, d_in, d_outs, seed=9100 + T, k=k), 1e-2)


@pytest.mark.parametrize("T,d_in,d_outs,N,r", [(48, 2048, (9216,), 28, 8),           # the first batch that leaves the streamed kernel
                                               (201, 2048, (7432,), 28, 8),          # ragged row pairs and tokens
                                               (256, 2048, (6144,), 28, 8),
                                               (96, 2120, (8456,), 12, 16),          # rank 16, a last k-step that is not full
                                               (112, 2048, (4096, 4360), 28, 8),     # two modules' token tiles side by side
                                               (256, 2048, (3072, 1544, 1544), 8, 8)])
def test_wide_batches_behind_token_tiles(T, d_in, d_outs, N, r):
    shape = mb.make_shape(T, d_in, d_outs[0], N, r, 2, torch.bfloat16)
    if len(d_outs) == 1:
        assert "launches=2" in mb.meteora_describe_plan(shape) and "persistent_pairs=" in mb.meteora_describe_plan(shape)
        w = workloads.make_workload("wide", T=T, d_in=d_in, d_out=d_outs[0], N=N, r=r, k=2, dtype="bf16", x_kind="rms", seed=9300 + T, b_std=0.3)
        check_group([w], 1e-2)
    else:
        assert mb.meteora_group_plan(T, d_in, list(d_outs), N, r, 2, torch.bfloat16) == 1
        check_group(make_group(T, d_in, d_outs, seed=9300 + T, N=N), 1e-2)


@pytest.mark.parametrize("T,d_in,d_out,N,r", [(257, 1024, 2560, 28, 8),       # two token tiles of 160, the second a short one
                                              (700, 520, 1800, 28, 8),        # a last k-step and a last row pair that are not full
                                              (1280, 512, 4096, 28, 8),       # a few tiles more than pairs
                                              (300, 512, 1024, 28, 32)])      # 8 tiles, rank 32
def test_short_prefill_walks_behind_its_routing(T, d_in, d_out, N, r):
    plan = mb.meteora_describe_plan(mb.make_shape(T, d_in, d_out, N, r, 2, torch.bfloat16))
    assert "path=chain" in plan and "persistent_pairs=" in plan, plan
    check_group([workloads.make_workload("short", T=T, d_in=d_in, d_out=d_out, N=N, r=r, k=2, dtype="bf16", x_kind="rms",
                                         seed=9500 + T, b_std=0.3)], 1e-2)
