"""The prefill base product on persistent pairs of SMs at the edges of its tiles, against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2405_13053_b200 import binding as mb
from paper_2405_13053_b200 import workloads
from .gpu_util import bf16_bound_ok, check_selection, rel_l2, to_dev
from .test_gpu_group import check_group, make_group

pytestmark = pytest.mark.gpu


# Tile widths 160 / 192 / 224 / 256 (257, 380, 1300, 1281 tokens), a last token tile with few tokens, odd numbers of row tiles and
# a ragged last one, axes of 5 k-steps and of no whole number, several adapters per block of expand columns (ranks 16 - 64), an
# odd number of blocks (33), fewer tiles than pairs, less and more than two rounds, whole rounds.
# With the routing in the walk (persist 2) and from kernels of its own (3: from 37 pair tiles on); 56 adapters: three pairs
# of stacked tiles, two lanes per token.
@pytest.mark.parametrize("persist,T,d_in,d_out,N,r,k", [(p, *c) for p in (2, 3) for c in [
    (257, 4096, 200, 28, 8, 2), (380, 2048, 384, 28, 8, 2), (512, 8192, 1024, 28, 8, 2), (700, 520, 2184, 28, 16, 2),
    (1281, 520, 2184, 28, 8, 2), (1300, 1024, 4096, 33, 8, 4), (1201, 1536, 5120, 5, 32, 2), (2560, 512, 2048, 28, 64, 2),
    (5000, 320, 2560, 28, 16, 2), (2400, 256, 1024, 100, 8, 2), (300, 320, 9472, 28, 8, 1), (1024, 640, 9472, 28, 8, 2),
    (600, 256, 3200, 56, 8, 2), (900, 512, 3200, 32, 8, 8),
] if p == 2 or (c[0] + 255) // 256 * ((c[2] + 255) // 256) > 37])
def test_persistent_pairs_match_oracle(persist, T, d_in, d_out, N, r, k):
    w = workloads.make_workload("persist", T=T, d_in=d_in, d_out=d_out, N=N, r=r, k=k, dtype="bf16", seed=90 + T, b_std=0.3)
    t = to_dev(w, "x", "W0", "A", "B", "Wg")
    mb.meteora_set_tuning("persist", persist)
    try:
        shape = mb.make_shape(T, d_in, d_out, N, r, k, torch.bfloat16)
        plan = mb.meteora_describe_plan(shape)
        whole = persist == 2 and N * (r + 1) <= 512 and N <= 64
        assert ("path=persistent_prefill" if whole else "path=chain") in plan and "persistent_pairs" in plan, plan
        ws = mb.alloc_workspace(shape)
        y, idx, _ = mb.meteora_linear_forward(*t, k, workspace=ws, return_routing=True)
        y, idx = y.float().cpu().numpy(), idx.cpu().numpy()
        assert mb.meteora_workspace_status(ws) == 0
        for _ in range(3):                               # sums in the same order, whatever the workspace holds
            again = mb.meteora_linear_forward(*t, k, workspace=ws)
        np.testing.assert_array_equal(y, again.float().cpu().numpy())
        assert mb.meteora_workspace_status(ws) == 0
    finally:
        mb.meteora_set_tuning("persist", 1)
    o_idx, _, o_logits = oracle.gate_topk(w["x"], w["Wg"], k)
    check_selection(idx, o_idx, o_logits, k)
    sel = np.unique(np.concatenate([np.arange(0, T, 61), np.arange(159, T, 160), np.arange(255, T, 256), [T - 1]]))
    ref = oracle.linear_forward_routed(w["x"][sel], w["W0"], w["A"], w["B"], w["Wg"], idx[sel])
    assert rel_l2(y[sel], ref) <= 5e-3
    assert bf16_bound_ok(y[sel], ref) <= 0.0


@pytest.mark.parametrize("T,d_in,d_outs", [(2100, 512, (2048, 512, 520)), (700, 1024, (4096, 4096)), (1500, 320, (256, 3000, 128, 2048))])
def test_a_prefill_group_is_one_walk(T, d_in, d_outs):
    ws_list = [workloads.make_workload("walk", T=T, d_in=d_in, d_out=d, dtype="bf16", seed=70, b_std=0.3) for d in d_outs]
    for m, w in enumerate(ws_list):                      # one x, weights of their own
        other = workloads.make_workload("walk", T=1, d_in=d_in, d_out=d_outs[m], dtype="bf16", seed=71 + m, b_std=0.3)
        w.tensors.update({n: other[n] for n in ("W0", "A", "B", "Wg")})
    x = to_dev(ws_list[0], "x")[0]
    dev = [to_dev(w, "W0", "A", "B", "Wg") for w in ws_list]
    assert mb.meteora_group_plan(T, d_in, list(d_outs), 28, 8, 2, torch.bfloat16) == 1
    W0s, As, Bs, Wgs = (list(t) for t in zip(*dev))
    ys, routing = mb.meteora_linear_forward_group(x, W0s, As, Bs, Wgs, 2, return_routing=True)
    ys2 = mb.meteora_linear_forward_group(x, W0s, As, Bs, Wgs, 2)
    sel = np.unique(np.concatenate([np.arange(0, T, 97), np.arange(255, T, 256), [T - 1]]))
    for w, y, y2, (idx, _) in zip(ws_list, ys, ys2, routing):
        assert torch.equal(y, y2)
        idx = idx.cpu().numpy()
        o_idx, _, o_logits = oracle.gate_topk(w["x"], w["Wg"], 2)
        check_selection(idx, o_idx, o_logits, 2)
        ref = oracle.linear_forward_routed(w["x"][sel], w["W0"], w["A"], w["B"], w["Wg"], idx[sel])
        assert rel_l2(y.float().cpu().numpy()[sel], ref) <= 5e-3


# Three and four tiles per pair with tiles of at most 64 tokens, which are one chunk of the epilogue: only one of its two groups has
# anything to read, and the accumulator's next tile waits for both.  Routing inside the walk (1 and 16 tokens, the groups) and ahead
# of it (17 on); 65 tokens are the first with more chunks than one.
@pytest.mark.parametrize("T,d_in,d_outs", [(1, 1024, (38664,)), (16, 2048, (38144,)), (17, 2048, (38664,)), (48, 2048, (38144,)),
                                           (64, 2048, (38664,)), (65, 2048, (38144,)), (13, 1024, (28672, 28680)), (64, 1024, (28680, 28672))])
def test_many_tiles_per_pair_of_one_chunk(T, d_in, d_outs):
    ws = make_group(T, d_in, d_outs, seed=9700 + T, N=12)
    if len(d_outs) == 1:
        shape = mb.make_shape(T, d_in, d_outs[0], 12, 8, 2, torch.bfloat16)
        assert "persistent_pairs=74 tiles=1" in mb.meteora_describe_plan(shape)
        t = to_dev(ws[0], "x", "W0", "A", "B", "Wg")
        workspace = mb.alloc_workspace(shape)
        mb.meteora_linear_forward(*t, 2, workspace=workspace)
        assert mb.meteora_workspace_status(workspace) == 0
    check_group(ws, 1e-2)


# The selection inside the walk: the sorted lists of 4 and of 8 (k up to 3 and 7), whole keys (k = 8, equal logits), one and two lanes
# per token, one to four pairs of stacked tiles (Wg in each), adapters of one 8-row block to 8; token counts of 5 to 8 chunks.
@pytest.mark.parametrize("T,d_in,d_out,N,r,k", [
    (300, 320, 9472, 28, 8, 1), (1250, 320, 2048, 28, 8, 3), (1250, 320, 2048, 28, 16, 4), (1250, 320, 2048, 9, 8, 7), (1250, 320, 2048, 8, 8, 8),
    (1250, 320, 2048, 28, 32, 2), (1100, 512, 2048, 12, 64, 2), (1250, 320, 2048, 64, 8, 3), (1100, 320, 2048, 33, 16, 8), (1250, 320, 2048, 48, 8, 5),
])
def test_selection_in_the_walk(T, d_in, d_out, N, r, k):
    w = workloads.make_workload("walk_pick", T=T, d_in=d_in, d_out=d_out, N=N, r=r, k=k, dtype="bf16", seed=190 + N + k, b_std=0.3)
    w["Wg"][N - 1] = w["Wg"][1]                          # two adapters that always tie
    w["x"][5] = 0.0                                      # a token whose logits all tie
    t = to_dev(w, "x", "W0", "A", "B", "Wg")
    mb.meteora_set_tuning("persist", 2)
    try:
        shape = mb.make_shape(T, d_in, d_out, N, r, k, torch.bfloat16)
        assert "path=persistent_prefill" in mb.meteora_describe_plan(shape)
        ws = mb.alloc_workspace(shape)
        y, idx, weight = mb.meteora_linear_forward(*t, k, workspace=ws, return_routing=True)
        again = mb.meteora_linear_forward(*t, k, workspace=ws)
        assert mb.meteora_workspace_status(ws) == 0
    finally:
        mb.meteora_set_tuning("persist", 1)
    assert torch.equal(y, again)
    y, idx, weight = y.float().cpu().numpy(), idx.cpu().numpy(), weight.cpu().numpy()
    o_idx, o_weight, o_logits = oracle.gate_topk(w["x"], w["Wg"], k)
    check_selection(idx, o_idx, o_logits, k)
    assert idx[5].tolist() == list(range(k))             # equal logits: the lower adapters, in order
    last = idx == N - 1
    tied = last.any(axis=1)
    assert (idx == 1).any(axis=1)[tied].all()            # never the higher one alone, nor ahead of the lower one
    assert (np.argmax(idx == 1, axis=1)[tied] < np.argmax(last, axis=1)[tied]).all()
    same = (idx == o_idx).all(axis=1)
    np.testing.assert_allclose(weight[same], o_weight[same], rtol=1e-4, atol=1e-5)
    sel = np.unique(np.concatenate([np.arange(0, T, 61), np.arange(255, T, 256), [5, T - 1]]))
    ref = oracle.linear_forward_routed(w["x"][sel], w["W0"], w["A"], w["B"], w["Wg"], idx[sel])
    assert rel_l2(y[sel], ref) <= 5e-3
    assert bf16_bound_ok(y[sel], ref) <= 0.0


# One token tile as wide as its tokens, in steps of 16: chunks of the epilogue that are whole, short and of one step; rows that end
# inside a tile and inside one of its halves of 64.
@pytest.mark.parametrize("T,d_out", [(49, 9216), (64, 9224), (72, 9288), (129, 9216), (200, 9408), (225, 9280), (240, 9352), (256, 9216)])
def test_single_token_tile(T, d_out):
    w = workloads.make_workload("one_tile", T=T, d_in=2048, d_out=d_out, dtype="bf16", seed=290 + T, b_std=0.3)
    t = to_dev(w, "x", "W0", "A", "B", "Wg")
    shape = mb.make_shape(T, 2048, d_out, 28, 8, 2, torch.bfloat16)
    assert f"tile=256x{(T + 15) // 16 * 16}" in mb.meteora_describe_plan(shape), mb.meteora_describe_plan(shape)
    ws = mb.alloc_workspace(shape)
    guard = torch.full((T + 64, d_out), 7.0, device="cuda", dtype=torch.bfloat16)
    y, idx, _ = mb.meteora_linear_forward(*t, 2, workspace=ws, return_routing=True, out=guard[:T])
    assert mb.meteora_workspace_status(ws) == 0
    assert (guard[T:] == 7.0).all()                      # nothing past the batch is written
    y, idx = y.float().cpu().numpy(), idx.cpu().numpy()
    o_idx, _, o_logits = oracle.gate_topk(w["x"], w["Wg"], 2)
    check_selection(idx, o_idx, o_logits, 2)
    sel = np.unique(np.concatenate([np.arange(0, T, 17), np.arange(15, T, 16), [T - 1]]))
    ref = oracle.linear_forward_routed(w["x"][sel], w["W0"], w["A"], w["B"], w["Wg"], idx[sel])
    assert rel_l2(y[sel], ref) <= 5e-3
    assert bf16_bound_ok(y[sel], ref) <= 0.0


# Decode batches of more than one round: tiles of fewer rows (8 to 56 less than 128 per CTA), ends inside and at the edge of a tile,
# adapters of one block and of two.
@pytest.mark.parametrize("T,d_in,d_outs,r", [(40, 2048, (14336, 14336), 8), (64, 2048, (11008, 11008), 8), (100, 2048, (13824, 13824), 8),
                                             (128, 2048, (19000, 504), 8), (33, 2048, (20480,), 8), (64, 2048, (25608,), 16), (90, 2048, (14336, 14344), 8)])
def test_tiles_of_fewer_rows(T, d_in, d_outs, r):
    ws = [workloads.make_workload(f"rows/{m}", T=T, d_in=d_in, d_out=d, N=12, r=r, k=2, dtype="bf16", seed=9800 + T + m, b_std=0.3)
          for m, d in enumerate(d_outs)]
    for w in ws[1:]:
        w.tensors["x"] = ws[0]["x"]
    if len(d_outs) == 1:
        t = to_dev(ws[0], "x", "W0", "A", "B", "Wg")
        guard = torch.full((T + 64, d_outs[0]), 7.0, device="cuda", dtype=torch.bfloat16)
        mb.meteora_linear_forward(*t, 2, out=guard[:T])
        assert (guard[T:] == 7.0).all()
    check_group(ws, 1e-2)


# Few tiles of a prefill batch on narrow ones: one and several token tiles per row pair, ragged last ones, an odd number of k-steps, rows
# that end inside a tile, us in one part and in three, adapters of 1, 2, 4 and 8 blocks.
@pytest.mark.parametrize("T,d_in,d_out,N,r,k,width", [
    (257, 320, 200, 28, 8, 2, 64), (300, 1088, 1024, 28, 8, 2, 64), (500, 2048, 1000, 28, 16, 4, 64), (700, 576, 2048, 12, 32, 2, 128),
    (1030, 1024, 1160, 28, 8, 1, 128), (2049, 512, 600, 28, 64, 2, 128), (290, 9024, 520, 28, 8, 2, 64), (1000, 320, 1928, 90, 8, 3, 128),
])
def test_few_tiles_are_narrow(T, d_in, d_out, N, r, k, width):
    w = workloads.make_workload("narrow", T=T, d_in=d_in, d_out=d_out, N=N, r=r, k=k, dtype="bf16", seed=390 + T, b_std=0.3)
    t = to_dev(w, "x", "W0", "A", "B", "Wg")
    shape = mb.make_shape(T, d_in, d_out, N, r, k, torch.bfloat16)
    tiles = (T + width - 1) // width
    assert f"tile=256x{((T + tiles - 1) // tiles + 31) // 32 * 32} " in mb.meteora_describe_plan(shape), mb.meteora_describe_plan(shape)
    ws = mb.alloc_workspace(shape)
    guard = torch.full((T + 128, d_out), 7.0, device="cuda", dtype=torch.bfloat16)
    y, idx, _ = mb.meteora_linear_forward(*t, k, workspace=ws, return_routing=True, out=guard[:T])
    assert mb.meteora_workspace_status(ws) == 0
    assert (guard[T:] == 7.0).all()
    y, idx = y.float().cpu().numpy(), idx.cpu().numpy()
    o_idx, _, o_logits = oracle.gate_topk(w["x"], w["Wg"], k)
    check_selection(idx, o_idx, o_logits, k)
    sel = np.unique(np.concatenate([np.arange(0, T, 31), np.arange(63, T, 64), [T - 1]]))
    ref = oracle.linear_forward_routed(w["x"][sel], w["W0"], w["A"], w["B"], w["Wg"], idx[sel])
    assert rel_l2(y[sel], ref) <= 5e-3
    assert bf16_bound_ok(y[sel], ref) <= 0.0


# Contraction axes of one iteration of the main loop (64 elements a step, two steps in the narrow walk), of a part of one, and of two
# and three: the expand may not come ahead of the step that clears the accumulator.  Narrow tiles of 64 and 128 tokens, 256-token tiles
# behind the routing kernels (us in one part and in three) and with the routing inside (knob 2).  W0 = 0 leaves the LoRA term alone, whose
# absence no tolerance can hide.
@pytest.mark.parametrize("T,d_in,d_out,N,r,k,persist", [
    (257, 64, 200, 28, 8, 2, 1), (300, 64, 256, 28, 8, 2, 1), (300, 128, 256, 28, 16, 2, 1), (300, 192, 256, 28, 8, 2, 1), (512, 128, 1024, 28, 8, 2, 1),
    (512, 64, 2048, 12, 64, 2, 1), (2048, 64, 1024, 28, 8, 2, 1), (600, 64, 256, 90, 8, 2, 1), (2048, 128, 520, 28, 64, 4, 1),
    (4096, 8, 1024, 28, 8, 2, 1), (4096, 56, 1024, 28, 16, 2, 1), (4096, 64, 1024, 28, 8, 2, 3), (4096, 72, 1024, 28, 8, 2, 1), (2048, 56, 768, 12, 64, 2, 1),
    (4096, 136, 1024, 28, 8, 2, 3), (512, 8, 2560, 100, 8, 2, 1), (4096, 64, 2048, 28, 8, 2, 2), (4096, 8, 2048, 28, 16, 2, 2), (4096, 72, 4096, 28, 8, 2, 2),
])
def test_short_contraction_axes_keep_the_lora_term(T, d_in, d_out, N, r, k, persist):
    w = workloads.make_workload("short_axis", T=T, d_in=d_in, d_out=d_out, N=N, r=r, k=k, dtype="bf16", seed=490 + T + d_in, b_std=0.3)
    x, W0, A, B, Wg = to_dev(w, "x", "W0", "A", "B", "Wg")
    mb.meteora_set_tuning("persist", persist)
    try:
        shape = mb.make_shape(T, d_in, d_out, N, r, k, torch.bfloat16)
        plan = mb.meteora_describe_plan(shape)
        assert "persistent_pairs=" in plan and ("path=persistent_prefill" in plan) == (persist == 2), plan
        ws = mb.alloc_workspace(shape)
        y, idx, _ = mb.meteora_linear_forward(x, W0, A, B, Wg, k, workspace=ws, return_routing=True)
        lora = mb.meteora_linear_forward(x, torch.zeros_like(W0), A, B, Wg, k, workspace=ws)
        assert mb.meteora_workspace_status(ws) == 0
    finally:
        mb.meteora_set_tuning("persist", 1)
    y, lora, idx = y.float().cpu().numpy(), lora.float().cpu().numpy(), idx.cpu().numpy()
    o_idx, _, o_logits = oracle.gate_topk(w["x"], w["Wg"], k)
    check_selection(idx, o_idx, o_logits, k)
    sel = np.unique(np.concatenate([np.arange(0, T, 61), np.arange(255, T, 256), [T - 1]]))
    ref = oracle.linear_forward_routed(w["x"][sel], w["W0"], w["A"], w["B"], w["Wg"], idx[sel])
    assert rel_l2(y[sel], ref) <= 5e-3
    ref = oracle.linear_forward_routed(w["x"][sel], 0 * w["W0"], w["A"], w["B"], w["Wg"], idx[sel])
    assert rel_l2(lora[sel], ref) <= 5e-3                # (us and y rounded to bf16 once each: 2 x 1.7e-3)


# The fp32 sums behind a bf16 y, made visible: equal tokens whose last four columns cancel the sum of the others (each weight the bf16 part
# that the ones before leave), so that y is the error.  The tensor cores cut off what they add: 2.1e-6 of the sum's size (rms) over 4096
# products in two accumulators, 4.4e-6 in one, with the expand of rank 16 in three parts as without one; in two over 14336 7.8e-6.
@pytest.mark.parametrize("T,d_in,d_out,r,b_std,limit", [(512, 4096, 1024, 8, 0.0, 3e-6), (700, 4096, 1024, 8, 0.0, 3e-6), (512, 4096, 1024, 16, 0.05, 3e-6),
                                                        (300, 4096, 1024, 64, 0.05, 3e-6), (512, 14336, 1024, 8, 0.0, 1.1e-5), (64, 4096, 14336, 8, 0.0, 3e-6)])
def test_narrow_tiles_sum_into_two_accumulators(T, d_in, d_out, r, b_std, limit):
    N, k = 28, 2
    g = torch.Generator(device="cuda").manual_seed(d_in + r)
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g)  # noqa: E731
    x, W0 = rand(d_in).bfloat16(), (0.02 * rand(d_out, d_in)).bfloat16()
    A, B, Wg = (rand(N, r, d_in) / d_in ** 0.5).bfloat16(), (b_std * rand(N, d_out, r)).bfloat16(), (rand(N, d_in) / d_in ** 0.5).bfloat16()
    x[-4:], W0[:, -4:] = 1, 0
    logits, idx = (Wg.double() @ x.double()).topk(k)
    w = torch.softmax(logits, 0)
    y = W0.double() @ x.double() + sum(w[j] * (B[idx[j]].double() @ (A[idx[j]].double() @ x.double())) for j in range(k))
    rest = -y
    for c in range(d_in - 4, d_in):
        W0[:, c] = rest.bfloat16()
        rest = rest - W0[:, c].double()
    got = mb.meteora_linear_forward(x.repeat(T, 1), W0, A, B, Wg, k)
    assert torch.equal(got, got[:1].expand(T, d_out))
    assert float((got[0].double() + rest).pow(2).mean().sqrt() / y.pow(2).mean().sqrt()) <= limit


# More than 512 rows of [Wg; A], or a round of tiles less with it: gate tiles select ahead, the walk's stacked tiles are A alone.  Error of the routing weights over
# 4096 products: 1.9e-6 from a stacked tile's one accumulator, 2^-25 per MMA (16 products) of a CTA from gate tiles.
@pytest.mark.parametrize("T,d_in,d_out,N,r,k,persist", [(1100, 512, 4352, 64, 8, 2, 1), (300, 200, 264, 64, 8, 8, 2), (513, 328, 520, 28, 32, 2, 2),
                                                        (257, 64, 256, 60, 8, 1, 2), (2048, 320, 4096, 50, 8, 2, 1), (700, 640, 1000, 48, 16, 3, 2), (700, 4096, 1024, 64, 8, 2, 2)])
def test_gate_tiles_ahead_of_the_walk(T, d_in, d_out, N, r, k, persist):
    g = torch.Generator(device="cuda").manual_seed(T + N)
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g)  # noqa: E731
    x, W0 = rand(T, d_in).bfloat16(), (rand(d_out, d_in) / d_in ** 0.5).bfloat16()
    A, B, Wg = (rand(N, r, d_in) / d_in ** 0.5).bfloat16(), (0.3 * rand(N, d_out, r)).bfloat16(), (rand(N, d_in) / d_in ** 0.5).bfloat16()
    shape = mb.make_shape(T, d_in, d_out, N, r, k, torch.bfloat16)
    ws = mb.alloc_workspace(shape)
    mb.meteora_set_tuning("persist", persist)
    try:
        assert "path=persistent_prefill launches=2 " in mb.meteora_describe_plan(shape)
        outs = []
        for W in (W0, 0 * W0, W0):
            y, idx, w = mb.meteora_linear_forward(x, W, A, B, Wg, k, workspace=ws, return_routing=True)
            outs.append((y, idx.clone(), w.clone()))
        assert mb.meteora_workspace_status(ws) == 0
        two = mb.meteora_linear_forward_group(x, [W0, W0], [A, A], [B, B], [Wg, Wg], k)
    finally:
        mb.meteora_set_tuning("persist", 1)
    y, idx, w = outs[0]
    assert torch.equal(y, outs[2][0]) and torch.equal(idx, outs[1][1])
    logits = x.double() @ Wg.double().T
    picked = logits.gather(1, idx.long())
    assert float((logits.topk(k, dim=1).values - picked).abs().max()) <= 1e-5      # (ties of fp32 sums apart)
    ref_w = torch.softmax(picked, dim=1)
    assert rel_l2(w.cpu().numpy(), ref_w.cpu().numpy()) <= 2.0 ** -25 * 32 + 2e-7
    mask = torch.zeros(T, N, dtype=torch.double, device="cuda").scatter_(1, idx.long(), w.double())
    u = (x.double() @ A.double().reshape(N * r, -1).T).view(T, N, r) * mask[:, :, None]
    lora = u.view(T, N * r) @ B.double().permute(0, 2, 1).reshape(N * r, -1)
    base = x.double() @ W0.double().T
    assert rel_l2(outs[1][0].float().cpu().numpy(), lora.cpu().numpy()) <= 5e-3    # (us and y rounded to bf16 once each: 2 x 1.7e-3)
    assert rel_l2(y.float().cpu().numpy(), (base + lora).cpu().numpy()) <= 5e-3
    for z in two:
        assert torch.equal(z, y)
