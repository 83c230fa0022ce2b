"""Token tiles (gate, selection and shrink of 128 tokens per cluster), the staged expand and the gate gradient's product at
the edges of their tiles, against the CPU oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2405_13053_b200 import binding as mb
from paper_2405_13053_b200 import workloads
from .gpu_util import check_selection, rel_l2, to_dev

pytestmark = pytest.mark.gpu


# 127 / 128 / 129 tokens: one tile, one tile exactly, a tile with one token; 4 tokens per warp of the expand; 1 k-step and an
# axis that is no multiple of 64; 28 adapters of rank 16 (two rounds of columns); 42 / 43 adapters around what dWg's product
# takes; d_out beyond a 128-row block by less than four outputs.
@pytest.mark.parametrize("T,d_in,d_out,N,r,k", [
    (1, 64, 8, 28, 8, 2), (3, 72, 136, 5, 8, 1), (127, 520, 264, 28, 8, 2), (128, 512, 130, 28, 8, 4), (129, 2048, 384, 28, 8, 2),
    (300, 1096, 512, 28, 16, 3), (257, 768, 200, 42, 8, 2), (200, 768, 256, 43, 8, 8), (65, 4096, 1024, 2, 64, 2), (700, 256, 640, 128, 8, 2),
])
def test_standalone_term_and_gate_gradient(T, d_in, d_out, N, r, k):
    w = workloads.make_workload("tile", T=T, d_in=d_in, d_out=d_out, N=N, r=r, k=k, dtype="bf16", seed=60 + T, b_std=0.3, temperature=2.0)
    x, A, B, Wg = to_dev(w, "x", "A", "B", "Wg")
    o_idx, o_w, o_logits = oracle.gate_topk(w["x"], w["Wg"], k, w.temperature)
    idx, wts, logits = mb.meteora_gate_topk(x, Wg, k, w.temperature, want_logits=True)
    clear = check_selection(idx.cpu().numpy(), o_idx, o_logits, k)
    np.testing.assert_allclose(logits.cpu().numpy(), o_logits, rtol=1e-4, atol=1e-5)
    np.testing.assert_allclose(wts.cpu().numpy()[clear], o_w[clear], rtol=1e-4, atol=1e-5)
    _, offsets, perm = mb.meteora_route(idx, N)
    delta = mb.meteora_lora_delta(x, A, B, idx, wts, offsets, perm)
    ref = oracle.lora_delta(w["x"], w["A"], w["B"], idx.cpu().numpy(), wts.cpu().numpy())
    assert rel_l2(delta.cpu().numpy(), ref) <= 1e-4
    dy = workloads.round_to_bf16(np.random.default_rng(7).standard_normal((T, d_out), dtype=np.float32))
    dWg, dlogit = mb.meteora_gate_backward(x, A, B, torch.from_numpy(dy).cuda().to(x.dtype), idx, wts, w.temperature)
    o_dlogit, o_dWg = oracle.gate_backward(w["x"], w["A"], w["B"], w["Wg"], dy, idx.cpu().numpy(), w.temperature)
    if k > 1:
        assert rel_l2(dlogit.cpu().numpy(), o_dlogit) <= 2e-3
        assert rel_l2(dWg.cpu().numpy(), o_dWg) <= 2e-3
    else:
        assert not dWg.any() and not dlogit.any()


@pytest.mark.parametrize("T,k,N", [(1, 1, 1), (31, 2, 28), (4096, 2, 28), (4097, 2, 28), (1024, 8, 128), (1025, 8, 3 + 8)])
def test_route_shares_of_the_warps(T, k, N):
    # 32 warps x 8 held steps x 32 slots = 8192 slots; one more takes the loop behind
    idx = np.random.default_rng(T).integers(0, N, (T, k)).astype(np.int32)
    counts, offsets, perm = (t.cpu().numpy() for t in mb.meteora_route(torch.from_numpy(idx).cuda(), N))
    np.testing.assert_array_equal(counts, np.bincount(idx.ravel(), minlength=N))
    np.testing.assert_array_equal(offsets, np.concatenate([[0], np.cumsum(counts)]))
    np.testing.assert_array_equal(perm, np.argsort(idx.ravel(), kind="stable"))
