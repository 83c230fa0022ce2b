"""The plain CUDA-core path (fp32 layers, shapes the tensor cores do not take) at the edges of its tiles."""
import numpy as np
import pytest
import torch

import oracle
from .gpu_util import check_selection, rel_l2, to_dev
from paper_2405_13053_b200 import binding as mb
from paper_2405_13053_b200 import workloads

pytestmark = pytest.mark.gpu


# Tiles are 64 rows x 16 tokens up to 16 tokens, 64 x 64 or 128 x 64 above; chunks of 16 elements, two at least per slice.
@pytest.mark.parametrize("T,d_in,d_out,N,r,k,dtype", [
    (1, 16, 1, 1, 1, 1, "f32"),               # the smallest of everything: one chunk, one slice
    (16, 33, 64, 4, 8, 2, "f32"),             # last token count of the narrow tile, rows not 16-byte aligned
    (17, 250, 63, 4, 8, 2, "f32"),            # first of the wide tile
    (65, 758, 1246, 8, 8, 2, "f32"),          # one token and part of a row tile beyond the last whole tile
    (130, 2048, 2000, 28, 8, 4, "f32"),       # 128-row tiles
    (512, 1031, 513, 128, 3, 8, "f32"),       # 128 adapters, rank 3, several slices
    (40, 1030, 100, 28, 64, 2, "f32"),        # the largest rank
    (33, 1027, 300, 28, 8, 2, "bf16"),        # bf16 rows of odd length
    (8, 2050, 130, 28, 5, 2, "bf16"),
    (8300, 20, 4000, 4, 8, 2, "f32"),         # several blocks of tokens on the same scratch
    (2300, 36, 30000, 4, 8, 1, "bf16"),
])
def test_plain_path_matches_oracle(T, d_in, d_out, N, r, k, dtype):
    w = workloads.make_workload("simt", T=T, d_in=d_in, d_out=d_out, N=N, r=r, k=k, dtype=dtype, seed=40 + T, b_std=0.3)
    t = to_dev(w, "x", "W0", "A", "B", "Wg")
    ws = mb.alloc_workspace(mb.make_shape(T, d_in, d_out, N, r, k, t[0].dtype))
    y, idx, wts = mb.meteora_linear_forward(*t, k, workspace=ws, return_routing=True)
    y1, idx = y.float().cpu().numpy(), idx.cpu().numpy()
    o_idx, o_w, o_logits = oracle.gate_topk(w["x"], w["Wg"], k)
    clear = check_selection(idx, o_idx, o_logits, k)
    np.testing.assert_allclose(wts.cpu().numpy()[clear], o_w[clear], rtol=1e-4, atol=1e-5)
    ref = oracle.linear_forward_routed(w["x"], w["W0"], w["A"], w["B"], w["Wg"], idx)
    assert rel_l2(y1, ref) <= (1e-5 if dtype == "f32" else 5e-3)
    np.testing.assert_array_equal(y1, mb.meteora_linear_forward(*t, k, workspace=ws).float().cpu().numpy())
