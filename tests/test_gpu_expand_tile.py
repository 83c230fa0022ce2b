"""The LoRA term's expand as a tensor-core product (B's rows against the masked w u in three parts), against fp64."""
import pytest
import torch

from paper_2405_13053_b200 import binding as mb

pytestmark = pytest.mark.gpu


def _problem(T, d_in, d_out, N, r, k, twice=False):
    g = torch.Generator(device="cuda").manual_seed(T + d_out)
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g)  # noqa: E731
    x, A, B = rand(T, d_in).bfloat16(), (rand(N, r, d_in) / d_in ** 0.5).bfloat16(), (0.3 * rand(N, d_out, r)).bfloat16()
    idx = torch.rand(T, N, device="cuda", generator=g).topk(k, dim=1).indices.int()
    if twice:
        idx[::3, -1] = idx[::3, 0]                               # picks of one token that name the same adapter add up
    return x, A, B, idx.contiguous(), torch.softmax(rand(T, k), dim=1)


def _reference(x, A, B, idx, w):
    u = torch.einsum("td,nrd->tnr", x.double(), A.double())
    out = torch.zeros(x.shape[0], B.shape[1], dtype=torch.double, device="cuda")
    for j in range(idx.shape[1]):
        for e in range(A.shape[0]):
            t = (idx[:, j] == e).nonzero()[:, 0]
            out[t] += w[t, j, None].double() * (u[t, e] @ B[e].double().T)
    return out


def _delta(x, A, B, idx, w):
    _, offsets, perm = mb.meteora_route(idx, A.shape[0])
    return mb.meteora_lora_delta(x, A, B, idx, w, offsets, perm)


# either side of the smallest work it takes (3 * 2^20 picks x outputs); one token beyond a tile of 32, a tile and a row block that are
# nearly empty; several rounds of the four operands; an odd number of columns of 8, ranks of several; most picks (several values
# per thread); the most columns that fit, and two more than that
@pytest.mark.parametrize("T,d_in,d_out,N,r,k", [
    (1, 64, 400000, 28, 8, 8), (50, 64, 32001, 28, 8, 2), (64, 64, 24575, 28, 8, 2), (64, 64, 24576, 28, 8, 2), (130, 72, 8193, 3, 8, 3),
    (620, 64, 1030, 7, 24, 5), (1573, 64, 4096, 28, 8, 2), (6100, 64, 520, 28, 8, 1), (300, 64, 20000, 28, 8, 8), (1500, 128, 264, 14, 16, 8),
    (5300, 64, 200, 3, 64, 3), (6000, 64, 200, 30, 8, 2),
])
@pytest.mark.parametrize("twice", [False, True])
def test_expand_tile(T, d_in, d_out, N, r, k, twice):
    x, A, B, idx, w = _problem(T, d_in, d_out, N, r, k, twice)
    ref = _reference(x, A, B, idx, w)
    # fp32 sums of 64 - 128 products in u and of k r in delta: about 2^-23 (sqrt(128) + sqrt(64)) / 4.  Without its third part
    # w u is off by up to 2^-16 of itself, 4e-6 on average.
    got = _delta(x, A, B, idx, w)
    assert float((got.double() - ref).norm() / ref.norm()) <= 1.5e-6
    assert float((got.double() - ref).abs().max()) <= 2.0 ** -19 * float(ref.abs().max()) * k
    assert torch.equal(got, _delta(x, A, B, idx, w))


def test_only_the_picks_count():
    x, A, B, idx, w = _problem(5300, 64, 300, 28, 8, 2)
    ref = _delta(x, A, B, idx, w)
    B2, x2 = B.clone(), x.clone()
    B2[5, 17, 3], B2[9, 140, 0], B2[11, 299, 7] = float("inf"), float("nan"), float("-inf")
    x2[70] = float("nan")
    got = _delta(x2, A, B2, idx, w)
    odd = torch.zeros_like(ref, dtype=torch.bool)
    for e, o in ((5, 17), (9, 140), (11, 299)):
        odd[(idx == e).any(dim=1), o] = True
    odd[70] = True
    assert torch.equal(~torch.isfinite(got), odd)
    # what was NaN in the product is computed again in another order: fp32 sums of 16 terms
    torch.testing.assert_close(got[~odd], ref[~odd], rtol=0, atol=float(2.0 ** -20 * ref.abs().max()))
    infinite = (idx == 5).any(dim=1) & (torch.arange(5300, device="cuda") != 70)
    assert torch.isinf(got[infinite, 17]).all()
