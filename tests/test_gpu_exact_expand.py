"""Where decode batches (and short prefill batches of larger ranks) run on persistent pairs, the LoRA expand keeps fp32's precision
and a token's y depends on the adapters it picked alone, as on the kernels that expand in fp32."""
import pytest
import torch

from paper_2405_13053_b200 import binding as mb

pytestmark = pytest.mark.gpu

# routing ahead of the walk (one token tile, several chunks), inside it (one and two pairs of stacked tiles, one chunk and several),
# groups of both kinds, short prefill batches of ranks 16 and 32
CASES = [(48, 2048, (9216,), 28, 8, 2), (201, 2048, (7432,), 28, 8, 4), (96, 2120, (8456,), 12, 16, 2), (16, 2048, (38144,), 12, 8, 2),
         (3, 1024, (38144,), 56, 8, 2), (20, 1024, (14336, 14336), 28, 8, 2), (112, 2048, (4096, 4360), 28, 8, 2),
         (140, 1024, (14344, 14336), 28, 8, 1), (300, 512, (1024,), 28, 32, 2), (513, 1024, (2048,), 28, 16, 2)]


def _module(g, d_in, d_out, N, r, zero_w0=False):
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g)  # noqa: E731
    W0 = torch.zeros(d_out, d_in, device="cuda") if zero_w0 else 0.02 * rand(d_out, d_in)
    return [t.bfloat16() for t in (W0, rand(N, r, d_in) / d_in ** 0.5, 0.3 * rand(N, d_out, r), rand(N, d_in) / d_in ** 0.5)]


def _run(x, mods, k):
    if len(mods) == 1:
        shape = mb.make_shape(x.shape[0], x.shape[1], mods[0][0].shape[0], *mods[0][1].shape[:2], k, torch.bfloat16)
        assert "persistent_pairs=" in mb.meteora_describe_plan(shape), mb.meteora_describe_plan(shape)
        y, idx, _ = mb.meteora_linear_forward(x, *mods[0], k, return_routing=True)
        return [(y, idx)]
    ys, routing = mb.meteora_linear_forward_group(x, *[list(t) for t in zip(*mods)], k, return_routing=True)
    return [(y, idx) for y, (idx, _) in zip(ys, routing)]


def _weighted(x, m, idx):
    """w_j (A_e x) and B_e of every slot, in fp64: [T, k, r], [T, k, d_out, r] by slot via index."""
    A, Wg = m[1].double(), m[3].double()
    w = torch.softmax((x.double() @ Wg.T).gather(1, idx.long()), dim=1)
    u = torch.einsum("td,nrd->tnr", x.double(), A).gather(1, idx.long()[:, :, None].expand(-1, -1, A.shape[1]))
    return w[:, :, None] * u


@pytest.mark.parametrize("T,d_in,d_outs,N,r,k", CASES)
def test_expand_holds_fp32(T, d_in, d_outs, N, r, k):
    # Without a base product y is the expand alone, rounded once: half a place of bf16 (8 bits: 2^(e - 9) for 2^(e - 1) <= |y| < 2^e)
    # plus what fp32 sums of d_in products leave in u (a few 2^-23 sqrt(d_in), below 2^-16) and in the k r products of the expand.
    # A bf16 operand would be off by up to 2^-8 of every product, which shows wherever the products cancel.
    g = torch.Generator(device="cuda").manual_seed(40 + T)
    mods = [_module(g, d_in, d, N, r, zero_w0=True) for d in d_outs]
    x = torch.randn(T, d_in, device="cuda", generator=g).bfloat16()
    for m, (y, idx) in zip(mods, _run(x, mods, k)):
        uw, B = _weighted(x, m, idx), m[2].double()
        ref, size = torch.zeros_like(y, dtype=torch.double), torch.zeros_like(y, dtype=torch.double)
        for j in range(k):
            for e in range(N):
                rows = (idx[:, j] == e).nonzero()[:, 0]
                ref[rows] += uw[rows, j] @ B[e].T
                size[rows] += uw[rows, j].abs() @ B[e].abs().T
        half_place = torch.ldexp(torch.ones_like(ref), torch.frexp(ref.abs() + 2.0 ** -14 * size)[1] - 9)
        worst = ((y.double() - ref).abs() - half_place - 2.0 ** -14 * size).max()
        assert float(worst) <= 0.0


@pytest.mark.parametrize("T,d_in,d_outs,N,r,k", CASES)
def test_an_adapter_that_was_not_picked_does_not_reach_y(T, d_in, d_outs, N, r, k):
    g = torch.Generator(device="cuda").manual_seed(50 + T)
    mods = [_module(g, d_in, d, N, r) for d in d_outs]
    x = torch.randn(T, d_in, device="cuda", generator=g).bfloat16()
    clean = [(y.clone(), idx.clone()) for y, idx in _run(x, mods, k)]
    bad, rows = int(clean[0][1][0, 0]), [0, 5, 131, mods[0][0].shape[0] - 1]      # an adapter that a token picked
    for m in mods:
        m[2][bad, rows[0], 0] = float("inf")
        m[2][bad, rows[1], r - 1] = float("nan")
        m[2][bad, rows[2]] = float("-inf")
        m[2][bad, -1, 1] = float("inf")
        rest = (bad + 1 + torch.arange(N - 1, device="cuda")) % N
        m[2][rest[-1], 7, 0] = float("nan")
    for m, (y0, idx0), (y, idx) in zip(mods, clean, _run(x, mods, k)):
        assert torch.equal(idx, idx0)
        hit = torch.zeros_like(y, dtype=torch.bool)
        for e in range(N):
            picked = (idx == e).any(dim=1)
            odd = ~torch.isfinite(m[2][e].float()).all(dim=1)
            hit |= picked[:, None] & odd[None, :]
        # the same sums in another order where the element was computed again: one place of bf16
        assert torch.isfinite(y[~hit]).all()
        assert torch.allclose(y[~hit].float(), y0[~hit].float(), rtol=2.0 ** -7, atol=1e-3)
        assert not torch.isfinite(y[hit]).any()
