"""The call on host buffers: pinned buffers that a kernel copies, and those that the copy engine does."""
import pytest
import torch

from paper_2405_13053_b200 import binding as mb

pytestmark = pytest.mark.gpu


def _host(T, d, dtype, how):
    if how == "pageable":
        return torch.empty(T, d, dtype=dtype)
    flat = torch.empty(T * d + 16, dtype=dtype).pin_memory()
    return flat[{"pinned": 0, "aligned_view": 16, "odd_view": 3}[how]:][:T * d].view(T, d)


# one vector; rows that are no whole vectors; some CTAs with a last vector; either side of the largest size that a kernel copies (512 KB)
@pytest.mark.parametrize("T,d_in,d_out,dtype", [(1, 8, 8, torch.bfloat16), (3, 7, 13, torch.float32), (5, 256, 1000, torch.float32),
                                               (33, 1024, 2056, torch.bfloat16), (32, 8192, 8192, torch.bfloat16),
                                               (33, 8192, 8192, torch.bfloat16)])
@pytest.mark.parametrize("how", ["pinned", "aligned_view", "odd_view", "pageable"])
def test_host_buffers(T, d_in, d_out, dtype, how):
    g = torch.Generator(device="cuda").manual_seed(T)
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g).to(dtype)  # noqa: E731
    W0, A, B, Wg = 0.02 * rand(d_out, d_in), 0.02 * rand(4, 8, d_in), rand(4, d_out, 8), rand(4, d_in)
    ws = mb.alloc_workspace(mb.make_shape(T, d_in, d_out, 4, 8, 2, dtype))
    x, y = _host(T, d_in, dtype, how), _host(T, d_out, dtype, how)
    for _ in range(2):
        x.copy_(rand(T, d_in))
        y.fill_(float("nan"))
        mb.meteora_linear_forward_host(x, W0, A, B, Wg, 2, y, ws)
        assert mb.meteora_workspace_status(ws) == 0              # synchronises
        ref = mb.meteora_linear_forward(x.cuda(), W0, A, B, Wg, 2)
        assert torch.equal(y, ref.cpu())


def test_calls_in_a_row_read_what_the_call_ahead_wrote():
    T, d, N = 40, 2048, 28
    g = torch.Generator(device="cuda").manual_seed(1)
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g).bfloat16()  # noqa: E731
    W0, A, B, Wg = d ** -0.5 * rand(d, d), 0.02 * rand(N, 8, d), 0.05 * rand(N, d, 8), rand(N, d)
    ws = mb.alloc_workspace(mb.make_shape(T, d, d, N, 8, 2, torch.bfloat16))
    bufs = [torch.randn(T, d).bfloat16().pin_memory()] + [torch.empty(T, d).bfloat16().pin_memory() for _ in range(6)]
    for x, y in zip(bufs, bufs[1:]):
        mb.meteora_linear_forward_host(x, W0, A, B, Wg, 2, y, ws)
    torch.cuda.synchronize()
    ref = bufs[0].cuda()
    for y in bufs[1:]:
        ref = mb.meteora_linear_forward(ref, W0, A, B, Wg, 2)
        assert torch.equal(y, ref.cpu())
