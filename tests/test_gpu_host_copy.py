"""The call on host buffers: pinned buffers that a kernel copies, and those that the copy engine does."""
import ctypes

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


def _graph_copies(graph):
    """How many of a captured call's nodes are copies by the copy engine."""
    rt, raw, n = ctypes.CDLL("libcudart.so.12"), ctypes.c_void_p(graph.raw_cuda_graph()), ctypes.c_size_t(0)
    assert rt.cudaGraphGetNodes(raw, None, ctypes.byref(n)) == 0
    nodes, kinds = (ctypes.c_void_p * n.value)(), []
    assert rt.cudaGraphGetNodes(raw, nodes, ctypes.byref(n)) == 0
    for node in nodes:
        kind = ctypes.c_int(-1)
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kinds.append(kind.value)
    return kinds.count(1)                                        # cudaGraphNodeTypeMemcpy


# a captured call, its nodes showing which copies a kernel makes: pinned buffers of whole aligned vectors up to 512 KB, each way by itself
@pytest.mark.parametrize("T,d_in,d_out,how,copies", [(1, 8, 8, "pinned", 0), (40, 1024, 2048, "aligned_view", 0), (32, 8192, 8192, "pinned", 0),
                                                     (33, 8192, 8192, "pinned", 2), (33, 8192, 1024, "pinned", 1), (33, 1024, 8192, "pinned", 1),
                                                     (40, 1024, 2048, "odd_view", 2)])
def test_captured_call_and_the_way_of_its_copies(T, d_in, d_out, how, copies):
    g = torch.Generator(device="cuda").manual_seed(d_out)
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g).bfloat16()  # noqa: E731
    W0, A, B, Wg = 0.02 * rand(d_out, d_in), 0.02 * rand(4, 8, d_in), rand(4, d_out, 8), rand(4, d_in)
    ws = mb.alloc_workspace(mb.make_shape(T, d_in, d_out, 4, 8, 2, torch.bfloat16))
    x, y = _host(T, d_in, torch.bfloat16, how), _host(T, d_out, torch.bfloat16, how)
    x.copy_(rand(T, d_in))
    mb.meteora_linear_forward_host(x, W0, A, B, Wg, 2, y, ws)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        mb.meteora_linear_forward_host(x, W0, A, B, Wg, 2, y, ws)
    assert _graph_copies(graph) == copies
    for _ in range(2):
        x.copy_(rand(T, d_in))
        y.fill_(float("nan"))
        torch.cuda.synchronize()
        graph.replay()
        assert mb.meteora_workspace_status(ws) == 0
        assert torch.equal(y, mb.meteora_linear_forward(x.cuda(), W0, A, B, Wg, 2).cpu())
