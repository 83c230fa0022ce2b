"""Calls whose CTAs wait for one another, on two streams of different priority at the same time: each launch holds all its SMs or none."""
import pytest
import torch

from paper_2405_13053_b200 import binding as mb

pytestmark = pytest.mark.gpu

GROUP, BATCH, PREFILL = (64, (1024, 512, 512)), (200, (2048,)), (600, (4096, 2048))


def _caller(T, d_outs, seed, d_in=2048, N=28, r=8, k=2):
    g = torch.Generator(device="cuda").manual_seed(seed)
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g)  # noqa: E731
    mods = [[t.bfloat16() for t in (0.02 * rand(d, d_in), rand(N, r, d_in) / d_in ** 0.5, 0.05 * rand(N, d, r), rand(N, d_in) / d_in ** 0.5)]
            for d in d_outs]
    x = rand(T, d_in).bfloat16()
    if len(d_outs) > 1:
        lists = [list(t) for t in zip(*mods)]
        return lambda: mb.meteora_linear_forward_group(x, *lists, k)
    workspace = mb.alloc_workspace(mb.make_shape(T, d_in, d_outs[0], N, r, k, torch.bfloat16))
    return lambda: [mb.meteora_linear_forward(x, *mods[0], k, workspace=workspace)]


@pytest.mark.parametrize("first,second", [(GROUP, BATCH), (BATCH, BATCH), (GROUP, PREFILL), (BATCH, PREFILL)])
def test_two_streams(first, second):
    calls = [_caller(*first, seed=1), _caller(*second, seed=2)]
    refs = [c() for c in calls]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(priority=0), torch.cuda.Stream(priority=-1)]
    for stream in streams:
        stream.wait_stream(torch.cuda.current_stream())
    results = [[], []]
    for _ in range(40):
        for i, stream in enumerate(streams):
            with torch.cuda.stream(stream):
                results[i].append(calls[i]())
    torch.cuda.synchronize()
    for ref, got in zip(refs, results):
        for ys in got:
            assert all(torch.equal(a, b) for a, b in zip(ref, ys))
