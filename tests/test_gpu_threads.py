"""The binding leaves other Python threads running while a call into the library blocks."""
import threading
import time

import pytest
import torch

from paper_2405_13053_b200 import binding as mb

pytestmark = pytest.mark.gpu


def test_a_blocking_call_does_not_stop_other_threads():
    T, d_in, d_out, N, r, k = 64, 1024, 1024, 28, 8, 2
    g = torch.Generator(device="cuda").manual_seed(3)
    rand = lambda *s: torch.randn(*s, device="cuda", generator=g).bfloat16()  # noqa: E731
    W0, A, B, Wg = rand(d_out, d_in), rand(N, r, d_in), rand(N, d_out, r), rand(N, d_in)
    x, y = torch.randn(T, d_in).bfloat16(), torch.empty(T, d_out, dtype=torch.bfloat16)      # pageable: the copies block
    workspace = mb.alloc_workspace(mb.make_shape(T, d_in, d_out, N, r, k, torch.bfloat16))
    mb.meteora_linear_forward_host(x, W0, A, B, Wg, k, y, workspace)
    torch.cuda.synchronize()
    expected, ticks, stop = y.clone(), [], threading.Event()

    def tick():
        while not stop.is_set():
            ticks.append(time.perf_counter())
            time.sleep(0.001)

    other = threading.Thread(target=tick)
    other.start()
    try:
        torch.cuda._sleep(600_000_000)                   # about 0.3 s of stream time ahead of the call
        begin = time.perf_counter()
        mb.meteora_linear_forward_host(x, W0, A, B, Wg, k, y, workspace)
        end = time.perf_counter()
    finally:
        stop.set()
        other.join()
    torch.cuda.synchronize()
    assert torch.equal(y, expected)
    assert end - begin > 0.1                             # the call did block
    assert sum(begin < t < end for t in ticks) > 20


def test_calls_from_several_threads():
    # a stream and a workspace for each thread: a decode group, a batch above 128 tokens, a prefill batch and the gate's gradient
    N, r, k, d_in = 28, 8, 2, 1024

    def make(i, T, d_outs):
        g = torch.Generator(device="cuda").manual_seed(20 + i)
        rand = lambda *s: torch.randn(*s, device="cuda", generator=g).bfloat16()  # noqa: E731
        mods = [(rand(d, d_in), rand(N, r, d_in), rand(N, d, r), rand(N, d_in)) for d in d_outs]
        x, dy = rand(T, d_in), rand(T, d_outs[0])

        def call():
            if len(d_outs) > 1:
                return mb.meteora_linear_forward_group(x, *[list(t) for t in zip(*mods)], k)
            W0, A, B, Wg = mods[0]
            idx, w, _ = mb.meteora_gate_topk(x, Wg, k)
            return [mb.meteora_linear_forward(x, W0, A, B, Wg, k), *mb.meteora_gate_backward(x, A, B, dy, idx, w)]

        return call

    calls = [make(i, *c) for i, c in enumerate([(64, (512, 256)), (200, (1024,)), (600, (2048,)), (300, (1024, 512))])]
    refs = [c() for c in calls]
    torch.cuda.synchronize()
    wrong = []

    def work(i):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            got = [calls[i]() for _ in range(25)]
        stream.synchronize()
        wrong.extend((i, n) for n, ys in enumerate(got) if not all(torch.equal(a, b) for a, b in zip(refs[i], ys)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
