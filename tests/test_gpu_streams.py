"""Calls without a Workspace on several streams and threads at once, and under graph capture: each has scratch of its own."""
import threading

import pytest

from paper_2607_17419_b200 import binding as kb

pytestmark = pytest.mark.gpu


def problem(dtype, H, T, d, seed):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return tuple(torch.randn(1, H, T, d, device="cuda", generator=gen).to(dtype) for _ in range(3))


def prefill(q, k, v):
    import torch
    H, d = q.shape[1], q.shape[-1]
    n = kb.decode_n_psi(d)
    S, Z = torch.empty(1, H, n, d, device="cuda"), torch.empty(1, H, n, device="cuda")
    return kb.kata_fwd_chunked(q, k, v, s_pre=S, z_pre=Z), S, Z


@pytest.mark.parametrize("what", ["state", "f32", "plain"])
def test_two_streams_at_once(what):
    """A long call on one stream and short ones on another while it runs: the same bits as one after the other."""
    import torch
    sizes, d, dt = ((2, 60000), (2, 2000)), 64, torch.bfloat16
    if what == "f32":
        sizes, d, dt = ((8, 30000), (2, 1200)), 16, torch.float32
    call = prefill if what == "state" else lambda q, k, v: (kb.kata_fwd_chunked(q, k, v),)
    probs = [problem(dt, H, T, d, T) for H, T in sizes]
    alone = [call(*p) for p in probs]
    streams = [torch.cuda.Stream() for _ in probs]
    torch.cuda.synchronize()
    got = [[], []]
    for _ in range(10):
        for i, times in ((0, 1), (1, 8)):
            with torch.cuda.stream(streams[i]):
                got[i] += [call(*probs[i]) for _ in range(times)]
    torch.cuda.synchronize()
    for i in range(2):
        for g in got[i]:
            assert all(torch.equal(a, b) for a, b in zip(alone[i], g))


def test_capture_without_a_workspace():
    """The scratch of a captured call stays the graph's: a larger call and new tensors later do not share its memory."""
    import torch
    q, k, v = problem(torch.bfloat16, 2, 3000, 64, 3)
    plain = prefill(q, k, v)[0]
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        out, S, Z = prefill(q, k, v)
    prefill(*problem(torch.bfloat16, 4, 9000, 64, 4))
    torch.cuda.synchronize()
    junk = [torch.full((n << 18,), 7, dtype=torch.int32, device="cuda") for n in (1, 2, 4, 8, 16, 24, 32) for _ in range(4)]
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, plain)
    assert all(bool((j == 7).all()) for j in junk)


def test_threads_have_scratch_of_their_own():
    import torch
    dev, seen = torch.device("cuda", torch.cuda.current_device()), []

    def use():
        torch.cuda.set_device(dev)
        q = torch.randn(1, 1, 1, 64, 64, device=dev).bfloat16()
        kb.kata_fwd_quadratic(q[0], q[0], q[0])
        torch.cuda.synchronize()
        seen.extend(held[0] for held in kb._default_scratch.bufs.values())

    use()
    t = threading.Thread(target=use)
    t.start()
    t.join()
    assert len(seen) >= 2 and len({b.data_ptr() for b in seen}) == len(seen)
