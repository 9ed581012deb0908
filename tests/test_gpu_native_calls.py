"""Tensor calls by the native module (csrc/kata_torch.cpp) against the same calls through ctypes (taken when a stream is named):
the same bits, the same errors, and the calls that it leaves alone."""
import pytest

from paper_2607_17419_b200 import binding as kb

pytestmark = pytest.mark.gpu


def tensors(shape, dtype, n=4, seed=0):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return [torch.randn(*shape, device="cuda", generator=gen).to(getattr(torch, dtype)) for _ in range(n)]


def state(B, H, d, **kw):
    import torch
    n = kb.decode_n_psi(d, **kw)
    gen = torch.Generator(device="cuda").manual_seed(9)
    return torch.rand(B, H, n, d, device="cuda", generator=gen), torch.rand(B, H, n, device="cuda", generator=gen) + 1


CALLS = {
    "quadratic": lambda s: kb.kata_fwd_quadratic(*tensors((2, 3, 300, 64), "bfloat16", 3), **s),
    "quadratic_f32": lambda s: kb.kata_fwd_quadratic(*tensors((1, 2, 65, 32), "float32", 3), **s),
    "chunked_groups": lambda s: kb.kata_fwd_chunked(*tensors((1, 2, 1500, 64), "bfloat16", 3), feature_groups=2, inter_chunk=kb.KATA_INTER_AUTO, **s),
    "chunked_scan": lambda s: kb.kata_fwd_chunked(*tensors((1, 2, 1500, 64), "bfloat16", 3), inter_chunk=kb.KATA_SCAN, scan_group=4, **s),
    "chunked_out": lambda s: kb.kata_fwd_chunked(*tensors((1, 2, 1500, 16), "float32", 4), **s),
    "scan_order1": lambda s: kb.kata_chunk_state_scan(*[x.abs() for x in tensors((1, 2, 700, 64), "bfloat16", 3)], C=128, feature_order=1, **s),
    "bwd_quadratic": lambda s: kb.kata_bwd_quadratic(*tensors((1, 2, 300, 64), "bfloat16"), **s),
    "bwd_chunked": lambda s: kb.kata_bwd_chunked(*tensors((1, 2, 600, 64), "bfloat16"), **s),
    "requires_grad": lambda s: kb.kata_fwd_quadratic(*[x.requires_grad_() for x in tensors((1, 2, 100, 64), "float32", 3)], **s),
}


def stream():
    import torch
    return {"stream": torch.cuda.current_stream().cuda_stream}


def as_tuple(x):
    return x if isinstance(x, tuple) else (x,)


@pytest.mark.parametrize("name", sorted(CALLS))
def test_same_bits(name, monkeypatch):
    import torch
    want = as_tuple(CALLS[name](stream()))            # (also leaves the scratch behind that the native call looks up)
    taken = []
    mod = kb.native()

    class Watch:
        def __getattr__(self, attr):
            def call(*a):
                taken.append(getattr(mod, attr)(*a))
                return taken[-1]
            return call

    monkeypatch.setattr(kb, "_native", Watch())
    got = as_tuple(CALLS[name]({}))
    assert len(taken) == 1 and taken[0] is not NotImplemented
    assert len(got) == len(want)
    for g, w in zip(got, want):
        assert g.dtype == w.dtype and g.shape == w.shape and not g.requires_grad and torch.equal(g, w)


@pytest.mark.parametrize("layout,groups,dtype", [(0, 1, "bfloat16"), (1, 2, "float32"), (1, 1, "bfloat16")])
def test_decode_and_prefill(layout, groups, dtype):
    import torch
    kw = dict(state_layout=layout, feature_groups=groups)
    q, k, v = tensors((2, 3, 64), dtype, 3)
    S, Z = state(2, 3, 64, state_layout=layout, feature_groups=groups)
    res = []
    for extra in (stream(), {}, {"out": torch.empty_like(v)}):
        S1, Z1 = S.clone(), Z.clone()
        o = kb.kata_decode_step(q, k, v, S1, Z1, **kw, **extra)
        assert "out" not in extra or o.data_ptr() == extra["out"].data_ptr()
        x = tensors((2, 3, 700, 64), dtype, 3, seed=1)
        p = kb.kata_fwd_chunked(*x, s_init=S1, z_init=Z1, s_pre=S1, z_pre=Z1, **kw, **{a: b for a, b in extra.items() if a == "stream"})
        res.append((o, p, S1, Z1))
    for other in res[1:]:
        assert all(torch.equal(a, b) for a, b in zip(res[0], other))


def bad_calls():
    import torch
    q, k, v, g = tensors((1, 2, 100, 64), "bfloat16")
    S, Z = state(1, 2, 64)
    t = tensors((1, 2, 64), "bfloat16", 3)
    return [
        lambda s: kb.kata_fwd_quadratic(q.transpose(1, 2), k, v, **s),
        lambda s: kb.kata_fwd_quadratic(q.half(), k.half(), v.half(), **s),
        lambda s: kb.kata_fwd_quadratic(q[0], k[0], v[0], **s),
        lambda s: kb.kata_fwd_quadratic(q, k, v, nonsense=1, **s),
        lambda s: kb.kata_fwd_quadratic(q, k, v, feature_groups=3, **s),
        lambda s: kb.kata_fwd_chunked(q, k, v, C=32, **s),
        lambda s: kb.kata_fwd_chunked(q, k, v, s_pre=S, **s),
        lambda s: kb.kata_fwd_chunked(q, k, v, feature_groups=2.0, **s),
        lambda s: kb.kata_fwd_chunked(q, k, v, impl=2, s_init=S, z_init=Z, feature_order=1, **s),
        lambda s: kb.kata_fwd_chunked(q.view(-1)[4:4 + 64 * 64].view(1, 1, 64, 64), k[:, :1, :64].contiguous(), v[:, :1, :64].contiguous(), **s),
        lambda s: kb.kata_decode_step(*t, S.half(), Z, **s),
        lambda s: kb.kata_decode_step(*t, S[:, :, 1:].contiguous(), Z, **s),
        lambda s: kb.kata_decode_step(*t, S, Z, s_pre=256, z_pre=256, **s),
        lambda s: kb.kata_bwd_quadratic(q, k, v, g.transpose(1, 2), **s),
        lambda s: kb.kata_bwd_chunked(q, k, v, g, C=128, **s),
        lambda s: kb.kata_bwd_quadratic(q, k, v, torch.stack([g, g])[:, 0, 0], out=None, **s),
        # tensors that the kernels would run over the end of, or misread (refused before the library is called)
        lambda s: kb.kata_fwd_quadratic(q, k[:, :, :50].contiguous(), v, **s),
        lambda s: kb.kata_fwd_chunked(q, k, v.float(), **s),
        lambda s: kb.kata_fwd_chunked(q, k, v, out=torch.empty(1, 2, 99, 64, dtype=torch.bfloat16, device="cuda"), **s),
        lambda s: kb.kata_fwd_chunked(q, k, v, out=torch.empty(1, 100, 2, 64, dtype=torch.bfloat16, device="cuda").transpose(1, 2), **s),
        lambda s: kb.kata_fwd_chunked(q, k, v, out=torch.empty_like(v, device="cpu"), **s),
        lambda s: kb.kata_fwd_chunked(q, k, v, s_pre=S[:, :1].contiguous(), z_pre=Z, **s),
        lambda s: kb.kata_chunk_state_scan(q, k, v, s_pre=S, z_pre=Z, **s),
        lambda s: kb.kata_decode_step(t[0], t[1][:, :1].contiguous(), t[2], S, Z, **s),
        lambda s: kb.kata_decode_step(*t, S, Z, out=torch.empty(1, 2, 32, dtype=torch.bfloat16, device="cuda"), **s),
        lambda s: kb.kata_bwd_quadratic(q, k, v, g[:, :, :50].contiguous(), **s),
        lambda s: kb.kata_bwd_chunked(q, k, v, g, dk=torch.empty(1, 2, 50, 64, dtype=torch.bfloat16, device="cuda"), **s),
    ]


def test_same_errors():
    for i, call in enumerate(bad_calls()):
        seen = []
        for s in (stream(), {}):
            with pytest.raises(Exception) as e:
                call(s)
            seen.append((type(e.value), str(e.value)))
        assert seen[0] == seen[1], i


def test_subclasses_and_function_modes_are_left_to_the_binding():
    import torch
    from torch.overrides import TorchFunctionMode
    q, k, v = tensors((1, 2, 100, 64), "bfloat16", 3)
    want = kb.kata_fwd_quadratic(q, k, v)

    class Mode(TorchFunctionMode):
        seen = 0

        def __torch_function__(self, func, types, args=(), kwargs=None):
            Mode.seen += func is torch.empty_like
            return func(*args, **(kwargs or {}))

    with Mode():
        got = kb.kata_fwd_quadratic(q, k, v)
    assert Mode.seen == 1 and torch.equal(got, want)
    par = torch.nn.Parameter(q)
    assert torch.equal(kb.kata_fwd_quadratic(par, k, v), want)
