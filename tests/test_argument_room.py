"""Tensors that a call would read or write beyond their end, or misread, are refused before anything is launched.  (Here on host
tensors, through the statements that every refused call ends in; on the device: test_gpu_native_calls.py.)"""
import pytest
import torch

from paper_2607_17419_b200 import binding as kb

B, H, T, D = 2, 3, 100, 64


def x(*shape, dtype=torch.float32):
    return torch.zeros(*shape, dtype=dtype)


def seq(**kw):
    return x(B, H, T, D, **kw)


def calls():
    n = kb.decode_n_psi(D)
    S, Z, t = x(B, H, n, D), x(B, H, n), [x(B, H, D) for _ in range(3)]
    short, half, strided, long = x(B, H, T - 1, D), seq(dtype=torch.bfloat16), x(B, T, H, D).transpose(1, 2), x(B, H, T + 1, D)
    fwd, bwd = kb.kata_fwd_chunked, kb.kata_bwd_quadratic
    bad = {"k": (short, half, long), "v": (short, half, long), "out": (short, half, strided)}
    for name, values in bad.items():
        for i, value in enumerate(values):
            for f in (kb.kata_fwd_quadratic, fwd, kb.kata_chunk_state_scan):
                args = {"q": seq(), "k": seq(), "v": seq(), name: value}
                yield f"{f.__name__} {name} {i}", lambda f=f, args=args: f(**args)
    yield "static k", lambda: kb.kata_chunk_state_scan_static(seq(), short, seq(), seq())
    yield "static out", lambda: kb.kata_chunk_state_scan_static(seq(), seq(), seq(), strided)
    yield "static q", lambda: kb.kata_chunk_state_scan_static(strided, seq(), seq(), seq())
    states = {"S": (S[:1], S.double(), S.transpose(2, 3)), "Z": (Z[:1], Z.double())}
    for which in ("pre", "init"):
        for name, values in states.items():
            for i, value in enumerate(values):
                kw = {f"s_{which}": S, f"z_{which}": Z, f"{name.lower()}_{which}": value}
                yield f"state {name} {which} {i}", lambda kw=kw: fwd(seq(), seq(), seq(), **kw)
    yield "layout", lambda: fwd(seq(), seq(), seq(), s_pre=x(B, H, 2080, D), z_pre=x(B, H, 2080))
    yield "per chunk", lambda: kb.kata_chunk_state_scan(seq(), seq(), seq(), s_pre=S, z_pre=Z)
    yield "status", lambda: fwd(seq(), seq(), seq(), device_status=x(0))
    for i, kw in enumerate([{"k": x(B, H, D - 1)}, {"v": half[:, :, 0]}, {"out": x(B, H - 1, D)}, {"out": x(D, H, B).permute(2, 1, 0)}]):
        yield f"decode {i}", lambda kw=kw: kb.kata_decode_step(**{"q": t[0], "k": t[1], "v": t[2], "S": S, "Z": Z, **kw})
    for f in (bwd, kb.kata_bwd_chunked):
        for name in ("k", "v", "dout", "dq", "dk", "dv"):
            for i, value in enumerate((short, half)):
                args = {"q": seq(), "k": seq(), "v": seq(), "dout": seq(), name: value}
                yield f"{f.__name__} {name} {i}", lambda f=f, args=args: f(**args)


CALLS = dict(calls())


@pytest.mark.parametrize("name", list(CALLS))
def test_refused(name):
    with pytest.raises(ValueError):
        CALLS[name]()


@pytest.mark.parametrize("kw", [{}, {"k": x(B * H, T, D)}, {"out": x(B * H * T * D + 5)}, {"s_pre": x(B, H, 2080, D), "z_pre": x(B, H, 2080),
                                "state_layout": kb.KATA_LAYOUT_PACKED}])
def test_taken_as_before(kw):
    """Other shapes of the same elements and outputs with room to spare pass (these calls end later, at the host tensors)."""
    with pytest.raises((RuntimeError, TypeError)):
        kb.kata_fwd_chunked(**{"q": seq(), "k": seq(), "v": seq(), **kw})


def test_one_head_may_have_more_keys():
    with pytest.raises((RuntimeError, TypeError)):
        kb.kata_fwd_chunked(x(1, 1, T, D), x(1, 1, T + 5, D), x(1, 1, T + 9, D))
