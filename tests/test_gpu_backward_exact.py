"""kata_bwd_chunked on the tensor cores (bf16, d = 64, 512 to 16384 tokens: the quadratic form with fp32 weights) at the edges
of its range and of its tiles (128 fixed rows, 64 streamed rows).

The operands are the bf16 inputs, the weights carry 24 bits and the sums are fp32, so beside the rounding of the stored
gradient (2^-9 of the entry) the error is that of fp32 sums: 1e-5 of the largest entry covers both sweeps' T terms.  The
plain FMA kernels of the same entry are held to the same bound."""
import numpy as np
import pytest

from oracle import kata_oracle as ko
from paper_2607_17419_b200 import binding as kb
from paper_2607_17419_b200 import inputs

from helpers import dev_tensors, to_numpy64
from test_gpu_backward import dout_for

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,zero", [(512, False), (513, True), (575, False), (577, False), (639, True), (641, False), (1100, True)])
def test_backward_exact(T, zero):
    import torch
    w = inputs.gaussian_workload(f"bwdx_{T}", "bf16", 1, 3, T, 64, 64, 64, 6100 + T)
    if zero:
        for arr in (w.k_ref, w.k_dev):
            arr[0, 0, [0, 127, 128, 300]] = 0
        for arr in (w.q_ref, w.q_dev):
            arr[0, 0, [5, 256, T - 1]] = 0
    q, k, v = dev_tensors(w)
    g, g_ref = dout_for(w, 5)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    grads = kb.kata_bwd_chunked(q, k, v, g, device_status=st)
    torch.cuda.synchronize()
    assert kb.kata_last_impl() == kb.KATA_IMPL_TENSOR and kb.kata_last_launch_count() == 3 and int(st.item()) == 0
    again = kb.kata_bwd_chunked(q, k, v, g, impl=kb.KATA_IMPL_TENSOR)
    plain = kb.kata_bwd_chunked(q, k, v, g, impl=kb.KATA_IMPL_SIMT)
    torch.cuda.synchronize()
    assert kb.kata_last_impl() == kb.KATA_IMPL_SIMT
    for h in range(w.H):
        ref = ko.kata_quadratic_bwd(w.q_ref[0, h], w.k_ref[0, h], w.v_ref[0, h], g_ref[0, h])
        for name, got, same, other, r in zip(("dq", "dk", "dv"), grads, again, plain, ref):
            assert torch.equal(got, same)
            for what, x in (("tensor", got), ("plain", other)):
                err = np.abs(to_numpy64(x[0, h]) - r)
                assert np.all(err <= 2.0 ** -8 * np.abs(r) + 1e-5 * np.abs(r).max()), (name, what, T, float(err.max()))


def test_rows_of_any_norm():
    """Rows scaled by powers of two (exact in bf16) whose squared norms fp32 holds, though not their products: out does not
    change, and the gradients are those of the unscaled rows divided by the powers, to the bit."""
    import torch
    T = 577
    w = inputs.gaussian_workload("bwdx_norm", "bf16", 1, 2, T, 64, 64, 64, 6900)
    q, k, v = dev_tensors(w)
    g, _ = dout_for(w, 6)
    k[0, 0, [0, 130]] = 0
    q[0, 1, 7] = 0
    base = kb.kata_bwd_chunked(q, k, v, g)
    gen = torch.Generator(device="cuda").manual_seed(1)
    for lo, hi in ((-55, -50), (40, 55), (-55, 55)):
        fq, fk = (torch.exp2(torch.randint(lo, hi, (1, 2, T, 1), device="cuda", generator=gen).float()) for _ in range(2))
        qs, ks = (q.float() * fq).bfloat16(), (k.float() * fk).bfloat16()
        dq, dk, dv = kb.kata_bwd_chunked(qs, ks, v, g)
        torch.cuda.synchronize()
        assert kb.kata_last_impl() == kb.KATA_IMPL_TENSOR
        for name, got, ref in (("dq", dq.float() * fq, base[0]), ("dk", dk.float() * fk, base[1]), ("dv", dv.float(), base[2])):
            assert torch.equal(got, ref.float()), (name, lo, hi)


@pytest.mark.parametrize("B,H,T", [(8, 16, 513), (8, 16, 577), (3, 40, 700)])
def test_many_heads(B, H, T):
    """Several items per CTA of both kernels (five to six tiles of 128 rows per head and 120 or 128 heads: four to five items each):
    the hand-over from one item to the next.  First, middle and last heads against the oracle, and the same bits every time."""
    import torch
    w = inputs.gaussian_workload(f"bwdx_heads_{B}_{H}_{T}", "bf16", B, H, T, 64, 64, 64, 6200 + T)
    q, k, v = dev_tensors(w)
    g = torch.from_numpy(inputs.normal(3, 8, B * H * T * 64).reshape(B, H, T, 64)).to(torch.bfloat16).cuda()
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    grads = kb.kata_bwd_chunked(q, k, v, g, device_status=st)
    for _ in range(10):
        assert all(torch.equal(a, b) for a, b in zip(grads, kb.kata_bwd_chunked(q, k, v, g, device_status=st)))
    torch.cuda.synchronize()
    assert kb.kata_last_impl() == kb.KATA_IMPL_TENSOR and int(st.item()) == 0
    for b, h in ((0, 0), (B // 2, H // 3), (B - 1, H - 1)):
        refs = ko.kata_quadratic_bwd(w.q_ref[b, h], w.k_ref[b, h], w.v_ref[b, h], to_numpy64(g[b, h]))
        for name, got, r in zip(("dq", "dk", "dv"), grads, refs):
            err = np.abs(to_numpy64(got[b, h]) - r)
            assert np.all(err <= 2.0 ** -8 * np.abs(r) + 1e-5 * np.abs(r).max()), (name, b, h, float(err.max()))


@pytest.mark.parametrize("T,impl", [(16384, "tensor"), (16385, "simt"), (511, "simt"), (512, "tensor")])
def test_ends_of_the_range(T, impl):
    """The last length of either route and the first of the other, sampled rows (dq row by row; dk and dv with every query
    behind the key) to the same bound."""
    import torch
    w = inputs.gaussian_workload(f"bwdx_end_{T}", "bf16", 1, 1, T, 64, 64, 64, 6300 + T)
    q, k, v = dev_tensors(w)
    g, g_ref = dout_for(w, 7)
    grads = kb.kata_bwd_chunked(q, k, v, g)
    torch.cuda.synchronize()
    assert kb.kata_last_impl() == (kb.KATA_IMPL_TENSOR if impl == "tensor" else kb.KATA_IMPL_SIMT)
    rows = [0, 1, 127, 128, T // 2, T - 129, T - 2, T - 1]
    refs = ko.kata_bwd_rows(w.q_ref[0, 0], w.k_ref[0, 0], w.v_ref[0, 0], g_ref[0, 0], rows, rows)
    for name, got, r in zip(("dq", "dk", "dv"), grads, refs):
        full = to_numpy64(got[0, 0])
        err = np.abs(full[rows] - r)
        assert np.all(err <= 2.0 ** -8 * np.abs(r) + 1e-5 * np.abs(full).max()), (name, T, float(err.max()))


@pytest.mark.parametrize("fn,T", [("kata_bwd_quadratic", 300), ("kata_bwd_chunked", 600)])
@pytest.mark.parametrize("which", [0, 1, 2])
def test_gradients_aligned_to_16_bytes_only(fn, T, which):
    """Gradient rows leave 32 bytes at a time where all three tensors allow it, 16 otherwise: the same bits."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(T)
    x = [torch.randn(1, 3, T, 64, device="cuda", generator=gen).bfloat16() for _ in range(4)]
    want = getattr(kb, fn)(*x)
    out = [torch.empty(3 * T * 64 + 8, dtype=torch.bfloat16, device="cuda")[8 * (i == which):][:3 * T * 64].view(1, 3, T, 64) for i in range(3)]
    assert out[which].data_ptr() % 32 == 16
    getattr(kb, fn)(*x, *out)
    assert all(torch.equal(a, b) for a, b in zip(want, out))
