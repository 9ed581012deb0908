"""GPU parity of the chunk-state and attend kernels (bf16): edges of chunks (512 or 1024 tokens), of blocks of 256 queries
and of the segments of the chunk axis, state in and out, one and several segments, narrow rows.

Tolerances: outputs as everywhere (2e-2).  Final state: operands are products of bf16 entries rounded twice (2^-8 each,
signs at random over the sum), so max |s - ref| <= 2e-2 of the largest entry."""
import numpy as np
import pytest

from oracle import kata_oracle as ko
from paper_2607_17419_b200 import binding as kb
from paper_2607_17419_b200 import inputs

from helpers import check, dev_tensors, oracle_full, oracle_rows, sample_picks, to_numpy64

pytestmark = pytest.mark.gpu


def feature_of(g, layout="psd_direct"):
    return layout if g == 1 else f"{layout}:g{g}"


# the smallest lengths that run as chunks without a state, and a few edges above them
@pytest.mark.parametrize("g,H,T,d", [(1, 1, 7169, 64), (1, 17, 7425, 64), (1, 2, 8192, 32), (2, 1, 3073, 64), (2, 30, 4097, 64),
                                     (4, 1, 1537, 64), (4, 2, 2048, 64), (4, 50, 2049, 64)])
def test_chunked_without_state(g, H, T, d):
    import torch
    w = inputs.gaussian_workload(f"chunks_{g}_{H}_{T}_{d}", "bf16", 1, H, T, d, d, 64, 5100 + T + g)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    q, k, v = dev_tensors(w)
    o = kb.kata_fwd_chunked(q, k, v, feature_groups=g, device_status=st)
    torch.cuda.synchronize()
    assert kb.kata_last_impl() == kb.KATA_IMPL_TENSOR and int(st.item()) == 0
    assert kb.kata_last_launch_count() in (3, 4), "key scales, chunk states (and their segments' sums), outputs"
    o2 = kb.kata_fwd_chunked(q, k, v, feature_groups=g)
    torch.cuda.synchronize()
    assert torch.equal(o, o2), "fixed summation order"
    picks = sample_picks(w, 64, T) + [(0, H - 1, t) for c in (512, 1024, 1536, 2048, T // 256 * 256) for t in (c - 1, c, c + 127, c + 128)
                                      if t < T]
    gpu = to_numpy64(o)
    check(np.stack([gpu[b, h, t] for b, h, t in picks]), oracle_rows(w, picks, feature_of(g)), "bf16", f"M{g} T={T} H={H} d={d}")


# rows of up to 32 entries: four of the eight runs of features, two block pairs of the last slice empty
@pytest.mark.parametrize("H,T,dk,dv", [(1, 4353, 32, 32), (64, 3601, 32, 32), (2, 5121, 16, 64), (3, 4608, 32, 64), (2, 4400, 16, 16)])
def test_narrow_rows(H, T, dk, dv):
    import torch
    w = inputs.gaussian_workload(f"narrow_{H}_{T}_{dk}_{dv}", "bf16", 1, H, T, dk, dv, 64, 5200 + T)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    o = kb.kata_fwd_chunked(*dev_tensors(w), device_status=st)
    torch.cuda.synchronize()
    assert kb.kata_last_impl() == kb.KATA_IMPL_TENSOR and int(st.item()) == 0
    assert kb.kata_last_launch_count() in (3, 4)
    picks = sample_picks(w, 64, T) + [(0, H - 1, t) for c in (512, 1024, 2048, 3072, 3584) for t in (c - 1, c, c + 127, c + 128) if t < T]
    gpu = to_numpy64(o)
    check(np.stack([gpu[b, h, t] for b, h, t in picks]), oracle_rows(w, picks, "psd_direct"), "bf16", f"narrow {dk}x{dv} T={T} H={H}")


@pytest.mark.parametrize("layout", ["psd_direct", "psd_packed"])
@pytest.mark.parametrize("g,H,cuts", [(1, 2, (513, 1537)), (1, 20, (100, 612)), (2, 3, (1024, 1025)), (4, 2, (700, 2300))])
def test_state_in_and_out(layout, g, H, cuts):
    """Two pieces, the state handed from one to the other in place, outputs and final state against the definition."""
    import torch
    T, d = cuts[1], 64
    w = inputs.gaussian_workload(f"hand_{g}_{H}_{T}", "bf16", 1, H, T, d, d, 64, 5300 + T + g)
    q, k, v = dev_tensors(w)
    code = kb.KATA_LAYOUT_PACKED if layout == "psd_packed" else kb.KATA_LAYOUT_DIRECT
    n = kb.decode_n_psi(d, 2, code, g)
    S, Z = torch.zeros(1, H, n, d, device="cuda"), torch.zeros(1, H, n, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    outs, a = [], 0
    for b in cuts:
        kw = dict(s_pre=S, z_pre=Z, state_layout=code, feature_groups=g, device_status=st)
        if a > 0:
            kw.update(s_init=S, z_init=Z)
        outs.append(kb.kata_fwd_chunked(*(x[:, :, a:b].contiguous() for x in (q, k, v)), **kw))
        assert kb.kata_last_impl() == kb.KATA_IMPL_TENSOR
        a = b
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    gpu = to_numpy64(torch.cat(outs, dim=2))
    for h in sorted({0, H - 1}):
        r = ko.kata_quadratic(w.q_ref[0, h], w.k_ref[0, h], w.v_ref[0, h], feature_of(g))[0]
        check(gpu[0, h], r, "bf16", f"M{g} pieces {cuts} head {h}")
        f = ko.apply_feature(w.k_ref[0, h], feature_of(g, layout))
        for got, ref in ((S, f.T @ w.v_ref[0, h]), (Z, f.sum(axis=0))):
            assert np.max(np.abs(to_numpy64(got[0, h]) - ref)) <= 2e-2 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("layout", ["psd_direct", "psd_packed"])
@pytest.mark.parametrize("g,H,T", [(1, 2, 700), (1, 20, 1500), (2, 3, 1500), (4, 40, 900)])
def test_exported_state_rounding(layout, g, H, T):
    """A term psi_f(k_t) v_t of the exported state is rounded to bf16 twice (r k_b and its product with k_a), as on the
    streaming kernel.  One rounding is off by 2^-8 / sqrt(3) x rms(1 / m) = 1.66e-3 (m, the mantissa, spread over its
    logarithm), independently from term to term: |S - ref| = 1.66e-3 sqrt(n) sqrt(sum |psi_t|^2 |v_t|^2) for n roundings.
    The bound lies at n = 2.45, between two and three."""
    import torch
    w = inputs.gaussian_workload(f"round_{g}_{H}_{T}", "bf16", 1, H, T, 64, 64, 64, 5400 + T + g)
    code = kb.KATA_LAYOUT_PACKED if layout == "psd_packed" else kb.KATA_LAYOUT_DIRECT
    n = kb.decode_n_psi(64, 2, code, g)
    S, Z = torch.empty(1, H, n, 64, device="cuda"), torch.empty(1, H, n, device="cuda")
    kb.kata_fwd_chunked(*dev_tensors(w), s_pre=S, z_pre=Z, state_layout=code, feature_groups=g)
    torch.cuda.synchronize()
    assert kb.kata_last_impl() == kb.KATA_IMPL_TENSOR and kb.kata_last_launch_count() >= 3
    eps = 2.0 ** -8 / np.sqrt(3.0) * np.sqrt(3.0 / (8.0 * np.log(2.0)))
    for h in (0, H - 1):
        v = w.v_ref[0, h]
        f = ko.apply_feature(w.k_ref[0, h], feature_of(g, layout))
        p2 = (f * f).sum(axis=1)
        for got, ref, terms in ((S, f.T @ v, p2 * (v * v).sum(axis=1)), (Z, f.sum(axis=0), p2)):
            err = np.linalg.norm(to_numpy64(got[0, h]) - ref)
            assert err <= eps * np.sqrt(2.45 * terms.sum()), (g, layout, h, err / (eps * np.sqrt(terms.sum())))


@pytest.mark.parametrize("g,H,T,state", [(1, 20, 600, True), (2, 3, 1000, False), (2, 20, 400, True), (4, 5, 1200, False)])
def test_weight_rounding(g, H, T, state):
    """Calls of one chunk with a state handed out or with feature groups: a weight r s^2 is rounded to bf16 once, so with the
    1.66e-3 of a rounding (above) an output row is off by 1.66e-3 sqrt(n sum (w / D)^2 |v - o|^2 + |o|^2), n = 1, the second
    term being the rounding of the result.  The bound lies at n = 2; s^2, r and their product rounded in turn are n = 3."""
    import torch
    w = inputs.gaussian_workload(f"weights_{g}_{H}_{T}", "bf16", 1, H, T, 64, 64, 64, 5500 + T + g)
    n = kb.decode_n_psi(64, 2, kb.KATA_LAYOUT_DIRECT, g)
    kw = dict(s_pre=torch.empty(1, H, n, 64, device="cuda"), z_pre=torch.empty(1, H, n, device="cuda")) if state else {}
    o = kb.kata_fwd_chunked(*dev_tensors(w), feature_groups=g, **kw)
    torch.cuda.synchronize()
    assert kb.kata_last_impl() == kb.KATA_IMPL_TENSOR and kb.kata_last_launch_count() == (3 if state else 2)
    eps = 2.0 ** -8 / np.sqrt(3.0) * np.sqrt(3.0 / (8.0 * np.log(2.0)))
    err = near = far = 0.0
    m = 64 // g
    for h in (0, H - 1):
        q, k, v = w.q_ref[0, h], w.k_ref[0, h], w.v_ref[0, h]
        p = sum((q[:, a:a + m] @ k[:, a:a + m].T) ** 2 for a in range(0, 64, m)) / (k * k).sum(axis=1)
        p = np.tril(p)
        p /= p.sum(axis=1, keepdims=True)
        r = p @ v
        err += ((to_numpy64(o[0, h]) - r) ** 2).sum()
        near += ((p * p) * ((v * v).sum(axis=1)[None, :] - 2 * (r @ v.T) + (r * r).sum(axis=1)[:, None])).sum()
        far += (r * r).sum()
    assert np.sqrt(err) <= eps * np.sqrt(2.0 * near + far), (g, H, T, (err / eps ** 2 - far) / near)


@pytest.mark.parametrize("dk,dv", [(32, 32), (32, 16), (16, 32), (16, 16), (32, 64)])
@pytest.mark.parametrize("H,T", [(1, 129), (2, 777), (40, 1153)])
def test_narrow_values(dk, dv, H, T):
    """Values of up to 32 entries have tiles of 32 columns, wider ones of 64: both halves on a block and the halves sharing its keys,
    the ring of stages past its end (several chunks: test_narrow_rows)."""
    import torch
    w = inputs.gaussian_workload(f"narrow_{dk}_{dv}_{H}_{T}", "bf16", 1, H, T, dk, dv, 64, 5700 + T + dv)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    q, k, v = dev_tensors(w)
    o = kb.kata_fwd_chunked(q, k, v, device_status=st)
    torch.cuda.synchronize()
    assert kb.kata_last_impl() == kb.KATA_IMPL_TENSOR and int(st.item()) == 0
    for (b, h), r in oracle_full(w, heads=[(0, 0), (0, H - 1)]).items():
        check(to_numpy64(o[b, h]), r, "bf16", f"T={T} d={dk},{dv} head {h}")


@pytest.mark.parametrize("H,T,dk,dv,state", [(3, 300, 64, 64, False), (1, 1300, 64, 64, False), (60, 700, 32, 16, False), (2, 2500, 64, 64, True)])
@pytest.mark.parametrize("layout", [kb.KATA_LAYOUT_DIRECT, kb.KATA_LAYOUT_PACKED])
def test_outputs_aligned_to_16_bytes_only(H, T, dk, dv, state, layout):
    """Output and state rows leave 32 bytes at a time where the tensors allow it, 16 otherwise: the same bits."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(T)
    q, k = (torch.randn(1, H, T, dk, device="cuda", generator=gen).bfloat16() for _ in range(2))
    v = torch.randn(1, H, T, dv, device="cuda", generator=gen).bfloat16()
    n = kb.decode_n_psi(dk, state_layout=layout)

    def run(shift):
        out = torch.empty(H * T * dv + 8, dtype=torch.bfloat16, device="cuda")[shift // 2:][:H * T * dv].view(1, H, T, dv)
        kw = {}
        if state:
            kw = {"s_pre": torch.empty(H * n * dv + 4, device="cuda")[shift // 4:][:H * n * dv].view(1, H, n, dv),
                  "z_pre": torch.empty(H * n + 4, device="cuda")[shift // 4:][:H * n].view(1, H, n), "state_layout": layout}
        assert out.data_ptr() % 32 == shift
        return (kb.kata_fwd_chunked(q, k, v, out=out, **kw), *[kw[x] for x in ("s_pre", "z_pre") if x in kw])

    for a, b in zip(run(0), run(16)):
        assert torch.equal(a, b)
