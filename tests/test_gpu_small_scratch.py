"""Calls with less scratch than kata_workspace_bytes asks for, that kernels with a smaller need serve: a state handed in or out,
fp32 rows, and the scan form's scratch under inter_chunk = AUTO.  They run, on those kernels, and give the same function."""
import pytest

from paper_2607_17419_b200 import binding as kb
from paper_2607_17419_b200 import inputs

from helpers import check, dev_tensors, oracle_rows, sample_picks, to_numpy64

import numpy as np

pytestmark = pytest.mark.gpu


class Capped(kb.Workspace):
    def __init__(self, cap):
        super().__init__()
        self.cap = cap

    def get(self, nbytes, device):
        assert nbytes > self.cap
        return super().get(self.cap, device)


def published(H, T):
    """Scratch of the sequential form with the state split over nine CTAs per head, which callers may have sized for."""
    al = lambda x: (x + 255) // 256 * 256
    nt = (T + 127) // 128
    return al((H * nt + 1) * 4) + al(H * T * 128) + al(H * T * 2) + al(H * 9 * nt * (128 * 128 + 128 * 8))


def scan_bytes(H, T):
    o = kb.make_opts(kb.KATA_BF16, inter_chunk=kb.KATA_SCAN)
    return kb.kata_workspace_bytes(kb.KATA_FN_CHUNKED, 1, H, T, 64, 64, 64, o)


@pytest.mark.parametrize("what,dtype,H,T,d,launches", [
    ("state", "bf16", 2, 1500, 64, 1), ("state", "bf16", 40, 300, 64, 1), ("plain", "f32", 2, 2000, 16, 1), ("plain", "f32", 3, 1700, 32, 1),
    ("published", "bf16", 1, 9000, 64, 4), ("auto", "bf16", 3, 30000, 64, None), ("published-auto", "bf16", 1, 1025, 64, 2)])
def test_small_scratch(what, dtype, H, T, d, launches):
    import torch
    w = inputs.gaussian_workload(f"small_{what}_{H}_{T}_{d}", dtype, 1, H, T, d, d, 64, 7300 + T)
    q, k, v = dev_tensors(w)
    kw = {}
    if what == "state":
        n = kb.decode_n_psi(d)
        kw = dict(s_pre=torch.empty(1, H, n, d, device="cuda"), z_pre=torch.empty(1, H, n, device="cuda"))
    cap = {"published": published, "published-auto": published, "auto": scan_bytes}.get(what, lambda H, T: 0)(H, T)
    if "auto" in what:
        kw["inter_chunk"] = kb.KATA_INTER_AUTO
    o = kb.kata_fwd_chunked(q, k, v, workspace=Capped(cap), **kw)
    torch.cuda.synchronize()
    if launches is not None:
        assert kb.kata_last_launch_count() == launches
    picks = sample_picks(w, 64, T)
    gpu = to_numpy64(o)
    check(np.stack([gpu[b, h, t] for b, h, t in picks]), oracle_rows(w, picks), dtype, f"{what} T={T} H={H}")
    if what == "state":                          # and the next piece, from that state, without scratch either
        o2 = kb.kata_fwd_chunked(q, k, v, workspace=Capped(0), s_init=kw["s_pre"], z_init=kw["z_pre"])
        full = kb.kata_fwd_chunked(q, k, v, s_init=kw["s_pre"], z_init=kw["z_pre"])
        torch.cuda.synchronize()
        diff = (o2.float() - full.float()).norm() / full.float().norm()
        assert float(diff) <= 2e-2


@pytest.mark.parametrize("H,T", [(50, 8192), (1, 16384), (2, 4097)])
def test_first_order_with_the_scratch_of_one_pass(H, T):
    """Sizes that are walked in groups now and were one pass per head: the scratch of one pass is still enough, and less is not."""
    import torch
    q, k = (torch.rand(1, H, T, 64, device="cuda").bfloat16() for _ in range(2))
    v = torch.randn(1, H, T, 64, device="cuda").bfloat16()
    o = kb.make_opts(kb.KATA_BF16, feature_order=1)
    one = kb.make_opts(kb.KATA_BF16, feature_order=1, scan_group=10 ** 6)
    need, least = (kb.kata_workspace_bytes(kb.KATA_FN_CHUNK_STATE_SCAN, 1, H, T, 64, 64, 128, x) for x in (o, one))
    assert kb.kata_scan_plan(kb.KATA_FN_CHUNK_STATE_SCAN, 1, H, T, 64, 64, 128, o)[0] > 1 and need > least > 0
    want = kb.kata_chunk_state_scan(q, k, v, feature_order=1, C=128, scan_group=10 ** 6)

    class Fixed:
        def __init__(self, n):
            self.buf = torch.empty(n, dtype=torch.uint8, device="cuda")

        def get(self, nbytes, device):
            return self.buf.data_ptr(), self.buf.numel()

    got = kb.kata_chunk_state_scan(q, k, v, feature_order=1, C=128, workspace=Fixed(least))
    assert torch.equal(got, want), "one pass per head is what runs"          # (its outputs: test_gpu_order1_tensor.py)
    own = kb.kata_chunk_state_scan(q, k, v, feature_order=1, C=128)
    assert torch.all((own.double() - want.double()).norm(dim=-1) <= 2e-2 * want.double().norm(dim=-1))
    with pytest.raises(kb.KataError) as e:
        kb.kata_chunk_state_scan(q, k, v, feature_order=1, C=128, workspace=Fixed(least - 256))
    assert e.value.status == kb.KATA_ERR_WORKSPACE_TOO_SMALL
