"""GPU parity of the fp32 chunked form on narrow rows (chunk states of 256 tokens, blocks of 32 or 64 queries, tiles of 32
keys): edges of the blocks, of the chunks and of the lengths that run as one chunk."""
import pytest

from paper_2607_17419_b200 import binding as kb
from paper_2607_17419_b200 import inputs

from helpers import check, dev_tensors, oracle_full, to_numpy64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dk,dv", [(16, 16), (16, 32), (32, 16), (32, 32)])
@pytest.mark.parametrize("T", [1, 31, 33, 64, 65, 1024, 1025, 1536, 1537, 2049, 2111])
def test_simt_attend(dk, dv, T):
    import torch
    w = inputs.gaussian_workload(f"sa_{dk}_{dv}_{T}", "f32", 1, 2, T, dk, dv, 64, 7000 + T + dk)
    for arr in (w.k_ref, w.k_dev):
        arr[0, 0, [0, T - 1]] = 0               # a first key of zero: normaliser 0, output 0
    q, k, v = dev_tensors(w)
    o = kb.kata_fwd_chunked(q, k, v)
    torch.cuda.synchronize()
    assert kb.kata_last_impl() == kb.KATA_IMPL_SIMT
    assert kb.kata_last_launch_count() == (3 if T > (1024 if dk == 16 else 1536) else 1)
    assert torch.equal(o, kb.kata_fwd_chunked(q, k, v)), "fixed summation order"
    assert torch.all(o[0, 0, 0] == 0)
    for (b, h), r in oracle_full(w).items():
        check(to_numpy64(o)[b, h], r, "f32", f"T={T} d={dk},{dv} head {h}")


@pytest.mark.parametrize("dk,T", [(16, 900), (16, 1200), (32, 1700)])
@pytest.mark.parametrize("scale", [1e-21, 1e18])
def test_queries_of_any_norm(dk, T, scale):
    """The norm of a query cancels: queries whose squares leave the range of fp32 give the answer of the unscaled ones (their
    squared norms, 1.6e-41 and up, do not leave it)."""
    import torch
    w = inputs.gaussian_workload(f"sa_norm_{dk}_{T}", "f32", 1, 2, T, dk, dk, 64, 7100 + T)
    q, k, v = dev_tensors(w)
    o = kb.kata_fwd_chunked(q * scale, k, v)
    torch.cuda.synchronize()
    for (b, h), r in oracle_full(w).items():
        check(to_numpy64(o)[b, h], r, "f32", f"T={T} d={dk} scale {scale} head {h}")


@pytest.mark.parametrize("dk,dv", [(16, 16), (16, 32), (32, 16), (32, 32)])
@pytest.mark.parametrize("T", [65, 511, 513, 1025, 1537, 2049])
def test_two_queries_per_lane(dk, dv, T):
    """Enough heads that blocks of 64 queries outnumber the SMs: two queries per lane, with one chunk and with several."""
    import torch
    H = 80
    assert (T + 63) // 64 * H > 148
    w = inputs.gaussian_workload(f"sa2_{dk}_{dv}_{T}", "f32", 1, H, T, dk, dv, 64, 7200 + T + dk)
    q, k, v = dev_tensors(w)
    o = kb.kata_fwd_chunked(q, k, v)
    torch.cuda.synchronize()
    assert kb.kata_last_impl() == kb.KATA_IMPL_SIMT
    one_chunk = 1536 if dk == 32 else 1024 if H * T <= 16384 else 512
    assert kb.kata_last_launch_count() == (3 if T > one_chunk else 1)
    assert torch.equal(o, kb.kata_fwd_chunked(q, k, v)), "fixed summation order"
    for (b, h), r in oracle_full(w, heads=[(0, 0), (0, H // 2), (0, H - 1)]).items():
        check(to_numpy64(o[b, h]), r, "f32", f"T={T} d={dk},{dv} head {h}")


@pytest.mark.parametrize("dk,dv,H,T", [(16, 16, 1, 7), (16, 16, 1, 1001), (16, 16, 2, 575), (16, 16, 3, 801), (16, 16, 5, 1024), (16, 16, 9, 513),
                                       (16, 16, 1, 2335), (16, 32, 1, 1000), (32, 16, 5, 400), (32, 32, 1, 9), (32, 32, 1, 1153), (32, 32, 2, 1160),
                                       (32, 32, 5, 900), (32, 32, 9, 1100), (32, 32, 1, 1700)])
def test_clusters_of_ctas_per_block(dk, dv, H, T):
    """Few blocks: two, four or eight CTAs share the keys of a block in tiles of 8, and the rows of its state; both sides of the
    counts of blocks at which the number changes."""
    import torch
    w = inputs.gaussian_workload(f"sac_{dk}_{dv}_{H}_{T}", "f32", 1, H, T, dk, dv, 64, 7300 + T + dk + H)
    for arr in (w.k_ref, w.k_dev):
        arr[0, 0, [0, T - 1]] = 0
    q, k, v = dev_tensors(w)
    o = kb.kata_fwd_chunked(q, k, v)
    torch.cuda.synchronize()
    assert kb.kata_last_impl() == kb.KATA_IMPL_SIMT
    assert torch.equal(o, kb.kata_fwd_chunked(q, k, v)), "fixed summation order"
    assert torch.all(o[0, 0, 0] == 0)
    for (b, h), r in oracle_full(w, heads=[(0, 0), (0, H - 1)]).items():
        check(to_numpy64(o)[b, h], r, "f32", f"T={T} d={dk},{dv} head {h}")
