"""Few blocks of 256 queries: the halves of a CTA share out the key tiles of 128 queries.  Odd and even numbers of tiles (a
first block that only one half works on), ragged ends, one and several items per CTA, either side of the rule (148 and 152
blocks, 192 and 200 with groups), feature groups, narrow rows, and the chunked entry's fp32 key scales."""
import numpy as np
import pytest

from oracle import kata_oracle as ko
from paper_2607_17419_b200 import binding as kb
from paper_2607_17419_b200 import inputs

from helpers import check, dev_tensors, to_numpy64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fn", ["kata_fwd_quadratic", "kata_fwd_chunked"])
@pytest.mark.parametrize("g,H,T,d", [(1, 1, 769, 64), (1, 1, 1000, 64), (1, 2, 1153, 64), (1, 37, 1024, 64), (1, 38, 1024, 64),
                                     (2, 1, 257, 64), (2, 3, 513, 64), (2, 48, 1000, 64), (2, 50, 1000, 64), (4, 2, 300, 64), (4, 29, 1200, 64),
                                     (1, 3, 1100, 32), (1, 36, 900, 16)])
def test_split_items(fn, g, H, T, d):
    import torch
    w = inputs.gaussian_workload(f"split_{g}_{H}_{T}_{d}", "bf16", 1, H, T, d, d, 64, 5600 + T + g)
    for arr in (w.k_ref, w.k_dev):
        arr[0, 0, [0, 128]] = 0                 # a first key of zero: normaliser 0, output 0
    q, k, v = dev_tensors(w)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    o = getattr(kb, fn)(q, k, v, feature_groups=g, device_status=st)
    torch.cuda.synchronize()
    assert kb.kata_last_impl() == kb.KATA_IMPL_TENSOR and kb.kata_last_launch_count() == 2 and int(st.item()) == 0
    assert torch.equal(o, getattr(kb, fn)(q, k, v, feature_groups=g)), "fixed summation order"
    assert torch.all(o[0, 0, 0] == 0)
    for h in sorted({0, H // 2, H - 1}):
        r = ko.kata_quadratic(w.q_ref[0, h], w.k_ref[0, h], w.v_ref[0, h], "psd_direct" if g == 1 else f"psd_direct:g{g}")[0]
        check(to_numpy64(o[0, h]), r, "bf16", f"M{g} T={T} H={H} d={d} head {h}")
