"""Performance cases: the calls a program that uses this library makes, over the range of sizes it makes them at.

Every case is a plain dict; ``prepare`` makes its inputs on the GPU from the seed, ``run`` is one pass through the public
entry points of ``paper_2607_17419_b200.binding``, ``work`` the bytes and operations the result cannot do without and
``tolerance`` how far two correct implementations of the same precision may be apart.

Keys of a case: ``path`` (which calls), ``B, H, T, d`` (d_k = d_v = d), ``dtype``, ``groups`` (blocks of the feature map),
and per path ``inter`` (how the chunk axis is walked), ``state`` (final state exported), ``layout`` (of a state),
``data`` (distribution of the inputs).
"""
import math

import torch

from paper_2607_17419_b200 import binding as kb

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
INTER = {"sequential": kb.KATA_SEQUENTIAL, "scan": kb.KATA_SCAN, "auto": kb.KATA_INTER_AUTO}
LAYOUT = {"direct": kb.KATA_LAYOUT_DIRECT, "packed": kb.KATA_LAYOUT_PACKED}


def _case(name, path, B, H, T, d, dtype="bf16", groups=1, inter="sequential", state=False, layout="direct", data="gauss"):
    return {"name": name, "path": path, "B": B, "H": H, "T": T, "d": d, "dtype": dtype, "groups": groups, "inter": inter,
            "state": state, "layout": layout, "data": data}


def listed():
    return [
        # one token of one sequence in an interactive session: latency of a small memory-bound step
        _case("decode_b1", "decode", 1, 16, 1, 64),
        # one token of a serving batch of sixteen sequences: the state streams from memory and back
        _case("decode_b16", "decode", 16, 16, 1, 64),
        # the tiny fp32 configuration: a small model in full precision, few launches of little work
        _case("chunked_tiny_f32", "chunked", 1, 2, 512, 16, dtype="f32"),
        # prompt processing before decoding: ragged length, the state after the last token is handed over
        _case("prefill_state", "chunked", 2, 16, 3001, 64, state=True),
        # a layer of a 340M-parameter model at its training shape
        _case("chunked_layer", "chunked", 8, 16, 4096, 64),
        # long context, one sequence: the headline workload
        _case("chunked_long", "chunked", 1, 16, 131072, 64),
        # long context with few heads on this GPU (heads sharded over others), blockwise map, the library picks the form
        _case("chunked_few_heads_m2", "chunked", 1, 4, 50001, 64, groups=2, inter="auto"),
        # recall workload: narrow heads, repeated keys, one-hot values
        _case("chunked_recall", "chunked", 16, 8, 2048, 32, data="recall"),
        # the definition evaluated tile by tile, for sequences of ordinary length
        _case("quadratic", "quadratic", 4, 16, 4096, 64),
        # a training step of one layer: forward and gradients
        _case("train_quadratic", "train_quadratic", 4, 16, 4096, 64),
        # a training step with the linear-time gradients
        _case("train_chunked", "train_chunked", 1, 16, 8192, 64),
        # already-mapped first-order features, one long sequence, chunk size 128
        _case("scan_order1", "order1", 1, 16, 131072, 64, data="nonneg"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges that the listed ones stand for."""
    path = rng.choice(["decode", "chunked", "chunked", "quadratic", "train_quadratic", "train_chunked", "order1"])
    c = _case("", path, 1, 1, 1, 64)
    del c["name"]
    if path == "decode":
        c["B"], c["H"] = _log_int(rng, 1, 24), rng.choice([4, 8, 12, 16])
        c["groups"] = rng.choice([1, 1, 2])
        c["layout"] = rng.choice(["direct", "packed"])
        c["dtype"] = rng.choice(["bf16", "bf16", "f32"])
        return c
    if path == "order1":
        tokens = _log_int(rng, 1 << 17, 1 << 21)            # tokens x heads
        c["T"] = _log_int(rng, 1024, 131072)
        c["data"] = "nonneg"
    elif path == "chunked":
        f32 = rng.random() < 0.2
        c["dtype"] = "f32" if f32 else "bf16"
        c["d"] = rng.choice([16, 32]) if f32 else rng.choice([64, 64, 64, 32])
        if c["d"] == 64:
            c["groups"] = rng.choice([1, 1, 1, 2, 4])
            c["state"] = rng.random() < 0.25
        c["layout"] = rng.choice(["direct", "packed"])
        if not c["state"]:
            c["inter"] = rng.choice(["sequential", "sequential", "auto"])
        tokens = _log_int(rng, 1 << 10, 1 << 18) if f32 else _log_int(rng, 1 << 14, 1 << 21)
        c["T"] = _log_int(rng, 256, 16384 if f32 else 131072)
        c["data"] = "recall" if c["d"] == 32 and not f32 else "gauss"
    elif path == "quadratic":
        tokens = _log_int(rng, 1 << 14, 1 << 19)
        c["T"] = _log_int(rng, 256, 8192)
        c["groups"] = rng.choice([1, 1, 2])
    elif path == "train_quadratic":
        tokens = _log_int(rng, 1 << 14, 1 << 19)
        c["T"] = _log_int(rng, 256, 8192)
        c["groups"] = rng.choice([1, 1, 2])
    else:                                                   # train_chunked
        tokens = _log_int(rng, 1 << 12, 1 << 17)
        c["T"] = _log_int(rng, 512, 8192)
    heads = max(1, tokens // c["T"])
    c["T"] = min(c["T"], tokens)
    c["H"] = min(heads, 16)
    c["B"] = max(1, heads // c["H"])
    return c


def _inputs(case, gen):
    B, H, T, d = case["B"], case["H"], case["T"], case["d"]
    dt = DTYPES[case["dtype"]]

    def normal(*shape):
        return torch.randn(*shape, device="cuda", generator=gen)

    if case["data"] == "recall":
        # keys from a dictionary of 256 unit vectors per head, one-hot values, queries = earlier keys plus noise
        dic = normal(B * H, 256, d)
        dic = dic / dic.norm(dim=-1, keepdim=True)
        ids = torch.randint(256, (B * H, T), device="cuda", generator=gen)
        k = torch.gather(dic, 1, ids[:, :, None].expand(-1, -1, d))
        v = torch.zeros(B * H, T, d, device="cuda")
        v.scatter_(2, torch.randint(d, (B * H, T, 1), device="cuda", generator=gen), 1.0)
        src = (torch.rand(B * H, T, device="cuda", generator=gen) * torch.arange(1, T + 1, device="cuda")).long()
        src = torch.minimum(src, torch.arange(T, device="cuda"))
        q = torch.gather(k, 1, src[:, :, None].expand(-1, -1, d)) + 0.1 * normal(B * H, T, d)
        return tuple(x.reshape(B, H, T, d).to(dt) for x in (q, k, v))
    q, k, v = (normal(B, H, T, d) for _ in range(3))
    if case["data"] == "nonneg":
        q, k = q.abs(), k.abs()
    return q.to(dt), k.to(dt), v.to(dt)


def _features(x, case):
    """Rows of a state for unit rows x [.., d] in the exported layouts: direct, or the packed upper triangle."""
    g = case["groups"]
    m = x.shape[-1] // g
    xb = x.reshape(*x.shape[:-1], g, m)
    full = xb[..., :, None] * xb[..., None, :]
    if case["layout"] == "direct":
        return full.reshape(*x.shape[:-1], g * m * m)
    a, b = torch.triu_indices(m, m, device=x.device)
    scale = torch.where(a == b, 1.0, math.sqrt(2.0))
    return (full[..., a, b] * scale).reshape(*x.shape[:-1], -1)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    state = {"case": dict(case)}
    q, k, v = _inputs(case, gen)
    if case["path"] == "decode":
        # the state of a sequence that has seen 256 tokens
        B, H, d = case["B"], case["H"], case["d"]
        n = kb.decode_n_psi(d, state_layout=LAYOUT[case["layout"]], feature_groups=case["groups"])
        S = torch.empty(B, H, n, d, device="cuda")
        Z = torch.empty(B, H, n, device="cuda")
        for b in range(B):
            past = torch.randn(H, 256, d, device="cuda", generator=gen)
            psi = _features(past / past.norm(dim=-1, keepdim=True), case)
            S[b] = psi.transpose(1, 2) @ torch.randn(H, 256, d, device="cuda", generator=gen)
            Z[b] = psi.sum(1)
        q, k, v = q[:, :, 0].contiguous(), k[:, :, 0].contiguous(), v[:, :, 0].contiguous()
        state.update(S=S, Z=Z)
    elif case["state"]:
        n = kb.decode_n_psi(case["d"], state_layout=LAYOUT[case["layout"]], feature_groups=case["groups"])
        state.update(S=torch.empty(case["B"], case["H"], n, case["d"], device="cuda"),
                     Z=torch.empty(case["B"], case["H"], n, device="cuda"))
    if case["path"].startswith("train"):
        state["dout"] = torch.randn(v.shape, device="cuda", generator=gen).to(v.dtype)
    state.update(q=q, k=k, v=v)
    return state


def run(state):
    case, q, k, v = state["case"], state["q"], state["k"], state["v"]
    path, g = case["path"], case["groups"]
    if path == "decode":
        out = kb.kata_decode_step(q, k, v, state["S"], state["Z"], feature_groups=g, state_layout=LAYOUT[case["layout"]])
        return out, state["S"], state["Z"]
    if path == "chunked":
        if case["state"]:
            out = kb.kata_fwd_chunked(q, k, v, feature_groups=g, state_layout=LAYOUT[case["layout"]], s_pre=state["S"],
                                      z_pre=state["Z"])
            return out, state["S"], state["Z"]
        return kb.kata_fwd_chunked(q, k, v, feature_groups=g, inter_chunk=INTER[case["inter"]])
    if path == "quadratic":
        return kb.kata_fwd_quadratic(q, k, v, feature_groups=g)
    if path == "train_quadratic":
        out = kb.kata_fwd_quadratic(q, k, v, feature_groups=g)
        return (out, *kb.kata_bwd_quadratic(q, k, v, state["dout"], feature_groups=g))
    if path == "train_chunked":
        out = kb.kata_fwd_chunked(q, k, v)
        return (out, *kb.kata_bwd_chunked(q, k, v, state["dout"]))
    return kb.kata_chunk_state_scan(q, k, v, feature_order=1, C=128)


def work(case):
    """Inputs read once, outputs written once; the operations of the cheaper of the two exact forms."""
    B, H, T, d, g = case["B"], case["H"], case["T"], case["d"], case["groups"]
    heads, eb = B * H, 4 if case["dtype"] == "f32" else 2
    m = d // g
    packed = g * m * (m + 1) // 2                           # independent features of the symmetric lift
    if case["path"] == "decode":
        n = kb.decode_n_psi(d, state_layout=LAYOUT[case["layout"]], feature_groups=g)
        return {"bytes": heads * (2 * n * (d + 1) * 4 + 4 * d * eb), "flops": heads * 4 * n * (d + 1)}
    io = heads * T * d * eb
    if case["path"] == "order1":
        return {"bytes": 4 * io, "flops": heads * T * 4 * d * (d + 1)}
    pairs = T * (T + 1) // 2
    update = T * 2 * packed * (d + 1)                       # one pass of feature times value, or of state times feature
    fwd = heads * min(pairs * 4 * d, 2 * update)
    bwd = heads * min(pairs * 10 * d, 5 * update)
    if case["path"].startswith("train"):
        return {"bytes": 11 * io, "flops": fwd + bwd}       # q, k, v, out; q, k, v, dout, dq, dk, dv
    out = {"bytes": 4 * io, "flops": fwd}
    if case["state"]:
        n = kb.decode_n_psi(d, state_layout=LAYOUT[case["layout"]], feature_groups=g)
        out = {"bytes": 4 * io + heads * n * (d + 1) * 4, "flops": heads * min(pairs * 4 * d + update, 2 * update)}
    return out


def tolerance(case):
    """About four times the relative 2-norm error against the same path in 64 bits, measured over the listed cases and two
    dozen drawn ones (largest seen: fp32 4.0e-7 at T = 3312, growing with the length; bf16 decode output 1.7e-3 and
    first-order output 2.0e-3, both little more than the rounding of the result; bf16 tensor-core outputs, states and
    gradients 3.4e-3: weights and state pass through bf16 operands)."""
    if case["dtype"] == "f32":
        return {"rel": 4e-6}
    return {"rel": 8e-3 if case["path"] in ("decode", "order1") else 1.3e-2}
