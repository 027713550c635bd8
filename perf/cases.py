"""Measured cases of the framework: the work its users have it do, through the public entry points.

Four kinds of pass, over the sizes of this repository's configurations, tests and benchmark:

  prefill   one layer's steered causal attention over the prompts (`seka_attention_fwd`; with several experts
            `seka_attention_fwd_routed`, which forms the routing coefficients in the call)
  edit      the key-editing hook alone, on a key cache (`seka_edit_keys`, in place or into a second tensor)
  decode    one generated token per sequence over the edited cache (`seka_decode_attention`)
  learn     offline learning of the projections of every (layer, KV head) slot (`seka_learn_projections`)

Inputs follow the recipes of `paper_2603_01281_b200/inputs.py` (unit-variance Q, K, V; orthonormal bases; highlighted
spans or short runs), drawn on the device.  What a serving program keeps between calls (bases, gains, shape, workspace,
output buffers) belongs to the state.
"""
import math

import numpy as np
import torch

from paper_2603_01281_b200 import binding

DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}
LEARN_CUT = 32          # columns of U that the learned projectors are formed from (the rank of the 8B configuration)


def _prefill(**kw):
    c = dict(kind="prefill", dtype="bf16", batch=1, seqlen=4096, min_len=0, q_heads=32, kv_heads=8, head_dim=128, rank=32,
             experts=1, mask="spans", highlight=0.10, gain=1.0)
    c.update(kw)
    return c


def _edit(**kw):
    c = dict(kind="edit", dtype="bf16", batch=4, seqlen=4096, min_len=0, q_heads=32, kv_heads=8, head_dim=128, rank=32, experts=1,
             mask="spans", highlight=0.10, gain=-0.4, in_place=True)
    c.update(kw)
    return c


def _decode(**kw):
    c = dict(kind="decode", batch=64, seqlen=4096, min_len=0, q_heads=32, kv_heads=8, head_dim=128)
    c.update(kw)
    return c


def _learn(**kw):
    c = dict(kind="learn", tokens=32768, slots=288, head_dim=128, gamma=0.7)
    c.update(kw)
    return c


def listed():
    return [
        # a toy layer in single precision: what a first try-out or a unit test of a user's model runs; launches count
        _prefill(name="prefill_toy_fp32", dtype="f32", seqlen=256, q_heads=4, kv_heads=4, head_dim=64, rank=8, highlight=0.125, gain=0.5),
        # one short prompt of odd length on the 8B shape: interactive use, a layer is a few tens of microseconds
        _prefill(name="prefill_short_prompt", seqlen=777),
        # one long-context sample of the length the paper's overhead run averages, most of it highlighted
        _prefill(name="prefill_mostly_highlighted", seqlen=4362, highlight=0.70),
        # the headline prefill: a batch of four prompts on the 8B shape, a tenth of the tokens highlighted
        _prefill(name="prefill_batch_8b", batch=4),
        # AdaSEKA on the 8B shape: four experts, coefficients routed in the call
        _prefill(name="prefill_adaseka", batch=2, seqlen=8192, experts=4),
        # long context, odd group size, strong gain: the largest prefill
        _prefill(name="prefill_long_context", seqlen=32768, q_heads=28, kv_heads=4, rank=64, highlight=0.05, gain=2.0),
        # a packed batch of a small model: ragged lengths, short highlighted runs in nearly every key tile
        _prefill(name="prefill_packed", batch=64, seqlen=2048, min_len=256, q_heads=16, kv_heads=16, head_dim=64, rank=16, mask="runs",
                 highlight=0.15),
        # the prompt keys of all 36 layers of an 8B model edited once, in place, before generation
        _edit(name="edit_cache_36_layers", batch=144),
        # single-precision keys of one layer of a small model into a second tensor (the cache itself stays as it is)
        _edit(name="edit_layer_fp32", dtype="f32", batch=4, seqlen=1500, q_heads=16, kv_heads=16, head_dim=64, rank=16, in_place=False, gain=1.0),
        # a generation step of a full batch: the cache is read once
        _decode(name="decode_batch_64"),
        # a generation step of a few users with contexts of very different length
        _decode(name="decode_few_ragged", batch=3, seqlen=6000, min_len=200),
        # projections of a whole 8B-shaped model from contrastive embeddings
        _learn(name="learn_8b_model"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["prefill"] * 6 + ["edit"] * 3 + ["decode"] * 3 + ["learn"])
    d = rng.choice([64, 128])
    kv = rng.choice([2, 4, 8, 16])
    group = rng.choice([1, 2, 4, 7])
    shape = dict(q_heads=kv * group, kv_heads=kv, head_dim=d)
    rank = rng.choice([8, 16, 24, 32, 64])
    mask = rng.choice(["spans", "spans", "runs"])
    if kind == "prefill":
        dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
        experts = rng.choice([1, 1, 4]) if dtype == "bf16" else 1
        while True:         # at most the work of the largest listed prefill, at most a batch's worth of tokens
            L, B = _log(rng, 64, 32768), _log(rng, 1, 64)
            if 2.0 * d * kv * group * B * L * L <= 7.0e12 and B * L <= 131072 and B * L * kv * group * d <= 2 ** 28:
                break
        ragged = B > 1 and rng.random() < 0.5
        return _prefill(dtype=dtype, batch=B, seqlen=L, min_len=max(1, L // 8) if ragged else 0, rank=rank, experts=experts, mask=mask,
                        highlight=round(rng.uniform(0.02, 1.0 if mask == "spans" else 0.3), 3), gain=rng.choice([0.25, 0.5, 1.0, 2.0, -0.5]), **shape)
    if kind == "edit":
        dtype = rng.choice(["bf16", "bf16", "f32"])
        experts = rng.choice([1, 1, 4]) if dtype == "bf16" else 1
        while True:         # at most half the bytes of the listed 36-layer cache (fp32: of a few layers)
            L, B = _log(rng, 100, 32768), _log(rng, 1, 144)
            if B * L * kv * d <= (2 ** 28 if dtype == "bf16" else 2 ** 24):
                break
        ragged = B > 1 and rng.random() < 0.3
        return _edit(dtype=dtype, batch=B, seqlen=L, min_len=max(1, L // 8) if ragged else 0, rank=min(rank, 32), experts=experts, mask=mask,
                     highlight=round(rng.uniform(0.02, 1.0 if mask == "spans" else 0.3), 3), gain=rng.choice([-0.4, -0.25, -0.6]),
                     in_place=rng.random() < 0.6, **shape)
    if kind == "decode":
        while True:
            L, B = _log(rng, 64, 65536), _log(rng, 1, 256)
            if B * L * kv * d <= 2 ** 28:
                break
        return _decode(batch=B, seqlen=L, min_len=max(1, L // 16) if B > 1 and rng.random() < 0.5 else 0, **shape)
    slots = 2 * _log(rng, 4, 100)
    return _learn(tokens=_log(rng, 2048, 32768), slots=slots, head_dim=d, gamma=rng.choice([0.5, 0.7, 0.9]))


def _lengths(case):
    """Lengths of the sequences: all `seqlen`, or uniform between `min_len` and `seqlen` for a packed batch (the same for
    every seed: the shape of the outputs belongs to the case)."""
    if case["min_len"] <= 0:
        return np.full(case["batch"], case["seqlen"], dtype=np.int64)
    rng = np.random.default_rng([case["batch"], case["seqlen"], case["min_len"]])
    return rng.integers(case["min_len"], case["seqlen"] + 1, size=case["batch"])


def _spans(rng, L, total):
    """One to three disjoint highlighted spans of `total` tokens in all."""
    m = np.zeros(L, dtype=np.uint8)
    total = max(1, min(L, total))
    n = min(int(rng.integers(1, 4)), total, L - total + 1)
    cuts = np.sort(rng.choice(np.arange(1, total), size=n - 1, replace=False)) if n > 1 else np.zeros(0, dtype=np.int64)
    parts = np.diff(np.concatenate([[0], cuts, [total]]))
    gaps = np.diff(np.concatenate([[0], np.sort(rng.integers(0, L - total - (n - 1) + 1, size=n))]))
    pos = 0
    for k, (gap, part) in enumerate(zip(gaps, parts)):
        pos += int(gap) + (1 if k else 0)
        m[pos:pos + int(part)] = 1
        pos += int(part)
    return m


def _runs(rng, L, p):
    """Consecutive runs of 1 to 16 tokens, each highlighted with probability p."""
    ln = rng.integers(1, 17, size=L // 8 + 32)
    on = rng.random(ln.size) < p
    m = np.repeat(on, ln).astype(np.uint8)
    while m.size < L:
        m = np.concatenate([m, m])
    return m[:L]


def _steering(case, lens, rng, gen, f32):
    """Highlight mask, bases, gains and, for several experts, singular values."""
    mask = np.concatenate([_spans(rng, int(n), int(round(case["highlight"] * n))) if case["mask"] == "spans" else _runs(rng, int(n), case["highlight"])
                           for n in lens])
    M, H, d, r = case["experts"], case["kv_heads"], case["head_dim"], case["rank"]
    U = torch.linalg.qr(torch.randn((M, H, d, d), generator=gen, **f32))[0][..., :r].contiguous()
    if case["mask"] == "runs" and case["gain"] > 0:     # packed batches of the small model: a gain of its own per sequence
        gain = torch.rand(case["batch"], generator=gen, **f32) * (1.75 * case["gain"]) + 0.25 * case["gain"]
    else:
        gain = torch.full((case["batch"],), case["gain"], **f32)
    sigma = None
    if M > 1:
        sigma = (torch.rand((M, H, 1), generator=gen, **f32) * 1.5 + 0.5) * 0.9 ** torch.arange(r, **f32)
    return torch.from_numpy(mask).cuda(), U, gain, sigma


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    f32 = dict(dtype=torch.float32, device="cuda")
    if case["kind"] == "learn":
        return _prepare_learn(case, gen, f32)
    dt = DTYPES[case.get("dtype", "bf16")]
    lens = _lengths(case)
    T, Hq, H, d = int(lens.sum()), case["q_heads"], case["kv_heads"], case["head_dim"]

    def rows(n, heads):
        return torch.randn((n, heads, d), generator=gen, **f32).to(dt)

    packed = case["min_len"] > 0
    cu = torch.from_numpy(np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)).cuda() if packed else None
    shape = binding.make_shape(batch=case["batch"], max_seqlen=int(lens.max()), n_q_heads=Hq, n_kv_heads=H, head_dim=d, rank=case.get("rank", 1),
                               n_experts=case.get("experts", 1), dtype=dt, total_tokens=T if packed else 0, cu_seqlens=cu)
    s = {"kind": case["kind"], "shape": shape}
    if case["kind"] == "decode":
        s.update(Q=rows(case["batch"], Hq), K=rows(T, H), V=rows(T, H))
        s.update(O=torch.empty_like(s["Q"]), lse=torch.empty((case["batch"], Hq), **f32),
                 ws=torch.zeros(binding.seka_decode_workspace_bytes(shape), dtype=torch.uint8, device="cuda"))
        return s
    s["mask"], s["U"], s["gain"], s["sigma"] = _steering(case, lens, rng, gen, f32)
    s["ws"] = binding.new_workspace(shape)
    s["K"] = rows(T, H)
    if case["kind"] == "edit":
        s["K_out"] = s["K"] if case["in_place"] else torch.empty_like(s["K"])
        s["alpha"] = None
        if case["experts"] > 1:
            s["alpha"] = torch.rand((case["batch"], H, case["experts"]), generator=gen, **f32)
        return s
    s.update(Q=rows(T, Hq), V=rows(T, H))
    s.update(O=torch.empty_like(s["Q"]), lse=torch.empty((T, Hq), **f32))
    if case["experts"] > 1:
        s["alpha"] = torch.empty((case["batch"], H, case["experts"]), **f32)
    return s


def _prepare_learn(case, gen, f32):
    """Contrastive key embeddings: per slot neutral keys with a decaying spread; positive / negative keys in which a planted
    rank-8 subspace is amplified / attenuated by a strength of the slot's own (every fourth slot does not react)."""
    n, slots, d = case["tokens"], case["slots"], case["head_dim"]
    decay = 0.98 ** torch.arange(d, **f32)
    B = torch.linalg.qr(torch.randn((slots, d, 8), generator=gen, **f32))[0]
    a = torch.rand(slots, generator=gen, **f32) * 1.2 + 0.3
    a[3::4] = 0.0
    h = torch.empty((n, slots, d), dtype=torch.bfloat16, device="cuda")
    hp, hn = torch.empty_like(h), torch.empty_like(h)
    for t in range(0, n, 4096):
        m = min(n, t + 4096) - t
        z = torch.randn((m, slots, d), generator=gen, **f32) * decay
        lift = torch.einsum("nsr,sdr->nsd", torch.einsum("nsd,sdr->nsr", z, B), B) * a[None, :, None]
        h[t:t + m] = z
        hp[t:t + m] = z + lift + 0.1 * torch.randn((m, slots, d), generator=gen, **f32)
        hn[t:t + m] = z - 0.5 * lift + 0.1 * torch.randn((m, slots, d), generator=gen, **f32)
    answer = (torch.rand(n, generator=gen, **f32) < 0.3).to(torch.uint8)
    return {"kind": "learn", "h": h, "hp": hp, "hn": hn, "answer": answer, "gamma": case["gamma"]}


def run(s):
    if s["kind"] == "prefill":
        if s["sigma"] is None:
            binding.seka_attention_fwd(s["shape"], s["Q"], s["K"], s["V"], s["O"], s["lse"], s["mask"], s["U"], None, s["gain"], None, s["ws"])
            return {"O": s["O"], "lse": s["lse"]}
        binding.seka_attention_fwd_routed(s["shape"], s["Q"], s["K"], s["V"], s["O"], s["lse"], s["mask"], s["U"], s["sigma"], 0, s["alpha"],
                                          s["gain"], None, s["ws"])
        return {"O": s["O"], "lse": s["lse"], "alpha": s["alpha"]}
    if s["kind"] == "edit":
        binding.seka_edit_keys(s["shape"], s["K"], s["K_out"], s["mask"], s["U"], s["alpha"], s["gain"], None, s["ws"])
        return {"K": s["K_out"]}
    if s["kind"] == "decode":
        binding.seka_decode_attention(s["shape"], s["Q"], s["K"], s["V"], s["O"], s["lse"], s["ws"])
        return {"O": s["O"], "lse": s["lse"]}
    out = binding.seka_learn_projections(s["h"], s["hp"], s["hn"], s["answer"], s["gamma"])
    # singular vectors are defined up to their sign: the bases come back as the projectors of Eq. 2 that they are learned
    # for (leading columns of U+, trailing columns of U-)
    Up, Un = out["U_pos"][..., :LEARN_CUT], out["U_neg"][..., LEARN_CUT:]
    return {"P_pos": Up @ Up.transpose(1, 2), "P_neg": Un @ Un.transpose(1, 2),
            **{k: out[k] for k in ("omega_pos", "omega_neg", "S_pos", "S_neg", "k_pos", "k_neg", "D")}}


def _mean_len(case):
    return case["seqlen"] if case["min_len"] <= 0 else 0.5 * (case["min_len"] + case["seqlen"])


def work(case):
    d = case["head_dim"]
    if case["kind"] == "learn":
        n, slots = case["tokens"], case["slots"]
        return {"bytes": 3.0 * n * slots * d * 2 + slots * (4.0 * d * d * 4 + 2 * d * 4), "flops": 4.0 * n * slots * d * d}
    B, L, Hq, H = case["batch"], _mean_len(case), case["q_heads"], case["kv_heads"]
    T = B * L
    if case["kind"] == "decode":
        return {"bytes": 2.0 * T * H * d * 2 + 2.0 * B * Hq * d * 2 + B * Hq * 4, "flops": 4.0 * T * Hq * d}
    e = 4 if case["dtype"] == "f32" else 2
    bank = case["experts"] * H * d * case["rank"] * 4.0
    hot = case["highlight"] * T
    edit = 4.0 * hot * H * d * case["rank"] * case["experts"]
    if case["kind"] == "edit":
        moved = 2.0 * (hot if case["in_place"] else T) * H * d * e
        return {"bytes": moved + T + bank, "flops": edit}
    squares = B * L * L if case["min_len"] <= 0 else B * (L * L + (case["seqlen"] - case["min_len"]) ** 2 / 12.0)     # E[len^2]
    return {"bytes": (2.0 * T * Hq + 2.0 * T * H) * d * e + T * Hq * 4 + T + bank, "flops": 2.0 * d * Hq * (squares + T) + edit}


def tolerance(case):
    """About four times the distance of the present path from the same computation in 64 bits (2-norm, largest)."""
    if case["kind"] == "learn":         # 32-bit sums over the tokens (1e-5), subspaces across a gap of the spectrum (1.2e-4)
        return {"rel": 4e-5, "max": 5e-4}
    if case["kind"] == "edit":
        if case["dtype"] == "f32":      # 32-bit sums over head_dim and rank (3e-8, 5e-7), or through U U^T in another order
            return {"rel": 5e-7, "max": 1e-5}
        return {"rel": 3e-3, "max": 1.6e-2}     # one rounding to bf16 of the edited rows (8e-4, 3.9e-3)
    if case.get("dtype") == "f32":      # inputs are rounded to bf16 on the way in (4.3e-3, 0.13)
        return {"rel": 1.6e-2, "max": 0.5}
    return {"rel": 1e-2, "max": 0.4}    # bf16 weights and output (2.1e-3 to 2.8e-3, up to 0.06)
