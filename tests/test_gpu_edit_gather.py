"""The gathering kernel of the key edit: both sides of its rule, one expert and several (projectors that stay on chip and projectors
that are replaced), many steps per CTA, consecutive and scattered tokens.  Rows are independent, so the fp64 oracle evaluates a
sample of the edited rows; every other row is compared bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_01281_b200 import binding

pytestmark = pytest.mark.gpu


def _mask(kind, T, rng):
    m = np.zeros(T, dtype=np.uint8)
    if kind == "all":
        m[:] = 1
    elif kind == "spans":                   # long spans at odd places, and single tokens
        for a in range(77, T - 700, max(1500, T // 40)):
            m[a:a + 1 + rng.integers(0, 700)] = 1
        m[rng.integers(0, T, 20)] = 1
    elif kind == "sparse":                  # about one token per segment of 1024: a step spans more than 100 segments
        m[rng.integers(0, T, T // 1024)] = 1
    else:                                   # short runs
        m[rng.random(T) < 0.2] = 1
    return m


@pytest.mark.parametrize("d,kv,lens,rank,experts,mask,in_place", [
    # one expert: rank 33 to 64 from 4096 units of 128 (8192 of 64) on
    (128, 16, [33000], 40, 1, "spans", True), (128, 16, [9000, 0, 1, 23998], 64, 1, "runs", False), (128, 16, [32640], 40, 1, "runs", True),
    (64, 16, [66000], 48, 1, "all", True), (64, 15, [30000, 45000], 33, 1, "spans", False), (64, 16, [65000], 48, 1, "spans", True),
    # beyond 64: every size
    (128, 3, [1], 65, 1, "all", True), (128, 2, [129, 500], 127, 1, "runs", True), (128, 7, [20000], 128, 1, "sparse", False),
    # up to 32: beyond 32768 units of 128
    (128, 16, [262200], 32, 1, "sparse", True), (128, 32, [65536, 65800], 9, 1, "spans", True),
    # several experts: all projectors stay / are replaced; groups of drain warps at head_dim 64 with every remainder of the experts
    (128, 2, [90000], 64, 2, "runs", True), (128, 2, [3000, 500], 128, 2, "spans", False), (128, 1, [40000], 128, 3, "spans", True),
    (128, 2, [700], 64, 8, "all", True), (64, 2, [80000], 64, 3, "runs", True), (64, 2, [70000], 64, 4, "spans", True), (64, 1, [90000], 64, 5, "all", True),
    (64, 2, [30000, 10000], 64, 8, "spans", False), (64, 3, [1000], 48, 7, "runs", True), (64, 2, [60000], 64, 1, "all", True)])
def test_gathered_edit(d, kv, lens, rank, experts, mask, in_place):
    rng = np.random.default_rng(rank + experts)
    gen = torch.Generator(device="cuda").manual_seed(rank)
    B, T = len(lens), int(sum(lens))
    m = _mask(mask, T, rng)
    cu = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    gain = np.linspace(1.0, -0.5, B).astype(np.float32)
    if B > 2:
        gain[-1] = 0.0                      # a sequence without a gain is not touched
    he = np.ones(kv, dtype=np.uint8)
    he[1::3] = 0
    alpha = rng.uniform(-1, 1, size=(B, kv, experts)).astype(np.float32)
    K = torch.randn((T, kv, d), generator=gen, dtype=torch.bfloat16, device="cuda")
    U = torch.linalg.qr(torch.randn((experts, kv, d, d), generator=gen, device="cuda"))[0][..., :rank].contiguous()
    shp = binding.make_shape(batch=B, max_seqlen=max(lens), n_q_heads=kv, n_kv_heads=kv, head_dim=d, rank=rank, n_experts=experts,
                             total_tokens=T, cu_seqlens=torch.from_numpy(cu).cuda())
    ws = binding.new_workspace(shp)
    out = K.clone() if in_place else torch.full_like(K, float("nan"))
    dev = [torch.from_numpy(x).cuda() for x in (m, alpha, gain, he)]
    binding.seka_edit_keys(shp, out if in_place else K, out, dev[0], U, dev[1], dev[2], dev[3], ws)
    assert binding.seka_poll_status(ws) == binding.SEKA_OK
    seq = np.repeat(np.arange(B), lens)
    hot = (m != 0) & (gain[seq] != 0)
    same = torch.from_numpy(~(hot[:, None] & (he != 0)[None, :])).cuda()
    assert torch.equal(out.view(torch.int16)[same], K.view(torch.int16)[same])
    # a sample of the edited tokens, their first and last among them
    idx = np.flatnonzero(hot)
    idx = np.unique(np.concatenate([idx[:40], idx[-40:], rng.choice(idx, min(idx.size, 400))]))
    n_of = np.bincount(seq[idx], minlength=B)
    Kh = K[torch.from_numpy(idx).cuda()].float().cpu().numpy()
    ref = oracle.edit_keys(Kh, np.ones(idx.size, dtype=np.uint8), np.concatenate([[0], np.cumsum(n_of)]).astype(np.int32), U.cpu().numpy(),
                           alpha=alpha, gain=gain, head_enable=he)
    got = out[torch.from_numpy(idx).cuda()].double().cpu().numpy()
    # one rounding of the result to bf16: half an ulp of the entry, at most 2^-8 of the row's largest
    assert (np.abs(got - ref) / np.abs(ref).max(axis=-1, keepdims=True)).max() <= 2.0 ** -8
    # ... for every edited row: k' lies within |g| sum |alpha| of k in length (orthonormal bases), and none was left out
    if he.any():
        on = torch.from_numpy(np.flatnonzero(he)).cuda()
        hd = torch.from_numpy(hot).cuda()
        delta = (out[hd][:, on].float() - K[hd][:, on].float()).norm(dim=-1)
        size = K[hd][:, on].float().norm(dim=-1)
        bound = torch.from_numpy(np.abs(gain[seq[hot]])[:, None] * np.abs(alpha[seq[hot]][:, he != 0]).sum(-1)).cuda()
        assert torch.isfinite(delta).all() and (delta <= (bound + 0.02) * (size + 1.0)).all()
        assert (delta > 0).float().mean() > 0.99
