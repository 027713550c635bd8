"""Tile kernels of the key edit at the edges of their 128-row steps, 64-column blocks of stacked U and dispatch rule, against the
fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_01281_b200 import binding, inputs

import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("d,rank,experts,kv,lens,mask", [
    (128, 32, 1, 2, [127], "all"), (128, 64, 1, 3, [128], "all"), (64, 16, 1, 2, [129], "all"), (64, 1, 1, 1, [1], "all"),
    (128, 65, 1, 2, [300, 0, 41], "runs"), (128, 24, 3, 2, [513, 70], "runs"), (64, 7, 9, 2, [200, 200], "spans"),
    (128, 128, 4, 2, [257], "spans"), (64, 64, 2, 5, [1024, 1025, 1], "runs"), (128, 16, 1, 2, [640], "none"),
    # both sides of a stacked rank of 32, where U changes its layout
    (128, 33, 1, 2, [300], "all"), (64, 32, 1, 2, [300, 77], "runs"), (64, 33, 1, 2, [300], "runs"), (128, 8, 4, 3, [257, 130], "spans"),
    (64, 11, 3, 2, [140], "all"), (128, 17, 1, 2, [190, 66], "all"), (64, 3, 10, 1, [513], "runs")])
def test_edit_steps_and_blocks(d, rank, experts, kv, lens, mask, in_place):
    w = inputs.make_custom(seed=90 + rank, dtype="bf16", lens=lens, n_q_heads=2 * kv, n_kv_heads=kv, head_dim=d, rank=rank,
                           n_experts=experts, mask_kind=mask, highlight=0.3, gain=np.linspace(1.0, -0.5, len(lens)))
    if len(lens) > 2:
        w.gain[-1] = 0.0                                        # a sequence without a gain is not touched
    alpha = np.random.default_rng(rank).uniform(-1, 1, size=(w.batch, kv, experts))
    he = np.ones(kv, dtype=np.uint8)
    he[-1] = kv == 1
    ref = oracle.edit_keys(w.K, w.mask, w.cu_seqlens, w.U, alpha=alpha, gain=w.gain, head_enable=he)
    got = H.run_edit(w, alpha=alpha, head_enable=he, in_place=in_place).double().cpu().numpy()
    # one rounding of the result to bf16: half an ulp of the entry, at most 2^-8 of the row's largest
    assert (np.abs(got - ref) / np.abs(ref).max(axis=-1, keepdims=True)).max() <= 2.0 ** -8
    seq_gain = np.repeat(w.gain, np.diff(w.cu_seqlens))
    same = ((w.mask == 0) | (seq_gain == 0))[:, None] | (he == 0)[None, :]
    assert np.array_equal(got[same], w.K.astype(np.float64)[same])


@pytest.mark.parametrize("d,seqs,kv,dtype", [(128, 74, 4, "bf16"), (128, 75, 4, "bf16"), (64, 111, 4, "bf16"), (64, 112, 4, "bf16"),
                                             (128, 75, 4, "f32"), (64, 112, 4, "f32")])
def test_preparation_on_both_sides_of_its_rule(d, seqs, kv, dtype):
    """Four key tiles a sequence, so that 74 | 75 (111 | 112) sequences lie on the two sides of the line between the chain and the
    pipelined preparation on a GPU of 148 SMs."""
    lens = [400 + (37 * i) % 113 for i in range(seqs - 1)] + [512]
    w = inputs.make_custom(seed=95, dtype=dtype, lens=lens, n_q_heads=kv, n_kv_heads=kv, head_dim=d, rank=16, mask_kind="runs",
                           highlight=0.1, gain=[(0.5, 2.0, 0.0)[i % 3] for i in range(seqs)])
    w.Q, w.K, w.V = (inputs.round_to_bf16(x) for x in (w.Q, w.K, w.V))      # (fp32 inputs are rounded on the way in)
    he = np.array([1, 0] + [1] * (kv - 2), dtype=np.uint8)
    rows = H.sampled_rows(w, 8, seed=1)
    O, LSE = H.run_fused(w, head_enable=he)
    Oref, Lref, idx = H.oracle_rows(w, rows, head_enable=he)
    H.check_attention(O[idx], Oref, "d%d %d sequences" % (d, seqs))
    np.testing.assert_allclose(LSE[idx], Lref, atol=2e-2)       # the bound of the other forward tests


@pytest.mark.parametrize("d,seqs,kv,L,rank,experts,dtype,varlen", [
    (128, 37, 4, 100, 32, 1, "bf16", False), (128, 38, 4, 100, 32, 1, "bf16", False),      # 148 | 152 steps: small form | not
    (64, 37, 4, 100, 16, 1, "bf16", False), (64, 38, 4, 100, 16, 1, "bf16", True),
    (128, 2, 2, 300, 65, 1, "bf16", True), (128, 3, 2, 129, 24, 3, "bf16", False),         # U in blocks that are replaced
    (64, 3, 3, 257, 33, 3, "bf16", True), (64, 2, 2, 128, 7, 1, "bf16", False),
    (64, 3, 4, 130, 8, 1, "f32", False), (128, 2, 3, 200, 16, 2, "f32", True)])
def test_small_preparation(d, seqs, kv, L, rank, experts, dtype, varlen):
    lens = [L if not varlen or i == 0 else (0 if i == 1 and seqs > 2 else max(1, L - 31 * i % L)) for i in range(seqs)]
    w = inputs.make_custom(seed=97, dtype=dtype, lens=lens, n_q_heads=2 * kv, n_kv_heads=kv, head_dim=d, rank=rank, n_experts=experts,
                           mask_kind="runs", highlight=0.2, gain=[(0.5, 2.0, 0.0)[i % 3] for i in range(seqs)])
    w.Q, w.K, w.V = (inputs.round_to_bf16(x) for x in (w.Q, w.K, w.V))      # (fp32 inputs are rounded on the way in)
    alpha = np.random.default_rng(rank).uniform(-1, 1, size=(w.batch, kv, experts)).astype(np.float32)
    he = np.array([1] * (kv - 1) + [0], dtype=np.uint8)
    rows = H.sampled_rows(w, 8, seed=1)
    O, LSE = H.run_fused(w, alpha=alpha, head_enable=he, force_varlen=varlen)
    Oref, Lref, idx = H.oracle_rows(w, rows, alpha=alpha, head_enable=he)
    H.check_attention(O[idx], Oref, "d%d %d sequences" % (d, seqs))
    np.testing.assert_allclose(LSE[idx], Lref, atol=2e-2)       # the bound of the other forward tests


@pytest.mark.parametrize("d,seqs,L,kv,rank,k_route", [
    (128, 25, 400, 4, 43, 43), (128, 25, 400, 4, 64, 16),       # 100 pairs, 400 steps: blocks of U stay, Eq. 6 by a launch of its own
    (128, 9, 1030, 4, 64, 64),                                  # 36 pairs: Eq. 6 in the CTAs
    (64, 25, 400, 4, 48, 48), (64, 25, 400, 4, 64, 64), (64, 5, 2100, 4, 48, 7), (64, 25, 400, 4, 33, 4)])
def test_wide_banks_with_many_steps(d, seqs, L, kv, rank, k_route):
    """One call with routing against the coefficients of adaseka_route given by hand: the same bits, and the oracle's rows."""
    w = inputs.make_custom(seed=98, dtype="bf16", lens=[L] * seqs, n_q_heads=kv, n_kv_heads=kv, head_dim=d, rank=rank, n_experts=4,
                           mask_kind="runs", highlight=0.2, gain=[(0.5, 2.0, 0.0)[i % 3] for i in range(seqs)])
    dev = H.device_tensors(w)
    shp = H.shape_of(w, dev)
    ws = binding.new_workspace(shp)
    sigma = torch.from_numpy((0.9 ** np.arange(rank) * np.ones((4, kv, 1))).astype(np.float32)).cuda()
    sigma *= torch.tensor([0.7, 1.0, 1.3, 0.9], device="cuda").view(4, 1, 1)
    alpha = torch.empty((seqs, kv, 4), dtype=torch.float32, device="cuda")
    binding.adaseka_route(shp, dev["Q"], dev["U"], sigma, k_route, alpha)
    O = torch.full_like(dev["Q"], float("nan"))
    for out in (torch.empty_like(alpha), None):
        binding.seka_attention_fwd_routed(shp, dev["Q"], dev["K"], dev["V"], O, None, dev["mask"], dev["U"], sigma, k_route, out, dev["gain"],
                                          None, ws)
        assert binding.seka_poll_status(ws) == binding.SEKA_OK
        assert out is None or torch.equal(out, alpha)
        rows = H.sampled_rows(w, 4, seed=1)
        Oref, _, idx = H.oracle_rows(w, rows, alpha=alpha.cpu().numpy())
        H.check_attention(O.double().cpu().numpy()[idx], Oref, "d%d rank %d" % (d, rank))


@pytest.mark.parametrize("d,lens,dtype", [
    (128, [512] * 74, "bf16"), (128, [512] * 75, "bf16"), (64, [512] * 112, "bf16"), (64, [512] * 112, "f32"),
    (64, [1 + i % 3 for i in range(600)], "bf16")])            # fewer tokens than (sequence, KV head) pairs
def test_one_routed_expert_on_both_sides_of_the_rule(d, lens, dtype):
    """One expert, four KV heads, on both sides of the line between the chain and the pipelined preparation: one call with routing gives
    the bits of adaseka_route followed by seka_attention_fwd."""
    w = inputs.make_custom(seed=99, dtype=dtype, lens=lens, n_q_heads=4, n_kv_heads=4, head_dim=d, rank=16, mask_kind="runs", highlight=0.3,
                           gain=[(0.5, 2.0, 0.0, -1.5)[i % 4] for i in range(len(lens))])
    dev = H.device_tensors(w)
    shp = H.shape_of(w, dev)
    sigma = torch.from_numpy(0.9 ** np.arange(16, dtype=np.float32) * np.ones((1, 4, 1), dtype=np.float32)).cuda()
    alpha = torch.empty((w.batch, 4, 1), dtype=torch.float32, device="cuda")
    binding.adaseka_route(shp, dev["Q"], dev["U"], sigma, 0, alpha)
    assert (alpha < 0).any() and (alpha > 0).any()
    bits = torch.int16 if dtype == "bf16" else torch.int32
    ref = torch.full_like(dev["Q"], float("nan"))
    ws = binding.new_workspace(shp)
    binding.seka_attention_fwd(shp, dev["Q"], dev["K"], dev["V"], ref, None, dev["mask"], dev["U"], alpha, dev["gain"], None, ws)
    assert binding.seka_poll_status(ws) == binding.SEKA_OK
    for out in (torch.full_like(alpha, float("nan")), None):
        O = torch.full_like(ref, float("nan"))
        ws = binding.new_workspace(shp)
        binding.seka_attention_fwd_routed(shp, dev["Q"], dev["K"], dev["V"], O, None, dev["mask"], dev["U"], sigma, 0, out, dev["gain"], None, ws)
        assert binding.seka_poll_status(ws) == binding.SEKA_OK
        assert out is None or torch.equal(out, alpha)
        assert torch.equal(O.view(bits), ref.view(bits))


@pytest.mark.parametrize("seqs,experts,rank,k_route,dtype,varlen", [
    (37, 4, 64, 64, "bf16", False), (38, 4, 64, 16, "bf16", False),            # 592 | 608 tiles: chain | pipeline
    (60, 2, 64, 64, "bf16", True), (45, 3, 57, 57, "bf16", False), (40, 5, 64, 3, "bf16", True), (70, 8, 64, 64, "bf16", False),
    (38, 8, 48, 48, "f32", True)])
def test_preparation_with_several_projectors(seqs, experts, rank, k_route, dtype, varlen):
    """Banks at head_dim 64 on both sides of the line between the chain and the pipelined preparation: the oracle's rows, and one call
    with routing gives the bits of the coefficients of adaseka_route given by hand."""
    lens = [512 if i == 0 or not varlen else 385 + (53 * i) % 127 for i in range(seqs)]
    w = inputs.make_custom(seed=96, dtype=dtype, lens=lens, n_q_heads=4, n_kv_heads=4, head_dim=64, rank=rank, n_experts=experts,
                           mask_kind="runs", highlight=0.15, gain=[(0.5, 2.0, 0.0, -1.0)[i % 4] for i in range(seqs)])
    w.Q, w.K, w.V = (inputs.round_to_bf16(x) for x in (w.Q, w.K, w.V))      # (fp32 inputs are rounded on the way in)
    dev = H.device_tensors(w)
    shp = H.shape_of(w, dev, force_varlen=varlen)
    he = torch.tensor([1, 1, 0, 1], dtype=torch.uint8, device="cuda")
    sigma = torch.rand((experts, 4, rank), generator=torch.Generator().manual_seed(1)).cuda() + 0.5
    alpha = torch.empty((seqs, 4, experts), dtype=torch.float32, device="cuda")
    binding.adaseka_route(shp, dev["Q"], dev["U"], sigma, k_route, alpha)
    ref = torch.full_like(dev["Q"], float("nan"))
    ws = binding.new_workspace(shp)
    binding.seka_attention_fwd(shp, dev["Q"], dev["K"], dev["V"], ref, None, dev["mask"], dev["U"], alpha, dev["gain"], he, ws)
    assert binding.seka_poll_status(ws) == binding.SEKA_OK
    rows = H.sampled_rows(w, 4, seed=1)
    Oref, _, idx = H.oracle_rows(w, rows, alpha=alpha.cpu().numpy(), head_enable=he.cpu().numpy())
    H.check_attention(ref.double().cpu().numpy()[idx], Oref, "%d experts of rank %d" % (experts, rank))
    bits = torch.int16 if dtype == "bf16" else torch.int32
    for out in (torch.full_like(alpha, float("nan")), None):
        O = torch.full_like(ref, float("nan"))
        ws = binding.new_workspace(shp)
        binding.seka_attention_fwd_routed(shp, dev["Q"], dev["K"], dev["V"], O, None, dev["mask"], dev["U"], sigma, k_route, out, dev["gain"], he, ws)
        assert binding.seka_poll_status(ws) == binding.SEKA_OK
        assert out is None or torch.equal(out, alpha)
        assert torch.equal(O.view(bits), ref.view(bits))
