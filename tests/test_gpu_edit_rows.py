"""fp32-arithmetic edit (fp32 tensors, wide banks, the workspace-free call) at the edges of its 64-token tiles and 32-column
rank chunks, against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_01281_b200 import binding, inputs

import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("in_place", [False, True])
@pytest.mark.parametrize("dtype,d,rank,experts,lens", [
    ("f32", 64, 1, 1, [1]), ("f32", 128, 8, 1, [63, 1]), ("f32", 64, 9, 1, [64, 65]), ("f32", 128, 33, 1, [200, 0, 57]),
    ("f32", 128, 128, 2, [129]), ("bf16", 128, 16, 5, [127, 66]), ("bf16", 64, 17, 9, [320]), ("f32", 64, 64, 3, [70] * 40)])
def test_row_edit_tiles_and_chunks(dtype, d, rank, experts, lens, in_place):
    w = inputs.make_custom(seed=70 + rank, dtype=dtype, lens=lens, n_q_heads=6, n_kv_heads=3, head_dim=d, rank=rank, n_experts=experts,
                           mask_kind="runs", highlight=0.4, gain=np.linspace(-0.5, 1.0, len(lens)))
    rng = np.random.default_rng(rank)
    alpha = rng.uniform(-1, 1, size=(w.batch, 3, experts)) if experts > 1 else None
    he = np.array([1, 0, 1], dtype=np.uint8)
    ref = oracle.edit_keys(w.K, w.mask, w.cu_seqlens, w.U, alpha=alpha, gain=w.gain, head_enable=he)
    scale = np.abs(ref).max(axis=-1, keepdims=True)
    # fp32: two dot products of length d and experts * rank, each off by at most its length in units of 2^-24 of the sum of
    # magnitudes, which stays below sqrt(d) * experts times the row maximum here; bf16: one rounding
    tol = 2.0 ** -24 * (d + experts * rank) * np.sqrt(d) * experts if dtype == "f32" else 2.0 ** -8
    outs = [H.run_edit(w, alpha=alpha, head_enable=he, in_place=in_place)]
    if experts == 1:
        dev = H.device_tensors(w)
        out = dev["K"].clone() if in_place else torch.full_like(dev["K"], float("nan"))
        binding.seka_edit_keys_static(H.shape_of(w, dev), out if in_place else dev["K"], out, dev["mask"], dev["U"], None, dev["gain"],
                                      torch.from_numpy(he).cuda())
        outs.append(out)
    for got in outs:
        got = got.double().cpu().numpy()
        assert (np.abs(got - ref) / scale).max() <= tol
        same = (w.mask == 0)[:, None] | (he == 0)[None, :]
        assert np.array_equal(got[same], w.K.astype(np.float64)[same])


@pytest.mark.parametrize("dtype,d,rank", [("f32", 64, 1), ("f32", 128, 3), ("f32", 64, 8), ("f32", 128, 13), ("f32", 64, 34), ("bf16", 64, 1), ("bf16", 128, 6)])
def test_row_edit_infinities_and_nan(dtype, d, rank):
    """A key with an infinity (or NaN) is edited as the sums over the stored columns say: the columns that fill up a chunk of the rank
    add nothing, and no other row is touched."""
    w = inputs.make_custom(seed=77, dtype=dtype, lens=[150], n_q_heads=2, n_kv_heads=2, head_dim=d, rank=rank, mask_kind="all", gain=0.5)
    w.K[3, 0, 5] = np.inf; w.K[70, 1, 1] = -np.inf; w.K[149, 0, 9] = np.nan
    with np.errstate(invalid="ignore"):
        ref = oracle_edit(w)
    for in_place in (False, True):
        dev = H.device_tensors(w)
        out = dev["K"] if in_place else torch.full_like(dev["K"], float("nan"))
        binding.seka_edit_keys_static(H.shape_of(w, dev), dev["K"], out, dev["mask"], dev["U"], None, dev["gain"], None)
        got = out.double().cpu().numpy()
        assert np.array_equal(np.isnan(got), np.isnan(ref))
        assert np.array_equal(np.isposinf(got), np.isposinf(ref)) and np.array_equal(np.isneginf(got), np.isneginf(ref))
        fin = np.isfinite(ref)
        assert np.isposinf(ref).any() or rank > 1
        # the tolerances of the test above (entries of a unit-variance row stay below 8)
        assert np.abs(got[fin] - ref[fin]).max() <= 8 * (2.0 ** -24 * (d + rank) * np.sqrt(d) if dtype == "f32" else 2.0 ** -8)


def oracle_edit(w):
    """k + g U (U^T k) in fp64, row by row (the oracle library is not asked for rows that are not finite)."""
    K, U = w.K.astype(np.float64), w.U[0].astype(np.float64)
    out = K.copy()
    for h in range(K.shape[1]):
        C = (K[:, h, :, None] * U[h][None]).sum(1)
        out[:, h] = K[:, h] + float(w.gain[0]) * (C[:, None, :] * U[h][None]).sum(-1)
    return out
