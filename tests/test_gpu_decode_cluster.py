"""The decode step on both sides of its dispatch: chunks of a (sequence, KV head) merged inside a cluster of 1, 2, 4 or 8 CTAs,
and by the second launch."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_01281_b200 import binding, inputs

import helpers as H
import test_gpu_decode as T

pytestmark = pytest.mark.gpu


def _launches(f):
    n = binding.load().seka_launch_count()
    out = f()
    return out, binding.load().seka_launch_count() - n


@pytest.mark.parametrize("d,Hq,Hkv,lens,launches", [
    (128, 1, 1, [128], 1), (128, 1, 1, [129], 1), (128, 4, 1, [1025, 0, 1, 128, 64], 1),        # clusters of 1, 2, 8 (ranks without tokens)
    (128, 16, 1, [8192], 1), (128, 9, 1, [8193], 2), (64, 2, 2, [8192], 1), (64, 2, 2, [8193], 2),      # longest chunk of few CTAs
    (128, 8, 8, [1500] * 5, 1), (128, 4, 4, [4500] * 11, 2), (128, 4, 4, [4500] * 12, 1),               # 176 | 192 CTAs in clusters of 4
    (128, 8, 8, [2200] * 9, 2), (128, 8, 8, [2200] * 8, 1),                                             # clusters of 4 fit | do not
    (128, 8, 8, [1100] * 37, 1), (128, 8, 8, [1100] * 38, 2),                                           # 296 | 304 pairs: one wave
    (64, 12, 12, [1100] * 37, 1), (64, 12, 12, [1100] * 38, 2),                                         # 444 | 456 pairs
    (128, 8, 8, [2560] + [30] * 36, 2), (128, 8, 8, [2560] * 20 + [30] * 17, 1),                        # uneven: far above an SM's share | not
    (128, 8, 8, [1000] + [60] * 17, 1), (128, 8, 8, [1100] + [60] * 17, 2),                             # uneven: clusters of 2, chunks of 512 | more
])
def test_decode_on_both_sides_of_its_dispatch(d, Hq, Hkv, lens, launches):
    w = inputs.make_custom(seed=41, dtype="bf16", lens=lens, n_q_heads=Hq, n_kv_heads=Hkv, head_dim=d, rank=8)
    dev = H.device_tensors(w)
    q = T._last_queries(w)
    (O, LSE), n = _launches(lambda: T._run_decode(w, dev, dev["K"], q))
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:
        assert n == launches, (n, launches)
    Oref, Lref = oracle.decode_attention(q, w.K, w.V, w.cu_seqlens)
    for b in np.flatnonzero(np.asarray(lens) == 0):
        assert np.all(O[b] == 0) and np.all(np.isneginf(LSE[b]))
    T._check(O, LSE, Oref, Lref)


@pytest.mark.parametrize("d,kv,lens,max_len,covered", [
    (128, 2, [3000] * 3, 129, 256), (64, 2, [3000, 20, 600], 500, 512),         # clusters of 2 and 4
    (128, 8, [4000] + [30] * 36, 2560, 3072)])                                  # two launches, chunks of 1024
def test_decode_of_lengths_beyond_max_seqlen(d, kv, lens, max_len, covered):
    """cu_seqlens that runs ahead of the shape's max_seqlen: the step attends to the tokens that its chunks cover and reads no
    chunk that does not exist."""
    w = inputs.make_custom(seed=43, dtype="bf16", lens=lens, n_q_heads=kv, n_kv_heads=kv, head_dim=d, rank=8)
    dev = H.device_tensors(w)
    q = T._last_queries(w)
    shp = H.shape_of(w, dev, force_varlen=True)
    shp.max_seqlen = max_len
    ws = torch.zeros(binding.seka_decode_workspace_bytes(shp), dtype=torch.uint8, device="cuda")
    qd = torch.from_numpy(q).to(device="cuda", dtype=torch.bfloat16)
    O = torch.full_like(qd, float("nan"))
    binding.seka_decode_attention(shp, qd, dev["K"], dev["V"], O, None, ws)
    assert binding.seka_poll_status(ws) == binding.SEKA_OK
    seen = np.minimum(lens, covered)
    rows = np.concatenate([s + np.arange(n) for s, n in zip(w.cu_seqlens[:-1].astype(np.int64), seen)])
    Oref, _ = oracle.decode_attention(q, w.K[rows], w.V[rows], np.concatenate([[0], np.cumsum(seen)]).astype(np.int32))
    err = np.abs(O.double().cpu().numpy() - Oref)
    assert err.max() <= 1e-2 and err.mean() <= 1e-3, (err.max(), err.mean())       # the bounds of the other decode tests
