"""Calls that follow one another in a stream without a host synchronisation between them, on data that changes: kernels may be
placed while the one before drains, so each has to wait for what it reads.  Each sequence of calls gives the bits of the same
sequence with a synchronisation after every call; once more on two streams with a workspace each, and captured into a graph."""
import pytest
import torch

from paper_2603_01281_b200 import binding

pytestmark = pytest.mark.gpu


class Setup:
    """A cache of `lens` tokens, its queries, and what the calls need (workspaces and outputs of its own)."""

    def __init__(self, seed, lens, d, kv, rank, experts=1):
        g = torch.Generator(device="cuda").manual_seed(seed)
        rnd = lambda *s: torch.randn(s, generator=g, dtype=torch.float32, device="cuda")       # noqa: E731
        T, B = sum(lens), len(lens)
        self.shp = binding.make_shape(batch=B, max_seqlen=max(lens), n_q_heads=2 * kv, n_kv_heads=kv, head_dim=d, rank=rank, n_experts=experts,
                                      total_tokens=T, cu_seqlens=torch.tensor([0] + torch.tensor(lens).cumsum(0).tolist(), dtype=torch.int32, device="cuda"))
        self.K0, self.V, self.Q, self.q1 = (x.bfloat16() for x in (rnd(T, kv, d), rnd(T, kv, d), rnd(T, 2 * kv, d), rnd(B, 2 * kv, d)))
        self.U = torch.linalg.qr(rnd(experts, kv, d, d))[0][..., :rank].contiguous()
        self.sigma = rnd(experts, kv, rank).abs() + 0.5
        self.masks = [(torch.rand(T, generator=g, device="cuda") < p).to(torch.uint8) for p in (0.3, 0.05, 0.8)]
        self.gain = torch.full((B,), -0.4, device="cuda")
        self.alpha = torch.empty((B, kv, experts), device="cuda")
        self.ws, self.dws = binding.new_workspace(self.shp), torch.zeros(binding.seka_decode_workspace_bytes(self.shp), dtype=torch.uint8, device="cuda")
        self.K, self.K2 = self.K0.clone(), torch.empty_like(self.K0)
        self.O, self.o1, self.lse = torch.empty_like(self.Q), torch.empty_like(self.q1), torch.empty((B, 2 * kv), device="cuda")
        self.out = []

    def calls(self):
        """Edit in place -> decode -> edit in place -> forward -> edit of the result into a second tensor -> decode over that."""
        for r in range(3):
            yield from self._round(*(self.masks[(r + i) % 3] for i in range(3)))

    def _round(self, m0, m1, m2):
        al = None if self.U.shape[0] == 1 else self.alpha
        if al is not None:
            yield lambda: binding.adaseka_route(self.shp, self.Q, self.U, self.sigma, 0, self.alpha)
        yield lambda: binding.seka_edit_keys(self.shp, self.K, self.K, m0, self.U, al, self.gain, None, self.ws)
        yield lambda: binding.seka_decode_attention(self.shp, self.q1, self.K, self.V, self.o1, self.lse, self.dws)
        yield lambda: self.out.append(self.o1.clone())
        yield lambda: binding.seka_edit_keys_static(self.shp, self.K, self.K, m1, self.U, al, self.gain, None)
        yield lambda: binding.seka_attention_fwd(self.shp, self.Q, self.K, self.V, self.O, None, m2, self.U, al, self.gain, None, self.ws)
        yield lambda: binding.seka_edit_keys(self.shp, self.K, self.K2, m2, self.U, al, self.gain, None, self.ws)
        yield lambda: binding.seka_decode_attention(self.shp, self.q1, self.K2, self.V, self.o1, self.lse, self.dws)
        yield lambda: self.out.extend([self.O.clone(), self.o1.clone(), self.K2.clone()])
        yield lambda: binding.seka_attention_fwd_routed(self.shp, self.Q, self.K2, self.V, self.O, None, m0, self.U, self.sigma, 0, self.alpha,
                                                        self.gain, None, self.ws)
        yield lambda: self.out.extend([self.O.clone(), self.alpha.clone(), self.K.clone()])

    def run(self, sync):
        self.K.copy_(self.K0)
        self.out = []
        for c in self.calls():
            c()
            if sync:
                torch.cuda.synchronize()
        return self.out


def _same(a, b):
    return len(a) == len(b) and all(torch.equal(x.view(torch.int16 if x.dtype == torch.bfloat16 else torch.int32), y.view(torch.int16 if y.dtype == torch.bfloat16 else torch.int32)) for x, y in zip(a, b))


CASES = [([300, 40], 128, 2, 32, 1), ([2000, 1500, 7], 128, 8, 70, 1), ([500] * 40, 64, 8, 16, 1), ([700, 1300], 64, 4, 64, 4), ([900] * 12, 128, 4, 24, 2)]


@pytest.mark.parametrize("lens,d,kv,rank,experts", CASES)
def test_calls_in_a_stream_keep_their_order(lens, d, kv, rank, experts):
    s = Setup(5, lens, d, kv, rank, experts)
    ref = s.run(sync=True)
    assert all(torch.isfinite(x.float()).all() for x in ref)
    for _ in range(5):
        assert _same(s.run(sync=False), ref)
    assert binding.seka_poll_status(s.ws) == binding.SEKA_OK and binding.seka_poll_status(s.dws) == binding.SEKA_OK


@pytest.mark.parametrize("lens,d,kv,rank,experts", CASES[:4])
def test_two_streams_with_workspaces_of_their_own(lens, d, kv, rank, experts):
    setups = [Setup(6 + i, lens, d, kv, rank, experts) for i in range(2)]
    refs = [s.run(sync=True) for s in setups]
    streams = [torch.cuda.Stream() for _ in setups]
    torch.cuda.synchronize()
    for _ in range(3):
        its = []
        for s, st in zip(setups, streams):
            with torch.cuda.stream(st):
                s.K.copy_(s.K0)
            s.out = []
            its.append(list(s.calls()))
        for pair in zip(*its):
            for c, st in zip(pair, streams):
                with torch.cuda.stream(st):
                    c()
        torch.cuda.synchronize()
        for s, ref in zip(setups, refs):
            assert _same(s.out, ref)


@pytest.mark.parametrize("lens,d,kv,rank,experts", CASES[:4])
def test_calls_captured_into_a_graph(lens, d, kv, rank, experts):
    s = Setup(8, lens, d, kv, rank, experts)
    ref = s.run(sync=True)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        out = s.run(sync=False)
    for _ in range(3):
        for x in out:
            x.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert _same(out, ref)
    assert binding.seka_poll_status(s.ws) == binding.SEKA_OK
