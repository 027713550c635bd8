"""The SVD of the learner on cross-covariances where its QR step and its rotations can go wrong: zero, of low rank (zero
singular values, exactly and to rounding), graded over many orders, with equal singular values, with a tiny scale."""
import numpy as np
import pytest
import torch

from paper_2603_01281_b200 import binding

pytestmark = pytest.mark.gpu


def _embeddings(kind, n, slots, d):
    rng = np.random.default_rng(17)
    h, hp, hn = (rng.standard_normal((n, slots, d)) for _ in range(3))
    hp += h
    hn -= 0.5 * h
    if kind == "zero":
        h[:] = 0.0
    elif kind == "zero_rows":           # rows of Omega that are exactly zero
        h[..., 5:] = 0.0
    elif kind == "zero_columns":        # columns of Omega that are exactly zero
        hp[..., 3:] = 0.0
        hn[..., :-1] = 0.0
    elif kind == "rank_deficient":      # fewer tokens than dimensions
        h[d // 3:] = 0.0
    elif kind == "graded":              # rows and columns from 1 to 2^-40, the large ones last
        g = 2.0 ** (40.0 * (np.arange(d) / (d - 1.0) - 1.0))
        h, hp, hn = h * g, hp * g, hn * g[::-1]
    elif kind == "equal":               # a multiple of the identity up to the order of its rows and signs
        h = np.zeros((n, slots, d))
        for t in range(d):
            h[t, :, t] = 1.0
        hp = np.roll(h, 3, axis=2)
        hn = -h
    elif kind == "tiny":
        h, hp, hn = h * 2.0 ** -55, hp * 2.0 ** -55, hn * 2.0 ** -55
    return h, hp, hn


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("kind", ["zero", "zero_rows", "zero_columns", "rank_deficient", "graded", "equal", "tiny"])
def test_svd_of_awkward_matrices(kind, d):
    n, slots, gamma = 192, 2, 0.6
    dev = [torch.from_numpy(x).to(device="cuda", dtype=torch.bfloat16) for x in _embeddings(kind, n, slots, d)]
    out = {k: v.double().cpu().numpy() for k, v in binding.seka_learn_projections(*dev, None, gamma).items() if k != "workspace"}
    for tag in ("pos", "neg"):
        for s in range(slots):
            Om, U, S = out["omega_" + tag][s], out["U_" + tag][s], out["S_" + tag][s]
            assert np.isfinite(U).all() and np.isfinite(S).all()
            _, S2, _ = np.linalg.svd(Om)
            # the bounds of the learner's other tests: fp32 outputs of an fp64 decomposition
            np.testing.assert_allclose(S, S2, rtol=2e-6, atol=2e-7 * S2[0])
            assert np.all(np.diff(S) <= 0)
            top = S2 > 1e-9 * S2[0] if S2[0] > 0 else np.zeros(d, bool)      # vectors of zero singular values are not determined
            np.testing.assert_allclose(U[:, top].T @ U[:, top], np.eye(int(top.sum())), atol=5e-6)
            # a left singular vector u of S: Omega^T u has the norm S; rounding u to fp32 (2^-24 per entry) moves it by
            # up to 2^-24 S2[0] against the leading directions
            np.testing.assert_allclose(np.linalg.norm(Om.T @ U[:, top], axis=0), S2[top], rtol=5e-6, atol=2.0 ** -22 * S2[0])
            np.testing.assert_allclose(Om @ (Om.T @ U[:, top]), (U * (S2 * S2))[:, top], atol=2e-5 * S2[0] ** 2)
            total = S2.sum()
            want = int(np.argmax(np.cumsum(S2) >= gamma * total)) + 1
            k = int(out["k_" + tag][s])
            assert k == want or abs(np.cumsum(S2)[k - 1] / total - gamma) < 1e-6
