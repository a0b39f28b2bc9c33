"""Predictor heads at the edges of their partition (eight CTAs share the hidden dimension, token sums in chunks beyond 128
tokens), against float64."""
import numpy as np
import pytest
import torch

from oracle import mixture_head as oracle_mix
from paper_2609_38090_b200 import inputs

pytestmark = pytest.mark.gpu

# Additions on the longest path of a score: a warp's tokens (at most 16, or 4 of a chunk's and 64 chunks), 8 warps, a lane's
# products (8 per vector, at most 8 vectors), 5 for the warp, 8 CTAs, the bias: below 160. Each rounds by 2^-24 of a partial sum that
# the sum of absolute values bounds.
ADDS = 160


def _head(C, E, seed):
    g = np.random.default_rng(seed)
    return inputs.round_to_bf16(0.02 * g.standard_normal((E, C)).astype(np.float32)), (0.02 * g.standard_normal(E)).astype(np.float32)


def _bound(x, w, b):
    return ADDS * 2.0 ** -24 * (np.abs(w).astype(np.float64) @ np.abs(x).astype(np.float64).mean(0) + np.abs(b))


@pytest.mark.parametrize("T,C,E", [(1, 64, 1), (3, 192, 7), (7, 2048, 64), (127, 320, 65), (128, 512, 8), (129, 512, 9), (1000, 2112, 60), (2048, 64, 256),
                                   (33, 16384, 13), (300, 16384, 3)])
def test_linear_head(T, C, E):
    from paper_2609_38090_b200 import binding as b
    g = np.random.default_rng(T + C + E)
    x = inputs.round_to_bf16((0.3 + g.standard_normal((T, C))).astype(np.float32))
    w, bias = _head(C, E, 5)
    m = b.Mira(C, 64, E, n_layers=8, max_tokens=T, max_top_k=1)
    xd, wd, bd = torch.from_numpy(x).cuda().bfloat16(), torch.from_numpy(w).cuda().bfloat16(), torch.from_numpy(bias).cuda()
    k = min(E, 16)
    ref = (x.astype(np.float64) @ w.astype(np.float64).T).mean(0)
    for bias_d, want in ((bd, ref + bias), (None, ref)):
        pooled, _, ids = m.predict(0, xd, wd, bias_d, k_pred=k)
        got = pooled.cpu().numpy()
        assert (np.abs(got - want) <= _bound(x, w, bias)).all()
        assert np.array_equal(ids.cpu().numpy(), np.argsort(-got, kind="stable")[:k])     # the selection of its own scores
        if T * E <= 65536:
            p2, i2 = b.predict_noalloc(xd, wd, bias_d, k_pred=k)
            assert torch.equal(p2, pooled) and torch.equal(i2, ids)


@pytest.mark.parametrize("C", [8, 24, 200])
def test_linear_head_on_hidden_sizes_below_one_vector_per_cta(C):
    from paper_2609_38090_b200 import binding as b
    g = np.random.default_rng(C)
    x = inputs.round_to_bf16(g.standard_normal((5, C)).astype(np.float32))
    w, bias = _head(C, 6, 1)
    pooled, _ = b.predict_noalloc(torch.from_numpy(x).cuda().bfloat16(), torch.from_numpy(w).cuda().bfloat16(), torch.from_numpy(bias).cuda(), k_pred=2)
    assert (np.abs(pooled.cpu().numpy() - ((x.astype(np.float64) @ w.astype(np.float64).T).mean(0) + bias)) <= _bound(x, w, bias)).all()


@pytest.mark.parametrize("T,C,E,offset", [(1, 64, 1, 0), (5, 192, 9, 0), (128, 256, 64, 0), (129, 256, 60, 0), (700, 512, 256, 0), (6, 256, 12, 1), (200, 256, 12, 3)])
def test_mixture_head(T, C, E, offset):
    """offset: the head's matrices start that many values behind a 16-byte boundary (rows are then read value by value)."""
    from paper_2609_38090_b200 import binding as b
    sh = inputs.LayerShape("mix", C=C, R=64, E=E, k=1, T=T, seed=T + E)
    h = inputs.mixture_head(sh)
    g = np.random.default_rng(T)
    x = inputs.hidden(sh, T)
    logits = g.standard_normal((T, E)).astype(np.float32)
    count = g.integers(0, 2 * T, E).astype(np.int32)

    def dev(n):
        if n == "b_g":
            return float(h[n])
        t = torch.from_numpy(np.asarray(h[n]))
        if n.startswith("b_"):
            return t.cuda()
        buf = torch.zeros(t.numel() + 16, dtype=torch.bfloat16, device="cuda")
        buf[offset:offset + t.numel()] = t.flatten().cuda().bfloat16()
        return buf[offset:offset + t.numel()].view(t.shape)
    hd = {n: dev(n) for n in h}
    k_top, k = min(E, 4), min(E, 4)
    m = b.Mira(C, 64, E, n_layers=8, max_tokens=T, max_top_k=1)
    scores, probs, alpha, ids = m.predict_mixture(0, torch.from_numpy(x).cuda().bfloat16(), torch.from_numpy(logits).cuda(), torch.from_numpy(count).cuda(),
                                                  k_top, hd, k)
    ref = oracle_mix.mixture_head(x, logits, count, k_top, h, k)
    got = scores.cpu().numpy()
    # both branches and the gate's own sums: ADDS roundings of 2^-24 of sums of absolute values below 10
    assert np.abs(got - ref["out"]).max() <= 1e-4 and abs(float(alpha) - ref["alpha"]) <= 1e-4
    assert np.abs(probs.cpu().numpy() - ref["prob"]).max() <= 1e-4
    assert np.array_equal(ids.cpu().numpy(), np.argsort(-got, kind="stable")[:k])
