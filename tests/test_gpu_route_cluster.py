"""Routing of 1 to 4 tokens, and of up to 8 with at most 16 experts, by one cluster of CTAs: numbers of experts around multiples of the cluster's size and of a warp's lanes,
hidden sizes around a warp's registers (512 vectors of eight), small and large top-k, shared experts; against the oracle, and the same scores
bit for bit as in a batch that another kernel routes."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import to_bf16_cuda
from paper_2609_38090_b200 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,C,E,k,ns", [(1, 64, 1, 1, 0), (4, 64, 7, 7, 1), (3, 192, 8, 2, 0), (2, 512, 9, 3, 3), (4, 2048, 60, 4, 4), (1, 4096, 8, 2, 0),
                                        (4, 4160, 17, 16, 0), (2, 8192, 33, 5, 2), (3, 16384, 65, 6, 0), (4, 1024, 127, 16, 1), (4, 320, 240, 8, 16),
                                        (4, 192, 240, 16, 16), (5, 2048, 16, 4, 4), (7, 8192, 16, 2, 0), (8, 8192, 9, 9, 1), (8, 4096, 8, 2, 0)])
def test_route_cluster(T, C, E, k, ns):
    from paper_2609_38090_b200 import binding as b
    g = np.random.default_rng(C + E)
    x = inputs.round_to_bf16(g.standard_normal((8, C)).astype(np.float32))
    w = inputs.round_to_bf16((0.05 * g.standard_normal((E, C))).astype(np.float32))
    bias = (0.1 * g.standard_normal(E)).astype(np.float32)
    x = np.concatenate([x, inputs.round_to_bf16(g.standard_normal((4, C)).astype(np.float32))])
    wd, bd = to_bf16_cuda(w), torch.from_numpy(bias).cuda()
    m = b.Mira(C, 64, E, n_shared=ns, max_tokens=12, max_top_k=k)
    r = m.route(to_bf16_cuda(x[:T]), wd, bd, k)
    got = {n: r[n].cpu().numpy().copy() for n in ("idx", "w", "count", "offset", "perm", "logits")}
    logits = oracle.linear_scores(x[:T], w, bias)
    # a lane adds C / 32 products, then five levels, the bias: each rounds by 2^-24 of what the absolute values bound
    bound = (C / 32 + 8) * 2.0 ** -24 * (np.abs(x[:T]).astype(np.float64) @ np.abs(w).astype(np.float64).T + np.abs(bias))
    assert (np.abs(got["logits"].reshape(-1)[:T * E].reshape(T, E) - logits) <= bound).all()
    idx, wts, _, margin = oracle.topk_softmax(logits, k)
    assert (margin > 2 * bound.max(1)).all()               # no near-ties in these seeded inputs
    assert np.array_equal(got["idx"].reshape(-1)[:T * k].reshape(T, k), idx)
    assert np.abs(got["w"].reshape(-1)[:T * k].reshape(T, k) - wts).max() <= 2 * bound.max() + 2.0 ** -20
    count, offset, perm, perm_sh = oracle.group(idx, E, ns)
    assert np.array_equal(got["count"], count) and np.array_equal(got["offset"], offset)
    assert np.array_equal(got["perm"].reshape(-1)[:T * (k + ns)].reshape(T, k + ns), np.concatenate([perm, perm_sh], axis=1))
    r8 = m.route(to_bf16_cuda(x), wd, bd, k)               # twelve tokens: another kernel
    assert np.array_equal(r8["logits"].cpu().numpy().reshape(-1)[:T * E], got["logits"].reshape(-1)[:T * E])
