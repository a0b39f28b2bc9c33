"""The weight-streaming expert kernels at the edges of their partition: digits made in the kernel up to 4 tokens and in token order up to 16, token tiles of up to
80, reduction boxes of 128 elements cut by the matrix, work items of four units that run into the next expert, slices of the
reduction beyond 4096 expert-hidden rows. Against float64 on the oracle's codes and routing."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import Workload
from paper_2609_38090_b200 import inputs

pytestmark = pytest.mark.gpu
NONE = 2 ** 31 - 1


def _uneven(sh, e):
    w1, w2, w3 = inputs.expert_weights(sh, e)
    g = np.random.default_rng(e)
    return w1 * np.exp(1.5 * g.standard_normal((sh.R, 1))).astype(np.float32), w2, w3


def _reference(wl, idx, w, act_on_w1, fp32_sums=0):
    """The layer in float64 and what the kernels may differ from it by. Activations are rounded to 2^-22 of their row's largest value
    on either side, the sums of products are exact and then converted to fp32 (2^-21 of the sum of absolute values covers both
    conversions; with fp32_sums, experts of the other kernels: 2^-23 for each of that many partial sums of 16 products);
    SwiGLU in fp32 to 2^-18; the intermediate is rounded to fp16, 2^-11, of values placed 22 binary digits above its subnormals'
    step; combination in fp32, weights to 2^-18."""
    sh = wl.shape
    y, dy = np.zeros((wl.T, sh.C)), np.zeros((wl.T, sh.C))
    x = wl.x.astype(np.float64)
    for e, blob in enumerate(wl.blobs):
        if e < sh.E:
            t, j = np.nonzero(idx == e)
            we = w[t, j].astype(np.float64)
        else:
            t, we = np.arange(wl.T), np.ones(wl.T)
        if len(t) == 0:
            continue
        u = oracle.unpack_expert_std(blob, sh.R, sh.C) if wl.fmt else oracle.unpack_expert(blob, sh.R, sh.C)
        w1, w2, w3 = (u[n].astype(np.float64) for n in ("w1", "w2", "w3"))
        xe = x[t]
        U, G = xe @ w1.T, xe @ w3.T
        top = np.abs(xe).max(1)[:, None]
        dU, dG = ((2.0 ** -21 + 2.0 ** -23 * fp32_sums) * (top * np.abs(m).sum(1) + np.abs(xe) @ np.abs(m).T) for m in (w1, w3))
        a, l, da, dl = (U, G, dU, dG) if act_on_w1 else (G, U, dG, dU)
        silu = a / (1 + np.exp(-a))
        h = silu * l
        dh = 1.1 * da * (np.abs(l) + dl) + np.abs(silu) * dl + np.abs(h) * (2.0 ** -18 + 2.0 ** -11)
        # the second projection's matrix with the scale on the side the kernels have it: s_r h_r is what is rounded
        s = np.ones(sh.R) if wl.fmt else u["s"].astype(np.float64)
        hs, q2 = h * s, np.abs(w2) / s
        dh_s = dh * s + 2.0 ** -20 * np.abs(hs).max(1)[:, None]
        ye = h @ w2.T
        dye = dh_s @ q2.T + (2.0 ** -18 + 2.0 ** -23 * fp32_sums) * (np.abs(hs) @ q2.T)
        np.add.at(y, t, we[:, None] * ye)
        np.add.at(dy, t, we[:, None] * dye)
    return y, dy


CASES = [  # C, R, experts, k, shared, tokens, format, thresholds (up, down): pairs from which an expert leaves the streaming kernels
    (64, 64, 3, 2, 0, 1, 0, (NONE, NONE)), (64, 64, 3, 2, 0, 16, 0, (NONE, NONE)), (64, 64, 3, 2, 0, 17, 0, (NONE, NONE)),
    (192, 320, 7, 3, 1, 4, 0, (NONE, NONE)), (320, 4224, 4, 2, 0, 4, 1, (NONE, NONE)), (64, 192, 200, 6, 2, 3, 0, (NONE, NONE)),
    (192, 320, 7, 3, 1, 5, 0, (NONE, NONE)), (192, 320, 7, 3, 1, 8, 0, (NONE, NONE)), (192, 320, 7, 3, 1, 9, 1, (NONE, NONE)), (192, 320, 7, 3, 1, 17, 1, (NONE, NONE)),
    (320, 192, 2, 2, 0, 80, 0, (NONE, NONE)), (320, 192, 2, 2, 0, 81, 0, (NONE, NONE)), (320, 192, 2, 2, 1, 160, 1, (NONE, NONE)),
    (320, 192, 2, 2, 0, 161, 0, (NONE, NONE)), (64, 4160, 3, 2, 1, 5, 0, (NONE, NONE)), (192, 8256, 2, 1, 0, 33, 0, (NONE, NONE)),
    (64, 192, 200, 6, 2, 16, 0, (NONE, NONE)), (192, 64, 200, 6, 2, 70, 0, (NONE, NONE)),
    (192, 320, 7, 3, 1, 40, 0, (NONE, 0)), (192, 320, 7, 3, 1, 40, 0, (0, NONE)), (192, 320, 7, 3, 1, 40, 0, (17, 9)),
]


@pytest.mark.parametrize("C,R,E,k,ns,T,fmt,mins", CASES)
@pytest.mark.parametrize("uneven", [False, True])
def test_streaming_kernels(C, R, E, k, ns, T, fmt, mins, uneven):
    from paper_2609_38090_b200 import binding as b
    sh = inputs.LayerShape("edges", C=C, R=R, E=E, k=k, T=T, n_shared=ns, zipf_a=1.1, seed=C + R + T)
    wl = Workload(sh, T, gen=_uneven if uneven else None, fmt=fmt)
    d = wl.device_inputs()
    m = b.Mira(C, R, E, n_shared=ns, max_tokens=T, max_top_k=k, out_fp32=True, act_on_w1=bool(fmt), fmt=fmt)
    blobs = m.quantize_experts(d["w1"], d["w2"], d["w3"])
    m.hybrid_min(*mins)
    slot_map = torch.arange(E + ns, dtype=torch.int32, device="cuda")
    out, dbg = m.moe_layer(d["x"], d["wr"], d["bias"], b.slot_table(blobs), slot_map, k, debug=True)
    torch.cuda.synchronize()
    assert m.poll_status()[0] == 0
    idx, w, _, _ = oracle.topk_softmax(oracle.linear_scores(wl.x, wl.wr, wl.bias), k)
    assert np.array_equal(dbg["idx"].cpu().numpy(), idx)
    ref, tol = _reference(wl, idx, w, bool(fmt), 0 if mins == (NONE, NONE) else max(C, R) // 16)
    err = np.abs(out.cpu().numpy() - ref)
    assert (err <= tol).all(), f"{(err / tol).max():.2f} of the bound"


@pytest.mark.parametrize("layout", [1, 2, 3, 4])
@pytest.mark.parametrize("C,R,T,slices", [(256, 128, 40, 1), (128, 192, 130, 1), (256, 1088, 200, 1), (256, 4224, 33, 2), (128, 8320, 70, 3)])
def test_weight_boxes_of_the_tensor_core_kernels(layout, C, R, T, slices):
    """The kernels for large batches load the weights in boxes of 128 codes, two blocks of the reduction: an odd number of blocks
    (R / 64), slices that begin at an odd one, rings that wrap inside a tile and between tiles, several token tiles per expert."""
    from paper_2609_38090_b200 import binding as b
    sh = inputs.LayerShape("boxes", C=C, R=R, E=3, k=2, T=T, n_shared=1, zipf_a=1.1, seed=R + T)
    wl = Workload(sh, T, gen=_uneven if R == 192 else None)
    d = wl.device_inputs()
    m = b.Mira(C, R, 3, n_shared=1, max_tokens=T, max_top_k=2, out_fp32=True)
    blobs = m.quantize_experts(d["w1"], d["w2"], d["w3"])
    m.hybrid_min(0, 0)
    m.tensor_layout(layout)
    m.down_slices(slices)
    out, dbg = m.moe_layer(d["x"], d["wr"], d["bias"], b.slot_table(blobs), torch.arange(4, dtype=torch.int32, device="cuda"), 2, debug=True)
    torch.cuda.synchronize()
    assert m.poll_status()[0] == 0
    idx, w, _, _ = oracle.topk_softmax(oracle.linear_scores(wl.x, wl.wr, wl.bias), 2)
    assert np.array_equal(dbg["idx"].cpu().numpy(), idx)
    ref, tol = _reference(wl, idx, w, False, max(C, R) // 16)
    err = np.abs(out.cpu().numpy() - ref)
    assert (err <= tol).all(), f"{(err / tol).max():.2f} of the bound"
