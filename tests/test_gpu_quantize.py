"""The quantizer's kernels at the edges of their partitions, bit for bit against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2609_38090_b200 import inputs

pytestmark = pytest.mark.gpu


def _weights(R, C, seed, dtype):
    """Gaussian weights, a row of zeros, one of very small values, and (bf16 has few distinct quotients anyway) values that
    lie exactly between two codes: (code + 1/2) times a power-of-two scale in a row whose largest value is 127 times it."""
    g = np.random.default_rng(seed)
    w = [0.02 * g.standard_normal(s).astype(np.float32) for s in ((R, C), (C, R), (R, C))]
    if R > 3:
        w[0][1], w[1][:, 1], w[2][1] = 0, 0, 0
        w[0][2] *= 1e-12; w[1][:, 2] *= 1e-12; w[2][2] *= 1e-12
        for m in (w[0], w[2]):
            m[3] = (g.integers(-126, 126, C) + 0.5) * 2.0 ** -10
        w[1][:, 3] = (g.integers(-126, 126, C) + 0.5) * 2.0 ** -10
        w[0][3, C // 2] = 127 * 2.0 ** -10
    return [inputs.round_to_bf16(m) for m in w] if dtype == "bf16" else w


# R: one strip of 32 / 64 rows, odd numbers of strips; C / 8 rows per CTA: 8, 24, more than one round of loads.
# Per-matrix rows: the lengths at which the number of threads per row steps up, and one 16-byte vector more.
@pytest.mark.parametrize("R,C", [(64, 64), (192, 192), (320, 2048), (64, 2112), (1088, 1024), (2112, 128), (64, 8256), (16384, 64), (192, 16384)])
@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("fmt", [0, 1])
def test_codes_and_scales_at_the_edges_of_the_partition(R, C, dtype, fmt):
    from paper_2609_38090_b200 import binding as b
    m = b.Mira(C, R, 2, max_tokens=1, max_top_k=1, fmt=fmt)
    ws = [_weights(R, C, 7 * R + C + e, dtype) for e in range(2)]
    dev = [torch.from_numpy(np.stack([w[i] for w in ws])).cuda().to(torch.bfloat16 if dtype == "bf16" else torch.float32) for i in range(3)]
    out = torch.full((3, m.expert_bytes), 0x5A, dtype=torch.uint8, device="cuda")
    m.quantize_experts(*dev, out=out)
    got = out.cpu().numpy()
    for e in range(2):
        assert np.array_equal(got[e], oracle.quantize_expert(*ws[e], fmt=fmt)), f"expert {e}"
    assert (got[2] == 0x5A).all()                    # nothing behind the call's blobs


def test_scales_whose_reciprocal_overflows():
    """With a tiny epsilon a row of subnormal weights gets a scale whose reciprocal is infinite: such rows are divided."""
    from paper_2609_38090_b200 import binding as b
    R, C, eps = 64, 128, 1e-38
    g = np.random.default_rng(3)
    w = [(0.02 * g.standard_normal(s)).astype(np.float32) for s in ((R, C), (C, R), (R, C))]
    w[0][5] *= 1e-37; w[1][:, 5] *= 1e-37; w[2][5] *= 1e-37
    w[0][6], w[1][:, 6], w[2][6] = 0, 0, 0
    m = b.Mira(C, R, 1, max_tokens=1, max_top_k=1, eps=eps)
    got = m.quantize_experts(*[torch.from_numpy(x[None]).cuda() for x in w]).cpu().numpy()[0]
    assert np.array_equal(got, oracle.quantize_expert(*w, eps=eps))
