"""The network's tensor-core kernels at the edges of their tiles (16 samples a warp, 128 a CTA, one and two
rounds of all CTAs, which is a chunk of the backward pass), against the FP64 oracle.

Tolerance: FP32 operands are split exactly into BF16 parts, so what is left are the roundings of blocks of
16 terms and of their sums.  Each of the five contractions in a row contributes at most 2^-22 of the
operands' size (a unit in the last place per block and per addition, mostly cancelling), the elementwise
functions a few units of 2^-24: 2e-6 of the gradient's norm, for targets that differ smoothly from the
output (a gradient of noise would cancel)."""
import numpy as np
import pytest

import paper_1411_4212_gb300 as rw
from oracle import mlp_oracle as mo

pytestmark = pytest.mark.gpu

SHIFT = np.array([-1.9, 0.19, 1.0, 0.4, 0.0, 0.0], dtype=np.float32)
SCALE = np.array([1 / 1.1, 20.0, 1.0, 5.0, 10.0, 1.0], dtype=np.float32)


def _sizes():
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 152
    round_of_ctas = sms * 8 * 16
    return [1, 15, 17, 127, 129, 16 * sms + 1, round_of_ctas - 1, 2 * round_of_ctas, 2 * round_of_ctas + 1]


@pytest.mark.parametrize("which", range(9))
def test_gradient_at_tile_and_chunk_edges(which):
    M = _sizes()[which]
    rng = np.random.default_rng(which)
    x = np.zeros((M, 6), dtype=np.float32)
    x[:, 0] = np.linspace(-3.3, -0.01, M)
    x[:, 1] = rng.choice([1 / 4, 1 / 5, 1 / 6], M)
    x[:, 2:4] = 1.0, 0.45
    x[:, 4] = 0.05
    t = (-0.3 * x[:, 0] ** 2 + x[:, 1]).astype(np.float32)
    seg = np.unique(np.concatenate([[0], np.linspace(0, M, min(M, 7) + 1).astype(int), [M]])).astype(np.int32)
    net = rw.Mlp(SHIFT, SCALE, seed=which)
    pb = net.params(bf16=True).astype(np.float64)
    sh, sc = SHIFT.astype(np.float64), SCALE.astype(np.float64)
    Lo, go = mo.loss_and_grad(pb, x.astype(np.float64), t.astype(np.float64), seg, sh, sc)
    yo, _ = mo.forward(pb, x.astype(np.float64), sh, sc)
    y = net.forward(x)
    assert np.linalg.norm(y - yo) <= 2e-6 * np.linalg.norm(yo) + 1e-7 * np.sqrt(M)
    L, g = net.gradient(x, t, seg)
    assert abs(L - Lo) <= 2e-6 * Lo + 1e-12
    assert np.linalg.norm(g - go) <= 2e-6 * np.linalg.norm(go) + 1e-9, np.linalg.norm(g - go) / np.linalg.norm(go)
    L2, g2 = net.gradient(x, t, seg)           # the chunks' sums start afresh
    assert L2 == L and np.array_equal(g.view(np.int32), g2.view(np.int32))
    net.close()
