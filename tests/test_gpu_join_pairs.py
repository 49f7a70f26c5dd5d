"""Joining on both sides of the rule that sends the pairs of windows through a launch of their own: one and many pairs
per warp, 32 and 33 of them, 1024 bins of all pairs and more.  Bit for bit the oracle's."""
import numpy as np
import pytest

import oracle
import paper_1411_4212_gb300 as rw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h,W,step", [(2, 1024, 300), (2, 1025, 300), (3, 512, 100), (3, 513, 100), (33, 32, 8), (33, 33, 8),
                                      (34, 30, 8), (32, 33, 20), (5, 3, 1)])
def test_join_of_few_windows(h, W, step):
    import torch
    starts = np.array([k * step for k in range(h)], dtype=np.int32)
    B = int(starts[-1]) + W
    rng = np.random.default_rng(h * W)
    base = np.cumsum(rng.normal(0.1, 1.0, B))
    frag = np.stack([base[s:s + W] + rng.normal(0, 2.0, (2, W)) + rng.normal(0, 50, (2, 1)) for s in starts])
    out = torch.empty(B, dtype=torch.float64, device="cuda")
    rw.stitch_device(torch.from_numpy(frag).cuda(), starts, B, out)
    ref = oracle.merge_fragments(frag, starts, B)
    ref = ref[0] if isinstance(ref, tuple) else ref
    assert np.array_equal(out.cpu().numpy().view(np.int64), np.asarray(ref).view(np.int64))
