"""Decode at the edges of its merges: more partials than one batch of the merging CTA, counts one below, at and above a
batch, one split (no merge through global memory), heads that fill one or two 8-head tiles or neither, both head dims."""
import numpy as np
import pytest
import torch

import paper_2609_13612_b200 as af
import parity_util as pu
from test_gpu_decode import draw, oracle_decode

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("group,Hkv,N,splits", [(1, 1, 6000, 47), (8, 1, 2700, 20), (9, 2, 2700, 21), (16, 1, 2500, 19), (3, 3, 640, 4), (5, 1, 641, 6),
                                                (7, 2, 15, 0), (2, 1, 5200, 41)])
def test_decode_merges(group, Hkv, N, splits, D):
    q, k, v = draw(2, group * Hkv, Hkv, N, D, 900 + group)
    mask = af.MaskSpec(True, -1, None)
    o, lse = af.decode(pu.to_dev(q), pu.to_dev(k), pu.to_dev(v), mask, D ** -0.5, n_splits=splits)
    torch.cuda.synchronize()
    assert af.device_status()[0] == 0
    want_o, want_l = oracle_decode(q, k, v, D ** -0.5)
    pu.assert_close("decode O", pu.to_np(o), want_o)
    assert np.abs(pu.to_np(lse) - want_l).max() <= pu.LSE_TOL
