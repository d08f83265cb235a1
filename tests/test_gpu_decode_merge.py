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


@pytest.mark.parametrize("D", [64, 128])
@pytest.mark.parametrize("splits", [1, 3, 19, 20, 21, 24])
def test_infinities_of_the_cache_stay_infinities(splits, D):
    """An infinity in V makes its head dim infinite (its weight is positive), whichever split holds it; the others stay
    finite."""
    N = 3000
    q, k, v = draw(1, 6, 2, N, D, 930)
    qd, kd, vd = pu.to_dev(q), pu.to_dev(k), pu.to_dev(v)
    vd[:, :, N - 2, 5] = float("inf")     # last split
    vd[:, :, 3, 9] = -float("inf")        # first
    vd[:, :, N // 2, 17] = float("inf")
    o, lse = af.decode(qd, kd, vd, af.MaskSpec(), 1.0 / 64, n_splits=splits)
    torch.cuda.synchronize()
    assert af.device_status()[0] == 0 and torch.isfinite(lse).all()
    for d in range(D):
        want = {5: float("inf"), 17: float("inf"), 9: -float("inf")}.get(d)
        assert torch.isfinite(o[..., d]).all() if want is None else (o[..., d] == want).all(), d


@pytest.mark.parametrize("D,N", [(128, 7812), (128, 7813), (64, 15626)])   # 4 MB of keys and values per CTA: dependent or plain launch
def test_long_splits(D, N):
    q, k, v = draw(1, 2, 1, N, D, 940)
    o, lse = af.decode(pu.to_dev(q), pu.to_dev(k), pu.to_dev(v), af.MaskSpec(), D ** -0.5, n_splits=1)
    torch.cuda.synchronize()
    assert af.device_status()[0] == 0
    want_o, want_l = oracle_decode(q, k, v, D ** -0.5)
    pu.assert_close("decode O", pu.to_np(o), want_o)
    assert np.abs(pu.to_np(lse) - want_l).max() <= pu.LSE_TOL
