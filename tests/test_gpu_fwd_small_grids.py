"""Forward on grids that leave SMs idle: one query tile per CTA, and key tiles shared out over a cluster of CTAs.  The sizes
reach every cluster size, shares that fall away (fewer tiles than CTAs), ragged lengths, windows (shares without a kept
pair for some rows), both output types, the hybrid arm and block lists; the last test keeps the two-tile kernels covered
at the sizes of the other tests."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_13612_b200 as af
from paper_2609_13612_b200 import synth
import parity_util as pu
from test_gpu_fwd import SMALL, run_case

pytestmark = pytest.mark.gpu
W = synth.Workload


@pytest.mark.parametrize("w", [
    W("one_head_long", 1, 1, 1, 3001, 128, theta=1e4, seed_id=801),
    W("gqa_ragged", 1, 4, 1, 1999, 64, theta=1e4, rotary_dim=32, alibi=True, seed_id=802),
    W("noncausal", 1, 2, 1, 1300, 128, theta=1e4, causal=False, seed_id=803),
    W("window_shares", 1, 2, 2, 2500, 128, theta=1e4, window=900, seed_id=804),
    W("no_rotation", 1, 3, 1, 2100, 64, rotary_dim=0, seed_id=805),
    W("two_parts", 1, 8, 2, 1000, 128, theta=1e4, seed_id=806),
], ids=lambda w: w.name)
@pytest.mark.parametrize("out_dtype", [torch.bfloat16, torch.float32], ids=["bf16", "fp32"])
def test_shared_key_tiles(w, out_dtype):
    t = synth.draw_all(w)
    dev = {k: pu.to_dev(v) for k, v in t.items()}
    o, lse = pu.gpu_fwd(w, dev, out_dtype=out_dtype)
    want_o, want_l = oracle.run_workload(w, t)
    pu.assert_close(w.name, pu.to_np(o), want_o)
    assert np.abs(pu.to_np(lse) - want_l).max() <= pu.LSE_TOL
    if w.R > 0:
        rope, mask = pu.specs(w)
        oh, lh = af.fwd_hybrid(dev["q"], dev["k"], dev["v"], rope, af.rope_table(rope, w.S), mask, w.scale, out_dtype=out_dtype)
        pu.assert_close(w.name + " hybrid", pu.to_np(oh), want_o)
        assert np.abs(pu.to_np(lh) - want_l).max() <= pu.LSE_TOL


@pytest.mark.parametrize("w", SMALL, ids=lambda w: w.name)
def test_forward_small_two_query_tiles_per_cta(w):
    with af.option(af.OPT_FWD_QTILES, 3):
        run_case(w)


@pytest.mark.parametrize("B,Hq,Hkv,S,causal,window,same_as", [
    (1, 20, 4, 1024, True, -1, 1),     # 160 tiles: the CTAs that follow others on an SM are the short ones
    (1, 20, 4, 1024, False, -1, 3),    # all alike: two waves of one tile would be slower than one of two
    (1, 2, 2, 10752, True, 300, 3),
    (1, 160, 8, 128, True, -1, 3),
    (1, 18, 6, 1024, False, -1, 1),    # 144 tiles: one wave either way
])
def test_query_tiles_per_cta_on_grids_a_little_larger_than_the_device(B, Hq, Hkv, S, causal, window, same_as):
    """The choice shows in the bits: with ALiBi the kernels for one and for two query tiles add the term in different places."""
    g = torch.Generator(device="cuda").manual_seed(808)
    q, k, v = (torch.randn(B, h, S, 128, generator=g, device="cuda").to(torch.bfloat16) for h in (Hq, Hkv, Hkv))
    slopes = torch.tensor([2.0 ** (-8.0 * (h + 1) / Hq) for h in range(Hq)], device="cuda")
    rope, mask = af.RopeSpec(theta=1e4, rotary_dim=128), af.MaskSpec(causal=causal, window=window, alibi_slopes=slopes)
    table = af.rope_table(rope, S)
    got = {}
    for option in (1, 2, 3):
        with af.option(af.OPT_FWD_QTILES, option):
            got[option] = af.fwd(q, k, v, rope, table, mask, 128 ** -0.5)[1]
    torch.cuda.synchronize()
    assert af.device_status()[0] == 0
    if torch.cuda.get_device_properties(0).multi_processor_count == 148:   # the line lies at the number of SMs
        assert not torch.equal(got[1], got[3])
        assert torch.equal(got[2], got[same_as])
