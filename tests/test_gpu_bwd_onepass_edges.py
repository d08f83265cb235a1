"""One-pass backward at the edges of its parts: the first query rows (fp32, beside the MMA work when dK and dV are fp32,
behind it when they are bf16), the set-up pass and the last pass of dQ - sequences shorter than, equal to and one past
the 16 first rows and the 128-row tile, every panel remainder of the query group, partial rotary widths."""
import pytest
import torch

import oracle
import paper_2609_13612_b200 as af
from paper_2609_13612_b200 import synth
import parity_util as pu

pytestmark = pytest.mark.gpu
W = synth.Workload


@pytest.mark.parametrize("dkv", [torch.float32, torch.bfloat16], ids=["fp32", "bf16"])
@pytest.mark.parametrize("S,group,D,R", [(7, 1, 128, 128), (16, 3, 64, 64), (17, 5, 128, 64), (129, 4, 64, 32), (300, 2, 128, 48), (260, 1, 64, 0)])
def test_onepass_edges(S, group, D, R, dkv):
    w = W("onepass_edge", 2, 2 * group, 2, S, D, theta=1e4, rotary_dim=R, backward=True, sigma=0.5, seed_id=700 + S + group)
    t = synth.draw_all(w)
    dev = {k: pu.to_dev(v) for k, v in t.items()}
    o, lse = pu.gpu_fwd(w, dev)
    with af.option(af.OPT_BWD_ONEPASS, 2):
        got = pu.gpu_bwd(w, dev, o, lse, dkv_dtype=dkv)
    want = oracle.run_workload(w, t, backward=True)
    for name, g, ref in zip(("dQ", "dK", "dV"), got, want):
        # (the bound of the parity tests; a bf16 dK or dV adds two roundings of half an ulp, 2^-8 of its value in all)
        pu.assert_close_scaled("%s %s" % (w.name, name), pu.to_np(g), ref)


@pytest.mark.parametrize("B,Hkv,group,S,D,causal,window", [
    (1, 1, 8, 600, 128, True, -1),      # clusters of 8; the last key tiles share out fewer than 8 ways
    (2, 2, 3, 777, 128, True, 300),     # 4, odd group: parts begin in the middle of a head
    (1, 1, 1, 640, 64, False, 100),     # few tiles per key tile, first ones not at the diagonal
    (1, 8, 4, 1530, 128, True, -1),     # 2
    (1, 4, 2, 1000, 64, False, -1),     # no mask at all
])
def test_key_tiles_shared_out_over_a_cluster(B, Hkv, group, S, D, causal, window):
    w = W("onepass_cluster", B, Hkv * group, Hkv, S, D, theta=1e4, causal=causal, window=window, alibi=causal, backward=True, seed_id=760 + S)
    t = synth.draw_all(w)
    dev = {k: pu.to_dev(v) for k, v in t.items()}
    o, lse = pu.gpu_fwd(w, dev)
    got = pu.gpu_bwd(w, dev, o, lse)
    again = pu.gpu_bwd(w, dev, o, lse)
    want = oracle.run_workload(w, t, backward=True)
    for name, g, ref in zip(("dQ", "dK", "dV"), got, want):
        pu.assert_close_scaled("%s %s" % (w.name, name), pu.to_np(g), ref)
    # the sums over the cluster run in rank order
    assert torch.equal(got[1], again[1]) and torch.equal(got[2], again[2])


def test_more_heads_than_a_grid_dimension_takes_in_groups():
    """The last pass of dQ takes the heads in groups of four along y (at most 65535)."""
    B, H, S, D = 4, 65540, 8, 64
    g = torch.Generator(device="cuda").manual_seed(811)
    q, k, v, do = (torch.randn(B, H, S, D, generator=g, device="cuda").to(torch.bfloat16) for _ in range(4))
    rope, mask = af.RopeSpec(), af.MaskSpec()
    o, lse = af.fwd(q, k, v, rope, None, mask, 0.125)
    got = af.bwd(q, k, v, o, lse, do, rope, None, mask, 0.125)
    torch.cuda.synchronize()
    assert af.device_status()[0] == 0
    for b in range(B):
        qf, kf, vf = (t[b].float().requires_grad_() for t in (q, k, v))
        s = (qf @ kf.transpose(1, 2) * 0.125).masked_fill(torch.ones(S, S, device="cuda").triu(1).bool(), float("-inf"))
        (torch.softmax(s, -1) @ vf).backward(do[b].float())
        for x, ref in zip(got, (qf.grad, kf.grad, vf.grad)):
            # (a bf16 dQ is off by half an ulp, 2^-9 of its value)
            assert ((x[b].float() - ref).abs() <= 2e-2 + pu.BF16_ULP * ref.abs()).all()


def test_as_many_key_tiles_as_a_grid_dimension_takes():
    """65535 key tiles: no row of the grid is left for the first query rows.  With a window the rows of a slice of the sequence
    are those of the whole, away from its ends."""
    S, D, W_, M = 65535 * 128, 64, 100, 1024
    g = torch.Generator(device="cuda").manual_seed(812)
    q, k, v, do = (torch.randn(1, 1, S, D, generator=g, device="cuda", dtype=torch.bfloat16) for _ in range(4))
    rope, mask = af.RopeSpec(), af.MaskSpec(window=W_)

    def run(a, b):
        x = [t[:, :, a:b].contiguous() for t in (q, k, v, do)]
        o, lse = af.fwd(x[0], x[1], x[2], rope, None, mask, 0.125)
        return (o,) + af.bwd(x[0], x[1], x[2], o, lse, x[3], rope, None, mask, 0.125)
    whole = run(0, S)
    torch.cuda.synchronize()
    assert af.device_status()[0] == 0
    for a in (0, S // 2 // 128 * 128, S - M):
        lo, hi = (0 if a == 0 else 2 * W_), (M if a + M == S else M - 2 * W_)
        for x, y in zip(whole, run(a, a + M)):
            x, y = x[:, :, a + lo:a + hi].float(), y[:, :, lo:hi].float()
            assert torch.isfinite(x).all() and ((x - y).abs() <= 2e-2 + pu.BF16_ULP * y.abs()).all()
