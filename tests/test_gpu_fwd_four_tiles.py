"""Forward with four query tiles per CTA (D = 64, dense masks, grids that fill the device): 64-key steps, groups that put four, two or
one head into a CTA, row blocks without rows, ragged lengths at the edges of steps and tiles, windows that start in the second half of
a key tile, both output types."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_13612_b200 as af
from paper_2609_13612_b200 import synth
import parity_util as pu

pytestmark = pytest.mark.gpu
W = synth.Workload


@pytest.mark.parametrize("w", [
    W("one_tile_each", 40, 8, 2, 65, 64, theta=1e4, seed_id=901),
    W("second_step_full", 40, 8, 8, 128, 64, theta=1e4, seed_id=902),
    W("rows_beyond_a_step", 32, 8, 4, 129, 64, theta=1e4, seed_id=903),
    W("two_heads_two_blocks", 16, 12, 2, 257, 64, theta=1e4, rotary_dim=32, seed_id=904),
    W("one_head_four_blocks", 16, 9, 3, 511, 64, theta=1e4, seed_id=905),
    W("fifth_block", 16, 6, 6, 577, 64, theta=1e4, rotary_dim=16, seed_id=906),
    W("window_in_second_half", 12, 8, 8, 700, 64, theta=1e4, window=70, seed_id=907),
    W("window_alibi", 12, 8, 4, 640, 64, theta=1e4, window=200, alibi=True, seed_id=908),
    W("window_zero", 24, 8, 8, 300, 64, theta=1e4, window=0, seed_id=909),
    W("noncausal", 12, 8, 1, 450, 64, theta=1e4, causal=False, seed_id=910),
    W("noncausal_window", 12, 9, 9, 500, 64, theta=1e4, causal=False, window=130, seed_id=911),
    W("no_rotation", 12, 16, 4, 520, 64, rotary_dim=0, seed_id=912),
    W("rotary_48", 12, 12, 12, 400, 64, theta=1e4, rotary_dim=48, seed_id=913),
    # (128 k - window) / 64 is odd where window mod 128 is 1 ... 64: a CTA's first step is the second half of a key tile
    W("odd_first_step", 6, 8, 2, 700, 64, theta=1e4, window=40, rotary_dim=32, seed_id=916),
    W("odd_first_step_rows", 4, 6, 6, 1300, 64, theta=1e4, window=130, rotary_dim=16, seed_id=917),
    W("odd_first_step_noncausal", 3, 9, 3, 1100, 64, theta=1e4, causal=False, window=150, seed_id=918),
    W("odd_first_step_alibi", 3, 4, 2, 900, 64, theta=1e4, window=300, alibi=True, seed_id=919),
], ids=lambda w: w.name)
@pytest.mark.parametrize("out_dtype", [torch.bfloat16, torch.float32], ids=["bf16", "fp32"])
def test_against_the_oracle_and_the_kernel_for_two(w, out_dtype):
    t = synth.draw_all(w)
    dev = {k: pu.to_dev(v) for k, v in t.items()}
    rope, mask = pu.specs(w)
    table = af.rope_table(rope, w.S)
    want_o, want_l = oracle.run_workload(w, t)
    # non-causal windows and ALiBi give few-key rows, whose outputs carry the roundings undivided: the generated examples' bound
    for call in (af.fwd, af.fwd_hybrid):
        o = torch.full((w.B, w.Hq, w.S, w.D), float("nan"), dtype=out_dtype, device="cuda")
        lse = torch.full((w.B, w.Hq, w.S), float("nan"), dtype=torch.float32, device="cuda")
        with af.option(af.OPT_FWD_QTILES, 4):
            call(dev["q"], dev["k"], dev["v"], rope, table, mask, w.scale, out=o, lse=lse)
        torch.cuda.synchronize()
        assert af.device_status()[0] == 0
        pu.assert_close_scaled(w.name, pu.to_np(o), want_o)
        assert np.abs(pu.to_np(lse) - want_l).max() <= pu.LSE_TOL
    with af.option(af.OPT_FWD_QTILES, 3):
        o2, _ = af.fwd(dev["q"], dev["k"], dev["v"], rope, table, mask, w.scale, out_dtype=out_dtype)
    torch.cuda.synchronize()
    pu.assert_close_scaled(w.name + " two", pu.to_np(o2), want_o)
    if w.S >= 128 and w.window != 0:   # (steps of 64 keys: other last bits, where rows have more than a step)
        assert not torch.equal(o, o2)


@pytest.mark.parametrize("B,Hq,Hkv,S,window,four", [
    (16, 16, 4, 600, -1, True), (4, 12, 12, 4096, -1, True), (8, 12, 12, 1024, -1, True), (16, 8, 4, 900, 70, True),
    (1, 16, 4, 2048, -1, False), (2, 12, 12, 4096, -1, False),
    # grids whose last wave decides (two / four: 58 / 75, 175 / 139, 64 / 51 us)
    (1, 8, 2, 6128, 2364, False), (4, 36, 12, 3270, 136, True), (8, 24, 8, 896, -1, True),
])
def test_which_calls_take_four(B, Hq, Hkv, S, window, four):
    g = torch.Generator(device="cuda").manual_seed(920)
    q, k, v = (torch.randn(B, h, S, 64, generator=g, device="cuda").to(torch.bfloat16) for h in (Hq, Hkv, Hkv))
    got = {}
    for option in (2, 3, 4):
        with af.option(af.OPT_FWD_QTILES, option):
            got[option] = af.fwd(q, k, v, af.RopeSpec(rotary_dim=0), None, af.MaskSpec(window=window), 0.125, out_dtype=torch.float32)[0]
    torch.cuda.synchronize()
    assert not torch.equal(got[3], got[4])
    assert torch.equal(got[2], got[4 if four else 3])
    assert af.device_status()[0] == 0


def test_infinite_and_nan_scores_as_in_the_kernel_for_two():
    """A key row of -inf takes part with weight zero (NaN where the products are), a NaN key row spoils the rows that see it."""
    g = torch.Generator(device="cuda").manual_seed(914)
    q, k, v = (torch.randn(16, h, 300, 64, generator=g, device="cuda").to(torch.bfloat16) for h in (8, 8, 8))
    q = q.abs()
    k[:, :, 7] = float("-inf")
    k[:, 1, 200] = float("nan")
    got = {}
    for option in (4, 3):
        with af.option(af.OPT_FWD_QTILES, option):
            got[option] = af.fwd(q, k, v, af.RopeSpec(rotary_dim=0), None, af.MaskSpec(), 0.125)
    torch.cuda.synchronize()
    assert af.device_status()[0] == 0
    for a, b in zip(got[4], got[3]):
        assert torch.equal(torch.isnan(a), torch.isnan(b)) and torch.equal(torch.isinf(a), torch.isinf(b))
        ok = torch.isfinite(b)
        assert (a[ok].float() - b[ok].float()).abs().max().item() <= 2.0 ** -6   # one bf16 ulp at |x| < 4, and P's rounding


def test_alibi_by_the_tensor_core_where_it_was_asked_for():
    """AF_OPT_FWD_ALIBI_MMA = 2 is for every forward kernel that can: with slopes it keeps away from the kernel for four, which cannot."""
    g = torch.Generator(device="cuda").manual_seed(915)
    q, k, v = (torch.randn(16, h, 600, 64, generator=g, device="cuda").to(torch.bfloat16) for h in (16, 4, 4))
    slopes = torch.tensor([2.0 ** -(h / 2 + 1) for h in range(16)], dtype=torch.float32, device="cuda")
    args = (q, k, v, af.RopeSpec(rotary_dim=0), None, af.MaskSpec(alibi_slopes=slopes), 0.125)
    with af.option(af.OPT_FWD_ALIBI_MMA, 2):
        got = af.fwd(*args)
        with af.option(af.OPT_FWD_QTILES, 3):
            want = af.fwd(*args)
    plain = af.fwd(*args)
    torch.cuda.synchronize()
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    assert not torch.equal(plain[0], want[0])   # (by itself this call takes four: other last bits)
    assert af.device_status()[0] == 0


@pytest.mark.parametrize("causal,window,alibi", [(True, -1, False), (True, 300, False), (True, 700, True), (True, -1, True), (False, -1, False),
                                                 (False, 200, False)])
def test_no_less_precise_than_two(causal, window, alibi):
    """Against fp64 on the same inputs.  Over 8e5 outputs the 2-norm of the error scatters by 0.1 %: five times that is allowed."""
    B, H, S = 1, 8, 1600
    g = torch.Generator(device="cuda").manual_seed(921)
    q, k, v = (torch.randn(B, H, S, 64, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    slopes = torch.tensor([2.0 ** -(h + 1) for h in range(H)], dtype=torch.float32, device="cuda") if alibi else None
    i, j = torch.arange(S, device="cuda")[:, None], torch.arange(S, device="cuda")
    s = q.double() @ k.double().transpose(2, 3) * 0.125
    if alibi:
        s = s + slopes.double()[None, :, None, None] * (j - i)
    keep = (j <= i) if causal else (j >= 0) & (i >= 0)
    if window >= 0:
        keep = keep & ((i - j).abs() <= window)
    want = torch.softmax(s.masked_fill(~keep, float("-inf")), -1) @ v.double()
    err = {}
    for option in (3, 4):
        with af.option(af.OPT_FWD_QTILES, option):
            o, _ = af.fwd(q, k, v, af.RopeSpec(rotary_dim=0), None, af.MaskSpec(causal=causal, window=window, alibi_slopes=slopes), 0.125,
                          out_dtype=torch.float32)
        err[option] = (o.double() - want).norm().item()
    assert af.device_status()[0] == 0
    assert err[4] <= 1.005 * err[3], err
