"""Forward with scratch memory: the keys rotated once, ahead of the kernel, have the bits of the on-chip rotation."""
import ctypes

import pytest
import torch

import paper_2609_13612_b200 as af
from paper_2609_13612_b200 import binding as b

pytestmark = pytest.mark.gpu


def scratch_bytes(B, Hq, Hkv, S, D, R, causal=True, window=-1, slopes=None):
    sh, r, m = b._Shape(B, Hq, Hkv, S, D), b._Rope(1e4, R, 0), b._Mask(int(causal), window, slopes)
    return af.lib().attnfuse_fwd_scratch_bytes(ctypes.byref(sh), ctypes.byref(r), ctypes.byref(m), Hq // Hkv)


@pytest.mark.parametrize("B,Hq,Hkv,S,D,R,causal", [
    (1, 32, 8, 2100, 128, 128, True),    # 17 key tiles: a second run of four, a last tile with few rows
    (2, 36, 12, 2049, 128, 64, True),    # odd number of tiles, columns that are copied
    (1, 40, 8, 5000, 128, 32, True),
    (2, 16, 4, 5200, 128, 16, False),
    (1, 32, 8, 2049, 128, 96, True),     # no angle-addition walk: the table is read for every row
    (4, 12, 12, 2300, 64, 64, True),
    (8, 12, 4, 1700, 64, 32, False),
])
def test_same_bits_as_on_chip(B, Hq, Hkv, S, D, R, causal):
    g = torch.Generator(device="cuda").manual_seed(921)
    assert scratch_bytes(B, Hq, Hkv, S, D, R, causal) == B * Hkv * S * D * 2
    q = torch.randn(B, Hq, S, D, generator=g, device="cuda").to(torch.bfloat16)
    kv = torch.randn(2, B, S, Hkv, D, generator=g, device="cuda").to(torch.bfloat16).transpose(2, 3)   # strided keys
    rope, mask = af.RopeSpec(theta=1e4, rotary_dim=R), af.MaskSpec(causal=causal)
    table = af.rope_table(rope, S)
    o, lse = torch.full_like(q, float("nan")), torch.full((B, Hq, S), float("nan"), device="cuda")
    before = kv.clone()
    af.fwd(q, kv[0], kv[1], rope, table, mask, D ** -0.5, out=o, lse=lse)
    want_o, want_l = af.fwd_variant(q, kv[0], kv[1], rope, table, mask, D ** -0.5)   # always on chip
    torch.cuda.synchronize()
    assert af.device_status()[0] == 0
    assert torch.equal(o, want_o) and torch.equal(lse, want_l) and torch.equal(kv, before)


@pytest.mark.parametrize("B,Hq,Hkv,S,R,causal", [(4, 16, 4, 2300, 64, True), (8, 16, 4, 2300, 32, True), (8, 16, 4, 4600, 16, True),
                                                 (4, 16, 4, 2300, 48, True), (4, 9, 9, 1900, 64, False), (4, 12, 6, 2111, 64, True)])
def test_same_bits_with_four_query_tiles(B, Hq, Hkv, S, R, causal):
    g = torch.Generator(device="cuda").manual_seed(923)
    q, k, v = (torch.randn(B, h, S, 64, generator=g, device="cuda").to(torch.bfloat16) for h in (Hq, Hkv, Hkv))
    rope, mask = af.RopeSpec(theta=1e4, rotary_dim=R), af.MaskSpec(causal=causal)
    args = (q, k, v, rope, af.rope_table(rope, S), mask, 0.125)
    with af.option(af.OPT_FWD_QTILES, 4):
        assert scratch_bytes(B, Hq, Hkv, S, 64, R, causal) == B * Hkv * S * 64 * 2
        got, want = af.fwd(*args), af.fwd_variant(*args)
    with af.option(af.OPT_FWD_QTILES, 3):
        two = af.fwd(*args)
    torch.cuda.synchronize()
    assert af.device_status()[0] == 0
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    assert not torch.equal(got[0], two[0])


def test_scratch_that_is_missing_short_or_misaligned():
    B, Hq, Hkv, S, D = 1, 16, 4, 3000, 128
    g = torch.Generator(device="cuda").manual_seed(924)
    q, k, v = (torch.randn(B, h, S, D, generator=g, device="cuda").to(torch.bfloat16) for h in (Hq, Hkv, Hkv))
    rope = af.RopeSpec(theta=1e4, rotary_dim=D)
    table = af.rope_table(rope, S)
    want = af.fwd_variant(q, k, v, rope, table, af.MaskSpec(), 0.09)
    n = scratch_bytes(B, Hq, Hkv, S, D, D)
    assert n > 0
    scratch = torch.empty(n + 16, dtype=torch.uint8, device="cuda")
    sh, r, m = b._Shape(B, Hq, Hkv, S, D), b._Rope(1e4, D, 0), b._Mask(1, -1, None)
    for at, size, status in ((None, 0, 0), (scratch.data_ptr(), n - 1, 0), (scratch.data_ptr(), n, 0), (scratch.data_ptr() + 8, n, 4)):
        scratch.fill_(7)
        o, lse = torch.full_like(q, 3.0), torch.full((B, Hq, S), 3.0, device="cuda")
        assert af.lib().attnfuse_fwd_scratch(ctypes.byref(sh), q.data_ptr(), k.data_ptr(), v.data_ptr(), None, None, ctypes.byref(r),
                                             table.data_ptr(), ctypes.byref(m), Hq // Hkv, 0.09, o.data_ptr(), 0, lse.data_ptr(), at, size,
                                             torch.cuda.current_stream().cuda_stream) == status
        torch.cuda.synchronize()
        if status:
            assert o.eq(3.0).all() and lse.eq(3.0).all()
        else:
            assert torch.equal(o, want[0]) and torch.equal(lse, want[1])
        used = not scratch[:n].eq(7).all()
        assert used == (size == n and status == 0) and scratch[n:].eq(7).all()
    assert af.device_status()[0] == 0


def test_where_no_scratch_is_used():
    assert scratch_bytes(1, 2, 2, 128, 64, 64) == 0           # small
    assert scratch_bytes(1, 32, 8, 4096, 128, 0) == 0         # nothing to rotate
    assert scratch_bytes(1, 32, 8, 4096, 128, 128, window=512) == 0
    assert scratch_bytes(1, 32, 8, 4096, 128, 128, window=4095) > 0
    assert scratch_bytes(1, 32, 7, 4096, 128, 128) == 0       # not a shape
    assert scratch_bytes(1, 32, 8, 4096, 128, 128, slopes=0x1000) == 0
    # a few rotated columns cost less on chip than a launch ahead (measured 26 / 31, 31 / 38 and 24 / 34 us)
    assert scratch_bytes(3, 12, 4, 1035, 128, 64) == 0
    assert scratch_bytes(1, 24, 12, 1430, 128, 32) == 0
    assert scratch_bytes(1, 32, 8, 1105, 128, 16) == 0
    with af.option(af.OPT_FWD_KEYS_BF16, 1):
        assert scratch_bytes(1, 32, 8, 4096, 128, 128) == 0


def test_captured_call_with_given_outputs_and_streams():
    g = torch.Generator(device="cuda").manual_seed(922)
    q, k, v = (torch.randn(1, h, 3000, 128, generator=g, device="cuda").to(torch.bfloat16) for h in (16, 4, 4))
    rope, mask = af.RopeSpec(theta=1e4, rotary_dim=128), af.MaskSpec()
    table = af.rope_table(rope, 3000)
    assert scratch_bytes(1, 16, 4, 3000, 128, 128) > 0
    want = af.fwd(q, k, v, rope, table, mask, 0.09)
    torch.cuda.synchronize()
    given = (torch.zeros_like(want[0]), torch.zeros_like(want[1]))
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.stream(side):
        with torch.cuda.graph(graph, stream=side):
            af.fwd(q, k, v, rope, table, mask, 0.09, out=given[0], lse=given[1])
            fresh = af.fwd(q, k, v, rope, table, mask, 0.09)
    graph.replay()
    outs = []
    for s in [torch.cuda.Stream() for _ in range(3)] * 3:   # scratch of calls in flight on several streams
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s):
            outs.append(af.fwd(q, k, v, rope, table, mask, 0.09))
    torch.cuda.synchronize()
    assert af.device_status()[0] == 0
    for got in [given, fresh] + outs:
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
