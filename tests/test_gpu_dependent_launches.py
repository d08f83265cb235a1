"""Every kernel starts as a programmatic dependent of the kernel before it in the stream, so what it reads must be read
behind its wait.  Here the inputs are written on the device by the launch right before the call: by the rotation pass,
which signals its dependents before it writes.  The buffers hold other valid contents beforehand, and the results must
be, bit for bit, those of the same inputs at rest."""
import pytest
import torch

import paper_2609_13612_b200 as af
from test_gpu_blocks import bigbird_blocks

pytestmark = pytest.mark.gpu
ROWS = 1 << 18   # of the tensor whose copy delivers the lists: its last row is written last


def normal(seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda").to(torch.bfloat16)


class Courier:
    """Up to 24 int32 values delivered by the rotation pass: in the unrotated columns 16..63 of the last row."""

    def __init__(self, values):
        assert values.numel() <= 24
        self.spec = af.RopeSpec(theta=1e4, rotary_dim=16)
        self.table = af.rope_table(self.spec, ROWS)
        self.src = torch.zeros(1, 1, ROWS, 64, dtype=torch.bfloat16, device="cuda")
        self.dst = torch.zeros_like(self.src)
        self.n = values.numel()
        self.view(self.src).copy_(values)

    def view(self, t):
        return t.view(torch.int32).view(-1)[-24:][:self.n]

    def deliver(self):
        af.rope(self.src, self.spec, self.table, out=self.dst)


@pytest.mark.parametrize("Hq,Hkv,D,qtiles", [(4, 2, 128, 3), (4, 2, 64, 2), (3, 3, 64, 3), (3, 1, 128, 2)],
                         ids=["head_pairs", "one_tile", "row_pairs", "one_tile_odd_group"])
def test_launch_order_of_block_lists_written_right_before_the_call(Hq, Hkv, D, qtiles):
    S = 128 * 20 + 40
    q, k, v = normal(1, 2, Hq, S, D), normal(2, 2, Hkv, S, D), normal(3, 2, Hkv, S, D)
    rope, mask = af.RopeSpec(theta=1e4, rotary_dim=D), af.MaskSpec(causal=False)
    table = af.rope_table(rope, S)
    bm = af.BlockMask(bigbird_blocks(21, seed=31))
    with af.option(af.OPT_FWD_QTILES, qtiles):
        want_o, want_l = af.fwd_blocks(q, k, v, rope, table, mask, D ** -0.5, bm)
        for name in ("row_order", "pair_order"):
            c = Courier(getattr(bm, name))
            setattr(bm, name, c.view(c.dst))
            for _ in range(4):
                c.dst.zero_()
                o, lse = torch.full_like(want_o, float("nan")), torch.full_like(want_l, float("nan"))
                torch.cuda.synchronize()
                c.deliver()
                af.fwd_blocks(q, k, v, rope, table, mask, D ** -0.5, bm, out=o, lse=lse)
                torch.cuda.synchronize()
                assert torch.equal(o, want_o) and torch.equal(lse, want_l), name
    assert af.device_status()[0] == 0


def test_inputs_written_right_before_the_call():
    """q, k, v, dO, the cache and the decoded query come out of the rotation pass that precedes each call, the slopes out of one
    before it; O and L of the backward come out of the forward, and a decode between writer and call hands the order on."""
    B, H, S, D = 2, 4, 1300, 128
    spec = af.RopeSpec(theta=1e4, rotary_dim=16)
    table16 = af.rope_table(spec, S)
    rope = af.RopeSpec(theta=1e4, rotary_dim=D)
    table = af.rope_table(rope, S)
    src = [normal(10 + i, B, H, S, D) for i in range(4)] + [normal(20, B, H, 1, D)]
    x, xk, xv, xd, xq = buf = [torch.empty_like(t) for t in src]
    slopes = Courier(torch.tensor([0.5, 0.25, 0.125, 0.0625], device="cuda").view(torch.int32))
    mask = af.MaskSpec(alibi_slopes=slopes.view(slopes.dst).view(torch.float32))
    bm = af.BlockMask(torch.ones(11, 11).tril().bool())
    ws = af.decode_workspace(B, H, H, S, D)
    bws = torch.empty(af.bwd_workspace_bytes(B, H, H, S, D), dtype=torch.uint8, device="cuda")
    o, lse = torch.empty_like(x), torch.empty(B, H, S, device="cuda")
    args = (rope, table, mask, 0.088)

    def decode():
        return af.decode(xq.view(B, H, D), xk, xv, mask, 0.088, workspace=ws)

    def step():
        af.fwd(x, xk, xv, *args, out=o, lse=lse)
        return af.bwd(x, xk, xv, o, lse, xd, *args, workspace=bws)[1:]   # (dQ: sums in no fixed order)

    def first(*i):   # the order of the writers: the last ones are the most likely to be overtaken
        return list(i) + [j for j in range(5) if j not in i]
    calls = [("fwd", first(1, 2), lambda: af.fwd(x, xk, xv, *args)),
             ("fwd_hybrid", first(1, 2, 3, 4), lambda: af.fwd_hybrid(x, xk, xv, *args)),
             ("fwd_blocks", first(0, 1), lambda: af.fwd_blocks(x, xk, xv, *args, bm)),
             ("decode", first(), decode),
             ("fwd and bwd", first(4, 0, 1, 2), step),
             ("decode, then fwd", first(3, 4), lambda: (decode(), af.fwd(x, xk, xv, *args))[1])]

    def fill(order):
        slopes.deliver()
        for i in order:
            af.rope(src[i], spec, table16, out=buf[i])

    def clear():
        for t in buf + [o, lse, slopes.dst]:
            t.zero_()
        torch.cuda.synchronize()

    for name, order, call in calls:
        fill(order)
        torch.cuda.synchronize()
        want = [t.clone() for t in call()]
        for _ in range(3):
            clear()
            fill(order)
            got = call()
            torch.cuda.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(got, want)), name
    assert af.device_status()[0] == 0
