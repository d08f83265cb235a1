"""A decode launch starts while the kernel in front of it ends: a cache that this kernel is still writing must be read as written."""
import pytest
import torch

import paper_2609_13612_b200 as af

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,Hq,Hkv,N", [(1, 32, 8, 4096), (2, 12, 4, 1333), (1, 8, 1, 20000), (1, 4, 4, 641)])
def test_cache_written_right_before_the_call(B, Hq, Hkv, N):
    g = torch.Generator(device="cuda").manual_seed(931)
    q = torch.randn(B, Hq, 128, generator=g, device="cuda").to(torch.bfloat16)
    src, v = (torch.randn(B, Hkv, N, 128, generator=g, device="cuda").to(torch.bfloat16) for _ in range(2))
    spec = af.RopeSpec(theta=1e4, rotary_dim=128)
    table = af.rope_table(spec, N)
    k, vv = torch.zeros_like(src), torch.zeros_like(v)
    ws = af.decode_workspace(B, Hq, Hkv, N, 128)
    af.rope(src, spec, table, out=k)
    af.rope(v, spec, table, out=vv)
    torch.cuda.synchronize()
    want_o, want_l = af.decode(q, k, vv, af.MaskSpec(), 0.088, workspace=ws)
    for _ in range(6):
        k.zero_()
        vv.zero_()
        torch.cuda.synchronize()
        af.rope(v, spec, table, out=vv)
        af.rope(src, spec, table, out=k)      # (signals its dependents before it writes)
        o, lse = af.decode(q, k, vv, af.MaskSpec(), 0.088, workspace=ws)
        torch.cuda.synchronize()
        assert torch.equal(o, want_o) and torch.equal(lse, want_l)
    assert af.device_status()[0] == 0
