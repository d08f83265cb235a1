"""The fp8 forward's two outputs: bf16 rows leave through shared memory and TMA (clipped at S), fp32 rows by direct stores.
Both come from the same fp32 accumulator, so the bf16 result has to be the fp32 one rounded to nearest even, bit for bit."""
import pytest
import torch

import paper_2609_13612_b200 as af

pytestmark = pytest.mark.gpu


# one short tile; a ragged second tile; an odd group (two row blocks per CTA, the second one past S); several CTAs per head
@pytest.mark.parametrize("B,Hq,Hkv,S,window,causal", [(1, 2, 2, 16, -1, True), (2, 4, 2, 144, -1, True), (1, 3, 1, 272, -1, False),
                                                      (1, 3, 3, 400, 100, True), (1, 8, 2, 2064, 512, True)])
def test_bf16_output_is_the_rounded_fp32_output(B, Hq, Hkv, S, window, causal):
    g = torch.Generator(device="cuda").manual_seed(907)
    enc = lambda *shape: torch.randn(shape, generator=g, device="cuda").to(torch.float8_e4m3fn).view(torch.uint8)
    q, k, vt = enc(B, Hq, S, 128), enc(B, Hkv, S, 128), enc(B, Hkv, 128, S)
    mask = af.MaskSpec(causal=causal, window=window)
    want, want_l = af.fwd_fp8(q, k, vt, mask, 0.088, 1.0, 1.0, 0.7, out_dtype=torch.float32)
    got, got_l = af.fwd_fp8(q, k, vt, mask, 0.088, 1.0, 1.0, 0.7, out_dtype=torch.bfloat16)
    torch.cuda.synchronize()
    assert af.device_status()[0] == 0
    assert torch.isfinite(want).all() and want.abs().max() > 0
    assert torch.equal(got, want.to(torch.bfloat16)) and torch.equal(got_l, want_l)
