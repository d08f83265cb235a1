"""Arguments of the native side of the Python binding: what it refuses (no GPU needed: nothing there reaches a launch) and what
it accepts."""
import numpy as np
import pytest
import torch

import paper_2609_13612_b200 as af

CPU = torch.zeros(1, 2, 128, 64, dtype=torch.bfloat16)
CODES = torch.zeros(1, 2, 128, 128, dtype=torch.uint8)
ROPE, MASK = af.RopeSpec(rotary_dim=0), af.MaskSpec()


@pytest.mark.parametrize("call", [
    lambda: af.fwd(CPU, CPU, CPU, ROPE, None, MASK, 0.1),
    lambda: af.fwd_hybrid(CPU, CPU, CPU, ROPE, None, MASK, 0.1),
    lambda: af.fwd_blocks(CPU, CPU, CPU, ROPE, None, MASK, 0.1, af.BlockMask([[True]], device="cpu")),
    lambda: af.fwd_fp8(CODES, CODES, CODES, MASK, 0.1),
    lambda: af.bwd(CPU, CPU, CPU, CPU, CPU, CPU, ROPE, None, MASK, 0.1),
    lambda: af.decode(CPU[:, :, 0], CPU, CPU, MASK, 0.1),
], ids=["fwd", "fwd_hybrid", "fwd_blocks", "fwd_fp8", "bwd", "decode"])
def test_tensors_off_the_device_are_refused(call):
    with pytest.raises(af.AttnFuseError) as e:
        call()
    assert e.value.code == -2


def test_tensors_without_storage_raise():
    """data_ptr() of a fake tensor throws: the exception has to reach the caller (and leave the interpreter lock held)."""
    from torch._subclasses.fake_tensor import FakeTensorMode
    with FakeTensorMode():
        q = torch.empty(1, 2, 128, 128, dtype=torch.bfloat16, device="cuda")
        lse, codes = torch.empty(1, 2, 128, device="cuda"), torch.empty(1, 2, 128, 128, dtype=torch.uint8, device="cuda")
        x = dict(out=torch.empty_like(q), lse=lse)
        calls = [lambda: af.fwd(q, q, q, ROPE, None, MASK, 0.1, **x),
                 lambda: af.fwd_hybrid(q, q, q, ROPE, None, MASK, 0.1, workspace=codes, **x),
                 lambda: af.fwd_fp8(codes, codes, codes, MASK, 0.1),
                 lambda: af.bwd(q, q, q, q, lse, q, ROPE, None, MASK, 0.1, workspace=codes),
                 lambda: af.decode(q[:, :, 0].contiguous(), q, q, MASK, 0.1, out=q[:, :, 0], lse=lse[:, :, 0], workspace=codes)]
        for call in calls:
            with pytest.raises(RuntimeError):
                call()


@pytest.mark.parametrize("bad", [None, 3.0, "q"])
def test_arguments_of_another_kind_are_refused(bad):
    with pytest.raises(TypeError):
        af.fwd(bad, CPU, CPU, ROPE, None, MASK, 0.1)


@pytest.mark.gpu
def test_numbers_and_codes_of_other_types_are_accepted():
    g = torch.Generator(device="cuda").manual_seed(5)
    q, k, v = (torch.randn(1, 2, 400, 64, generator=g, device="cuda").to(torch.bfloat16) for _ in range(3))
    want = af.fwd(q, k, v, ROPE, None, af.MaskSpec(window=300), 0.125)
    for window, scale in ((300.0, 0.125), ("300", "0.125"), (torch.tensor(300), torch.tensor(0.125)), (np.float32(300), np.float64(0.125))):
        got = af.fwd(q, k, v, ROPE, None, af.MaskSpec(window=window), scale)
        assert all(torch.equal(x, y) for x, y in zip(got, want))
    codes = [torch.randn(*s, generator=g, device="cuda").to(torch.float8_e4m3fn) for s in ((1, 2, 400, 128), (1, 2, 400, 128), (1, 2, 128, 400))]
    want = af.fwd_fp8(*codes, MASK, 0.1)
    for dt in (torch.uint8, torch.int8, torch.int16, torch.int32, torch.bfloat16):
        got = af.fwd_fp8(*(c.view(dt) for c in codes), MASK, "0.1", scale_q=1)
        assert all(torch.equal(x, y) for x, y in zip(got, want)), dt
    assert af.device_status()[0] == 0


def test_a_binding_built_for_another_torch_is_stale(monkeypatch):
    from paper_2609_13612_b200 import binding, build
    assert not build.binding_is_stale() and binding._load_native().ABI_TAG == build.abi_tag()
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    assert build.binding_is_stale()
    monkeypatch.setattr(binding, "_native", None)
    with pytest.raises(af.AttnFuseError, match="torch 0.0.1"):
        binding._load_native()
