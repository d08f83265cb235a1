"""Where the binding's forward gets its scratch memory: a call that can do without must not break somebody's capture."""
import threading

import pytest
import torch

import paper_2609_13612_b200 as af

pytestmark = pytest.mark.gpu
SHAPE = (1, 16, 4, 3000, 128)


def problem(seed):
    B, Hq, Hkv, S, D = SHAPE
    g = torch.Generator(device="cuda").manual_seed(seed)
    q, k, v = (torch.randn(B, h, S, D, generator=g, device="cuda").to(torch.bfloat16) for h in (Hq, Hkv, Hkv))
    rope = af.RopeSpec(theta=1e4, rotary_dim=D)
    return q, k, v, rope, af.rope_table(rope, S), af.MaskSpec(), 0.09


def test_another_threads_capture_survives_a_first_call():
    """Given outputs, scratch memory that has to come from cudaMalloc, and a capture in the global mode at the same time."""
    args = problem(931)
    want = af.fwd(*args)
    out, lse = torch.zeros_like(want[0]), torch.zeros_like(want[1])
    x = torch.zeros(1000, device="cuda")
    worker, capture, failed = torch.cuda.Stream(), torch.cuda.Stream(), []
    torch.cuda.synchronize()
    torch.cuda.empty_cache()

    def call():
        try:
            with torch.cuda.stream(worker):   # a stream without memory of its own yet
                af.fwd(*args, out=out, lse=lse)
        except Exception as e:   # noqa: BLE001
            failed.append(e)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=capture):
        x.add_(1.0)
        t = threading.Thread(target=call)
        t.start()
        t.join()
        x.add_(1.0)
    graph.replay()
    torch.cuda.synchronize()
    assert not failed and x.eq(2.0).all()
    assert torch.equal(out, want[0]) and torch.equal(lse, want[1])
    assert af.device_status()[0] == 0
