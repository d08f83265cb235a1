"""Where the binding's forward gets its scratch memory: a call that can do without must not break somebody's capture, fail with the
allocator, or leave memory to others that a captured graph still writes."""
import ctypes
import os
import subprocess
import sys
import textwrap
import threading

import pytest
import torch

import paper_2609_13612_b200 as af

pytestmark = pytest.mark.gpu
SHAPE = (1, 16, 4, 3000, 128)
SCRATCH = 4 * 3000 * 128 * 2


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


ALLOCATOR = r"""
#include <cuda_runtime.h>
#include <stdexcept>
#include <sys/types.h>
extern "C" {
ssize_t watched = -1;   // a size that this allocator has trouble with
int mode = 0, hits = 0;
void* take(ssize_t size, int, cudaStream_t) {
    void* p = nullptr;
    if (size == watched) {
        ++hits;
        if (mode == 0) throw std::runtime_error("no memory of this size");
        if (cudaMalloc(&p, size + 256) != cudaSuccess) return nullptr;
        return static_cast<char*>(p) + 8;
    }
    return cudaMalloc(&p, size) == cudaSuccess ? p : nullptr;
}
void give(void* p, ssize_t size, int, cudaStream_t) {
    cudaDeviceSynchronize();
    cudaFree(size == watched && mode == 1 ? static_cast<char*>(p) - 8 : p);
}
}
"""


def test_an_allocator_that_fails_in_its_own_way(tmp_path):
    """Memory that a call can do without: neither another exception than torch's nor a misaligned block may fail it."""
    src, so = tmp_path / "allocator.cpp", tmp_path / "allocator.so"
    src.write_text(ALLOCATOR)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I" + cuda + "/include", "-o", str(so), str(src), "-L" + cuda + "/lib64", "-lcudart"], check=True)
    code = textwrap.dedent("""
        import ctypes, sys, torch
        sys.path[:0] = [%r, %r]
        lib = ctypes.CDLL(%r)
        torch.cuda.memory.change_current_allocator(torch.cuda.memory.CUDAPluggableAllocator(%r, "take", "give"))
        import paper_2609_13612_b200 as af
        import test_gpu_fwd_scratch_memory as t
        args = t.problem(933)
        out, lse = torch.zeros_like(args[0]), torch.zeros(t.SHAPE[0], t.SHAPE[1], t.SHAPE[3], device="cuda")
        want = af.fwd_variant(*args)   # on chip, the same bits
        for mode in (0, 1):
            out.zero_()
            ctypes.c_int.in_dll(lib, "mode").value = mode
            ctypes.c_ssize_t.in_dll(lib, "watched").value = t.SCRATCH
            af.fwd(*args, out=out, lse=lse)
            torch.cuda.synchronize()
            ctypes.c_ssize_t.in_dll(lib, "watched").value = -1
            assert torch.equal(out, want[0]) and torch.equal(lse, want[1]), mode
        assert ctypes.c_int.in_dll(lib, "hits").value == 2 and af.device_status()[0] == 0
        print("allocator ok")
    """) % (os.path.dirname(os.path.dirname(os.path.abspath(__file__))), os.path.dirname(os.path.abspath(__file__)), str(so), str(so))
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "allocator ok" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]


def test_a_capture_that_torch_does_not_know_of():
    """Outputs allocated by the call, memory from torch's ordinary pool: what the call returns to the pool goes to others, and a
    replay must not write there."""
    rt = ctypes.CDLL("libcudart.so.12")
    args = problem(932)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        want = af.fwd(*args)
        warm = af.fwd(*args)
        s.synchronize()
        del warm   # (its memory and the scratch memory are in the stream's pool now)
        handle, graph, exe = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p(), ctypes.c_void_p()
        assert rt.cudaStreamBeginCapture(handle, 1) == 0   # thread-local mode
        got = af.fwd(*args)
        assert rt.cudaStreamEndCapture(handle, ctypes.byref(graph)) == 0
        others = [torch.full((SCRATCH,), 7, dtype=torch.uint8, device="cuda") for _ in range(8)]
        for x in got:
            x.zero_()
        assert rt.cudaGraphInstantiate(ctypes.byref(exe), graph, ctypes.c_ulonglong(0)) == 0
        assert rt.cudaGraphLaunch(exe, handle) == 0
        s.synchronize()
    assert rt.cudaGraphExecDestroy(exe) == 0 and rt.cudaGraphDestroy(graph) == 0
    assert all(x.eq(7).all() for x in others)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    assert af.device_status()[0] == 0


def test_a_graph_of_torchs_own_is_still_lent_memory():
    """The same bits, and the graph holds the launch that rotates the keys, too."""
    args = problem(934)
    want = af.fwd(*args)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        got = af.fwd(*args)
    nodes = ctypes.c_size_t()
    assert ctypes.CDLL("libcudart.so.12").cudaGraphGetNodes(ctypes.c_void_p(graph.raw_cuda_graph()), None, ctypes.byref(nodes)) == 0
    assert nodes.value == 2
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    assert af.device_status()[0] == 0
