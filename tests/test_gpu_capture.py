"""Evaluation step calls under stream capture: a graph of one call gives the call's results."""
import ctypes
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MEMORY_NODES = {10, 11}  # cudaGraphNodeTypeMemAlloc, cudaGraphNodeTypeMemFree
# name: net, population, batch
CALLS = {"u8": ([784, 112, 10], 200, 100), "u8_odd": ([784, 100, 10], 620, 60), "u8_large": ([784, 112, 10], 310, 512),
         "f32": ([784, 112, 10], 620, 100), "bf16": ([784, 112, 10], 400, 100)}


def _runtime():
    import torch  # noqa: F401  (brings the CUDA runtime into the process)
    with open("/proc/self/maps") as fh:
        name = next(line.split()[-1] for line in fh if "libcudart.so" in line)
    return ctypes.CDLL(name)


def _setup(gpu, name):
    """(call(stream, f), pop) of a named call on seeded inputs."""
    import torch
    dims, pop, batch = CALLS[name]
    g = torch.Generator(device="cuda").manual_seed(5)
    pd = torch.zeros((pop, gpu.leea_padded_params(dims)), device="cuda").normal_(0.0, 0.03, generator=g)
    lv = torch.randint(0, 256, (batch, dims[0]), device="cuda", dtype=torch.uint8, generator=g)
    y = torch.randint(0, dims[2], (batch,), device="cuda", dtype=torch.int32, generator=g)
    x = lv.float() / 255.0
    if name == "bf16":
        sh = torch.empty((pop, gpu.leea_shadow_stride(dims, 1)), dtype=torch.uint8, device="cuda")
        amax, cor = torch.empty(pop, device="cuda"), torch.empty(pop, dtype=torch.int32, device="cuda")
        gpu.leea_make_shadow(pop, dims, 1, pd, sh, None, amax)

    def call(stream, f):
        if name == "f32":
            gpu.leea_evaluate(pop, dims, pd, x, y, batch, 1.0, None, f, None, stream=stream)
        elif name == "bf16":
            gpu.leea_evaluate_shadow_u8(pop, dims, pd, 1, sh, None, lv, 255.0, y, batch, 1.0, None, f, None, cor, None,
                                        stream=stream)
        else:
            gpu.leea_evaluate_u8(pop, dims, pd, lv, 255.0, y, batch, 1.0, None, f, None, stream=stream)

    return call, pop


def _capture(rt, call, stream, f):
    handle, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    assert rt.cudaStreamBeginCapture(handle, 0) == 0  # the strictest mode
    call(stream, f)
    assert rt.cudaStreamEndCapture(handle, ctypes.byref(graph)) == 0
    return graph


def _launch(rt, graph, stream):
    ex = ctypes.c_void_p()
    assert rt.cudaGraphInstantiate(ctypes.byref(ex), graph, ctypes.c_ulonglong(0)) == 0
    assert rt.cudaGraphLaunch(ex, ctypes.c_void_p(stream.cuda_stream)) == 0
    stream.synchronize()
    return ex


FIRST_CALL = """
import sys
sys.path[:0] = [{root!r}, {tests!r}]
import torch
from paper_1806_09819_gb300 import leea
import test_gpu_capture as T
call, pop = T._setup(leea, {name!r})
f, s, rt = torch.zeros(pop, device="cuda"), torch.cuda.Stream(), T._runtime()
torch.cuda.synchronize()
T._launch(rt, T._capture(rt, call, s, f), s)
assert bool((f < 0).all()) and leea.leea_device_status() == 0
"""


@pytest.mark.parametrize("name", ["u8", "f32"])
def test_first_call_of_a_process(gpu, name):
    code = FIRST_CALL.format(root=ROOT, tests=os.path.join(ROOT, "tests"), name=name)
    res = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=ROOT, timeout=120)
    assert res.returncode == 0, res.stderr[-2000:]


@pytest.mark.parametrize("name", list(CALLS))
def test_captured_call(gpu, name):
    """The same results to a rounding as outside, launched again and again; and where the call has a way without scratch
    memory no memory nodes, so that the graph can be instantiated more than once."""
    import torch
    rt = _runtime()
    call, pop = _setup(gpu, name)
    s = torch.cuda.Stream()
    direct, f = torch.zeros(pop, device="cuda"), torch.zeros(pop, device="cuda")
    torch.cuda.synchronize()
    call(s, direct)
    s.synchronize()
    graph = _capture(rt, call, s, f)
    n = ctypes.c_size_t(0)
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes, kinds = (ctypes.c_void_p * n.value)(), []
    assert rt.cudaGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    for node in nodes:
        t = ctypes.c_int()
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(t)) == 0
        kinds.append(t.value)
    memory = bool(MEMORY_NODES & set(kinds))
    assert memory == (name == "u8")
    for _ in range(1 if memory else 2):
        f.zero_()
        torch.cuda.synchronize()
        ex = _launch(rt, graph, s)
        # FP32 evaluations of the same fitness: each within 1e-6 relative of it
        assert torch.allclose(f, direct, rtol=2e-6, atol=0)
        f.zero_()
        torch.cuda.synchronize()
        assert rt.cudaGraphLaunch(ex, ctypes.c_void_p(s.cuda_stream)) == 0
        s.synchronize()
        assert torch.allclose(f, direct, rtol=2e-6, atol=0)
    assert gpu.leea_device_status() == 0
