"""A minibatch written by the kernel just before the call on the same stream, one that lets its successors start long
before it writes (programmatic dependent launch): every evaluation that stages its batch must wait for it.  The results
are those of the same call on a batch that was there from the start, bit for bit."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_1806_09819_gb300 import build as B
from paper_1806_09819_gb300 import synthetic

pytestmark = pytest.mark.gpu

# Lets its dependents start, lets 200 us pass, then copies.
PRODUCER = r"""
#include <cstdint>
__global__ void late_copy(const unsigned char* src, unsigned char* dst, long long n)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    uint64_t t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (int i = 0; i < 100000; ++i) {
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 > 200000u) break;
        __nanosleep(500);
    }
    for (long long i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}
extern "C" int launch_late_copy(const void* src, void* dst, long long n, void* stream)
{
    late_copy<<<1, 512, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<const unsigned char*>(src),
                                                               static_cast<unsigned char*>(dst), n);
    return static_cast<int>(cudaGetLastError());
}
"""


@pytest.fixture(scope="module")
def late_copy(gpu, tmp_path_factory):
    import torch
    d = tmp_path_factory.mktemp("late_copy")
    src, lib = d / "late_copy.cu", d / "late_copy.so"
    src.write_text(PRODUCER)
    subprocess.run([B.nvcc(), *B.ARCH, "-shared", "-Xcompiler", "-fPIC", "-cudart", "shared", str(src), "-o", str(lib)],
                   check=True)
    fn = ctypes.CDLL(str(lib)).launch_late_copy
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong, ctypes.c_void_p]

    def run(src_t, dst):
        n = src_t.numel() * src_t.element_size()
        dst = dst if isinstance(dst, int) else dst.data_ptr()
        assert fn(src_t.data_ptr(), dst, n, torch.cuda.current_stream().cuda_stream) == 0

    return run


def _batch(batch, k, floats):
    import torch
    rng = np.random.default_rng(batch + k)
    lv = rng.integers(0, 256, size=(batch, k)).astype(np.uint8)
    x = torch.from_numpy(lv.astype(np.float32) / 255.0 if floats else lv).cuda()
    return x, torch.from_numpy(rng.integers(0, 10, size=batch).astype(np.int32)).cuda()


# kind, hidden units, population, batch
STEP = [("f32", 64, 600, 100), ("f32", 64, 300, 300), ("u8", 64, 300, 100), ("u8", 50, 700, 100), ("u8", 64, 400, 300),
        ("bf16", 64, 400, 100), ("fp8", 64, 400, 200)]


@pytest.mark.parametrize("kind,h,pop,batch", STEP)
def test_step_call_waits_for_its_batch(gpu, late_copy, kind, h, pop, batch):
    import torch
    dims = [784, h, 10]
    c, cp = gpu.leea_layout_num_params(dims), gpu.leea_padded_params(dims)
    popv = torch.zeros((pop, cp), device="cuda")
    popv[:, :c] = torch.from_numpy(synthetic.random_population(pop, c, seed=3, scale=0.1)).cuda()
    x, y = _batch(batch, 784, kind == "f32")
    late = torch.zeros_like(x)
    prec = {"bf16": 1, "fp8": 2}.get(kind, 0)
    if prec:
        sh = torch.empty((pop, gpu.leea_shadow_stride(dims, prec)), dtype=torch.uint8, device="cuda")
        se, am = torch.zeros(pop, dtype=torch.int32, device="cuda"), torch.empty(pop, device="cuda")
        gpu.leea_make_shadow(pop, dims, prec, popv, sh, se, am)
        n = gpu.leea_shadow_scratch_bytes(pop, batch)
        scratch = torch.empty(n // 4, device="cuda") if n else None
    cor = torch.empty(pop, dtype=torch.int32, device="cuda")

    def call(xd, f):
        if kind == "f32":
            gpu.leea_evaluate(pop, dims, popv, xd, y, batch, 1.0, None, f, None)
        elif kind == "u8":
            gpu.leea_evaluate_u8(pop, dims, popv, xd, 255.0, y, batch, 1.0, None, f, None)
        else:
            gpu.leea_evaluate_shadow_u8(pop, dims, popv, prec, sh, se, xd, 255.0, y, batch, 1.0, None, f, None, cor,
                                        scratch)

    want, got = torch.empty(pop, device="cuda"), torch.empty(pop, device="cuda")
    call(x, want)
    call(late, got)  # the scratch is there, and nothing of the call is lazy any more
    torch.cuda.synchronize()
    assert not torch.equal(want, got)
    late_copy(x, late)
    call(late, got)
    assert gpu.leea_device_status() == 0
    assert torch.equal(want, got)


@pytest.mark.parametrize("kind,h,pop,batch", [("u8", 64, 600, 100), ("u8", 50, 600, 200), ("f32", 64, 600, 100),
                                              ("bf16", 64, 600, 200), ("fp8", 144, 600, 100), ("u8", 64, 200, 100)])
def test_generation_waits_for_its_batch(gpu, late_copy, kind, h, pop, batch):
    import torch
    dims = [784, h, 10]
    xs = [_batch(batch + i, 784, kind == "f32") for i in range(3)]
    xs = [(x[:batch].contiguous(), y[:batch].contiguous()) for x, y in xs]
    out = []
    for is_late in (False, True):
        st = gpu.LeeaState(pop, dims, gpu.Params(precision={"bf16": 1, "fp8": 2}.get(kind, 0), n_elite=1), seed=5)
        try:
            for x, y in xs:  # the initial evaluation, then two bred generations
                xd = torch.zeros_like(x) if is_late else x
                torch.cuda.synchronize()
                if is_late:
                    late_copy(x, xd)
                if kind == "f32":
                    st.leea_generation(xd, y)
                else:
                    st.leea_generation_u8(xd, y)
                torch.cuda.synchronize()
            assert gpu.leea_device_status() == 0
            out.append((st.leea_fitness(), st.leea_get_population()))
        finally:
            st.close()
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("kind,h,pop,batch", [("fused", 64, 200, 100), ("bf16", 64, 60, 100), ("fp8", 160, 60, 200)])
def test_kernels_that_load_the_batch_themselves(gpu, late_copy, kind, h, pop, batch):
    """The fused breed + evaluate step and the chunked shadow evaluation."""
    import torch
    dims = [784, h, 10]
    c, cp = gpu.leea_layout_num_params(dims), gpu.leea_padded_params(dims)
    popv = torch.zeros((pop, cp), device="cuda")
    popv[:, :c] = torch.from_numpy(synthetic.random_population(pop, c, seed=3, scale=0.1)).cuda()
    x, y = _batch(batch, 784, False)
    late = torch.zeros_like(x)
    cor = torch.empty(pop, dtype=torch.int32, device="cuda")
    prec = {"bf16": 1, "fp8": 2}.get(kind, 0)
    if prec:
        sh = torch.empty((pop, gpu.leea_shadow_stride(dims, prec)), dtype=torch.uint8, device="cuda")
        se, am = torch.zeros(pop, dtype=torch.int32, device="cuda"), torch.empty(pop, device="cuda")
        gpu.leea_make_shadow(pop, dims, prec, popv, sh, se, am)
    par = torch.arange(pop, dtype=torch.int32, device="cuda")
    two = torch.full((pop,), 2, dtype=torch.int32, device="cuda")
    kids = torch.zeros_like(popv)

    def call(xd, f):
        if kind == "fused":
            gpu.leea_breed_evaluate_u8(pop, dims, gpu.Params(mut_rate=0.1), 4, 1, popv, par, par, two, kids, xd, 255.0, y,
                                       batch, 1.0, None, f, None, None)
        else:
            gpu.leea_evaluate_shadow_u8_noalloc(pop, dims, popv, prec, sh, se, xd, 255.0, y, batch, 1.0, None, f, None, cor)

    want, got = torch.empty(pop, device="cuda"), torch.empty(pop, device="cuda")
    call(x, want)
    call(late, got)
    torch.cuda.synchronize()
    assert not torch.equal(want, got)
    late_copy(x, late)
    call(late, got)
    assert gpu.leea_device_status() == 0
    assert torch.equal(want, got)


def test_runs_wait_for_their_first_batch(gpu, late_copy):
    """The batching form reads its first minibatch where the caller writes it, in the object's own buffers."""
    import torch
    specs = [gpu.RunSpec(60, 32, 64, seed=1), gpu.RunSpec(50, 48, 40, seed=2)]
    out = []
    for is_late in (False, True):
        m = gpu.MultiRun(specs, 784, 10, gpu.Params(precision=1, n_elite=1))
        try:
            rows = m.total_rows
            g = torch.Generator(device="cuda").manual_seed(1)
            x = torch.randint(0, 256, (rows, 784), device="cuda", dtype=torch.uint8, generator=g)
            y = torch.randint(0, 10, (rows,), device="cuda", dtype=torch.int32, generator=g)
            xb, yb = m.batch_buffers()
            late_copy(torch.zeros_like(x), xb)
            late_copy(y, yb)
            torch.cuda.synchronize()
            late_copy(x, xb)
            if not is_late:
                torch.cuda.synchronize()
            assert m.lib.leea_multi_generation_u8(m._h, xb, 255.0, yb) == 0
            out.append(np.asarray(m.fitness()))
        finally:
            m.close()
    np.testing.assert_array_equal(out[0], out[1])
