"""leea_evaluate_shadow_u8 on both sides of its switch to two individuals per MMA (populations times 128-sample tiles
of two per SM): the same bits as the allocation-free entry point, which always takes the chunked kernel."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("dims,per_sm,extra,batch", [([784, 112, 10], 2, -1, 100), ([784, 112, 10], 2, 0, 128),
                                                     ([784, 128, 16], 2, 1, 1), ([96, 16, 3], 1, 0, 129),
                                                     ([16, 48, 10], 1, -1, 256), ([784, 32, 10], 1, 1, 300)])
def test_pair_call_keeps_the_bits(gpu, dims, per_sm, extra, batch, precision):
    import torch
    pop = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + extra
    rng = np.random.default_rng(pop + batch)
    c, cp = gpu.leea_layout_num_params(dims), gpu.leea_padded_params(dims)
    pd = torch.zeros((pop, cp), device="cuda")
    pd[:, :c] = torch.from_numpy(rng.normal(0, 0.1, size=(pop, c)).astype(np.float32)).cuda()
    sh = torch.zeros((pop, gpu.leea_shadow_stride(dims, precision)), dtype=torch.uint8, device="cuda")
    se, am = torch.zeros(pop, dtype=torch.int32, device="cuda"), torch.zeros(pop, device="cuda")
    gpu.leea_make_shadow(pop, dims, precision, pd, sh, se, am)
    x = torch.from_numpy(rng.integers(0, 256, size=(batch, dims[0])).astype(np.uint8)).cuda()
    y = torch.from_numpy(rng.integers(0, dims[2], size=batch).astype(np.int32)).cuda()
    f_inh = torch.from_numpy(rng.normal(size=pop).astype(np.float32)).cuda()
    nbytes = gpu.leea_shadow_scratch_bytes(pop, batch)
    scratch = torch.empty(nbytes // 4, device="cuda") if nbytes else None
    out = []
    for noalloc in (False, True):
        f_raw, f_adj = (torch.full((pop,), float("nan"), device="cuda") for _ in range(2))
        cor = torch.full((pop,), -1, dtype=torch.int32, device="cuda")
        args = (pop, dims, pd, precision, sh, se, x, 255.0, y, batch, 0.25, f_inh, f_raw, f_adj, cor)
        if noalloc:
            gpu.leea_evaluate_shadow_u8_noalloc(*args)
        else:
            gpu.leea_evaluate_shadow_u8(*args, scratch)
        assert gpu.leea_device_status() == 0
        out.append([t.cpu().numpy() for t in (f_raw, f_adj, cor)])
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
