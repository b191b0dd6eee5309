"""Inheritance in place: f_adj may be the array that f_inh is read from, also where the tensor-core evaluation marks
individuals for the kernel that follows it.  The same bits as into an array of its own."""
import numpy as np
import pytest

from helpers import to_device_pop

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,dims,pop,batch", [("f32", [784, 112, 10], 300, 100), ("f32", [784, 48, 10], 200, 300),
                                                 ("u8", [784, 100, 10], 333, 50), ("u8", [784, 112, 10], 160, 300),
                                                 ("u8", [784, 112, 10], 160, 100)])
def test_in_place(gpu, kind, dims, pop, batch):
    import torch
    rng = np.random.default_rng(batch)
    popv = rng.normal(0.0, 0.05, size=(pop, gpu.leea_layout_num_params(dims))).astype(np.float32)
    popv[1, 7], popv[4, 3000], popv[pop - 1, 0] = 200.0, -130.0, 500.0  # outside the pieces' range
    pd = to_device_pop(popv, gpu.leea_padded_params(dims))
    lv = torch.from_numpy(rng.integers(0, 256, size=(batch, dims[0])).astype(np.uint8)).cuda()
    y = torch.from_numpy(rng.integers(0, dims[2], size=batch).astype(np.int32)).cuda()
    f_inh = torch.from_numpy(rng.normal(-2.3, 0.1, size=pop).astype(np.float32)).cuda()
    out = []
    for in_place in (False, True):
        raw, adj = torch.empty(pop, device="cuda"), torch.empty(pop, device="cuda")
        inh = f_inh.clone()
        if in_place:
            adj = inh
        if kind == "f32":
            gpu.leea_evaluate(pop, dims, pd, lv.float() / 255.0, y, batch, 0.3, inh, raw, adj)
        else:
            gpu.leea_evaluate_u8(pop, dims, pd, lv, 255.0, y, batch, 0.3, inh, raw, adj)
        assert gpu.leea_device_status() == 0
        out.append((raw.cpu().numpy(), adj.cpu().numpy()))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])
