"""The tensor-core evaluation of nets with three hidden layers at the edges of its plan: individuals shared by several
CTAs, last input blocks of 16, 32 and 48 inputs, widths on both sides of the stacked weight slots, nets whose layers share
accumulator columns, and both orders of the products.  Against the FP64 oracle with the fitness tolerance."""
import numpy as np
import pytest

from helpers import assert_correct_close, assert_fitness_close, to_device_pop

pytestmark = pytest.mark.gpu

CASES = [  # dims, pop, batch
    ([196, 256, 128, 64, 10], 160, 300), ([196, 256, 128, 64, 10], 3, 1024), ([256, 256, 256, 256, 16], 5, 260),
    ([48, 16, 16, 16, 2], 200, 129), ([80, 128, 144, 48, 7], 33, 400), ([32, 240, 256, 16, 3], 20, 200),
    ([196, 256, 128, 64, 10], 160, 15), ([196, 256, 128, 64, 10], 160, 16), ([64, 256, 256, 112, 10], 33, 13),
    ([36, 80, 128, 128, 16], 310, 8), ([64, 64, 64, 64, 10], 1, 2000), ([200, 256, 192, 32, 10], 155, 128), ([4, 16, 256, 240, 5], 7, 1),
]


@pytest.mark.parametrize("dims,pop,batch", CASES, ids=[f"{d}-{p}-{b}" for d, p, b in CASES])
def test_units_match_oracle(gpu, oracle_mod, dims, pop, batch):
    import torch
    rng = np.random.default_rng(dims[2] * 1000 + batch)
    popv = rng.normal(0.0, 0.1, size=(pop, gpu.leea_layout_num_params(dims))).astype(np.float32)
    if pop > 4:
        popv[1, -1 - dims[4]] = 150.0                # a last-layer weight outside the pieces' range
        popv[2] *= np.float32(12.0)                  # activations outside it
        popv[4] = popv[0]
    levels = rng.integers(0, 256, size=(batch, dims[0])).astype(np.uint8)
    y = rng.integers(0, dims[4], size=batch).astype(np.int32)
    f_inh = rng.normal(-2.3, 0.1, size=pop).astype(np.float32)
    f, fa = (torch.empty(pop, device="cuda") for _ in range(2))
    cor = torch.empty(pop, dtype=torch.int32, device="cuda")
    gpu.leea_evaluate_u8(pop, dims, to_device_pop(popv, gpu.leea_padded_params(dims)), torch.from_numpy(levels).cuda(),
                         255.0, torch.from_numpy(y).cuda(), batch, 0.3, torch.from_numpy(f_inh).cuda(), f, fa, cor,
                         gpu.EVAL_TENSOR)
    assert gpu.leea_device_status() == 0
    f_ref, cor_ref, logits = oracle_mod.evaluate(popv.astype(np.float64), dims, levels.astype(np.float64) / 255.0, y,
                                                 want_logits=True)
    assert_fitness_close(f.cpu().numpy(), f_ref)
    assert_correct_close(cor.cpu().numpy(), cor_ref, logits)
    adj_ref = oracle_mod.inherit(float(np.float32(0.3)), f_inh.astype(np.float64), f_ref, first=False)
    assert_fitness_close(fa.cpu().numpy(), adj_ref, "f_adj")
    if pop > 4:
        assert f[0] == f[4]
