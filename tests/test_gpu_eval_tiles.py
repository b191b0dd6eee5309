"""Evaluation of batches of several 128-sample tiles for every number of output groups (a lane of the epilogue takes
four samples and a quarter of the hidden units), with one and two individuals per unit.  Against the FP64 oracle with
the fitness tolerance, 8-bit levels and floats."""
import numpy as np
import pytest

from helpers import assert_correct_close, assert_fitness_close, to_device_pop

pytestmark = pytest.mark.gpu

CASES = [  # dims, pop, batch
    ([52, 48, 4], 700, 300), ([64, 112, 8], 400, 257), ([784, 80, 12], 9, 512), ([784, 112, 13], 320, 260),
    ([300, 96, 2], 310, 129), ([36, 130, 16], 320, 200),
]


@pytest.mark.parametrize("floats", [False, True], ids=["u8", "f32"])
@pytest.mark.parametrize("dims,pop,batch", CASES, ids=[f"{d}-{p}-{b}" for d, p, b in CASES])
def test_tiles_match_oracle(gpu, oracle_mod, dims, pop, batch, floats):
    import torch
    rng = np.random.default_rng(dims[1] * 1000 + batch)
    popv = rng.normal(0.0, 0.15, size=(pop, gpu.leea_layout_num_params(dims))).astype(np.float32)
    popv[1, 0] = -300.0  # outside the pieces' range
    levels = rng.integers(0, 256, size=(batch, dims[0])).astype(np.uint8)
    x = levels.astype(np.float32) / np.float32(255.0) if floats else levels
    y = rng.integers(0, dims[2], size=batch).astype(np.int32)
    popd = to_device_pop(popv, gpu.leea_padded_params(dims))
    f, fa = (torch.empty(pop, device="cuda") for _ in range(2))
    cor = torch.empty(pop, dtype=torch.int32, device="cuda")
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    if floats:
        gpu.leea_evaluate(pop, dims, popd, xd, yd, batch, 1.0, None, f, fa, cor)
    else:
        gpu.leea_evaluate_u8(pop, dims, popd, xd, 255.0, yd, batch, 1.0, None, f, fa, cor)
    assert gpu.leea_device_status() == 0
    ref_x = x.astype(np.float64) if floats else levels.astype(np.float64) / 255.0
    f_ref, cor_ref, logits = oracle_mod.evaluate(popv.astype(np.float64), dims, ref_x, y, want_logits=True)
    assert_fitness_close(f.cpu().numpy(), f_ref)
    assert_correct_close(cor.cpu().numpy(), cor_ref, logits)
