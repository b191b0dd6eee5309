"""Evaluation through FP16 pieces where inputs and weights differ widely in scale: features of very different size with
weights in proportion, small features beside a large one, tiny first layers with large second ones, levels of a tiny
x_div.  What the pieces cannot carry has to come from the kernel that takes the call otherwise: against the FP64 oracle
with the fitness tolerance, and for floats the same bits as that kernel where every individual is of that kind."""
import numpy as np
import pytest

from helpers import assert_correct_close, assert_fitness_close, to_device_pop

pytestmark = pytest.mark.gpu


def _floats(gpu, dims, popd, x, y, path=0):
    import torch
    f = torch.empty(popd.shape[0], device="cuda")
    cor = torch.empty(popd.shape[0], dtype=torch.int32, device="cuda")
    gpu.leea_evaluate(popd.shape[0], dims, popd, torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), len(y), 1.0, None,
                      f, None, cor, path)
    assert gpu.leea_device_status() == 0
    return f.cpu().numpy(), cor.cpu().numpy()


def _population(gpu, dims, pop, rng):
    k, h, d = dims
    popv = np.zeros((pop, gpu.leea_layout_num_params(dims)), dtype=np.float32)
    popv[:, :k * h] = rng.normal(0.0, k ** -0.5, size=(pop, k * h))
    popv[:, k * h:k * h + h] = rng.normal(0.0, 0.01, size=(pop, h))
    popv[:, k * h + h:] = rng.normal(0.0, h ** -0.5, size=(pop, d * h + d))
    return popv


CASES = ["large_features", "small_beside_large", "one_unit_large", "tiny_first_layer"]


@pytest.mark.parametrize("batch", [60, 300])
@pytest.mark.parametrize("case", CASES)
def test_floats(gpu, oracle_mod, case, batch):
    dims, pop = [784, 112, 10], 310
    k, h, d = dims
    rng = np.random.default_rng(CASES.index(case) * 1000 + batch)
    popv = _population(gpu, dims, pop, rng)
    w1 = popv[:, :k * h].reshape(pop, h, k)
    w2 = popv[:, k * h + h:k * h + h + d * h].reshape(pop, d, h)
    x = rng.random((batch, k)).astype(np.float32)
    if case == "large_features":          # 8 columns of 1e7 with weights in proportion
        x[:, :8] *= np.float32(1e7)
        w1[:, :, :8] *= np.float32(1e-7)
    elif case == "small_beside_large":    # one input that no weight reads, the others small
        x *= np.float32(1e-3)
        x[:, 5] = 1e6
        w1[:, :, 5] = 0.0
        w2 *= np.float32(1e3)
    elif case == "one_unit_large":        # one hidden unit reads the large columns, the others hardly
        x[:, :8] *= np.float32(1e7)
        w1[:, 1:, :8] *= np.float32(1e-7)
        w2[:, :, 0] *= np.float32(1e-6)
    else:                                 # weights below 2^-11 but for one, second layers to match
        w1 *= np.float32(1e-6)
        w1[:, 3, 3] = 0.05
        w2 *= np.float32(1e6)
        w2[:, :, 3] *= np.float32(1e-6)
    y = rng.integers(0, d, size=batch).astype(np.int32)
    popd = to_device_pop(popv, gpu.leea_padded_params(dims))
    f, cor = _floats(gpu, dims, popd, x, y)
    f_ref, cor_ref, logits = oracle_mod.evaluate(popv.astype(np.float64), dims, x.astype(np.float64), y, want_logits=True)
    assert_fitness_close(f, f_ref)
    assert_correct_close(cor, cor_ref, logits)
    f_tf32, cor_tf32 = _floats(gpu, dims, popd, x, y, gpu.EVAL_TENSOR)
    np.testing.assert_array_equal(f, f_tf32)
    np.testing.assert_array_equal(cor, cor_tf32)


def test_even_scales_keep_the_pieces(gpu):
    """Images, and images without their division by 255: no individual is evaluated twice."""
    dims, pop, batch = [784, 112, 10], 310, 100
    rng = np.random.default_rng(1)
    popd = to_device_pop(_population(gpu, dims, pop, rng), gpu.leea_padded_params(dims))
    y = rng.integers(0, 10, size=batch).astype(np.int32)
    for scale in (1.0, 255.0):
        x = (rng.random((batch, 784)) * scale).astype(np.float32)
        f, _ = _floats(gpu, dims, popd, x, y)
        f_tf32, _ = _floats(gpu, dims, popd, x, y, gpu.EVAL_TENSOR)
        assert (f != f_tf32).mean() > 0.9  # other roundings: the pieces' own


@pytest.mark.parametrize("dims,pop,batch", [([784, 100, 10], 620, 60), ([784, 112, 10], 310, 300)])
@pytest.mark.parametrize("case", ["tiny_first_layer", "tiny_x_div"])
def test_levels(gpu, oracle_mod, case, dims, pop, batch):
    import torch
    k, h, d = dims
    rng = np.random.default_rng(batch + len(case))
    popv = _population(gpu, dims, pop, rng)
    w1 = popv[:, :k * h]
    x_div = 255.0
    if case == "tiny_first_layer":
        w1 *= np.float32(1e-6)
        popv[:, k * h + h:k * h + h + d * h] *= np.float32(1e6)
        popv[:, k * h:k * h + h] *= np.float32(1e-6)
    else:
        w1 *= np.float32(1e-6)
        x_div = 255.0e-6
    lv = rng.integers(0, 256, size=(batch, k)).astype(np.uint8)
    y = rng.integers(0, d, size=batch).astype(np.int32)
    f = torch.empty(pop, device="cuda")
    cor = torch.empty(pop, dtype=torch.int32, device="cuda")
    gpu.leea_evaluate_u8(pop, dims, to_device_pop(popv, gpu.leea_padded_params(dims)), torch.from_numpy(lv).cuda(), x_div,
                         torch.from_numpy(y).cuda(), batch, 1.0, None, f, None, cor)
    assert gpu.leea_device_status() == 0
    f_ref, cor_ref, logits = oracle_mod.evaluate(popv.astype(np.float64), dims, lv.astype(np.float64) / x_div, y,
                                                 want_logits=True)
    assert_fitness_close(f.cpu().numpy(), f_ref)
    assert_correct_close(cor.cpu().numpy(), cor_ref, logits)
