"""How the tensor-core evaluation of deeper nets adds up an individual's loss: identical individuals get identical bits."""
import numpy as np
import pytest

from helpers import assert_fitness_close, to_device_pop

pytestmark = pytest.mark.gpu


def _evaluate(gpu, dims, pd, levels, y):
    import torch
    pop = pd.shape[0]
    f = torch.full((pop,), float("nan"), device="cuda")
    cor = torch.full((pop,), -1, dtype=torch.int32, device="cuda")
    gpu.leea_evaluate_u8(pop, dims, pd, torch.from_numpy(levels).cuda(), 255.0, torch.from_numpy(y).cuda(), len(y), 1.0,
                         None, f, None, cor, gpu.EVAL_TENSOR)
    assert gpu.leea_device_status() == 0
    return f.cpu().numpy(), cor.cpu().numpy()


@pytest.mark.parametrize("dims,batch", [([16, 16, 16, 16, 2], 128), ([32, 16, 16, 16, 10], 1), ([64, 32, 16, 32, 5], 77)])
def test_many_small_nets_of_one_tile(gpu, dims, batch):
    """Net after net on every CTA with little between them: each one's sum holds all of its samples and no other's, so
    that it has the bits of the net alone on a CTA (which the oracle checks elsewhere)."""
    pop, kinds = 12000, 7
    rng = np.random.default_rng(batch)
    nets = rng.normal(0.0, 0.5, size=(kinds, gpu.leea_layout_num_params(dims))).astype(np.float32)
    which = rng.integers(0, kinds, size=pop)
    levels = rng.integers(0, 256, size=(batch, dims[0])).astype(np.uint8)
    y = rng.integers(0, dims[-1], size=batch).astype(np.int32)
    cp = gpu.leea_padded_params(dims)
    alone, cor_alone = _evaluate(gpu, dims, to_device_pop(nets, cp), levels, y)
    pd = to_device_pop(nets[which], cp)
    for _ in range(3):
        f, cor = _evaluate(gpu, dims, pd, levels, y)
        np.testing.assert_array_equal(f, alone[which])
        np.testing.assert_array_equal(cor, cor_alone[which])


def test_twins_split_differently_among_ctas(gpu):
    """Twins on three tiles, of which some lie within a CTA and others in two or three.  The losses make the order of the
    sum visible in the result: 3 2^58 and 3 2^34 in the first tile, whose quotient by the 384 samples is a tie between two
    floats, and 64, half an ulp of their FP64 sum, in each of the others."""
    dims, pop, batch = [64, 16, 16, 16, 10], 228, 384
    net = np.zeros(gpu.leea_layout_num_params(dims), dtype=np.float32)
    net[-10:] = [0.0, -3.0 * 2.0 ** 58, -3.0 * 2.0 ** 34, -64.0] + [-200.0] * 6  # the output layer's biases
    y = np.zeros(batch, dtype=np.int32)  # class 0: loss 0; class o: minus its bias
    y[0], y[1], y[128 + 5], y[256 + 5] = 1, 2, 3, 3
    levels = np.zeros((batch, dims[0]), dtype=np.uint8)
    f, cor = _evaluate(gpu, dims, to_device_pop(np.tile(net, (pop, 1)), gpu.leea_padded_params(dims)), levels, y)
    total = ((3.0 * 2.0 ** 58 + 3.0 * 2.0 ** 34) + 64.0) + 64.0
    np.testing.assert_array_equal(f, np.full(pop, -np.float32(total / batch)))
    assert (cor == batch - 4).all()


@pytest.mark.parametrize("batch", [5, 40, 200])
def test_last_layer_is_fp32(gpu, oracle_mod, batch):
    """Last-layer weights of 24 bits that nearly cancel in pairs: 64 (1 + 2^-12 + 2^-23) - 64 (1 + 2^-12), eight times, a
    logit of 2^-14 that weights of 22 bits lose."""
    dims = [16, 16, 16, 16, 2]
    net = np.zeros(gpu.leea_layout_num_params(dims), dtype=np.float32)
    b3 = 3 * (16 * 16 + 16) - 16
    net[b3:b3 + 16] = 64.0  # layer 3's activations
    w4 = net[b3 + 16:b3 + 16 + 32].reshape(2, 16)
    w4[0, 0::2] = 1.0 + 2.0 ** -12 + 2.0 ** -23
    w4[0, 1::2] = -(1.0 + 2.0 ** -12)
    levels, y = np.full((batch, 16), 7, dtype=np.uint8), np.zeros(batch, dtype=np.int32)
    f, _ = _evaluate(gpu, dims, to_device_pop(np.tile(net, (3, 1)), gpu.leea_padded_params(dims)), levels, y)
    ref, _ = oracle_mod.evaluate(np.tile(net, (3, 1)).astype(np.float64), dims, levels.astype(np.float64) / 255.0, y)
    assert abs(ref[0] + np.log1p(np.exp(-2.0 ** -14))) < 1e-12  # the oracle's sum of `batch` equal losses
    assert_fitness_close(f, ref)
