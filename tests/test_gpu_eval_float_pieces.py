"""Evaluation of float inputs through FP16 pieces: edges of tiles, units and K stages, samples of very different
magnitudes, and the individuals and samples that the pieces cannot carry.  Against the FP64 oracle with the fitness
tolerance; for infinite and NaN inputs against the TF32 path."""
import numpy as np
import pytest

from helpers import assert_correct_close, assert_fitness_close, to_device_pop

pytestmark = pytest.mark.gpu

CASES = [  # dims, pop, batch
    ([784, 112, 10], 155, 100), ([784, 100, 10], 333, 50), ([784, 1, 10], 5, 3), ([4, 17, 2], 3, 1),
    ([20, 129, 16], 7, 130), ([784, 256, 16], 4, 256), ([784, 112, 10], 1, 1000), ([52, 112, 10], 305, 128),
    ([36, 127, 5], 307, 257), ([68, 16, 10], 2400, 127), ([784, 33, 10], 3, 1025), ([100, 128, 10], 153, 129),
    ([20, 128, 16], 700, 130), ([36, 112, 5], 400, 257), ([784, 32, 10], 300, 1025), ([784, 16, 10], 170, 3),
]


def _run(gpu, dims, popd, x, y, path=0, alpha=1.0, f_inh=None):
    import torch
    pop = popd.shape[0]
    f, fa = (torch.empty(pop, device="cuda") for _ in range(2))
    cor = torch.empty(pop, dtype=torch.int32, device="cuda")
    gpu.leea_evaluate(pop, dims, popd, torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), len(y), alpha,
                      None if f_inh is None else torch.from_numpy(f_inh).cuda(), f, fa, cor, path)
    assert gpu.leea_device_status() == 0
    return f.cpu().numpy(), fa.cpu().numpy(), cor.cpu().numpy()


def _population(gpu, dims, pop, rng):
    popv = rng.normal(0.0, 0.15, size=(pop, gpu.leea_layout_num_params(dims))).astype(np.float32)
    if pop > 3:
        w1 = dims[0] * dims[1]
        popv[1, w1 // 2] = 200.0                 # above the pieces' range
        popv[2] = popv[0]                        # the same individual elsewhere in a unit
        popv[3, :w1] *= np.float32(1e-6)         # below the pieces' resolution
        popv[pop - 1, :w1] = 0.0
    return popv


@pytest.mark.parametrize("dims,pop,batch", CASES, ids=[f"{d}-{p}-{b}" for d, p, b in CASES])
def test_float_pieces_match_oracle(gpu, oracle_mod, dims, pop, batch):
    rng = np.random.default_rng(dims[1] * 1000 + batch)
    popv = _population(gpu, dims, pop, rng)
    x = rng.normal(0.0, 1.0, size=(batch, dims[0])).astype(np.float32)
    x *= (10.0 ** rng.uniform(-12, 1, size=(batch, 1))).astype(np.float32)
    x[0] = 0.0
    if batch > 2:
        x[1, 1:] *= np.float32(1e-7)             # one input far above the sample's others
        x[2] = np.float32(1e-42)                 # subnormal
    y = rng.integers(0, dims[2], size=batch).astype(np.int32)
    f_inh = rng.normal(-2.3, 0.1, size=pop).astype(np.float32)
    f, fa, cor = _run(gpu, dims, to_device_pop(popv, gpu.leea_padded_params(dims)), x, y, 0, 0.3, f_inh)
    f_ref, cor_ref, logits = oracle_mod.evaluate(popv.astype(np.float64), dims, x.astype(np.float64), y, want_logits=True)
    assert_fitness_close(f, f_ref)
    assert_correct_close(cor, cor_ref, logits)
    adj_ref = oracle_mod.inherit(float(np.float32(0.3)), f_inh.astype(np.float64), f_ref, first=False)
    assert_fitness_close(fa, adj_ref, "f_adj")
    if pop > 3:
        assert f[0] == f[2]


@pytest.mark.parametrize("dims,pop", [([784, 112, 10], 40), ([36, 64, 5], 400)])
def test_float_pieces_non_finite_inputs(gpu, dims, pop):
    """Bit for bit what the TF32 kernel gives."""
    rng = np.random.default_rng(3)
    popd = to_device_pop(_population(gpu, dims, pop, rng), gpu.leea_padded_params(dims))
    y = rng.integers(0, dims[2], size=70).astype(np.int32)
    for v in (np.inf, -np.inf, np.nan):
        x = rng.random((70, dims[0])).astype(np.float32)
        x[33, 5] = v
        for a, b in zip(_run(gpu, dims, popd, x, y, 0), _run(gpu, dims, popd, x, y, gpu.EVAL_TENSOR)):
            np.testing.assert_array_equal(a, b)
