"""The tensor-core evaluation of 8-bit inputs beyond the shapes that eval_path TENSOR promises: hidden widths off the
MMA's 16, up to 256, and batches of several 128-sample tiles, at the edges of tiles, units and CTAs.  Against the FP64
oracle with the fitness tolerance, and bit for bit where the same individual or sample tile appears twice."""
import numpy as np
import pytest

from helpers import assert_correct_close, assert_fitness_close, to_device_pop

pytestmark = pytest.mark.gpu

CASES = [  # dims, pop, batch
    ([784, 100, 10], 333, 50), ([784, 1, 10], 5, 3), ([4, 17, 2], 3, 1), ([20, 129, 16], 7, 130), ([784, 255, 3], 3, 7),
    ([784, 256, 16], 2, 256), ([784, 112, 10], 1, 1000), ([784, 112, 10], 155, 384), ([52, 112, 10], 153, 129),
    ([36, 127, 5], 307, 257), ([68, 16, 10], 400, 512), ([784, 33, 10], 2, 1025),
    ([784, 100, 10], 333, 47), ([784, 100, 10], 333, 48),
]


def _run(gpu, dims, popd, levels, y, alpha=1.0, f_inh=None):
    import torch
    pop = popd.shape[0]
    f, fa = (torch.empty(pop, device="cuda") for _ in range(2))
    cor = torch.empty(pop, dtype=torch.int32, device="cuda")
    gpu.leea_evaluate_u8(pop, dims, popd, torch.from_numpy(levels).cuda(), 255.0, torch.from_numpy(y).cuda(),
                         len(y), alpha, None if f_inh is None else torch.from_numpy(f_inh).cuda(), f, fa, cor)
    assert gpu.leea_device_status() == 0
    return f.cpu().numpy(), fa.cpu().numpy(), cor.cpu().numpy()


@pytest.mark.parametrize("dims,pop,batch", CASES, ids=[f"{d}-{p}-{b}" for d, p, b in CASES])
def test_wide_matches_oracle(gpu, oracle_mod, dims, pop, batch):
    rng = np.random.default_rng(dims[1] * 1000 + batch)
    c, cp = gpu.leea_layout_num_params(dims), gpu.leea_padded_params(dims)
    popv = rng.normal(0.0, 0.15, size=(pop, c)).astype(np.float32)
    if pop > 2:
        popv[1, (dims[0] * dims[1]) // 2] = 200.0    # outside the FP16 pieces' range: FP32 layer 1
        popv[2] = popv[0]                            # the same individual elsewhere in a unit
    levels = rng.integers(0, 256, size=(batch, dims[0])).astype(np.uint8)
    y = rng.integers(0, dims[2], size=batch).astype(np.int32)
    f_inh = rng.normal(-2.3, 0.1, size=pop).astype(np.float32)
    f, fa, cor = _run(gpu, dims, to_device_pop(popv, cp), levels, y, 0.3, f_inh)
    f_ref, cor_ref, logits = oracle_mod.evaluate(popv.astype(np.float64), dims, levels.astype(np.float64) / 255.0, y,
                                                 want_logits=True)
    assert_fitness_close(f, f_ref)
    assert_correct_close(cor, cor_ref, logits)
    adj_ref = oracle_mod.inherit(float(np.float32(0.3)), f_inh.astype(np.float64), f_ref, first=False)
    assert_fitness_close(fa, adj_ref, "f_adj")
    if pop > 2:
        assert f[0] == f[2]


def test_wide_state_object_grows_with_the_batch(gpu, oracle_mod):
    """One FP32 state object over batches on both sides of a tile, each generation's fitness against the oracle."""
    import torch
    dims, pop = [784, 48, 10], 100
    st = gpu.LeeaState(pop, dims, gpu.Params(sigma=0.01, mut_rate=0.1, n_elite=1), seed=11)
    rng = np.random.default_rng(5)
    for batch in (100, 300, 129, 700, 128):
        levels = rng.integers(0, 256, size=(batch, 784)).astype(np.uint8)
        y = rng.integers(0, 10, size=batch).astype(np.int32)
        st.leea_generation_u8(torch.from_numpy(levels).cuda(), torch.from_numpy(y).cuda())
        f_ref, _ = oracle_mod.evaluate(st.leea_get_population().astype(np.float64), dims,
                                       levels.astype(np.float64) / 255.0, y)
        assert_fitness_close(st.leea_raw_fitness(), f_ref)
    st.close()
