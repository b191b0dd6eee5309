"""The tensor-core probe's ways of mutating (none, listed pairs, all pairs with masks, every gene) and the edges of its
tasks: a short last K block of 1, 3 and 4 sixteens, one K block, more warps than tasks, a tail that ends inside a unit,
populations that are only 16-byte aligned.  Against the children that leea_breed_entities makes (checked against the
oracle elsewhere), rounded to BF16 and evaluated by the oracle, with the descriptor tolerances."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [([784, 16, 10], 32), ([112, 48, 3], 5), ([64, 16, 1], 1), ([256, 128, 16], 32), ([80, 32, 7], 31)]


@pytest.mark.parametrize("rate", [0.0, 0.1, 0.349, 0.351, 1.0])
@pytest.mark.parametrize("dims,n_probe", SHAPES, ids=[str(d) for d, _ in SHAPES])
def test_probe_paths(gpu, oracle_mod, dims, n_probe, rate):
    import torch
    pop, n = 9, 160  # more recipes than SMs: some CTAs take two
    kw = dict(sigma=0.05, mut_rate=rate, xo_gene_p=0.3)
    c, cp = gpu.leea_layout_num_params(dims), gpu.leea_padded_params(dims)
    rng = np.random.default_rng(dims[0] + dims[1])
    parents = rng.normal(0, 0.1, size=(pop, c)).astype(np.float32)
    p1, p2 = (rng.integers(0, pop, size=n).astype(np.int32) for _ in range(2))
    kind = (np.arange(n) % 3).astype(np.int32)
    ent = (np.arange(n) + 2 ** 30).astype(np.int32)
    f, f_inh = rng.normal(size=pop).astype(np.float32), rng.normal(size=n).astype(np.float32)
    probe = (rng.integers(0, 256, size=(n_probe, dims[0])) / 255.0).astype(np.float32)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    got = []
    for skip in (0, 4):
        par = torch.zeros(pop * cp + 8, device="cuda")[skip:skip + pop * cp].view(pop, cp)
        par[:, :c] = t(parents)
        desc = torch.empty((n, 5 + n_probe * dims[2]), device="cuda")
        gpu.leea_descriptors(pop, dims, gpu.Params(precision=1, **kw), 7, 3, par, t(f), t(p1), t(p2), t(kind), t(f_inh),
                             t(ent), n, t(probe), n_probe, desc)
        assert gpu.leea_device_status() == 0
        got.append(desc.cpu().numpy())
    np.testing.assert_array_equal(got[0], got[1])
    d = got[0].astype(np.float64)
    kids = torch.zeros((n, cp), device="cuda")
    gpu.leea_breed_entities(pop, dims, gpu.Params(**kw), 7, 3, par.clone(), t(p1), t(p2), t(kind), t(ent), n, kids)
    kids = kids[:, :c].cpu().numpy().astype(np.float64)
    pa, pb = parents[p1].astype(np.float64), parents[p2].astype(np.float64)
    np.testing.assert_array_equal(d[:, 0], f[p1])
    np.testing.assert_array_equal(d[:, 1], f[p2])
    np.testing.assert_array_equal(d[:, 2], f_inh)
    frac = np.where((kids == pb) & (pa != pb), 1, 0).mean(axis=1)
    xo = (kind == 1) & (p1 != p2)  # the parents differ in every gene
    np.testing.assert_allclose(d[xo, 3], frac[xo], rtol=1e-6)
    assert (d[kind != 1, 3] == 0).all() and (d[kind != 2, 4] == 0).all()
    step = np.sqrt(((kids - pa) ** 2).sum(axis=1))
    # the step recovered from rounded children: half an ulp (2^-25) of genes of at most 0.6 in each
    np.testing.assert_allclose(d[kind == 2, 4], step[kind == 2], rtol=1e-5, atol=2.0 ** -25 * np.sqrt(c))
    q = oracle_mod.quantize_w1(kids, dims, 1, None)
    _, _, ref = oracle_mod.evaluate(q, dims, probe.astype(np.float64), np.zeros(n_probe, dtype=np.int32),
                                    want_logits=True)
    np.testing.assert_allclose(d[:, 5:], ref.reshape(n, -1), rtol=1e-4, atol=1e-5 * np.abs(ref).max())
