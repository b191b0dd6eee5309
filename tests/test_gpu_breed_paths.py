"""The breeding kernel's three ways of mutating (listed pairs, all pairs with masks, every gene) and its edges:
genomes of one partial chunk (32 genes), one chunk less or more than 512 genes, a last chunk with padding, rates on
both sides of the switch, buffers that are only 16-byte aligned.  Against the oracle with the breeding tolerance."""
import numpy as np
import pytest

from helpers import assert_genes_close
from paper_1806_09819_gb300 import synthetic

pytestmark = pytest.mark.gpu

# c = 12, 482, 517, 513, 1054, 9010
SHAPES = [([2, 2, 2], 5), ([21, 20, 2], 7), ([52, 9, 4], 6), ([14, 32, 1], 4), ([100, 10, 4], 9), ([89, 99, 1], 3)]


@pytest.mark.parametrize("rate", [0.0, 2.0 ** -16, 0.1, 0.349, 0.351, 0.9999, 1.0])
@pytest.mark.parametrize("dims,pop", SHAPES, ids=[f"{d}-{p}" for d, p in SHAPES])
def test_breed_paths_match_oracle(gpu, oracle_mod, dims, pop, rate):
    import torch
    kw = dict(xo_gene_p=0.3, n_elite=1, p_c=0.3, sigma=0.02, mut_rate=rate)
    c, cp = gpu.leea_layout_num_params(dims), gpu.leea_padded_params(dims)
    parents = synthetic.random_population(pop, c, seed=c, scale=0.2)
    f = np.random.default_rng(c).normal(size=pop)
    prm = oracle_mod.Params(**kw)
    p1, p2, kind, _ = oracle_mod.select(prm, f, oracle_mod.rank(f), 9, 3)
    ref = oracle_mod.breed(prm, dims, 9, 3, parents.astype(np.float64), p1, p2, kind)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.int32)).cuda()
    got = []
    for skip in (0, 4):  # 32-byte aligned populations, and 16 bytes past that
        par = torch.full((pop * cp + 8,), 5.0, device="cuda")[skip:skip + pop * cp].view(pop, cp)
        par[:, :c] = torch.from_numpy(parents).cuda()  # the parents' padding is not zero: the children's is
        kid = torch.full((pop * cp + 8,), 3.0, device="cuda")[skip:skip + pop * cp].view(pop, cp)
        gpu.leea_breed(pop, dims, gpu.Params(**kw), 9, 3, par, t(p1), t(p2), t(kind), kid)
        got.append(kid.cpu().numpy())
    assert (got[0][:, c:] == 0).all()
    assert_genes_close(got[0][:, :c], ref, prm.sigma)
    np.testing.assert_array_equal(got[0], got[1])


def test_breed_invalid_parent_gives_nan(gpu):
    import torch
    dims, pop = [64, 16, 2], 4
    c, cp = gpu.leea_layout_num_params(dims), gpu.leea_padded_params(dims)
    par = torch.ones((pop, cp), device="cuda")
    kid = torch.zeros((pop, cp), device="cuda")
    i = lambda *v: torch.tensor(v, dtype=torch.int32, device="cuda")
    gpu.leea_breed(pop, dims, gpu.Params(sigma=0.0, mut_rate=0.5), 1, 1, par, i(0, pop, 1, 2), i(0, 0, -1, 2),
                   i(0, 2, 1, 2), kid)
    got = kid.cpu().numpy()
    assert (got[[0, 3], :c] == 1).all() and np.isnan(got[[1, 2], :c]).all() and (got[:, c:] == 0).all()
