"""Tensor-core descriptors at the shapes with the shortest ring of operand blocks for the way between two tasks of a
warp, several recipes per CTA: against the children that leea_breed_entities makes (checked against the oracle
elsewhere), rounded to BF16 and evaluated by the oracle, with the descriptor tolerances."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [[1024, 16, 10], [960, 48, 10], [960, 64, 10], [832, 128, 10], [16, 16, 10]], ids=str)
def test_probe_ring(gpu, oracle_mod, dims):
    import torch
    pop, n, n_probe = 7, 760, 4
    prm = dict(sigma=0.05, mut_rate=0.1, xo_gene_p=0.5)
    c, cp = gpu.leea_layout_num_params(dims), gpu.leea_padded_params(dims)
    rng = np.random.default_rng(dims[0] + dims[1])
    parents = rng.normal(0, 0.1, size=(pop, c)).astype(np.float32)
    p1, p2 = (rng.integers(0, pop, size=n).astype(np.int32) for _ in range(2))
    kind = (np.arange(n) % 3).astype(np.int32)
    ent = np.arange(n).astype(np.int32)
    f, f_inh = rng.normal(size=pop).astype(np.float32), rng.normal(size=n).astype(np.float32)
    probe = (rng.integers(0, 256, size=(n_probe, dims[0])) / 255.0).astype(np.float32)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    par = torch.zeros((pop, cp), device="cuda")
    par[:, :c] = t(parents)
    desc = torch.empty((n, 5 + n_probe * dims[2]), device="cuda")
    gpu.leea_descriptors(pop, dims, gpu.Params(precision=1, **prm), 7, 3, par, t(f), t(p1), t(p2), t(kind), t(f_inh),
                         t(ent), n, t(probe), n_probe, desc)
    assert gpu.leea_device_status() == 0
    kids = torch.zeros((n, cp), device="cuda")
    gpu.leea_breed_entities(pop, dims, gpu.Params(**prm), 7, 3, par, t(p1), t(p2), t(kind), t(ent), n, kids)
    q = oracle_mod.quantize_w1(kids[:, :c].cpu().numpy().astype(np.float64), dims, 1, None)
    _, _, ref = oracle_mod.evaluate(q, dims, probe.astype(np.float64), np.zeros(n_probe, dtype=np.int32),
                                    want_logits=True)
    np.testing.assert_allclose(desc[:, 5:].cpu().numpy(), ref.reshape(n, -1), rtol=1e-4, atol=1e-5 * np.abs(ref).max())
