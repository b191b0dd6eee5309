"""Performance cases: the work a user of the library has it do, through its public entry points.

Whole calls (the state objects, several generations and then the reads a training loop makes):

* ``generation``  Algorithm 1 on the library-owned state object, FP32 or with BF16 / FP8 shadows of W1
* ``batching``    many independent runs of uneven sizes advanced together

Single steps on caller-owned device buffers (a caller that composes its own generation):

* ``breed``       crossover and mutation of a whole population (Section 3.2)
* ``evaluate``    fitness of a whole population on one minibatch (Eq. 1), 8-bit or float inputs
* ``shadow``      the same through BF16 / FP8 shadows of W1
* ``descriptors`` the surrogate form's fused breed + probe pass over a generation's recipes

Nets are 784-h-10 (28x28 images) or the paper's 196-256-128-64-10 behind 2x2 pooling.  Inputs are the synthetic
28x28 images of ``paper_1806_09819_gb300.synthetic``; populations are N(0, 1/fan_in) weights with small biases, which
is where a run starts and, with mutation steps of 0.001-0.005, about where it stays.
"""
import math
import random

import numpy as np
import torch

from paper_1806_09819_gb300 import leea, synthetic

PAPER_NET = "196-256-128-64-10"
DEVICE = torch.device("cuda", 0)
N_PROBE = 32
RECIPE_ENTITY0 = 1 << 30  # Philox entity of recipe 0


# ---- the cases ---------------------------------------------------------------------
def listed():
    return [
        # The smallest run: a generation is a chain of latencies.  20 generations, then fitness and the best net.
        dict(name="generation_small", kind="generation", precision=0, pop=32, hidden=32, batch=16, gens=20),
        # The benchmark's run: FP32, 1000 nets of 89,050 genes, a minibatch of 100.
        dict(name="generation_plain", kind="generation", precision=0, pop=1000, hidden=112, batch=100, gens=10),
        # The precision form at its benchmark size.
        dict(name="generation_bf16", kind="generation", precision=1, pop=4096, hidden=112, batch=256, gens=3),
        # A parameter study: 16 runs of uneven population, width and batch advanced together.
        dict(name="batching_16", kind="batching", precision=1, runs=16, pop_max=2000, spec_seed=4242, gens=2),
        # The breeding step of the benchmark's run: one gene in ten mutates.
        dict(name="breed_plain", kind="breed", net="784-112-10", pop=1000, p_c=0.5, xo_op=0, mut_rate=0.1),
        # The paper's operators on the paper's network: every gene of a mutation child mutates.
        dict(name="breed_every_gene", kind="breed", net=PAPER_NET, pop=1000, p_c=0.5, xo_op=0, mut_rate=1.0),
        # Float inputs (data that are no 8-bit images).
        dict(name="evaluate_f32", kind="evaluate", net="784-112-10", pop=1000, batch=100, inputs="f32"),
        # The paper's default minibatch of 512 (Section 4) on 8-bit images.
        dict(name="evaluate_batch512", kind="evaluate", net="784-112-10", pop=1000, batch=512, inputs="u8"),
        # A hidden width and a batch off every tile: 100 hidden units, 50 samples, 333 nets.
        dict(name="evaluate_odd", kind="evaluate", net="784-100-10", pop=333, batch=50, inputs="u8"),
        # The paper's network, population and batch of its comparison with SGD (Section 4.5).
        dict(name="evaluate_paper_net", kind="evaluate", net=PAPER_NET, pop=2000, batch=1024, inputs="u8"),
        # The precision form's evaluation as a step call, FP8.
        dict(name="shadow_fp8", kind="shadow", precision=2, pop=2048, hidden=112, batch=256),
        # The surrogate form's benchmark size: 4 recipes per offspring slot of 2048 nets.
        dict(name="descriptors", kind="descriptors", pop=2048, hidden=112, mult=4),
    ]


def _logu(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["generation", "batching", "breed", "evaluate", "evaluate", "shadow", "descriptors"])
    if kind == "generation":
        precision = rng.choice([0, 0, 1, 2])
        pop = _logu(rng, 32, 1000 if precision == 0 else 4096)
        return dict(kind=kind, precision=precision, pop=pop, hidden=16 * _logu(rng, 1, 8),
                    batch=_logu(rng, 8, 128 if precision == 0 else 256), gens=max(1, min(10, 4000 // pop)))
    if kind == "batching":
        return dict(kind=kind, precision=rng.choice([1, 1, 2]), runs=rng.randint(4, 12), pop_max=_logu(rng, 100, 1500),
                    spec_seed=rng.randrange(1 << 20), gens=2)
    if kind == "breed":
        net = rng.choice([PAPER_NET, "784-%d-10" % _logu(rng, 16, 256)])
        most = 1000 * 89050 // _genes(_dims(net))
        return dict(kind=kind, net=net, pop=_logu(rng, 32, min(4096, most)), p_c=rng.choice([0.0, 0.5, 0.75]),
                    xo_op=rng.choice([0, 0, 1]), mut_rate=rng.choice([0.1, 0.3, 1.0]))
    if kind == "evaluate":
        inputs = rng.choice(["u8", "u8", "f32"])
        net = rng.choice([PAPER_NET, "784-%d-10" % _logu(rng, 16, 256), "784-%d-10" % (16 * _logu(rng, 1, 16))])
        batch = _logu(rng, 8, 1024)
        flops = _flops(_dims(net))
        # At most the work of the dearest listed case on the same units.
        most = (2000 * 1024 if inputs == "u8" else 60000) if net == PAPER_NET else 1000 * 512 * 112 * 794 * 2 // flops
        return dict(kind=kind, net=net, pop=min(2000, max(16, min(_logu(rng, 16, 2000), most // batch))), batch=batch,
                    inputs=inputs)
    if kind == "shadow":
        return dict(kind=kind, precision=rng.choice([1, 2]), pop=_logu(rng, 32, 2048), hidden=16 * _logu(rng, 1, 8),
                    batch=_logu(rng, 8, 256))
    return dict(kind=kind, pop=_logu(rng, 64, 2048), hidden=16 * _logu(rng, 1, 7), mult=rng.randint(1, 4))


# ---- sizes -------------------------------------------------------------------------
def _dims(net):
    return [int(v) for v in net.split("-")]


def _genes(dims):
    return sum(dims[i + 1] * dims[i] + dims[i + 1] for i in range(len(dims) - 1))


def _padded(dims):
    return -(-_genes(dims) // 32) * 32


def _flops(dims):
    """Per net and sample: two per weight."""
    return 2 * sum(dims[i + 1] * dims[i] for i in range(len(dims) - 1))


def _net_of(case):
    return _dims(case["net"]) if "net" in case else [784, case["hidden"], 10]


def _counts(pop, p_c, n_elite=1):
    """Elites, crossover children and mutation children."""
    nc = min(int(math.floor(p_c * pop + 0.5)), pop - n_elite)
    return n_elite, nc, pop - n_elite - nc


def _run_specs(case):
    """Populations, hidden widths and batches of a batching case, log-uniform over the benchmark's ranges."""
    rng = random.Random(case["spec_seed"])
    return [(_logu(rng, 50, case["pop_max"]), min(256, max(16, 16 * round(_logu(rng, 16, 256) / 16))),
             _logu(rng, 8, 512)) for _ in range(case["runs"])]


def _params(case):
    """The benchmark's operators."""
    return leea.Params(n_elite=1, p_c=case.get("p_c", 0.5), sigma=0.005, mut_rate=case.get("mut_rate", 0.1),
                       xo_op=case.get("xo_op", 0), precision=case.get("precision", 0))


# ---- inputs ------------------------------------------------------------------------
def _generator(seed):
    return torch.Generator(device=DEVICE).manual_seed(int(seed) * 1000003 % (1 << 62))


def _population(pop, dims, seed):
    """float32[pop][c_pad]: weights N(0, 1/fan_in), biases N(0, 0.01^2), zero padding."""
    g = _generator(seed)
    out = torch.zeros((pop, _padded(dims)), device=DEVICE)
    off = 0
    for i in range(len(dims) - 1):
        n = dims[i + 1] * dims[i]
        out[:, off:off + n].normal_(0.0, dims[i] ** -0.5, generator=g)
        out[:, off + n:off + n + dims[i + 1]].normal_(0.0, 0.01, generator=g)
        off += n + dims[i + 1]
    return out


def _images(n, d_in, seed):
    """(levels uint8[n][d_in], labels int32[n]) on the GPU, 28x28 or pooled 2x2."""
    x, y = synthetic.make_split(n, int(seed) % (1 << 31), synthetic.templates())
    lv = synthetic.to_levels(x)
    if d_in == 196:
        lv = lv.reshape(n, 14, 2, 14, 2).max(axis=(2, 4)).reshape(n, 196)
    return torch.from_numpy(np.ascontiguousarray(lv)).to(DEVICE), torch.from_numpy(y).to(DEVICE)


def _selection(pop, n, n_cross, n_elite, f, g):
    """Parents, kinds and inherited fitness of n children: truncation to the better half of pop (Section 3.1)."""
    order = torch.argsort(f, descending=True)
    pool = order[:max(1, pop // 2)]
    par1 = pool[torch.randint(len(pool), (n,), generator=g, device=DEVICE)]
    par2 = pool[torch.randint(len(pool), (n,), generator=g, device=DEVICE)]
    kind = torch.full((n,), 2, dtype=torch.int32, device=DEVICE)
    kind[:n_elite + n_cross] = 1
    kind[:n_elite] = 0
    par1[:n_elite] = order[:n_elite]
    par2 = torch.where(kind == 1, par2, par1)
    f_inh = (f[par1] + f[par2]) / 2
    return par1.int(), par2.int(), kind, f_inh


def prepare(case, seed):
    s = dict(case=case, seed=int(seed))
    kind = case["kind"]
    if kind == "generation":
        dims = _net_of(case)
        x, y = _images(case["batch"] * (case["gens"] + 1), dims[0], seed)
        n = case["batch"]
        s["x"] = [x[i * n:(i + 1) * n].clone() for i in range(case["gens"] + 1)]
        s["y"] = [y[i * n:(i + 1) * n].clone() for i in range(case["gens"] + 1)]
        s["state"] = leea.LeeaState(case["pop"], dims, _params(case), int(seed))
        s["state"].leea_generation_u8(s["x"][0], s["y"][0])  # evaluates the initial population
    elif kind == "batching":
        specs = [leea.RunSpec(p, h, b, seed=int(seed) * 1000 + r) for r, (p, h, b) in enumerate(_run_specs(case))]
        s["state"] = leea.MultiRun(specs, 784, 10, _params(case))
        rows = s["state"].total_rows
        x, y = _images(rows * (case["gens"] + 1), 784, seed)
        s["x"] = [x[i * rows:(i + 1) * rows].clone() for i in range(case["gens"] + 1)]
        s["y"] = [y[i * rows:(i + 1) * rows].clone() for i in range(case["gens"] + 1)]
        for i in range(case["gens"] + 1):  # the initial evaluation, and both buffer parities
            s["state"].generation_u8(s["x"][i], s["y"][i])
    elif kind == "breed":
        dims, pop = _net_of(case), case["pop"]
        s["prm"] = _params(case)
        s["parents"] = _population(pop, dims, seed)
        g = _generator(seed + 1)
        f = torch.randn(pop, generator=g, device=DEVICE) * 0.1 - 2.3
        ne, nc, _ = _counts(pop, case["p_c"])
        s["par1"], s["par2"], s["kind"], _ = _selection(pop, pop, nc, ne, f, g)
        s["children"] = torch.zeros_like(s["parents"])
    elif kind in ("evaluate", "shadow"):
        dims, pop, batch = _net_of(case), case["pop"], case["batch"]
        s["pop"] = _population(pop, dims, seed)
        s["x"], s["y"] = _images(batch, dims[0], seed)
        g = _generator(seed + 1)
        s["f_inh"] = torch.randn(pop, generator=g, device=DEVICE) * 0.1 - 2.3
        s["f_raw"], s["f_adj"] = torch.empty(pop, device=DEVICE), torch.empty(pop, device=DEVICE)
        if case.get("inputs") == "f32":
            s["x"] = s["x"].float() / 255.0
        if kind == "shadow":
            prec = case["precision"]
            s["shadow"] = torch.empty((pop, leea.leea_shadow_stride(dims, prec)), dtype=torch.uint8, device=DEVICE)
            s["scale"] = torch.zeros(pop, dtype=torch.int32, device=DEVICE)
            s["amax"] = torch.empty(pop, device=DEVICE)
            leea.leea_make_shadow(pop, dims, prec, s["pop"], s["shadow"], s["scale"], s["amax"])
            s["correct"] = torch.empty(pop, dtype=torch.int32, device=DEVICE)
            nbytes = leea.leea_shadow_scratch_bytes(pop, batch)
            s["scratch"] = torch.empty(nbytes // 4, device=DEVICE) if nbytes else None
    else:
        dims, pop = _net_of(case), case["pop"]
        _, nc, nm = _counts(pop, 0.5)
        n = case["mult"] * (nc + nm)
        g = _generator(seed + 1)
        s["prm"] = leea.Params(n_elite=1, p_c=0.5, sigma=0.005, mut_rate=0.1, precision=1)
        s["parents"] = _population(pop, dims, seed)
        s["f"] = torch.randn(pop, generator=g, device=DEVICE) * 0.1 - 2.3
        s["par1"], s["par2"], s["kind"], s["f_inh"] = _selection(pop, n, case["mult"] * nc, 0, s["f"], g)
        s["entity"] = torch.arange(RECIPE_ENTITY0, RECIPE_ENTITY0 + n, dtype=torch.int64, device=DEVICE).int()
        lv, _ = _images(N_PROBE, 784, seed)
        s["probe"] = lv.float() / 255.0
        s["desc"] = torch.empty((n, 5 + N_PROBE * dims[-1]), device=DEVICE)
    return s


# ---- one pass ----------------------------------------------------------------------
def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "generation":
        st = state["state"]
        for i in range(1, case["gens"] + 1):
            st.leea_generation_u8(state["x"][i], state["y"][i])
        f, correct = st.leea_fitness(with_correct=True)
        return {"f_adj": f, "correct": correct, "best": st.leea_best_params()}
    if kind == "batching":
        st = state["state"]
        for i in range(1, case["gens"] + 1):
            st.generation_u8(state["x"][i], state["y"][i])
        f, correct = st.fitness(with_correct=True)
        return {"f_adj": f, "correct": correct}
    dims, pop = _net_of(case), case["pop"]
    if kind == "breed":
        leea.leea_breed(pop, dims, state["prm"], state["seed"], 1, state["parents"], state["par1"], state["par2"],
                        state["kind"], state["children"])
        return state["children"]
    if kind == "evaluate":
        if case["inputs"] == "u8":
            leea.leea_evaluate_u8(pop, dims, state["pop"], state["x"], 255.0, state["y"], case["batch"], 0.5,
                                  state["f_inh"], state["f_raw"], state["f_adj"])
        else:
            leea.leea_evaluate(pop, dims, state["pop"], state["x"], state["y"], case["batch"], 0.5, state["f_inh"],
                               state["f_raw"], state["f_adj"])
        return {"f_raw": state["f_raw"], "f_adj": state["f_adj"]}
    if kind == "shadow":
        leea.leea_evaluate_shadow_u8(pop, dims, state["pop"], case["precision"], state["shadow"], state["scale"],
                                     state["x"], 255.0, state["y"], case["batch"], 0.5, state["f_inh"],
                                     state["f_raw"], state["f_adj"], state["correct"], state["scratch"])
        return {"f_raw": state["f_raw"], "f_adj": state["f_adj"], "correct": state["correct"]}
    leea.leea_descriptors(pop, dims, state["prm"], state["seed"], 1, state["parents"], state["f"], state["par1"],
                          state["par2"], state["kind"], state["f_inh"], state["entity"], state["desc"].shape[0],
                          state["probe"], N_PROBE, state["desc"])
    return state["desc"]


# ---- what a pass cannot do without ---------------------------------------------------
def _generation_work(pop, dims, batch, precision):
    """One read and one write of every child's genes, the shadow written and read, the evaluation's products."""
    c, w1 = _genes(dims), dims[0] * dims[1]
    shadow = (0, 2, 1)[precision] * w1
    # The evaluation reads the genes again (FP32), or the shadow and the genes past W1.
    read = 4 * c if precision == 0 else shadow + 4 * (c - w1)
    return pop * (8 * c + shadow + read), pop * batch * _flops(dims)


def work(case):
    kind = case["kind"]
    if kind == "generation":
        b, f = _generation_work(case["pop"], _net_of(case), case["batch"], case["precision"])
        return {"bytes": case["gens"] * b, "flops": case["gens"] * f}
    if kind == "batching":
        got = [_generation_work(p, [784, h, 10], n, case["precision"]) for p, h, n in _run_specs(case)]
        return {"bytes": case["gens"] * sum(b for b, _ in got), "flops": case["gens"] * sum(f for _, f in got)}
    dims, pop = _net_of(case), case["pop"]
    c = _genes(dims)
    if kind == "breed":
        return {"bytes": 8 * c * pop, "flops": 0}
    if kind == "evaluate":
        size = 1 if case["inputs"] == "u8" else 4
        return {"bytes": 4 * c * pop + size * case["batch"] * dims[0] + 12 * pop, "flops": pop * case["batch"] * _flops(dims)}
    if kind == "shadow":
        w1 = dims[0] * dims[1]
        per = (2 if case["precision"] == 1 else 1) * w1 + 4 * (c - w1)
        return {"bytes": per * pop + case["batch"] * dims[0] + 16 * pop, "flops": pop * case["batch"] * _flops(dims)}
    _, nc, nm = _counts(pop, 0.5)
    n = case["mult"] * (nc + nm)
    return {"bytes": 4 * c * pop + 4 * n * (5 + N_PROBE * dims[-1]), "flops": n * N_PROBE * _flops(dims)}


# ---- the same in 64 bits ---------------------------------------------------------------
def _philox(blk, ent, gen, tag, seed):
    """Philox4x32-10 (Salmon et al., SC'11) on int64 tensors holding 32-bit words: four words per counter."""
    lo = 0xFFFFFFFF
    shape = torch.broadcast_shapes(blk.shape, ent.shape)
    c = [blk.expand(shape), ent.expand(shape), torch.full(shape, gen, device=DEVICE), torch.full(shape, tag, device=DEVICE)]
    k0, k1 = seed & lo, (seed >> 32) & lo
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & lo) ^ c[1] ^ k0, p1 & lo, ((p0 >> 32) & lo) ^ c[3] ^ k1, p0 & lo]
        k0, k1 = (k0 + 0x9E3779B9) & lo, (k1 + 0xBB67AE85) & lo
    return c


def _mask(n, ent, tag, seed, q):
    """bool[len(ent)][n]: 16-bit draws below floor(q 2^16)."""
    if q >= 1.0:
        return torch.ones((len(ent), n), dtype=torch.bool, device=DEVICE)
    blk = torch.arange(-(-n // 8), device=DEVICE)[None, :]
    w = _philox(blk, ent[:, None], 1, tag, seed)
    halves = torch.stack([v for x in w for v in (x & 0xFFFF, x >> 16)], dim=-1)
    return halves.reshape(len(ent), -1)[:, :n] < int(math.floor(q * 65536.0))


def _normals(n, ent, seed):
    """float64[len(ent)][n] Box-Muller normals of the NORMAL stream."""
    blk = torch.arange(-(-n // 4), device=DEVICE)[None, :]
    w = [(2 * (x >> 9) + 1).double() * 2.0 ** -24 for x in _philox(blk, ent[:, None], 1, 5, seed)]
    out = []
    for a, b in ((w[0], w[1]), (w[2], w[3])):
        r = torch.sqrt(-2.0 * torch.log(a))
        out += [r * torch.cos(2.0 * math.pi * b), r * torch.sin(2.0 * math.pi * b)]
    return torch.stack(out, dim=-1).reshape(len(ent), -1)[:, :n]


def _child_genes(parents, par1, par2, kind, ent, c, prm, seed):
    """float64[n][c] children of a chunk, and per child the crossover hits and sum z^2 over mutated genes."""
    v = parents[par1.long(), :c].double()
    hits = torch.zeros(len(ent), dtype=torch.float64, device=DEVICE)
    z2 = torch.zeros_like(hits)
    xo, mu = (kind == 1).nonzero()[:, 0], (kind == 2).nonzero()[:, 0]
    if len(xo):
        b = parents[par2[xo].long(), :c].double()
        if prm.xo_op == 0:
            m = _mask(c, ent[xo], 3, seed, prm.xo_gene_p)
            v[xo] = torch.where(m, b, v[xo])
            hits[xo] = m.double().mean(dim=1)
        else:
            v[xo] = (v[xo] + b) / 2
            hits[xo] = 0.5
    if len(mu):
        z = _normals(c, ent[mu], seed) * _mask(c, ent[mu], 4, seed, prm.mut_rate)
        v[mu] += float(np.float32(prm.sigma)) * z
        z2[mu] = (z * z).sum(dim=1)
    return v, hits, z2


def _logits(w, dims, x, w1=None):
    """float64[n][batch][d_out] of nets w[n][c] on x[batch][d_0]; w1 in place of the first layer's weights."""
    a, off = x.double()[None].expand(w.shape[0], -1, -1), 0
    for i in range(len(dims) - 1):
        n = dims[i + 1] * dims[i]
        m = (w1 if i == 0 and w1 is not None else w[:, off:off + n].double()).reshape(-1, dims[i + 1], dims[i])
        a = torch.bmm(a, m.transpose(1, 2)) + w[:, off + n:off + n + dims[i + 1]].double()[:, None, :]
        off += n + dims[i + 1]
        if i + 2 < len(dims):
            a = a.relu_()
    return a


def exact(case, seed):
    kind = case["kind"]
    if kind in ("generation", "batching"):
        return None  # every generation follows from the ranking of the one before
    s = prepare(case, seed)
    dims, pop = _net_of(case), case["pop"]
    c = _genes(dims)
    if kind == "breed":
        out = torch.zeros(s["children"].shape, dtype=torch.float64, device=DEVICE)
        for i in range(0, pop, 64):
            j = slice(i, min(pop, i + 64))
            ent = torch.arange(pop, device=DEVICE)[j]
            out[j, :c] = _child_genes(s["parents"], s["par1"][j], s["par2"][j], s["kind"][j], ent, c, s["prm"],
                                      s["seed"])[0]
        return out
    if kind == "descriptors":
        n, prm = s["desc"].shape[0], s["prm"]
        out = torch.empty(s["desc"].shape, dtype=torch.float64, device=DEVICE)
        for i in range(0, n, 64):
            j = slice(i, min(n, i + 64))
            v, hits, z2 = _child_genes(s["parents"], s["par1"][j], s["par2"][j], s["kind"][j], s["entity"][j].long(), c,
                                       prm, s["seed"])
            out[j, 0], out[j, 1] = s["f"][s["par1"][j].long()].double(), s["f"][s["par2"][j].long()].double()
            out[j, 2], out[j, 3] = s["f_inh"][j].double(), hits
            out[j, 4] = float(np.float32(prm.sigma)) * z2.sqrt()
            # The child is an FP32 net whose first-layer weights are held in BF16.
            v = v.float()
            w1 = v[:, :dims[0] * dims[1]].bfloat16().double()
            out[j, 5:] = _logits(v, dims, s["probe"], w1).reshape(v.shape[0], -1)
        return out
    x = s["x"].double() / 255.0 if s["x"].dtype == torch.uint8 else s["x"].double()
    f = torch.empty(pop, dtype=torch.float64, device=DEVICE)
    step = max(1, min(pop, 200_000_000 // (case["batch"] * 784 * 8)))
    n1 = dims[0] * dims[1]
    for i in range(0, pop, step):
        w, w1 = s["pop"][i:i + step, :c], None
        if kind == "shadow" and case["precision"] == 1:
            w1 = w[:, :n1].bfloat16().double()
        elif kind == "shadow":
            e = torch.ldexp(torch.ones(1, dtype=torch.float64, device=DEVICE), s["scale"][i:i + step])[:, None]
            w1 = (w[:, :n1].double() / e).clamp(-448.0, 448.0).float().to(torch.float8_e4m3fn).double() * e
        z = _logits(w, dims, x, w1)
        f[i:i + step] = -(torch.logsumexp(z, dim=2) - z.gather(2, s["y"].long()[None, :, None].expand(
            z.shape[0], -1, -1))[:, :, 0]).mean(dim=1)
    got = {"f_raw": f, "f_adj": 0.5 * s["f_inh"].double() + 0.5 * f}
    if kind == "shadow":
        got["correct"] = None
    return got
