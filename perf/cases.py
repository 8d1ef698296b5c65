"""The work a user of the library has it do, as cases that can be timed and compared.

A case is one call (or the two calls of one step) through the package's public entry points: CSR build, GCN /
GraphSAGE / GAT aggregation, edge softmax, whole layers, the dense transform and the one-shot path.  Graphs,
widths, heads and dtypes are those of the repository's own configurations (``graphgen``), the vertex and edge
counts of the paper's three data sets among them, and odd sizes between.  Inputs are made on the GPU from the seed
alone, by the recipes ``graphgen`` uses on the host (power-law in-degrees with sources drawn by degree, or RMAT;
shuffled edge order, relabelled vertices).

A case's fields: ``kind`` what is called, ``graph`` ("power" or "rmat"), ``n`` vertices, ``e`` input edges, ``flags``
the build options as letters (l = add self-loops, s = symmetrise, d = remove duplicates), ``ids`` edge id type,
``model``, ``f`` columns aggregated (``heads`` * ``dim`` for GAT), ``ld`` row pitch of the features in elements,
``cw`` chunk width, ``dtype`` of the features, ``f_in`` / ``mode`` of the dense transform.
"""
import math

import torch

import paper_2104_03058_b200 as g

FLAG = {"l": 1, "d": 2, "s": 4}        # GNNFD_CSR_ADD_SELF_LOOPS, _DEDUP, _SYMMETRIZE
FIELDS = {"kind": "aggregate", "graph": "power", "n": 0, "e": 0, "flags": "", "ids": "i32", "model": "gcn", "f": 0, "ld": 0,
          "cw": 0, "heads": 0, "dim": 0, "dtype": "f32", "f_in": 0, "mode": "fp32"}
MOST_EDGES, MOST_WORK = 115_000_000, 115_000_000 * 602      # of the largest listed case: input edges, edges x columns


def _case(name=None, **fields):
    c = dict(FIELDS, **fields)
    if c["model"] == "gat" and not c["f"]:
        c["f"] = c["heads"] * c["dim"]
    c["cw"] = c["cw"] or c["f"]
    c["ld"] = c["ld"] or c["f_in"] or c["f"]
    return dict(c, name=name) if name else c


def listed():
    return [
        # one hidden-layer aggregation on a few thousand vertices: what counts is the latency of the call
        _case("gcn_4k_f16", n=4096, e=40_000, flags="l", f=16),
        # a citation-sized graph (19,717 vertices, 88,676 edges, 64-bit ids) that arrives per request: build and aggregate
        _case("step_20k_f32_i64", kind="step", n=19_717, e=88_676, flags="l", ids="i64", f=32),
        # GraphSAGE mean on a sparse graph of ordinary size, input features of 128 columns in two layers of 64
        _case("sage_100k_f128", n=100_000, e=2_000_000, model="sage", f=128, cw=64),
        # multi-head attention on a sparse graph: 8 heads of 8 columns, scores and fused softmax aggregation
        _case("gat_200k_8x8", n=200_000, e=3_000_000, flags="l", model="gat", heads=8, dim=8),
        # output layer of an odd number of classes: rows of 41 floats, as a linear layer leaves them (no padding)
        _case("gcn_133k_f41", n=132_534, e=39_561_252, flags="l", f=41),
        # attention coefficients written out (for inspection or a custom message step), 8 heads
        _case("softmax_233k_h8", kind="softmax", n=232_965, e=114_615_892, flags="l", model="gat", heads=8, dim=8),
        # the benchmark's step: build of the large dense-ish graph and input-layer aggregation of 602 columns, rows padded to 608
        _case("step_233k_f602", kind="step", n=232_965, e=114_615_892, flags="l", f=602, ld=608, cw=64),
        # a whole layer 602 -> 64 on the same graph, the transform ahead of the aggregation, fp32-faithful
        _case("layer_gcn_233k", kind="layer", n=232_965, e=114_615_892, flags="l", f_in=602, ld=608, f=64),
        # a whole attention layer in bf16: 128 -> 8 heads of 16
        _case("layer_gat_133k_bf16", kind="layer", n=132_534, e=39_561_252, flags="l", model="gat", heads=8, dim=16, dtype="bf16",
              f_in=128),
        # set-up of a large skewed graph given as an undirected edge list with repeats
        _case("build_rmat21", kind="build", graph="rmat", n=1 << 21, e=60_000_000, flags="lsd"),
        # hidden layer of 64 bf16 columns on that graph
        _case("gcn_rmat21_f64_bf16", graph="rmat", n=1 << 21, e=60_000_000, flags="lsd", f=64, dtype="bf16"),
        # a graph used once: edge list in, aggregated hidden layer out
        _case("oneshot_sage_133k", kind="oneshot", n=132_534, e=39_561_252, model="sage", f=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["aggregate", "aggregate", "aggregate", "step", "layer", "softmax", "build", "oneshot", "combine"])
    graph = rng.choice(["power", "power", "power", "rmat"])
    n = 1 << rng.randint(12, 21) if graph == "rmat" else _log(rng, 4_000, 240_000)
    e = min(MOST_EDGES // 2 if graph == "rmat" else MOST_EDGES, int(n * math.exp(rng.uniform(math.log(4), math.log(500)))), n * (n // 50))
    flags = "lsd" if graph == "rmat" else rng.choice(["l", "l", "", "ls"])
    if "s" in flags:
        e = min(e, MOST_EDGES // 2)
    model = rng.choice(["gcn", "sage", "gat"])
    dtype = rng.choice(["f32", "f32", "bf16"])
    align = 4 if dtype == "f32" else 8
    c = {"kind": kind, "graph": graph, "n": n, "e": e, "flags": flags, "ids": rng.choice(["i32", "i32", "i64"]), "model": model,
         "dtype": dtype}
    if kind == "oneshot" and "d" in flags:
        c["flags"] = "ls"
    if kind == "softmax":
        return _case(**dict(c, model="gat", heads=rng.choice([1, 2, 3, 4, 6, 8]), dim=8, dtype="f32"))
    if kind == "build":
        return _case(**c)
    if model == "gat":
        heads, dim = rng.choice([1, 2, 4, 6, 8]), rng.choice([4, 7, 8, 16, 32])
        f = heads * dim
        c.update(heads=heads, dim=dim)
        cw = rng.choice([f, f, dim])
    else:
        f = rng.choice([8, 16, 32, 64, _log(rng, 8, 128)]) if kind in ("layer", "combine") else \
            rng.choice([8, 16, 32, 64, 128, 256, _log(rng, 8, 602), _log(rng, 8, 602)])
        cw = rng.choice([f, f, min(f, 64), min(f, 32)])
    c["e"] = min(c["e"], int(MOST_WORK / 4 / f))
    if kind in ("layer", "combine"):
        f_in = _log(rng, 16, 602)
        c.update(f_in=f_in, ld=-(-f_in // align) * align, mode=rng.choice(["fp32", "fp32", "tf32"]))
        if kind == "combine":
            c.update(model="gcn", graph="power", heads=0, dim=0, e=0, flags="", ids="i32")
    else:
        c["ld"] = f if rng.random() < 0.6 else -(-f // align) * align
    return _case(**dict(c, f=f, cw=cw))


# ---------------------------------------------------------------- inputs

def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed(seed * 64 + stream)


def _power_graph(n, e, seed, ids):
    """Directed power-law graph of exactly e distinct edges without loops: in-degrees x0 * U^(-1/1.1) between 1 and 20,000,
    sources drawn in proportion to degree, ids relabelled, edge order shuffled."""
    rnd = _gen(seed, 1)
    u = torch.rand(n, generator=rnd, device="cuda", dtype=torch.float64).clamp_min(1e-12).pow_(-1 / 1.1)
    top = float(min(20_000, n - 1))
    budget, keys = e * 1.05, None
    while keys is None or keys.numel() < e:         # repeats and loops fall away: draw again with more
        lo, hi = 1e-3, top
        for _ in range(50):
            x0 = (lo + hi) / 2
            lo, hi = (x0, hi) if float((u * x0).clamp_(1, top).sum()) < budget else (lo, x0)
        deg = (u * hi).clamp_(1, top).to(torch.int64)
        dst = torch.repeat_interleave(torch.arange(n, device="cuda"), deg)
        src = dst[torch.randint(dst.numel(), (dst.numel(),), generator=rnd, device="cuda")]
        keys = torch.unique((dst * n + src)[dst != src])
        budget *= 1.15
    keys = keys[torch.randperm(keys.numel(), generator=rnd, device="cuda")[:e]]
    label = torch.randperm(n, generator=rnd, device="cuda").to(ids)
    return label[keys % n], label[keys // n]


def _rmat_graph(n, e, seed, ids):
    """RMAT with (0.57, 0.19, 0.19, 0.05), one quadrant draw per level, ids relabelled, as an undirected edge list of e
    entries: 9 of 10 are distinct pairs without loops (as many as 60 million draws on 2^21 vertices give, give or take),
    the rest repeats of them, each in either direction."""
    rnd = _gen(seed, 1)
    distinct, pairs = _distinct(e), torch.empty(0, dtype=torch.int64, device="cuda")
    while pairs.numel() < distinct:
        src = torch.zeros(e, dtype=torch.int64, device="cuda")
        dst = torch.zeros(e, dtype=torch.int64, device="cuda")
        for _ in range(n.bit_length() - 1):
            u = torch.rand(e, generator=rnd, device="cuda")
            src = src * 2 + (u >= 0.76)
            dst = dst * 2 + (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
        keys = torch.minimum(src, dst) * n + torch.maximum(src, dst)
        pairs = torch.unique(torch.cat([pairs, keys[src != dst]]))
    pairs = pairs[torch.randperm(pairs.numel(), generator=rnd, device="cuda")[:distinct]]
    keys = torch.cat([pairs, pairs[torch.randint(distinct, (e - distinct,), generator=rnd, device="cuda")]])
    keys = keys[torch.randperm(e, generator=rnd, device="cuda")]
    label = torch.randperm(n, generator=rnd, device="cuda").to(ids)
    a, b = label[keys // n], label[keys % n]
    turn = torch.rand(e, generator=rnd, device="cuda") < 0.5
    return torch.where(turn, a, b), torch.where(turn, b, a)


def _distinct(e):
    return e * 9 // 10


def _matrix(rows, cols, ld, dtype, seed, stream, scale=1.0):
    """Normal values in the first `cols` of `ld` columns; the padding is left as zeros."""
    t = torch.zeros((rows, ld), dtype=torch.float32, device="cuda")
    t[:, :cols] = torch.randn((rows, cols), generator=_gen(seed, stream), device="cuda") * scale
    return t.to(torch.bfloat16) if dtype == "bf16" else t


def prepare(case, seed):
    c, s = case, dict(case)
    flags = s["bits"] = sum(FLAG[x] for x in c["flags"])
    if c["kind"] != "combine":
        make = _rmat_graph if c["graph"] == "rmat" else _power_graph
        src, dst = make(c["n"], c["e"], seed, torch.int64 if c["ids"] == "i64" else torch.int32)
        if c["kind"] in ("build", "step", "oneshot"):
            s["src"], s["dst"] = src, dst
        else:
            s["csr"] = g.build_csr(c["n"], src, dst, flags)      # a program keeps the handle of a graph it goes on using
    if c["kind"] == "softmax":
        s["s_src"], s["s_dst"] = (_matrix(c["n"], c["heads"], c["heads"], "f32", seed, k) for k in (2, 3))
    elif c["kind"] != "build":
        s["x"] = _matrix(c["n"], c["f_in"] or c["f"], c["ld"], c["dtype"], seed, 2)
    if c["f_in"]:
        s["w_t"] = _matrix(c["f"], c["f_in"], c["ld"], c["dtype"], seed, 4, c["f_in"] ** -0.5)
    if c["model"] == "gat":
        s["a_src"], s["a_dst"] = (_matrix(c["heads"], c["dim"], c["dim"], "f32", seed, k, 0.1) for k in (5, 6))
    return s


# ---------------------------------------------------------------- one pass

def _aggregate(s, csr):
    if s["model"] == "gat":
        return g.aggregate_gat(csr, s["x"], s["a_src"], s["a_dst"], s["heads"], s["dim"], 0.2, chunk_width=s["cw"])
    return (g.aggregate_gcn if s["model"] == "gcn" else g.aggregate_sage)(csr, s["x"], f=s["f"], chunk_width=s["cw"])


def run(state):
    s, kind = state, state["kind"]
    if kind == "aggregate":
        return _aggregate(s, s["csr"])
    if kind == "softmax":
        return g.edge_softmax(s["csr"], s["s_src"], s["s_dst"], 0.2)
    if kind == "layer":
        gat = dict(a_src=s["a_src"], a_dst=s["a_dst"], heads=s["heads"], dim=s["dim"]) if s["model"] == "gat" else {}
        return g.layer(s["csr"], s["model"], s["x"], s["w_t"], f_in=s["f_in"], mode=s["mode"], chunk_width=s["cw"], **gat)
    if kind == "combine":
        return g.combine(s["x"], s["w_t"], f_in=s["f_in"], mode=s["mode"])
    if kind == "oneshot":
        if s["model"] == "gat":
            return g.oneshot_gat(s["n"], s["src"], s["dst"], s["x"], s["a_src"], s["a_dst"], s["heads"], s["dim"], 0.2, flags=s["bits"],
                                 chunk_width=s["cw"])
        return g.oneshot(s["model"], s["n"], s["src"], s["dst"], s["x"], flags=s["bits"], f=s["f"], chunk_width=s["cw"])
    csr = g.build_csr(s["n"], s["src"], s["dst"], s["bits"])
    if kind == "step":
        return _aggregate(s, csr)
    return {"row_ptr": csr.row_ptr, "col_idx": csr.col_idx, "perm": csr.perm, "edge_weight": csr.edge_weight,
            "dinv_sqrt": csr.dinv_sqrt, "rdeg": csr.rdeg, "row_order": csr.row_order}


# ---------------------------------------------------------------- the same results in 64 bits

def _csr64(c, seed):
    """(row pointers, sources, destinations) of the entries in (destination, source) order, as torch makes them."""
    make = _rmat_graph if c["graph"] == "rmat" else _power_graph
    src, dst = make(c["n"], c["e"], seed, torch.int64)
    if "s" in c["flags"]:
        loop = src == dst
        src, dst = torch.cat([src, dst[~loop]]), torch.cat([dst, src[~loop]])
    if "l" in c["flags"]:
        keep, own = src != dst, torch.arange(c["n"], device="cuda")
        src, dst = torch.cat([src[keep], own]), torch.cat([dst[keep], own])
    keys = dst * c["n"] + src
    keys = torch.unique(keys) if "d" in c["flags"] else keys.sort().values
    dst = keys // c["n"]
    row_ptr = torch.searchsorted(dst, torch.arange(c["n"] + 1, device="cuda"))
    return row_ptr, keys % c["n"], dst


def _attention64(c, col, row, s_src, s_dst):
    """Edge softmax of LeakyReLU(s_src[source] + s_dst[destination]), slope 0.2, one head after the other."""
    alpha = torch.empty((col.numel(), s_src.shape[1]), dtype=torch.float64, device="cuda")
    for h in range(s_src.shape[1]):
        logit = torch.nn.functional.leaky_relu(s_src[col, h] + s_dst[row, h], 0.2)
        top = torch.full((c["n"],), -math.inf, dtype=torch.float64, device="cuda").scatter_reduce_(0, row, logit, "amax")
        value = (logit - top[row]).exp_()
        alpha[:, h] = value / torch.zeros(c["n"], dtype=torch.float64, device="cuda").index_add_(0, row, value)[row]
    return alpha


def _sum64(row_ptr, col, weight, x):
    """Rows' weighted sums of x, 64 columns at a time."""
    a = torch.sparse_csr_tensor(row_ptr, col, weight, size=(row_ptr.numel() - 1, x.shape[0]))
    return torch.cat([a @ part.contiguous() for part in x.split(64, dim=1)], dim=1)


def exact(case, seed):
    c = case
    if c["kind"] not in ("softmax", "build"):
        x = _matrix(c["n"], c["f_in"] or c["f"], c["ld"], c["dtype"], seed, 2)[:, :c["f_in"] or c["f"]].double()
    if c["f_in"]:
        w_t = _matrix(c["f"], c["f_in"], c["ld"], c["dtype"], seed, 4, c["f_in"] ** -0.5)[:, :c["f_in"]].double()
        z = x @ w_t.T
        if c["kind"] == "combine":
            return z
        x = z.to(torch.bfloat16).double() if c["dtype"] == "bf16" else z      # a layer keeps z in the features' type
    row_ptr, col, row = _csr64(c, seed)
    deg = (row_ptr[1:] - row_ptr[:-1]).double()
    dinv, rdeg = (torch.where(deg > 0, deg.clamp_min(1) ** p, 0.0) for p in (-0.5, -1.0))
    if c["kind"] == "build":
        return {"row_ptr": None, "col_idx": None, "perm": None, "edge_weight": dinv[col] * dinv[row], "dinv_sqrt": dinv,
                "rdeg": rdeg, "row_order": None}
    if c["kind"] == "softmax":
        return _attention64(c, col, row, *(_matrix(c["n"], c["heads"], c["heads"], "f32", seed, k).double() for k in (2, 3)))
    if c["model"] == "gat":
        a_src, a_dst = (_matrix(c["heads"], c["dim"], c["dim"], "f32", seed, k, 0.1).double() for k in (5, 6))
        heads = x.reshape(c["n"], c["heads"], c["dim"])
        alpha = _attention64(c, col, row, (heads * a_src).sum(2), (heads * a_dst).sum(2))
        return torch.cat([_sum64(row_ptr, col, alpha[:, h].contiguous(), heads[:, h]) for h in range(c["heads"])], dim=1)
    return _sum64(row_ptr, col, dinv[col] * dinv[row] if c["model"] == "gcn" else rdeg[row], x)


# ---------------------------------------------------------------- floors and tolerances

def work(case):
    c = case
    n, f, elem = c["n"], c["f"], 2 if c["dtype"] == "bf16" else 4
    kept = _distinct(c["e"]) if "d" in c["flags"] else c["e"]
    nnz = kept * (2 if "s" in c["flags"] else 1) + (n if "l" in c["flags"] else 0)
    edges = c["e"] * 2 * (8 if c["ids"] == "i64" else 4)                                       # the edge list as given
    csr = 4 * (n + 1) + 4 * nnz                                                                # row pointers and columns
    if c["kind"] == "build":
        return {"bytes": edges + csr + 8 * nnz + 12 * n, "flops": 0}                           # perm, weights, normalisers, row order
    if c["kind"] == "softmax":
        return {"bytes": csr + 8 * n * c["heads"] + 4 * nnz * c["heads"], "flops": 8 * nnz * c["heads"]}
    if c["kind"] == "combine":
        return {"bytes": n * c["f_in"] * elem + f * c["f_in"] * elem + 4 * n * f, "flops": 2 * n * f * c["f_in"]}
    graph = edges if c["kind"] in ("step", "oneshot") else csr
    flops = nnz * (2 * f + (8 * c["heads"] if c["model"] == "gat" else 0)) + (2 * n * f * c["f_in"] if c["f_in"] else 0)
    return {"bytes": graph + n * (c["f_in"] or f) * elem + 4 * n * f + f * c["f_in"] * elem, "flops": flops}


def tolerance(case):
    # About four times what each path differs by from its evaluation in 64 bits (rel / max): sums and GAT 1.5e-7 / 2e-6,
    # fp32-faithful transform 1.7e-6 / 5e-6, bf16 layers (the transformed features are rounded to bf16, and a sum that
    # falls on the other side moves a value by 2^-8) 2e-5 / 3e-3; tf32 operands keep 10 mantissa bits, cut or rounded;
    # softmax values carry the rounding of logits of up to about 10 and of the exponential.
    if case["kind"] == "softmax":
        return {"rel": 2e-6, "max": 2e-5}
    if case["kind"] in ("layer", "combine"):
        if case["dtype"] == "f32":
            return {"rel": 2e-3, "max": 2e-2} if case["mode"] == "tf32" else {"rel": 1e-5, "max": 5e-5}
        if case["kind"] == "layer":
            return {"rel": 1e-4, "max": 1.5e-2}
    return {"rel": 1e-6, "max": 1e-5, "differ": 0.0}
