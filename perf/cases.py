"""Performance cases: what a user of the Stop-and-Stare library has it do.

A case names one kind of call ("op") and its sizes:

  solve     one SSA / D-SSA query on a kept solver (graph resident, workspaces kept)
  pool      the hot-path steps one by one: create a pool, grow it, count, pick seeds, check them
  estimate  Estimate-Inf of a seed set that the caller already has
  load      host edge arrays to an answer: upload, CSR build, one-shot solve
  serve     a burst of mixed queries through the serving loop, all answers awaited
  cover     the allocation-free coverage count over a device-held pool

Graphs are directed R-MAT graphs (a, b, c, d = 0.57, 0.19, 0.19, 0.05), the
stand-in for social networks that the tests and the benchmark use: generated on
the device for 2^scale nodes, or drawn here and loaded as an edge list where
the node count is odd or the weights are explicit.  Everything is made from the
seed: the graph, the weights, the benefits and the queries' Philox seeds.
"""
import math

import numpy as np
import torch

import paper_1605_07990_gb300 as P

WEIGHTS = {"wc": P.SSA_W_WC, "tri": P.SSA_W_TRIVALENCY, "explicit": P.SSA_W_EXPLICIT}
MODELS = {"ic": P.SSA_IC, "lt": P.SSA_LT}
ALGOS = {"ssa": P.SSA_ALGO_SSA, "dssa": P.SSA_ALGO_DSSA}
RMAT = (0.57, 0.19, 0.19)


def _solve(name, algo, model, weights, n, m, k, eps, targeted=False, captured=False):
    return {"name": name, "op": "solve", "algo": algo, "model": model, "weights": weights, "n": n, "m": m, "k": k,
            "eps": eps, "targeted": targeted, "captured": captured}


def listed():
    return [
        # a small network (NetHEPT's scale): plain SSA, the whole call is a few milliseconds
        _solve("solve_ssa_ic_wc_2e14", "ssa", "ic", "wc", 1 << 14, 1 << 17, 50, 0.1),
        # the smallest query: LT, ten seeds, rounds as captured CUDA graphs (the server's setting)
        _solve("solve_dssa_lt_wc_2e14", "dssa", "lt", "wc", 1 << 14, 1 << 17, 10, 0.2, captured=True),
        # a targeted (benefit-weighted) query on a mid-size network, as the serving mix asks it
        _solve("solve_dssa_targeted_2e20", "dssa", "ic", "wc", 1 << 20, 1 << 24, 100, 0.1, targeted=True),
        # trivalency weights: few huge RR sets, per-edge coins
        _solve("solve_dssa_ic_tri_2e20", "dssa", "ic", "tri", 1 << 20, 1 << 24, 100, 0.1),
        # a large network under LT with many seeds and a tight bound
        _solve("solve_dssa_lt_wc_2e23", "dssa", "lt", "wc", 1 << 23, 1 << 27, 500, 0.05),
        # the same network, the serving mix's largest seed count, captured rounds
        _solve("solve_dssa_ic_wc_2e23", "dssa", "ic", "wc", 1 << 23, 1 << 27, 1000, 0.1, captured=True),
        # the billion-edge network of the benchmark
        _solve("solve_ssa_ic_wc_2e25", "ssa", "ic", "wc", 1 << 25, 1_300_000_000, 100, 0.1),
        # the steps one by one on a loaded graph of odd size with learned (explicit) probabilities
        {"name": "pool_ic_explicit_odd", "op": "pool", "model": "ic", "weights": "explicit", "n": 300_007,
         "m": 3_000_001, "sets": 100_003, "k": 77, "targeted": False},
        # checking a seed set found elsewhere on the mid-size network
        {"name": "estimate_ic_wc_2e20", "op": "estimate", "model": "ic", "weights": "wc", "n": 1 << 20, "m": 1 << 24,
         "k": 100, "hits": 20_000, "targeted": False},
        # an edge list from a file: load it and ask once, LT with general in-weights
        {"name": "load_lt_explicit_odd", "op": "load", "algo": "dssa", "model": "lt", "weights": "explicit",
         "n": 1_000_003, "m": 10_000_019, "k": 20, "eps": 0.1},
        # a burst of 24 mixed queries over two resident graphs, with the server's default slots
        {"name": "serve_mix_24", "op": "serve", "n": 1 << 20, "m": 1 << 24, "n2": 1 << 21, "m2": 1 << 25,
         "queries": 24, "slots": 4},
        # the stare count over a pool that the caller holds
        {"name": "cover_20m", "op": "cover", "n": 1 << 20, "entries": 20_000_003, "sets": 1_000_003, "k": 100},
    ]


def _log(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _graph(rng, weights, most):
    """n and m of up to `most` drawn edges: a power of two generated on the device, or an odd size that is loaded."""
    m = _log(rng, 1 << 15, most)
    n = max(2048, int(m / math.exp(rng.uniform(math.log(4), math.log(24)))))
    if weights != "explicit":
        n = 1 << max(11, min(23, int(round(math.log2(n)))))
    return n, m


def draw(rng):
    op = rng.choice(["solve", "solve", "solve", "pool", "estimate", "load", "cover"])
    weights = rng.choice(["wc", "wc", "wc", "tri", "explicit"])
    # per-edge coins and host edge lists keep to smaller graphs, as their cost grows with the edges
    n, m = _graph(rng, weights, {"wc": 1 << 27, "tri": 1 << 21, "explicit": 1 << 21}[weights])
    model = "ic" if weights == "tri" else rng.choice(["ic", "lt"])
    k = min(_log(rng, 1, 1000), n)
    if op == "solve":
        # plain SSA draws several times the sets of D-SSA: with per-edge coins it is asked loosely
        algo = rng.choice(["ssa", "dssa"])
        tight = weights == "wc" and algo == "dssa"
        eps = rng.choice([0.05, 0.1, 0.2]) if tight else rng.choice([0.1, 0.2]) if weights == "wc" else 0.2
        return {"op": "solve", "algo": algo, "model": model, "weights": weights, "n": n, "m": m, "k": k, "eps": eps,
                "targeted": rng.random() < 0.3, "captured": rng.random() < 0.4}
    if op == "pool":
        return {"op": "pool", "model": model, "weights": weights, "n": n, "m": m,
                "sets": _log(rng, 2000, 500_000 if weights == "wc" else 20_000), "k": k, "targeted": rng.random() < 0.3}
    if op == "estimate":
        return {"op": "estimate", "model": model, "weights": weights, "n": n, "m": m, "k": k,
                "hits": _log(rng, 500, 50_000 if weights == "wc" else 5000), "targeted": rng.random() < 0.3}
    if op == "load":
        m = _log(rng, 1 << 15, 1 << 22)
        n = max(2048, int(m / math.exp(rng.uniform(math.log(4), math.log(24)))))
        weights = rng.choice(["wc", "explicit"])
        return {"op": "load", "algo": "dssa", "model": rng.choice(["ic", "lt"]), "weights": weights, "n": n, "m": m,
                "k": min(k, n), "eps": rng.choice([0.1, 0.2])}
    entries = _log(rng, 1 << 12, 20_000_000)
    return {"op": "cover", "n": _log(rng, 1000, 10_000_000), "entries": entries,
            "sets": max(1, int(entries / rng.uniform(1.5, 60))), "k": k}


# ---- inputs ----

def _edges(n, m, gen):
    """An R-MAT edge list over n nodes (any n): draws outside [0, n) and self-loops are dropped."""
    src = torch.zeros(m, dtype=torch.int32, device="cuda")
    dst = torch.zeros(m, dtype=torch.int32, device="cuda")
    a, b, c = RMAT
    for _ in range(max(1, math.ceil(math.log2(n)))):
        u = torch.rand(m, device="cuda", generator=gen)
        src = src * 2 + (u >= a + b)
        dst = dst * 2 + ((u >= a) & (u < a + b) | (u >= a + b + c))
    keep = (src < n) & (dst < n) & (src != dst)
    return src[keep].int(), dst[keep].int()


def _in_weights(n, dst, gen):
    """General in-weights as 32-bit thresholds: each node's sum lies between 0.6 and 1."""
    w = torch.randint(1 << 20, 10 << 20, (dst.numel(),), device="cuda", generator=gen, dtype=torch.int64)
    total = torch.zeros(n, device="cuda", dtype=torch.int64).index_add_(0, dst.long(), w).clamp_min(1)
    share = torch.rand(n, device="cuda", generator=gen, dtype=torch.float64) * 0.4 + 0.6
    t = (w * (share / total)[dst.long()] * 2.0 ** 32).floor().clamp_max(2.0 ** 32 - 1)
    return t.to(torch.int64)


def _host_edges(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    src, dst = _edges(case["n"], case["m"], gen)
    thr = _in_weights(case["n"], dst, gen).cpu().numpy().astype(np.uint32) if case["weights"] == "explicit" else None
    return src.cpu().numpy(), dst.cpu().numpy(), thr


def _make_graph(case, seed):
    n, m = case["n"], case["m"]
    if case["weights"] != "explicit" and n & (n - 1) == 0:
        return P.ssa_gen_rmat(n.bit_length() - 1, m, *RMAT, seed=seed, weighting=WEIGHTS[case["weights"]],
                              weight_seed=seed + 1)
    src, dst, thr = _host_edges(case, seed)
    return P.ssa_load_graph(n, src, dst, thr, WEIGHTS[case["weights"]], seed + 1)


def _benefit(n, seed):
    """Zipf (s = 1.2) benefits max(1, floor(2^20 / rank^1.2)) over a random ranking."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rank = torch.randperm(n, device="cuda", generator=gen).double() + 1
    return (2.0 ** 20 / rank.pow(1.2)).floor().clamp_min(1).to(torch.int64).cpu().numpy().astype(np.uint32)


def prepare(case, seed):
    op = case["op"]
    s = {"op": op, "case": case, "seed": seed + 1}
    if op == "cover":
        # a flat pool as the library's own look: entries of a set together, low node ids the hubs
        gen = torch.Generator(device="cuda").manual_seed(seed)
        u = torch.rand(case["entries"], device="cuda", generator=gen)
        s["nodes"] = (u.pow(4) * case["n"]).int().clamp_max(case["n"] - 1)
        s["samp"] = torch.sort(torch.randint(case["sets"], (case["entries"],), device="cuda", generator=gen,
                                             dtype=torch.int32)).values
        s["seeds"] = torch.randint(case["n"], (case["k"],), device="cuda", generator=gen, dtype=torch.int32)
        torch.cuda.synchronize()
        return s
    if op == "load":
        s["src"], s["dst"], s["thr"] = _host_edges(case, seed)
        return s
    if op == "serve":
        gs = [P.ssa_gen_rmat(n.bit_length() - 1, m, *RMAT, seed=seed, weighting=P.SSA_W_WC)
              for n, m in ((case["n"], case["m"]), (case["n2"], case["m2"]))]
        ben = [_benefit(g.n, seed + i) for i, g in enumerate(gs)]
        rng = np.random.default_rng(seed)
        s["graphs"], s["queries"] = gs, []
        for i in range(case["queries"]):
            # every pairing of graph, model, seed count and bound, every other one targeted
            g = i % 2
            s["queries"].append((g, P.SSA_ALGO_DSSA, (i // 2) % 2, [1, 10, 100, 1000][(i // 4) % 4],
                                 [0.1, 0.05, 0.2][(i // 8) % 3], 1.0 / gs[g].n, int(rng.integers(1 << 40)),
                                 ben[g] if (i // 2) % 3 == 1 else None))
        s["server"] = P.Server(gs, slots=case["slots"])
        return s
    g = s["graph"] = _make_graph(case, seed)
    s["benefit"] = _benefit(g.n, seed) if case["targeted"] else None
    if case["model"] == "ic":
        P.ssa_autotune(g, P.SSA_IC)
    if op == "solve":
        s["solver"] = P.Solver(g).set_graphs(case["captured"])
    if op == "estimate":
        p = P.Pool(g, MODELS[case["model"]], seed, 0, s["benefit"]).grow(4000)
        s["seeds"] = p.max_coverage(4000, case["k"])[0]
        # a node set that covers a share of the sample reaches `hits` after about hits / share sets
        share = max(p.coverage(0, 4000, s["seeds"]), 1) / 4000
        s["t_max"] = int(2 * case["hits"] / share) + 1000
        p.free()
    return s


# ---- one pass ----

def _answer(r):
    # the rounds' counts and figures, in arrays of one shape however many rounds there were
    counts, figures = np.zeros((64, 4), np.int64), np.zeros((64, 4))
    for i, t in enumerate(r.trace):
        counts[i] = t["n_sets"], t["cov"], t["check_cov"], t["check_T"]
        figures[i] = t["stat"], t["eps1"], t["eps2"], t["eps3"]
    return {"seeds": r.seeds, "influence": r.influence, "n_rr": r.n_rr, "rounds": counts, "stats": figures}


def run(s):
    c, op = s["case"], s["op"]
    if op == "solve":
        return _answer(s["solver"].solve(ALGOS[c["algo"]], MODELS[c["model"]], c["k"], c["eps"], 1.0 / c["n"],
                                         s["seed"], benefit=s["benefit"]))
    if op == "pool":
        N = c["sets"]
        train = N * 2 // 3
        p = P.Pool(s["graph"], MODELS[c["model"]], s["seed"], 0, s["benefit"]).grow(N)
        seeds, gains, cov = p.max_coverage(train, c["k"])
        out = {"seeds": seeds, "gains": gains, "cov": cov, "held_out": p.coverage(train, N - train, seeds),
               "counts": p.counts(N), "sizes": p.set_sizes()}
        p.free()
        return out
    if op == "estimate":
        return list(P.ssa_estimate_inf(s["graph"], MODELS[c["model"]], s["seed"], 1, s["seeds"], float(c["hits"]),
                                       s["t_max"], benefit=s["benefit"]))
    if op == "load":
        g = P.ssa_load_graph(c["n"], s["src"], s["dst"], s["thr"], WEIGHTS[c["weights"]], 1)
        r = P.ssa_solve(g, ALGOS[c["algo"]], MODELS[c["model"]], c["k"], c["eps"], 1.0 / c["n"], s["seed"])
        g.free()
        return _answer(r)
    if op == "serve":
        srv = s["server"]
        tickets = [srv.submit(*q[:7], benefit=q[7]) for q in s["queries"]]
        got = [srv.wait(t) for t in tickets]
        return {"seeds": np.concatenate([r.seeds for r in got]), "influence": np.array([r.influence for r in got]),
                "n_rr": np.array([r.n_rr for r in got])}
    return P.ssa_coverage_noalloc(c["n"], s["nodes"].data_ptr(), s["samp"].data_ptr(), c["entries"], 0, c["sets"],
                                  s["seeds"].data_ptr(), c["k"], torch.cuda.current_stream().cuda_stream)


def _csr_bytes(weights, n, m):
    # weighted cascade needs no stored weight: it follows from the in-degree
    return (4 if weights == "wc" else 8) * m + 4 * n


def work(case):
    """The graph (or pool) read once and the answer written once.  Sampling reads no more than the
    graph's parts that its sets reach, but reads those once per set: how often is the random outcome."""
    op = case["op"]
    if op == "cover":
        return {"bytes": 8 * case["entries"] + 4 * case["k"] + 8, "flops": 0}
    if op == "serve":
        return {"bytes": case["queries"] // 2 * (_csr_bytes("wc", case["n"], case["m"])
                                                 + _csr_bytes("wc", case["n2"], case["m2"])), "flops": 0}
    b = _csr_bytes(case["weights"], case["n"], case["m"]) + 12 * case["k"]
    if op == "load":
        b += (12 if case["weights"] == "explicit" else 8) * case["m"]
    if op == "pool":
        # each set holds a node at least: stored once, counted once; counts and sizes come back
        b += case["sets"] * (4 + 4 + 8) + 4 * case["n"]
    return {"bytes": b, "flops": 0}


def exact(case, seed):
    """Seeds, counts and sets are whole numbers, which have to be equal; a solve's few FP64 figures are
    quotients of its counts.  Only the coverage count has a plain restatement that is quick."""
    if case["op"] != "cover":
        return None
    s = prepare(case, seed)
    is_seed = torch.zeros(case["n"], dtype=torch.bool, device="cuda")
    is_seed[s["seeds"].long()] = True
    hit = torch.zeros(case["sets"], dtype=torch.bool, device="cuda")
    hit[s["samp"][is_seed[s["nodes"].long()]].long()] = True
    return int(hit.sum())
