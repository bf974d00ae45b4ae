"""What this library's users wait for, as timed cases.

Two kinds of call carry the work.  A whole fixpoint: an engine is created on
input columns that already lie in device memory, the program is declared, run
and its derived relations are exported to device columns (what bench.py's
step does, with the results kept).  And one step of a round through the
single-step calls: sort + unique, difference + merge, join.  The learned
join-size estimator's training adds the floating-point gradient.

Sizes are the benchmark's workloads, the micro-benchmark's sizes and small
or ragged ones beside them; draw() spreads over the same ranges.
"""
import math

import numpy as np
import torch

from paper_2501_13051_gb300 import cdl
from paper_2501_13051_gb300 import workloads as W


def listed():
    return [
        # the smallest whole call: the paper's transitive closure on a graph
        # of a thousand nodes, rounds in one captured CUDA graph
        {"name": "tc-er-1000-graph", "kind": "tc", "n": 1000, "m": 1500, "graph": True},
        # the same closure on a larger graph in the engine's default form
        # (rounds driven by the host), an odd number of nodes
        {"name": "tc-er-4001", "kind": "tc", "n": 4001, "m": 6007, "graph": False},
        # same generation as the paper prints it (a filter in both rules), an
        # ordinary size
        {"name": "sg-paper-20011", "kind": "sg", "n": 20011, "paper": True},
        # the benchmark's default workload, the largest fixpoint listed
        {"name": "sg-200k", "kind": "sg", "n": 200000, "paper": False},
        # points-to analysis: mutual recursion, Zipf hubs, joins that mostly
        # repeat tuples
        {"name": "points-to-2e-7", "kind": "pt", "scale": 2.0 ** -7},
        # knowledge-graph reasoning: 193 rules over 202 relations
        {"name": "owl-rl-20m", "kind": "owl", "triples": 20_000_000},
        # many independent fixpoints served as one batched run
        {"name": "batched-512", "kind": "batch", "count": 512, "lo": 1e3, "hi": 5e5, "graph": True},
        # single steps: a call where latency and launches are everything
        {"name": "sort-1000-pairs", "kind": "sort", "n": 1000, "arity": 2, "bits": 18},
        # a round's new pairs of a large fixpoint (18-bit ids)
        {"name": "sort-16m-pairs", "kind": "sort", "n": 16_777_259, "arity": 2, "bits": 18},
        # merge of a large Full with an eighth of new tuples, half repeats
        {"name": "merge-50m", "kind": "merge", "n_full": 50_000_000, "n_new": 6_250_000, "arity": 2},
        # a join of 16M probe rows with a 16M-row index built in the call
        {"name": "join-16m", "kind": "join", "n_probe": 16_000_003, "n_build": 16_777_216, "fan": 1, "zipf": False},
        # one training step's forward and backward of the join-size network
        {"name": "estimator-grad-3000", "kind": "mlp", "n": 3000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["tc", "sg", "pt", "owl", "batch", "sort", "sort", "merge", "merge", "join", "join", "mlp"])
    if kind == "tc":
        n = _log(rng, 200, 12000)
        return {"kind": kind, "n": n, "m": int(n * rng.uniform(1.1, 1.6)), "graph": rng.random() < 0.5}
    if kind == "sg":
        return {"kind": kind, "n": _log(rng, 1000, 120000), "paper": rng.random() < 0.4}
    if kind == "pt":
        return {"kind": kind, "scale": math.exp(rng.uniform(math.log(2.0 ** -12), math.log(2.0 ** -7)))}
    if kind == "owl":
        return {"kind": kind, "triples": _log(rng, 100_000, 18_000_000)}
    if kind == "batch":
        return {"kind": kind, "count": _log(rng, 2, 480), "lo": 1e3, "hi": float(_log(rng, 5000, 450_000)),
                "graph": rng.random() < 0.6}
    if kind == "sort":
        arity = rng.choice([1, 2, 2, 2, 3, 3, 4, 6, 8])
        return {"kind": kind, "n": _log(rng, 50, 40_000_000 // arity), "arity": arity,
                "bits": rng.choice([9, 14, 16, 18, 21, 24, 31, 32])}
    if kind == "merge":
        arity = rng.choice([1, 2, 2, 2, 3, 4])
        nf = _log(rng, 500, 90_000_000 // arity)
        return {"kind": kind, "n_full": nf, "n_new": max(1, int(nf * math.exp(rng.uniform(math.log(0.002), math.log(1.0))))),
                "arity": arity}
    if kind == "join":
        return {"kind": kind, "n_probe": _log(rng, 300, 16_000_000), "n_build": _log(rng, 300, 16_000_000),
                "fan": rng.choice([1, 1, 2, 5]), "zipf": rng.random() < 0.4}
    return {"kind": "mlp", "n": _log(rng, 20, 6000)}


# ------------------------------------------------------------------- inputs
# A case fixes the shape of its data (the benchmark's generator seeds 1..5),
# the seed gives it other ids and another row order: a seed's outputs are
# other tuples, as many of them.

def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda()


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _below(g, n, m):
    """n integers uniform in [0, m)."""
    return torch.randint(0, int(m), (int(n),), generator=g, device="cuda", dtype=torch.int64)


def _perm(g, n):
    return torch.randperm(int(n), generator=g, device="cuda")


def _u32(t):
    """int64 values below 2^32 as the int32 columns the library takes."""
    return torch.where(t >= 1 << 31, t - (1 << 32), t).to(torch.int32).contiguous()


def _zipf(g, n, universe, s=1.1):
    """n ids Zipf(s) over [0, universe), hot ids scattered."""
    w = torch.arange(1, universe + 1, dtype=torch.float64, device="cuda") ** -s
    cdf = torch.cumsum(w, 0)
    cdf /= cdf[-1].clone()
    r = torch.searchsorted(cdf, torch.rand(n, generator=g, device="cuda", dtype=torch.float64), right=True)
    return _perm(g, universe)[r.clamp_(max=universe - 1)]


def _split(keys, bits):
    return [_u32(keys >> bits), _u32(keys & ((1 << bits) - 1))]


def _graph_program(program, nodes, seed):
    """A workloads.Program over node ids, its input relations as device
    columns, the nodes renamed and the rows shuffled."""
    g = _gen(seed)
    name = _perm(g, nodes)
    edb = {}
    for nm, rows in program.edb.items():
        order = _perm(g, len(rows))
        r = torch.from_numpy(rows.astype(np.int64)).cuda()[order]
        edb[nm] = [_u32(name[r[:, k]]) for k in range(program.arity[nm])]
    return {"arity": program.arity, "rules": program.rules, "edb": edb, "derived": program.idb()}


def _owl(triples, seed):
    """The OWL-RL-style workload (workloads.owl_triples' shapes: a quarter
    type triples, Zipf subjects, uniform classes, properties and objects)
    with its data drawn on the GPU; the schema is the workload's own."""
    n_ent = max(1000, int(5_000_000 * triples / 20_000_000))
    _, sch = W.owl_triples(40, 4, n_entities=1000)
    shift = n_ent - 1000  # class ids follow the entities
    sch.class_base = n_ent
    sch.sub_class = [(a + shift, b + shift) for a, b in sch.sub_class]
    sch.domain = [(p, c + shift) for p, c in sch.domain]
    sch.range_ = [(p, c + shift) for p, c in sch.range_]
    g, name = _gen(4), _perm(_gen(seed), n_ent)
    n_type = triples // 4
    n_prop = triples - n_type
    b = max(1, (n_ent + sch.n_classes).bit_length())
    typ = torch.unique((name[_zipf(g, n_type, n_ent)] << b) | (n_ent + _below(g, n_type, sch.n_classes)))
    p_of = _below(g, n_prop, sch.n_props)
    keys = torch.unique((((p_of << b) | name[_zipf(g, n_prop, n_ent)]) << b) | name[_below(g, n_prop, n_ent)])
    at = torch.searchsorted(keys >> (2 * b), torch.arange(sch.n_props + 1, device="cuda")).tolist()
    low = keys & ((1 << (2 * b)) - 1)
    edb = {"type": _split(typ, b)}
    for p in range(sch.n_props):
        edb["p%d" % p] = _split(low[at[p]:at[p + 1]], b)
    edb["sc"] = [_dev(np.array(c, dtype=np.uint32)) for c in zip(*sorted(set(sch.sub_class)))]
    program = W.owl_program({nm: np.zeros((0, 2), np.uint32) for nm in edb}, sch)
    return {"arity": program.arity, "rules": program.rules, "edb": edb, "derived": program.idb()}


def _batch(case, seed):
    """Independent instances, TC on even and SG on odd ones, log-uniform edge
    counts, mean out-degree 0.9 (workloads.batched_instances' shapes)."""
    g = _gen(5)
    sizes = torch.from_numpy(W.batched_graph_sizes(case["count"], 5, case["lo"], case["hi"])).cuda()
    nodes = torch.ceil(sizes / 0.9).to(torch.int64)
    inst = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), sizes)
    n = nodes[inst].to(torch.float64)
    u = (torch.rand(len(inst), generator=g, device="cuda", dtype=torch.float64) * n).to(torch.int64)
    v = (torch.rand(len(inst), generator=g, device="cuda", dtype=torch.float64) * n).to(torch.int64)
    # the nodes of each instance renamed among themselves
    node_inst = torch.repeat_interleave(torch.arange(len(nodes), device="cuda"), nodes)
    key = torch.rand(len(node_inst), generator=_gen(seed), device="cuda", dtype=torch.float64) + node_inst
    first = torch.cumsum(nodes, 0) - nodes
    name = torch.argsort(key) - first[node_inst]
    ok = u != v
    inst, u, v = inst[ok], u[ok], v[ok]
    keys = torch.unique(((inst << 21) | name[first[inst] + u]) << 21 | name[first[inst] + v])
    inst, u, v = keys >> 42, (keys >> 21) & ((1 << 21) - 1), keys & ((1 << 21) - 1)
    program = W.batched_program([], [])
    edb = {}
    for nm, odd in (("tc_edge", 0), ("sg_edge", 1)):
        pick = (inst & 1) == odd
        edb[nm] = [_u32(inst[pick]), _u32(u[pick]), _u32(v[pick])]
    return {"arity": program.arity, "rules": program.rules, "edb": edb, "derived": program.idb()}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "tc":
        program = W.tc_program(W.er_graph(case["n"], case["m"], 1))
        return dict(_graph_program(program, case["n"], seed), opts={"graph": case["graph"]})
    if kind == "sg":
        make = W.sg_paper_program if case["paper"] else W.sg_program
        return dict(_graph_program(make(W.random_forest(case["n"], 2)), case["n"], seed), opts={})
    if kind == "pt":
        program = W.points_to_program(W.points_to_edb(case["scale"], 3))
        return dict(_graph_program(program, max(2, int(round(2_000_000 * case["scale"]))), seed), opts={})
    if kind == "owl":
        return dict(_owl(case["triples"], seed), opts={})
    if kind == "batch":
        return dict(_batch(case, seed), opts={"n_instances": case["count"], "graph": case["graph"]})
    g, own = _gen(case.get("n", case.get("n_full", 0)) + 6), _gen(seed)
    if kind == "sort":
        # uniform values; the seed flips bits of a column's values alike
        order = _perm(own, case["n"])
        flip = _below(own, case["arity"], 1 << case["bits"]).tolist()
        return {"sort": [_u32((_below(g, case["n"], 1 << case["bits"]) ^ f)[order]) for f in flip]}
    if kind == "merge":
        k = case["arity"]
        b = {1: 31, 2: 18, 3: 12, 4: 9}[k]
        want = min(case["n_full"], 1 << (k * b - 1))
        full = torch.unique(_below(g, int(want * 1.03) + 8, 1 << (k * b)))
        full = full[_perm(g, len(full))[:want]]
        half = case["n_new"] // 2
        new = torch.cat([full[_below(g, half, len(full))], _below(g, case["n_new"] - half, 1 << (k * b))])
        flip = _below(own, 1, 1 << (k * b))
        cols = lambda t: [_u32((t >> (b * (k - 1 - i))) & ((1 << b) - 1)) for i in range(k)]
        return {"full": cols(torch.sort(full ^ flip)[0]), "new": cols(torch.sort(new ^ flip)[0])}
    if kind == "join":
        # build rows sorted by key, about `fan` rows a key; every probe row matches
        distinct = max(1, case["n_build"] // case["fan"])
        bits = (2 * distinct - 1).bit_length()
        key = torch.unique(_below(g, distinct, 1 << bits))
        key = key[_perm(g, len(key))]
        build = key[torch.arange(case["n_build"], device="cuda") % len(key)] if case["fan"] > 1 else key
        pick = _zipf(g, case["n_probe"], len(key)) if case["zipf"] else _below(g, case["n_probe"], len(key))
        flip = _below(own, 1, 1 << bits)
        return {"probe": [_u32((key[pick] ^ flip)[_perm(own, case["n_probe"])]), _u32(_below(own, case["n_probe"], 1 << 30))],
                "build": [_u32(torch.sort(build ^ flip)[0]), _u32(_below(own, len(build), 1 << 30))]}
    # the network's parameters as training starts from them, features and
    # targets in the ranges of logged joins
    n = case["n"]
    u = lambda *shape: torch.rand(*shape, generator=own, device="cuda", dtype=torch.float32)
    he = lambda rows, fan_in: ((2 * u(rows * fan_in) - 1) * math.sqrt(6.0 / fan_in))
    zero = lambda k: torch.zeros(k, device="cuda")
    params = torch.cat([he(64, 16), zero(64), he(64, 64), zero(64), he(1, 64), zero(1)])
    scale = torch.tensor([25, 25, 28, 11, 11, 8, 28, 1, 1, 5, 5, 1, 40, 28, 26, 1], device="cuda", dtype=torch.float32)
    return {"params": params, "X": (u(n, 16) * scale).contiguous(), "y": u(n) * 28}


# --------------------------------------------------------------------- calls

def run(state):
    if "rules" in state:
        with cdl.Engine(**state["opts"]) as e:
            for name, arity in state["arity"].items():
                e.relation(name, arity)
            e.load_many(state["edb"])
            for r in state["rules"]:
                e.rule(r.head, r.body, r.neq)
            st = e.run()
            out = {name: e.export(name, device=True) for name in state["derived"]}
        props = [nm for nm in out if nm.startswith("p") and nm[1:].isdigit()]
        if props:  # a triple store's program puts the properties into one table of triples
            parts = [out.pop(nm) for nm in props]
            out["triples"] = [torch.cat([p[k] for p in parts]) for k in range(2)]
            out["sizes"] = np.array([len(p[0]) for p in parts], dtype=np.int64)
        out["rounds"] = np.array([st.iterations, st.rounds, st.derived_tuples] + list(st.delta_per_round), dtype=np.int64)
        if st.iters_per_instance:
            out["instances"] = np.array(st.iters_per_instance, dtype=np.int64)
        return out
    if "sort" in state:
        return cdl.sort_unique(state["sort"])
    if "full" in state:
        delta, merged = cdl.diff_merge(state["full"], state["new"])
        return {"delta": delta, "merged": merged}
    if "probe" in state:
        return cdl.join(state["probe"], 0, state["build"], 0, [(0, 1), (1, 1)])
    pred, grad = cdl.mlp_gradient(state["params"], state["X"], state["y"])
    return {"pred": pred, "grad": grad}


def work(case):
    """Bytes of the inputs read once and the results written once (the
    derived relations' sizes as the generators give them on average)."""
    kind = case["kind"]
    flops = 0.0
    if kind == "tc":
        reach = max(0.0, 1.0 - 0.5 ** ((case["m"] / case["n"] - 0.9) / 0.75 + 0.5)) ** 2
        total = 8.0 * case["m"] + 8.0 * (reach * case["n"] ** 2 + case["m"])
    elif kind == "sg":
        total = 8.0 * case["n"] + 8.0 * 0.045 * case["n"] ** 2
    elif kind == "pt":
        total = 8.0 * 5e6 * case["scale"] + 8.0 * 0.09 * (2e6 * case["scale"]) ** 2
    elif kind == "owl":
        total = 8.0 * case["triples"] * (1.0 + 5.3)
    elif kind == "batch":
        edges = case["count"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        total = 12.0 * edges * (1.0 + 6.8)
    elif kind == "sort":
        total = 8.0 * case["arity"] * case["n"]
    elif kind == "merge":
        total = 4.0 * case["arity"] * (2.0 * case["n_full"] + 2.0 * case["n_new"])
    elif kind == "join":
        total = 8.0 * (2.0 * case["n_probe"] * case["fan"] + case["n_build"])
    else:
        total = 4.0 * (18.0 * case["n"] + 2 * cdl.MLP_PARAMS)
        flops = 6.0 * cdl.MLP_PARAMS * case["n"]
    return {"bytes": total, "flops": flops}


def exact(case, seed):
    """The gradient in 64 bits; every other result is whole numbers."""
    if case["kind"] != "mlp":
        return None
    s = prepare(case, seed)
    th = s["params"].double().requires_grad_(True)
    X, y = s["X"].double(), s["y"].double()
    w1, b1 = th[:1024].reshape(64, 16), th[1024:1088]
    w2, b2 = th[1088:5184].reshape(64, 64), th[5184:5248]
    w3, b3 = th[5248:5312], th[5312]
    h1 = torch.relu(X @ w1.T + b1)
    h2 = torch.relu(h1 @ w2.T + b2)
    pred = h2 @ w3 + b3
    r = y - pred
    loss = torch.where(r > 0, 0.9 * r, -0.1 * r).mean()
    loss.backward()
    return {"pred": pred.detach(), "grad": th.grad}
