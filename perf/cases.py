"""What a user of the engine has it do, as measurable cases.

A case is one pass through the public entry points: reset the engine, load the
input facts from device memory, run the program to its fixpoint and read the
derived relations back to device memory (discrete runs and inference), or one
forward + backward through ``autograd.fixpoint`` (training).  Sizes are those
of this repository's configurations, benchmark and tests, and of the ranges
between their smallest and largest instances.

``exact`` computes tags and gradients in 64 bits with plain torch, without the
engine: layered sums for add-mult, bottleneck paths over ranked inputs for
max-min, most likely paths for top-1 proofs.
"""
from __future__ import annotations

import functools

import numpy as np
import torch

from paper_2503_21937_gb300 import Engine, lobster
from paper_2503_21937_gb300 import workloads as W
from paper_2503_21937_gb300.autograd import fixpoint

HOP_PROGRAM = ("hop(x,y,1) :- edge(x,y).\n"
               "hop(x,z,d + 1) :- hop(x,y,d), edge(y,z), d < {hops}.\n")


def listed():
    return [
        # An interactive query on a handful of facts: launches and host work are all there is.
        {"name": "tc_small", "kind": "tc_er", "nodes": 67, "edges": 131},
        # The 1,000-node / 3,000-edge random digraph of the configurations: many short iterations.
        {"name": "tc_er_1k", "kind": "tc_er", "nodes": 1000, "edges": 3000},
        # Reachability over a graph with hubs, the benchmark's closure: hundreds of millions of facts.
        {"name": "tc_power_20k", "kind": "tc_power", "nodes": 20000, "edges": 100000},
        # Same generation over a 50,000-node hierarchy, the benchmark's other half: the largest result.
        {"name": "sg_tree_50k", "kind": "sg_tree", "nodes": 50000},
        # Points-to analysis of a program: four rules, three-way joins, most candidates known already.
        {"name": "andersen_200k", "kind": "andersen", "vars": 200000, "stmts": 400000},
        # One probabilistic grid, forward and backward, as a training step on a single sample runs it.
        {"name": "grid_64_max_min", "kind": "reach", "side": 64, "semiring": "diff_max_min"},
        {"name": "grid_64_add_mult", "kind": "reach", "side": 64, "semiring": "diff_add_mult"},
        # The batched training step: 512 samples of uneven size, reachability and kinship together.
        {"name": "batch_512_max_min", "kind": "batch", "samples": 512, "semiring": "diff_max_min"},
        {"name": "batch_512_add_mult", "kind": "batch", "samples": 512, "semiring": "diff_add_mult"},
        # The fixpoint of a Pathfinder training step with one proof per fact (the paper's semiring for it).
        {"name": "proofs_64x16", "kind": "proofs", "batch": 64, "side": 16},
        # Inference with a computed column: best path of every length up to a bound, 64-bit keys.
        {"name": "hops_max_min", "kind": "hops", "nodes": 500, "edges": 2000, "hops": 8},
        # Deduplication where nothing may be allocated: the shortest call of the library.
        {"name": "unique_rows", "kind": "unique", "rows": 100003, "arity": 2},
    ]


def _log(rng, lo, hi):
    """An integer of [lo, hi], spread over its logarithm."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["tc_er", "tc_power", "sg_tree", "andersen", "reach", "batch", "proofs", "hops", "unique"])
    if kind == "tc_er":
        n = _log(rng, 40, 3000)
        return {"kind": kind, "nodes": n, "edges": int(n * rng.uniform(1.5, 4.0))}
    if kind == "tc_power":
        n = _log(rng, 500, 20000)
        return {"kind": kind, "nodes": n, "edges": int(n * rng.uniform(3.0, 5.0))}
    if kind == "sg_tree":
        return {"kind": kind, "nodes": _log(rng, 300, 50000)}
    if kind == "andersen":
        n = _log(rng, 2000, 200000)
        return {"kind": kind, "vars": n, "stmts": int(n * rng.uniform(1.2, 2.0))}
    if kind == "reach":
        return {"kind": kind, "side": _log(rng, 5, 64), "semiring": rng.choice(["diff_max_min", "diff_add_mult"])}
    if kind == "batch":
        return {"kind": kind, "samples": _log(rng, 9, 512), "semiring": rng.choice(["diff_max_min", "diff_add_mult"])}
    if kind == "proofs":
        return {"kind": kind, "batch": rng.randint(8, 64), "side": rng.randint(6, 32)}
    if kind == "hops":
        n = _log(rng, 50, 700)
        return {"kind": kind, "nodes": n, "edges": int(n * rng.uniform(1.5, 4.0)), "hops": rng.randint(3, 10)}
    return {"kind": kind, "rows": _log(rng, 100, lobster.NOALLOC_MAX_ROWS), "arity": rng.randint(1, 2)}


# ---------------------------------------------------------------------------
# inputs: host columns from the seed, and the state a program keeps
# ---------------------------------------------------------------------------
_STRUCTURE = 1000  # one structure per case; the seed draws its labels, row order and probabilities


def _ints(a):
    return torch.from_numpy(np.ascontiguousarray(a).astype(np.int32)).cuda()


def _floats(a):
    return torch.from_numpy(np.ascontiguousarray(a).astype(np.float32)).cuda()


def _relabelled(cols, n, s):
    """The same relation over relabelled ids, rows in another order."""
    return s.permutation(n)[np.stack(cols)][:, s.permutation(len(cols[0]))]


def _facts(case, seed):
    """relation -> (columns (arity, n), probabilities or None, sample ids or None), on the host."""
    kind, s = case["kind"], W.stream(_STRUCTURE + 1 + int(seed))
    if kind == "tc_er":
        edges = W.erdos_renyi(case["nodes"], case["edges"], seed_index=_STRUCTURE)
        return {"edge": (_relabelled(edges, case["nodes"], s), None, None)}
    if kind == "tc_power":
        edges = W.chung_lu_power_law(case["nodes"], case["edges"], seed_index=_STRUCTURE)
        return {"edge": (_relabelled(edges, case["nodes"], s), None, None)}
    if kind == "sg_tree":
        parent, child, _ = W.random_tree(case["nodes"], seed_index=_STRUCTURE)
        return {"parent": (_relabelled((parent, child), case["nodes"], s), None, None)}
    if kind == "andersen":
        stmts = W.andersen_program(case["vars"], case["stmts"], seed_index=_STRUCTURE)
        ids = s.permutation(case["vars"])
        return {k: (ids[np.stack(v)][:, s.permutation(len(v[0]))], None, None) for k, v in stmts.items()}
    if kind == "reach":
        src, dst, _ = W.grid_reach_instance(case["side"])["edge"]
        return {"edge": (np.stack([src, dst]), np.repeat(s.prob(len(src) // 2), 2), None),
                "start": (np.zeros((1, 1), np.uint32), None, None)}
    if kind == "batch":
        b = W.batched_instance(case["samples"], seed_index=_STRUCTURE)
        e, st, f, c = b["edge"], b["start"], b["fact"], b["comp"]
        ids = s.permutation(case["samples"])  # the samples come in another order
        return {"edge": (np.stack(e[:2]), np.repeat(s.prob(len(e[0]) // 2), 2), ids[e[3]]),
                "start": (st[0][None, :], None, ids[st[2]]),
                "fact": (np.stack(f[:3]), s.prob(len(f[0])), ids[f[4]]),
                "comp": (np.stack(c[:3]), None, ids[c[4]])}
    if kind == "proofs":
        # the probabilities a partly trained edge predictor gives: most edges near 0.1 or 0.9
        side, batch = case["side"], case["batch"]
        u, v = W.grid_edges(side)
        lit = s.unit(batch * len(u)) < 0.4
        logit = np.where(lit, 2.0, -2.0) + 0.8 * s.normal(batch * len(u))
        p = (1.0 / (1.0 + np.exp(-logit))).astype(np.float32).reshape(batch, -1)
        start = s.below(batch, side * side)
        cols = np.stack([np.tile(np.concatenate([u, v]), batch), np.tile(np.concatenate([v, u]), batch)])
        ids = np.arange(batch, dtype=np.uint32)
        return {"edge": (cols, np.concatenate([p, p], axis=1).ravel(), np.repeat(ids, 2 * len(u))),
                "start": (start[None, :], None, ids)}
    if kind == "hops":
        edges = W.erdos_renyi(case["nodes"], case["edges"], seed_index=_STRUCTURE)
        return {"edge": (_relabelled(edges, case["nodes"], s), s.prob(case["edges"]), None)}
    raise ValueError(kind)


# program, semiring and the relations read back, per kind of engine run
_PROGRAMS = {"tc_er": (W.TC_PROGRAM, "unit", "path"), "tc_power": (W.TC_PROGRAM, "unit", "path"),
             "sg_tree": (W.SG_PROGRAM, "unit", "sg"), "andersen": (W.ANDERSEN_PROGRAM, "unit", "pt"),
             "hops": (HOP_PROGRAM, "max_min", "hop")}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "unique":
        # about a third of the rows are repeats
        n, arity, s = case["rows"], case["arity"], W.stream(_STRUCTURE + 1 + int(seed))
        rows = np.stack([s.below(n, max(2, n)) for _ in range(arity)])
        if arity == 2:
            again = s.below(n // 3, n)
            rows[:, : n // 3] = rows[:, again]
        return {"kind": kind, "cols": _ints(rows), "out": torch.zeros((arity, n), dtype=torch.int32, device="cuda"),
                "n_out": torch.zeros(1, dtype=torch.int64, device="cuda")}
    facts = {k: (_ints(c), None if p is None else _floats(p), None if s is None else _ints(s))
             for k, (c, p, s) in _facts(case, seed).items()}
    state = {"kind": kind, "facts": facts}
    if kind in _PROGRAMS:
        program, semiring, out = _PROGRAMS[kind]
        e = Engine()
        e.program(program.format(hops=case["hops"]) if kind == "hops" else program)
        state.update(engine=e, semiring=semiring, out=out)
    elif kind == "reach":
        state.update(program=W.REACH_PROGRAM, semiring=case["semiring"], outputs=["reach"])
    elif kind == "batch":
        state.update(program=W.REACH_PROGRAM + W.KIN_PROGRAM, semiring=case["semiring"], outputs=["reach", "kin"])
    else:
        state.update(program=W.REACH_PROGRAM, semiring="diff_top1_proofs", outputs=["reach"])
    return state


def run(state):
    if state["kind"] == "unique":
        lobster.unique_rows_noalloc(state["cols"], state["out"], state["n_out"])
        return {"rows": state["out"], "count": state["n_out"]}
    if "engine" in state:
        e = state["engine"]
        e.reset()
        for name, (cols, probs, samples) in state["facts"].items():
            e.load(name, cols, probs, samples)
        e.run(state["semiring"])
        r = e.read(state["out"], device=True)
        return {"cols": r.cols} if state["semiring"] == "unit" else {"cols": r.cols, "tags": r.tags}
    leaves = {k: v[1].detach().requires_grad_(True) for k, v in state["facts"].items() if v[1] is not None}
    got = fixpoint(state["program"], {k: (v[0], leaves.get(k), v[2]) for k, v in state["facts"].items()},
                   state["semiring"], outputs=state["outputs"])
    loss = sum(0.5 * got[o][1].square().sum() for o in state["outputs"])
    loss.backward()
    res = {}
    for o in state["outputs"]:
        res[o] = {"cols": got[o][0], "tags": got[o][1].detach(), "samples": got[o][2]}
    for k, p in leaves.items():
        res["grad_" + k] = p.grad
    return res


# ---------------------------------------------------------------------------
# the least traffic of a pass: inputs once, outputs once
# ---------------------------------------------------------------------------
def _closure_pairs(src, dst, n):
    """Reachable pairs through the strongly connected core around the node of
    highest degree: (nodes that reach it) x (nodes it reaches), which is all
    but a small share of a random graph's closure."""
    hub = int(np.argmax(np.minimum(np.bincount(src, minlength=n), np.bincount(dst, minlength=n))))

    def cone(a, b):
        seen = np.zeros(n, bool)
        seen[hub] = True
        while True:
            new = b[seen[a] & ~seen[b]]
            if not len(new):
                return int(seen.sum())
            seen[new] = True

    return cone(src, dst) * cone(dst, src)


def work(case):
    kind = case["kind"]
    if kind == "unique":
        n, a = case["rows"], case["arity"]
        return {"bytes": n * a * 4 + (2 * n // 3) * a * 4, "flops": 0}
    facts = _facts(case, 0)
    n_in = sum(c.size * 4 + (0 if p is None else p.size * 4) + (0 if s is None else s.size * 4)
               for c, p, s in facts.values())
    grads = sum(0 if p is None else p.size * 4 for _, p, _ in facts.values())
    flops = 0
    if kind in ("tc_er", "tc_power"):
        (src, dst), _, _ = facts["edge"]
        out = 8 * _closure_pairs(src, dst, case["nodes"])
    elif kind == "sg_tree":
        _, _, depth = W.random_tree(case["nodes"], seed_index=_STRUCTURE)
        level = np.bincount(depth)[1:].astype(np.int64)
        out = 8 * int((level * (level - 1)).sum())
    elif kind == "andersen":
        # points-to facts per distinct address-of statement, as measured on these programs
        out = 8 * 300 * len(np.unique(facts["addr"][0], axis=1).T)
    elif kind == "hops":
        # nearly every pair is joined by some walk of the longer lengths
        n, m, k = case["nodes"], case["edges"], case["hops"]
        pairs = sum(min(n * (m / n) ** d, n * n * 0.9) for d in range(1, k + 1))
        out, flops = int(16 * pairs), 0
    else:
        nodes = (case["side"] ** 2 if kind == "reach" else case["batch"] * case["side"] ** 2 if kind == "proofs"
                 else int((_sides(case["samples"]) ** 2).sum()))
        out = 12 * nodes + grads
        if kind == "batch":
            out += case["samples"] * 11400 * 20  # kinship facts of a sample, about 11,400
            flops = case["samples"] * 9.0e6 * (6 if case["semiring"] == "diff_add_mult" else 0)
    return {"bytes": n_in + out, "flops": flops}


@functools.lru_cache(maxsize=4)
def _sides(samples):
    return W.batched_instance(samples, seed_index=_STRUCTURE)["sides"]


# ---------------------------------------------------------------------------
# the same answers in 64 bits
# ---------------------------------------------------------------------------
def _long(a):
    return torch.from_numpy(np.ascontiguousarray(a).astype(np.int64)).cuda()


def _ranks(p):
    """1..n by (probability, then earlier row higher): the order of (value, input id) tags."""
    p = torch.from_numpy(np.asarray(p, np.float32)).cuda()
    n = len(p)
    order = (n - 1) - torch.argsort(p.flip(0), stable=True)
    rank = torch.empty(n, dtype=torch.int64, device="cuda")
    rank[order] = torch.arange(1, n + 1, device="cuda")
    return rank, order


def _max_min_result(rank, present, order, p, grad_rows):
    """Tags of the present facts from their ranks (the top rank: tag 1, no
    input), and the gradient of half the sum of squares."""
    r = rank[present]
    p64 = torch.from_numpy(np.asarray(p, np.float32)).cuda().double()
    top = len(p64) + 1
    fact = order[(r - 1).clamp(max=len(p64) - 1)]
    tags = torch.where(r == top, torch.ones((), dtype=torch.float64, device="cuda"), p64[fact])
    grad = torch.zeros(grad_rows, dtype=torch.float64, device="cuda")
    grad.index_add_(0, fact, torch.where(r == top, torch.zeros_like(tags), tags))
    return tags, grad


def _reach_max_min(src, dst, p, starts, n):
    rank, order = _ranks(p)
    t = torch.zeros(n, dtype=torch.int64, device="cuda")
    t[starts] = len(p) + 1
    while True:
        u = t.scatter_reduce(0, dst, torch.minimum(t[src], rank), "amax")
        if torch.equal(u, t):
            break
        t = u
    return _max_min_result(t, t > 0, order, p, len(p))


def _reach_add_mult(src, dst, p, starts, n):
    p = torch.from_numpy(np.asarray(p, np.float32)).cuda().double().requires_grad_(True)
    t = torch.zeros(n, dtype=torch.float64, device="cuda")
    t[starts] = 1.0
    seen = t > 0
    while True:  # a fact's tag is the clamped sum over the derivations of its first iteration
        use = torch.nonzero(seen[src] & ~seen[dst]).squeeze(1)
        if not len(use):
            break
        d = dst[use]
        s = torch.zeros(n, dtype=torch.float64, device="cuda").index_add(0, d, t[src[use]] * p[use])
        t = t + s.clamp(max=1.0)
        seen = seen.clone()
        seen[d] = True
    tags = t[seen]
    (0.5 * tags.square().sum()).backward()
    return tags.detach(), p.grad


def _reach_proofs(src, dst, p, starts, n):
    p = torch.from_numpy(np.asarray(p, np.float32)).cuda().double().requires_grad_(True)
    q = p.detach()
    t = torch.zeros(n, dtype=torch.float64, device="cuda")
    t[starts] = 1.0
    while True:
        u = t.scatter_reduce(0, dst, t[src] * q, "amax")
        if torch.equal(u, t):
            break
        t = u
    # the last edge of each fact's most likely path, then the products along the paths
    is_start = torch.zeros(n, dtype=torch.bool, device="cuda")
    is_start[starts] = True
    best = torch.nonzero((t[src] * q == t[dst]) & (t[dst] > 0) & ~is_start[dst]).squeeze(1)
    last = torch.full((n,), -1, dtype=torch.int64, device="cuda")
    last[dst[best]] = best
    prob = torch.zeros(n, dtype=torch.float64, device="cuda")
    prob[starts] = 1.0
    done, node = is_start.clone(), torch.arange(n, device="cuda")
    todo = node[(last >= 0) & ~done]
    while len(todo):
        ready = todo[done[src[last[todo]]]]
        if not len(ready):
            break
        prob = prob.index_copy(0, ready, prob[src[last[ready]]] * p[last[ready]])
        done = done.index_fill(0, ready, True)
        todo = todo[~done[todo]]
    tags = prob[t > 0]
    (0.5 * tags.square().sum()).backward()
    return tags.detach(), p.grad


def _kinship(facts, comp, samples, semiring):
    """Tags of kin in (sample, r, x, y) order and the gradient of the fact rows,
    on dense (sample, label, person, person) arrays, 32 samples at a time."""
    (r, a, b), p, sid = facts
    n, labels = 40, 20
    table = np.zeros((labels, labels), np.int64)
    table[comp[0], comp[1]] = comp[2]
    head = torch.from_numpy(table.reshape(-1)).cuda()
    r, a, b, sid = _long(r), _long(a), _long(b), _long(sid)
    off = ~torch.eye(n, dtype=torch.bool, device="cuda")
    max_min = semiring == "diff_max_min"
    if max_min:
        rank, order = _ranks(p)
    else:
        p64 = torch.from_numpy(np.asarray(p, np.float32)).cuda().double().requires_grad_(True)
    tags = []
    grad = torch.zeros(len(p), dtype=torch.float64, device="cuda")
    step = 32
    for s0 in range(0, samples, step):
        m = min(step, samples - s0)
        rows = torch.nonzero((sid >= s0) & (sid < s0 + m)).squeeze(1)
        at = (((sid[rows] - s0) * labels + r[rows]) * n + a[rows]) * n + b[rows]
        size = m * labels * n * n
        if max_min:
            k = torch.zeros(size, dtype=torch.int64, device="cuda").scatter_reduce(0, at, rank[rows], "amax")
            k = k.view(m, labels, n, n).int()
            while True:
                left = k.permute(0, 1, 2, 3).reshape(m, labels * n, n)
                right = k.permute(0, 2, 1, 3).reshape(m, n, labels * n)
                best = torch.zeros(m, labels * n, labels * n, dtype=torch.int32, device="cuda")
                for y in range(n):
                    best = torch.maximum(best, torch.minimum(left[:, :, y, None], right[:, y, None, :]))
                best = best.view(m, labels, n, labels, n).permute(0, 1, 3, 2, 4).reshape(m, labels * labels, n, n)
                new = torch.zeros_like(k).index_reduce(1, head, best, "amax") * off
                new = torch.maximum(k, new)
                if torch.equal(new, k):
                    break
                k = new
            k = k.long()
            t, g = _max_min_result(k, k > 0, order, p, len(p))
            tags.append(t)
            grad += g
            continue
        k = torch.zeros(size, dtype=torch.float64, device="cuda").index_add(0, at, p64[rows]).clamp(max=1.0)
        k = k.view(m, labels, n, n)
        seen = torch.zeros(size, dtype=torch.bool, device="cuda").index_fill(0, at, True).view(m, labels, n, n)
        while True:
            def product(x):
                left = x.reshape(m, labels * n, n)
                right = x.permute(0, 2, 1, 3).reshape(m, n, labels * n)
                z = (left @ right).view(m, labels, n, labels, n).permute(0, 1, 3, 2, 4)
                z = z.reshape(m, labels * labels, n, n)
                return torch.zeros_like(x).index_add(1, head, z) * off

            new = (product(seen.float()) > 0) & ~seen
            if not bool(new.any()):
                break
            k = k + torch.where(new, product(k).clamp(max=1.0), torch.zeros((), dtype=torch.float64, device="cuda"))
            seen = seen | new
        t = k[seen]
        g, = torch.autograd.grad(0.5 * t.square().sum(), p64)
        tags.append(t.detach())
        grad += g
    return torch.cat(tags), grad


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("reach", "batch", "proofs", "hops"):
        return None  # whole numbers only
    facts = _facts(case, seed)
    if kind == "hops":
        (src, dst), p, _ = facts["edge"]
        n, k = case["nodes"], case["hops"]
        e = torch.zeros(n, n, dtype=torch.float64, device="cuda")
        e[_long(src), _long(dst)] = torch.from_numpy(p).cuda().double()  # rows are distinct
        layers = [e]
        for _ in range(k - 1):
            nxt = torch.zeros_like(e)
            for y in range(n):
                nxt = torch.maximum(nxt, torch.minimum(layers[-1][:, y, None], e[y, None, :]))
            layers.append(nxt)
        t = torch.stack(layers, dim=2)
        return {"cols": None, "tags": t[t > 0]}
    (src, dst), p, sid = facts["edge"]
    width = {"reach": case.get("side", 0) ** 2, "batch": 48 * 48, "proofs": case.get("side", 0) ** 2}[kind]
    samples = {"reach": 1, "batch": case.get("samples"), "proofs": case.get("batch")}[kind]
    sample = _long(np.zeros(len(p)) if sid is None else sid)
    ssid = facts["start"][2]
    starts = _long(facts["start"][0][0]) + width * _long(np.zeros(1) if ssid is None else ssid)
    reach = (_reach_proofs if kind == "proofs" else
             _reach_max_min if case["semiring"] == "diff_max_min" else _reach_add_mult)
    tags, grad = reach(_long(src) + width * sample, _long(dst) + width * sample, p, starts, width * samples)
    res = {"reach": {"cols": None, "tags": tags, "samples": None}, "grad_edge": grad}
    if kind == "batch":
        comp = facts["comp"]
        first = comp[2] == comp[2][0]  # the table is the same for every sample
        tags, grad = _kinship(facts["fact"], comp[0][:, first], samples, case["semiring"])
        res["kin"] = {"cols": None, "tags": tags, "samples": None}
        res["grad_fact"] = grad
    return res
