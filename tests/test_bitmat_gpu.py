"""Chain programs on bit matrices (unit semiring) against the oracle and
against the general path (option bit_matrix = 0): relations, iterations,
derivations and new facts are equal on every program shape, both storage
orientations, renumbered ids, long rows and listed (large) matrices."""
import numpy as np
import pytest

from paper_2503_21937_gb300 import workloads as W
from tests.common import compare, engine_run

pytestmark = pytest.mark.gpu

PROGRAMS = {
    "left": W.TC_PROGRAM,
    "right": "path(x,y) :- edge(x,y).\npath(x,z) :- edge(x,y), path(y,z).\n",
    "nonlinear": "path(x,y) :- edge(x,y).\npath(x,z) :- path(x,y), path(y,z).\n",
    "same_generation": "path(x,y) :- edge(p,x), edge(p,y), x != y.\npath(x,y) :- edge(a,x), path(a,b), edge(b,y).\n",
    "reversed": "path(y,x) :- edge(x,y).\npath(x,z) :- path(y,x), edge(y,z), x != z.\n",
    "four_atoms": "path(x,y) :- edge(x,y).\npath(x,w) :- edge(x,y), path(z,y), edge(z,v), path(v,w).\n",
    "loops": "path(x,y) :- edge(x,y).\npath(x,z) :- path(x,y), edge(y,z).\nback(x,y) :- path(x,z), path(z,y), x == y.\n",
    "mutual": "odd(x,y) :- edge(x,y).\nodd(x,z) :- even(x,y), edge(y,z).\neven(x,z) :- odd(x,y), edge(y,z).\n",
    "two_rules": "path(x,y) :- edge(x,y).\npath(x,y) :- edge(y,x).\npath(x,z) :- path(x,y), edge(y,z).\n"
                 "path(x,z) :- path(x,y), edge(z,y).\n",
}


def same_as_general(program, inputs, **kw):
    outs = []
    for on in (1, 0):
        e, st, got = engine_run(program, inputs, options={"bit_matrix": on}, **kw)
        outs.append((st, got))
        e.close()
    (a, ga), (b, gb) = outs
    for k in ("iterations", "derived", "candidates", "new_facts"):
        assert a[k] == b[k], (k, a[k], b[k])
    for name in gb:
        assert np.array_equal(ga[name].cols, gb[name].cols), name
        assert np.array_equal(ga[name].tags, gb[name].tags), name
        assert np.array_equal(ga[name].samples, gb[name].samples), name
    return a


@pytest.mark.parametrize("name", list(PROGRAMS))
@pytest.mark.parametrize("n,m,scale", [(2, 1, 1), (31, 40, 1), (33, 60, 1), (127, 200, 40000), (129, 180, 1)])
def test_program_shapes(name, n, m, scale):
    """Rows of one word group and just past one, ids dense and spread out
    (renumbered), every rule shape; duplicates among the input rows."""
    s = W.stream(7100 + n)
    a, b = s.below(m, n) * np.uint32(scale), s.below(m, n) * np.uint32(scale)
    inputs = {"edge": ((np.concatenate([a, a[:5]]), np.concatenate([b, b[:5]])),)}
    compare(PROGRAMS[name], inputs)
    same_as_general(PROGRAMS[name], inputs)


@pytest.mark.parametrize("name", ["left", "right", "nonlinear", "mutual", "same_generation"])
def test_facts_loaded_into_derived_relations(name):
    s = W.stream(7200)
    a, b, c, d = (s.below(60, 50) for _ in range(4))
    head = "odd" if name == "mutual" else "path"
    inputs = {"edge": ((a, b),), head: ((c[:9], d[:9]),)}
    compare(PROGRAMS[name], inputs)
    same_as_general(PROGRAMS[name], inputs)


@pytest.mark.parametrize("n", [12000, 17000])
@pytest.mark.parametrize("name", ["left", "right", "same_generation", "two_rules"])
def test_listed_rows_and_long_rows(name, n):
    """Matrices beyond the listing threshold (12,000 values) and the one for wide
    rows (17,000), rows of more than 512 entries in both directions (a hub), most
    rows idle in most iterations."""
    s = W.stream(7300)
    parent, child, _ = W.random_tree(n, seed_index=7301)
    hub = np.full(700, 5, np.uint32)
    leaf = s.below(700, n)
    a = np.concatenate([parent, hub, leaf[:600]])
    b = np.concatenate([child, leaf, hub[:600]])
    if name == "same_generation":
        a, b = parent, child
    if name == "two_rules":
        a, b = a[:3000], b[:3000]
    same_as_general(PROGRAMS[name], {"edge": ((a, b),)})


def test_points_to_and_iteration_limit():
    A = W.andersen_program(60000, 3000, seed_index=7400)
    inputs = {k: ((v[0], v[1]),) for k, v in A.items()}
    compare(W.ANDERSEN_PROGRAM, inputs, rels=["pt"])
    same_as_general(W.ANDERSEN_PROGRAM, inputs)
    from paper_2503_21937_gb300 import Engine, LobsterError
    got = []
    for on in (1, 0):
        e = Engine()
        e.program(W.TC_PROGRAM)
        e.set_option("bit_matrix", on)
        e.load("edge", W.ktree_chain(60))
        with pytest.raises(LobsterError, match="MAXITER"):
            e.run("unit", max_iters=7)
        got.append(e.read("path").cols)
        e.close()
    assert np.array_equal(got[0], got[1])


def _profiled(program, inputs, on):
    e, st, _ = engine_run(program, inputs, options={"bit_matrix": on, "profile": 1}, read=[])
    kernels = e.profile()
    e.close()
    assert sum(k["ms"] for k in kernels.values()) <= st["ms"]  # a second start counts
    assert sum(k["launches"] for k in kernels.values()) <= st["kernel_launches"]
    return st, {k for k in kernels if k.startswith(("bit_gather", "bit_scatter"))}, \
        {k for k in kernels if k.startswith(("join", "pwarp", "cross"))}


def _forest(n, chain, seed):
    """Trees (or chains) of 40 nodes over n nodes."""
    i = np.arange(n, dtype=np.uint32)
    k = i[i % 40 != 0]
    up = np.ones(len(k), np.uint32) if chain else (k % 40) - W.stream(seed).below(len(k), k % 40)
    return k - up, k


@pytest.mark.parametrize("name,n,chain", [("left", 60000, True), ("left", 80001, False), ("right", 70001, True),
                                          ("nonlinear", 12640, True), ("same_generation", 80001, False),
                                          ("two_rules", 33840, False), ("loops", 60000, False)])
def test_sparse_programs_keep_the_general_path(name, n, chain):
    """Few facts over many values: no product of matrices is formed, and the relations
    and statistics are those of bit_matrix = 0."""
    inputs = {"edge": (_forest(n, chain, 7600),)}
    assert not _profiled(PROGRAMS[name], inputs, 1)[1]
    same_as_general(PROGRAMS[name], inputs)


@pytest.mark.parametrize("name,n,m", [("left", 45000, 54000), ("right", 60000, 70000), ("same_generation", 50001, 0),
                                      ("left", 70000, 60000)])
def test_programs_run_on_matrices_from_the_start(name, n, m):
    """Many facts over many values, or few in few rows and many iterations, as the
    count of walks tells: matrices only."""
    edges = W.erdos_renyi(n, m, seed_index=7601) if m else W.random_tree(n, seed_index=7602)[:2]
    st, bits, joins = _profiled(PROGRAMS[name], {"edge": (edges,)}, 1)
    assert bits and not joins
    want, none, _ = _profiled(PROGRAMS[name], {"edge": (edges,)}, 0)
    assert not none and all(st[k] == want[k] for k in ("iterations", "derived", "candidates", "new_facts"))


@pytest.mark.parametrize("name,n", [("nonlinear", 14000), ("mutual", 40000)])
def test_programs_that_turn_out_dense_start_again_on_matrices(name, n):
    """Programs whose walks are not counted: general until they are about to derive a
    32nd of the pairs.  The closure's pairs are those of the left-recursive rule."""
    inputs = {"edge": (W.erdos_renyi(n, int(1.3 * n), seed_index=7603),)}
    st, bits, joins = _profiled(PROGRAMS[name], inputs, 1)
    assert bits and joins
    if name == "nonlinear":
        assert st["derived"] == _profiled(PROGRAMS["left"], inputs, 1)[0]["derived"]
    else:
        want = _profiled(PROGRAMS[name], inputs, 0)[0]
        assert all(st[k] == want[k] for k in ("iterations", "derived", "candidates", "new_facts"))


def test_matrices_are_bounded_in_all():
    """15 derived relations over 32,700 values, each read both ways: 75 matrices of 134
    MB.  The general path runs instead, in a fraction of that."""
    text = "r0(x,y) :- edge(x,y).\n" + "".join(
        f"r{i}(x,z) :- r{i - 1}(x,y), edge(y,z).\nr{i}(x,z) :- r{i - 1}(y,x), edge(y,z).\n" for i in range(1, 15))
    i = np.arange(32700 // 2, dtype=np.uint32)
    e, st, _ = engine_run(text, {"edge": ((2 * i, 2 * i + 1),)}, read=[])
    assert st["peak_bytes"] < 4 << 30
    assert e.size("r0") == len(i)
    e.close()


POINTS_TO = ("pt(p,q) :- addr(p,q).\npt(p,q) :- assign(p,r), pt(r,q).\npt(p,q) :- load(p,r), pt(r,s), pt(s,q).\n"
             "pt(r,q) :- store(p,s), pt(p,r), pt(s,q).\n")


@pytest.mark.parametrize("name,n", [(name, n) for name in ("nonlinear", "four_atoms", "loops", "points_to")
                                    for n in (4200, 5000, 12200)] + [("four_atoms", 13000)])
def test_products_of_derived_relations_over_many_values(name, n):
    """Rules that join derived relations over more than 4,096 values (several chunks of
    a row) and over listed matrices (12,200): index rows in bits over temporaries,
    transposed full sets, skipped arms, rows that no later product reads.  On 13,000
    values the general path starts, cannot hold a hub's join, and gives up."""
    s = W.stream(7700 + n)
    if name == "points_to":
        stmt = lambda m: (s.below(m, n), s.below(m, n))
        inputs = {"addr": ((s.below(n, n), s.below(n, n)),), "assign": (stmt(n // 3),), "load": (stmt(n // 20),),
                  "store": (stmt(n // 20),)}
        program = POINTS_TO
    else:
        parent, child, _ = W.random_tree(n, seed_index=7701)
        hub, leaf = np.full(560, 5, np.uint32), s.below(560, n)
        inputs = {"edge": ((np.concatenate([parent, hub]), np.concatenate([child, leaf])),)}
        program = PROGRAMS[name]
    e, _, _ = engine_run(program, inputs, options={"profile": 1}, read=[])
    assert "bit_gather" in e.profile()
    e.close()
    if name != "four_atoms":
        same_as_general(program, inputs)
        return
    # (on 12,200 values the general path would need 393 GB for the bindings of a step)
    import torch
    edge = torch.zeros((n, n), device="cuda")
    edge[tuple(torch.from_numpy(c.astype(np.int64)).cuda() for c in inputs["edge"][0])] = 1.0
    path, size = edge, -1
    while int(path.sum(dtype=torch.float64)) != size:
        size = int(path.sum(dtype=torch.float64))
        step = edge
        for m in (path.T, edge, path):
            step = ((step @ m) > 0).float()
        path = torch.maximum(path, step)
    e, st, got = engine_run(program, inputs, read=["path"])
    e.close()
    assert np.array_equal(got["path"].cols.astype(np.int64), torch.nonzero(path).T.cpu().numpy())
