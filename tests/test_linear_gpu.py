"""Linear components of tagged programs in one launch (option driver = 2, from
the first run on) against the oracle and against the host-driven loop
(driver = 0): relations, tags, iterations, candidates, new facts, gradients."""
import numpy as np
import pytest

from paper_2503_21937_gb300 import workloads as W
from tests.common import compare, engine_run

pytestmark = pytest.mark.gpu

SEMIRINGS = ["max_min", "add_mult", "diff_max_min", "diff_add_mult"]
TURNS = ("a(x) :- start(x).\nb(y) :- a(x), edge(x,y).\na(y) :- b(x), edge(x,y), x != y.\n")
TAILED = W.REACH_PROGRAM + "pair(x,y) :- edge(x,y).\npair(x,z) :- pair(x,y), pair(y,z), x != z.\n"


def both(program, inputs, semiring, rels, grad=None, max_iters=1 << 30):
    """driver 2 and driver 0: same statistics and relations; add-mult tags agree
    within the reordering of FP64 sums rounded once to f32 (1 ulp = 1.2e-7)."""
    runs = []
    for driver in (2, 0):
        e, st, got = engine_run(program, inputs, semiring, options={"driver": driver}, read=rels, max_iters=max_iters)
        g = None
        if grad:
            g = np.zeros(len(inputs[grad][0][0]), np.float32)
            for r in rels:
                e.backward(r, np.linspace(-1, 1, got[r].cols.shape[1]).astype(np.float32), {grad: g})
        e.close()
        runs.append((st, got, g))
    (a, ga, da), (b, gb, db) = runs
    for k in ("iterations", "derived", "candidates", "new_facts"):
        assert a[k] == b[k], (k, a[k], b[k])
    for r in rels:
        assert np.array_equal(ga[r].cols, gb[r].cols) and np.array_equal(ga[r].samples, gb[r].samples)
        if "add_mult" in semiring:
            np.testing.assert_allclose(ga[r].tags, gb[r].tags, rtol=3e-7, atol=0)
        else:
            assert np.array_equal(ga[r].tags, gb[r].tags)
    if grad:
        np.testing.assert_allclose(da, db, rtol=1e-4, atol=1e-5 * max(1.0, float(np.abs(db).max())))
    return a


@pytest.mark.parametrize("semiring", SEMIRINGS)
@pytest.mark.parametrize("side", [1, 2, 3, 17])
def test_grids_against_the_oracle(semiring, side):
    g = W.grid_reach_instance(side, sub=801)
    src, dst, p = g["edge"]
    if side == 1:
        src, dst, p = np.array([0], np.uint32), np.array([0], np.uint32), np.array([0.5], np.float32)
    compare(W.REACH_PROGRAM, {"edge": ((src, dst), p), "start": (g["start"],)}, semiring, options={"driver": 2})


@pytest.mark.parametrize("semiring", SEMIRINGS)
def test_mutually_recursive_and_two_column_relations(semiring):
    s = W.stream(802)
    src, dst, p = s.below(150, 40), s.below(150, 40), (s.prob(150) * 0.4).astype(np.float32)
    start = ((np.array([3, 9], np.uint32),), np.array([0.25, 0.75], np.float32))
    inputs = {"edge": ((src, dst), p), "start": start}
    st, _ = compare(TURNS, inputs, semiring, options={"driver": 2})
    assert st["device_iterations"] > 0 and st["graph_launches"] == 1
    compare(W.TC_PROGRAM, {"edge": ((src, dst), p)}, semiring, options={"driver": 2})
    # facts loaded into the derived relation as well
    loaded = {"edge": ((src, dst), p), "path": ((dst[:20], src[:20]), p[:20])}
    compare(W.TC_PROGRAM, loaded, semiring, options={"driver": 2})


@pytest.mark.parametrize("semiring", SEMIRINGS)
def test_linear_component_beside_a_nonlinear_one(semiring):
    """Two components of one program: the linear one in its own launch, the
    other by the graph or the host; batched samples of uneven size."""
    B = W.batched_instance(7, side_lo=3, side_hi=13)
    e, st, f, c = B["edge"], B["start"], B["fact"], B["comp"]
    inputs = {"edge": (e[:2], e[2], e[3]), "start": ((st[0],), None, st[2]), "fact": (f[:3], f[3], f[4]),
              "comp": (c[:3], None, c[4])}
    diff = semiring.startswith("diff")
    both(W.REACH_PROGRAM + W.KIN_PROGRAM, inputs, semiring, ["reach", "kin"])
    both(W.REACH_PROGRAM, {k: inputs[k] for k in ("edge", "start")}, semiring, ["reach"], "edge" if diff else None)
    s = W.stream(803)
    src, dst, p = s.below(60, 30), s.below(60, 30), (s.prob(60) * 0.3).astype(np.float32)
    both(TAILED, {"edge": ((src, dst), p), "start": ((src[:1],),)}, semiring, ["reach", "pair"], "edge" if diff else None)


@pytest.mark.parametrize("semiring", SEMIRINGS)
def test_several_blocks_and_a_hub(semiring):
    """200,000 input facts (12 blocks and their barrier), one of the nodes with
    3,000 neighbours."""
    s = W.stream(804)
    n = 30000
    src = np.concatenate([s.below(200000, n), np.full(3000, 7, np.uint32)])
    dst = np.concatenate([s.below(200000, n), s.below(3000, n)])
    p = (s.prob(len(src)) * 0.2).astype(np.float32)
    inputs = {"edge": ((src, dst), p), "start": ((np.array([7, 11], np.uint32),),)}
    both(W.REACH_PROGRAM, inputs, semiring, ["reach"], "edge" if semiring.startswith("diff") else None)


def _proofs(program, inputs, rels, options):
    e, st, got = engine_run(program, inputs, "diff_top1_proofs", options=options, read=rels)
    out = [(got[r].cols, got[r].samples, got[r].tags, [list(p) for p in e.proofs(r)]) for r in rels]
    e.close()
    return st, out


@pytest.mark.parametrize("program,rels", [(W.REACH_PROGRAM, ["reach"]), (TURNS, ["a", "b"]), (W.TC_PROGRAM, ["path"])])
@pytest.mark.parametrize("n,m,words,lo,hi", [(6, 9, 1 << 22, 0.0, 1.0), (40, 150, 1 << 22, 0.0, 1.0), (40, 150, 64, 0.5, 1.0),
                                             (300, 7000, 1 << 22, 0.9, 1.0), (64, 63, 1 << 22, 0.9, 1.0),
                                             (64, 63, 256, 0.0, 0.01), (12, 30, 1 << 22, 1.0, 1.3)])
def test_proofs_of_linear_components(program, rels, n, m, words, lo, hi):
    """The likeliest proof of every fact (driver 2) against the general steps
    (driver 0): tags bit for bit, the same proofs, iterations and candidates.
    m = n - 1: a chain, proofs of up to 63 facts; a small arena runs out and the
    loop runs again; tags that underflow, tags of 0, probabilities above 1."""
    s = W.stream(810 + n)
    src, dst = (np.arange(m, dtype=np.uint32), np.arange(1, m + 1, dtype=np.uint32)) if m == n - 1 else (s.below(m, n), s.below(m, n))
    p = (lo + (hi - lo) * s.prob(m)).astype(np.float32)
    if lo == 0.0:
        p[::7] = 0.0
    inputs = {"edge": ((src, dst), p), "start": ((np.array([0, 3], np.uint32),), np.array([0.5, 0.75], np.float32))}
    if program is W.TC_PROGRAM:
        inputs.pop("start")
        if m > 1000:
            return
    (a, ga), (b, gb) = (_proofs(program, inputs, rels, {"driver": d, "proof_arena_words": words}) for d in (2, 0))
    assert a["device_iterations"] > 0 and b["device_iterations"] == 0
    for k in ("iterations", "derived", "candidates", "new_facts"):
        assert a[k] == b[k], (k, a[k], b[k])
    for x, y in zip(ga, gb):
        assert np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1])
        assert np.array_equal(x[2].view(np.uint32), y[2].view(np.uint32))
        likely = x[2] > 0.0  # proofs of probability 0 tie; the others have distinct probabilities
        assert [q for q, t in zip(x[3], likely) if t] == [q for q, t in zip(y[3], likely) if t]


@pytest.mark.parametrize("driver", [0, 2])
def test_proof_cap_in_the_linear_loop(driver):
    """A chain of nine facts below 0.5: a cap of seven is an error, of eight is not."""
    from paper_2503_21937_gb300 import LobsterError
    a, b = W.ktree_chain(9)
    inputs = {"edge": ((a, b), np.full(8, 0.5, np.float32)), "start": ((np.array([0], np.uint32),),)}
    with pytest.raises(LobsterError) as ei:
        engine_run(W.REACH_PROGRAM, inputs, "top1_proofs", options={"driver": driver, "proof_cap": 7})
    assert ei.value.code == -9
    _, st, got = engine_run(W.REACH_PROGRAM, inputs, "top1_proofs", options={"driver": driver, "proof_cap": 8})
    assert got["reach"].tags.tolist() == [0.5 ** k for k in range(9)]


def test_backward_replays_only_what_the_output_depends_on():
    """Two components that share no rule: the backward pass of one leaves the other's
    launch out, and gives the same gradients as in a program of its own.  An arm over
    an input relation, all of whose facts are recent, sorts nothing by stamp."""
    s = W.stream(805)
    src, dst, p = s.below(60, 30), s.below(60, 30), (s.prob(60) * 0.3).astype(np.float32)
    inputs = {"edge": ((src, dst), p), "start": ((src[:1],),)}
    e, _, got = engine_run(TAILED, inputs, "diff_add_mult", options={"driver": 2}, read=["reach", "pair"])
    e.set_option("profile", 1)

    def backward(en, rel):
        g = np.zeros(len(src), np.float32)
        en.profile_reset()
        en.backward(rel, np.linspace(-1, 1, en.size(rel)).astype(np.float32), {"edge": g})
        return g, en.profile()

    g, kernels = backward(e, "pair")
    assert "linear_backward" not in kernels
    assert "linear_backward" in backward(e, "reach")[1]
    e.close()
    pair = TAILED[len(W.REACH_PROGRAM):]
    e, _, _ = engine_run(pair, {"edge": inputs["edge"]}, "diff_add_mult", options={"driver": 2}, read=[])
    want = np.zeros(len(src), np.float32)
    e.backward("pair", np.linspace(-1, 1, e.size("pair")).astype(np.float32), {"edge": want})
    e.close()
    np.testing.assert_allclose(g, want, rtol=1e-6, atol=1e-6 * float(np.abs(want).max()))
    e, _, _ = engine_run("two(x,z) :- edge(x,y), edge(y,z).\n", {"edge": inputs["edge"]}, "diff_add_mult", read=[])
    e.set_option("profile", 1)
    g, kernels = backward(e, "two")
    assert g.any() and "radix_sort" not in kernels, kernels
    e.close()
