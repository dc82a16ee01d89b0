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
