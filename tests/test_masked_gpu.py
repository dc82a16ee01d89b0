"""Masked last join steps (tagged semirings: the last probe leaves one column
of at most 6 bits free) against the oracle and against the general kernels:
row widths from 1 to 6 bits and just past, filters, transposed and constant
head columns, samples, old-fact arms, gradients, both iteration drivers."""
import numpy as np
import pytest

from paper_2503_21937_gb300 import workloads as W
from tests.common import compare, engine_run

pytestmark = pytest.mark.gpu

PROGRAMS = {
    "nonlinear": "p(x,y) :- e(x,y).\np(x,z) :- p(x,y), p(y,z).\n",
    "transposed": "p(x,y) :- e(x,y).\np(z,x) :- p(x,y), p(y,z), x != z.\n",
    "constant": "p(x,y) :- e(x,y).\nq(7,z) :- p(x,y), p(y,z).\nq(z,3) :- q(x,y), e(x,z).\n",
    "three": "p(x,y) :- e(x,y).\np(x,w) :- p(x,y), e(y,z), p(z,w), x != w.\n",
}


def _facts(n, m, seed, scale):
    s = W.stream(seed)
    return s.below(m, n), s.below(m, n), (s.prob(m) * scale).astype(np.float32)


@pytest.mark.parametrize("name", list(PROGRAMS))
@pytest.mark.parametrize("n", [2, 3, 7, 15, 31, 33, 62, 63, 64])
def test_row_widths(name, n):
    a, b, p = _facts(n, 2 * n + 3, 900 + n, 0.3)
    p[:: 5] = 0.0  # a fact of tag 0 is a fact
    for semiring in ("add_mult", "max_min", "diff_max_min"):
        for driver in (0, 2):
            compare(PROGRAMS[name], {"e": ((a, b), p)}, semiring, options={"driver": driver})


@pytest.mark.parametrize("semiring", ["add_mult", "diff_add_mult", "max_min", "diff_max_min"])
@pytest.mark.parametrize("program", ["kinship", "nonlinear", "three"])
def test_same_as_the_general_kernels(program, semiring):
    """Statistics equal, tags within the reordering of FP64 sums rounded once to
    f32, gradients within 1e-4 (as against the oracle)."""
    if program == "kinship":
        B = W.batched_instance(40)
        f, c = B["fact"], B["comp"]
        text, rel, grad = W.KIN_PROGRAM, "kin", "fact"
        inputs = {"fact": (f[:3], f[3], f[4]), "comp": (c[:3], None, c[4])}
    else:
        a, b, p = _facts(60, 200, 950, 0.2)
        sid = (np.arange(200) % 3).astype(np.uint32)
        text, rel, grad = PROGRAMS[program], "p", "e"
        inputs = {"e": ((a, b), p, sid), "p": ((b[:9], a[:9]), p[:9], sid[:9])}
    runs = []
    for opts in ({"packed_join": 0, "driver": 0}, {"driver": 0}, {"driver": 2}):
        e, st, got = engine_run(text, inputs, semiring, options=opts, read=[rel])
        g = np.zeros(len(inputs[grad][0][0]), np.float32)
        if semiring.startswith("diff"):
            e.backward(rel, np.linspace(-1, 1, got[rel].cols.shape[1]).astype(np.float32), {grad: g})
        e.close()
        runs.append((st, got[rel], g))
    (a, ra, ga) = runs[0]
    for st, r, g in runs[1:]:
        for k in ("iterations", "derived", "candidates", "new_facts"):
            assert st[k] == a[k], (k, st[k], a[k])
        assert np.array_equal(r.cols, ra.cols) and np.array_equal(r.samples, ra.samples)
        np.testing.assert_allclose(r.tags, ra.tags, rtol=3e-7 if "add" in semiring else 0, atol=0)
        np.testing.assert_allclose(g, ga, rtol=1e-4, atol=1e-5 * max(1.0, float(np.abs(ga).max())))


@pytest.mark.parametrize("semiring", ["max_min", "diff_max_min"])
@pytest.mark.parametrize("rows", [1, 33, 255, 257, 152 * 256 + 1, 152 * 4096 - 1, 152 * 4096 + 41])
def test_rows_grouped_by_head(rows, semiring):
    """Input rows just past the smallest tiles, one wave of full tiles and two
    waves; heads of 64 rows (two items) and of one."""
    s = W.stream(960)
    i = np.arange(rows, dtype=np.uint32)
    a = (i // 64, i % 64)
    if rows > 64:
        a[0][-3:], a[1][-3:] = rows + np.arange(3), 5  # heads of a single row
    b = (s.below(700, 64), s.below(700, 50))
    inputs = {"a": (a, s.prob(rows)), "b": (b, s.prob(700))}
    text = "q(x,z) :- a(x,y), b(y,z), y != z.\n"
    got = []
    for opts in ({"packed_join": 0}, {}):
        e, st, g = engine_run(text, inputs, semiring, options=opts, read=["q"])
        e.close()
        got.append((st, g["q"]))
    (x, p), (y, q) = got
    for k in ("iterations", "derived", "candidates", "new_facts"):
        assert x[k] == y[k], (k, x[k], y[k])
    assert np.array_equal(p.cols, q.cols) and np.array_equal(p.tags, q.tags)


@pytest.mark.parametrize("semiring", ["max_min", "diff_max_min"])
@pytest.mark.parametrize("rows", [1, 33, 255, 257, 152 * 256 + 1, 152 * 4096 - 1, 152 * 4096 + 41])
def test_rows_of_a_derived_relation_grouped_by_head(rows, semiring):
    """The masked step with exactly `rows` input rows: the delta atom is derived, so
    that the step of iteration 2 is a masked one (a rule over input relations alone,
    as in the test before, never is), and the loop in one launch is off.  Rows just
    past the smallest tiles, one wave of full tiles and two waves; heads of 64 rows
    (two items) and of one."""
    s = W.stream(961)
    i = np.arange(rows, dtype=np.uint32)
    a = (i // 64, i % 64)
    if rows > 64:
        a[0][-3:], a[1][-3:] = rows + np.arange(3), 5  # heads of a single row
    b = (s.below(700, 64), s.below(700, 50))
    inputs = {"a": (a, s.prob(rows)), "b": (b, s.prob(700))}
    text = "p(x,y) :- a(x,y).\nq(x,z) :- p(x,y), b(y,z), y != z.\n"
    got = []
    for opts in ({"packed_join": 0, "driver": 0}, {"driver": 0, "profile": 1}):
        e, st, g = engine_run(text, inputs, semiring, options=opts, read=["q"])
        got.append((st, g["q"], e.profile()))
        e.close()
    (x, p, _), (y, q, kernels) = got
    assert kernels["join_masked"]["launches"] == 1
    for k in ("iterations", "derived", "candidates", "new_facts"):
        assert x[k] == y[k], (k, x[k], y[k])
    assert np.array_equal(p.cols, q.cols) and np.array_equal(p.tags, q.tags)
