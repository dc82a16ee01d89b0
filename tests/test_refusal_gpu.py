"""Device memory refused on the host side (no GPU fault): a run that loses any one
of its requests ends with the right relations or a clean LOB_E_OOM."""
import numpy as np
import pytest

from paper_2503_21937_gb300 import workloads as W
from tests.common import oracle_run

pytestmark = pytest.mark.gpu


class Refusing:
    """An allocator that refuses the request numbered `at` (from 1, counted while
    armed), and every one that would take more than `budget` bytes in all."""

    def __init__(self):
        self.live, self.armed, self.at, self.seen, self.refused = {}, False, 0, 0, 0
        self.held, self.peak, self.budget = 0, 0, 1 << 62

    def alloc(self, nbytes, stream):
        import torch
        self.seen += self.armed
        if self.armed and (self.seen == self.at or self.held + nbytes > self.budget):
            self.refused += 1
            return 0
        p = torch.cuda.caching_allocator_alloc(nbytes, stream=stream)
        self.live[p] = nbytes
        self.held += nbytes
        self.peak = max(self.peak, self.held)
        return p

    def release(self, p, nbytes, stream):
        import torch
        self.held -= self.live.pop(p)
        torch.cuda.caching_allocator_delete(p)

    def arm(self, at=0):
        self.armed, self.at, self.seen, self.refused = True, at, 0, 0


def loaded_engine(program, inputs, options, A):
    from paper_2503_21937_gb300 import Engine
    e = Engine(allocator=(A.alloc, A.release))
    e.program(program)
    for k, v in options.items():
        e.set_option(k, v)
    for name, spec in inputs.items():
        e.load(name, *spec)
    return e


NONLINEAR = "path(x,y) :- edge(x,y).\npath(x,z) :- path(x,y), path(y,z).\n"
SAME_GENERATION = "path(x,y) :- edge(p,x), edge(p,y), x != y.\npath(x,y) :- edge(a,x), path(a,b), edge(b,y).\n"


@pytest.mark.parametrize("loaded", [False, True])
@pytest.mark.parametrize("program,n", [(W.TC_PROGRAM, 60), (NONLINEAR, 60), (SAME_GENERATION, 60), (W.TC_PROGRAM, 5000)])
def test_bit_matrices_with_a_request_refused(program, n, loaded):
    """Every single request of a run on bit matrices refused in turn, in the one-launch
    form (60 values) and the queued one (5,000, renumbered): the general path takes
    over from the loaded facts.  After an LOB_E_OOM the engine runs again."""
    from paper_2503_21937_gb300 import LobsterError
    s = W.stream(7500)
    m, scale = (80, 1) if n == 60 else (4000, 7)
    a, b, c, d = (s.below(m, n) * np.uint32(scale) for _ in range(4))
    inputs = {"edge": ((a, b),)}
    if loaded:
        inputs["path"] = ((c[:9], d[:9]),)
    want = oracle_run(program, inputs).relation("path").cols
    clean, at = False, 0
    while not clean:
        at += 1
        A = Refusing()
        e = loaded_engine(program, inputs, {}, A)
        A.arm(at)
        try:
            e.run("unit")
        except LobsterError as x:
            assert x.code == -5
            A.armed = False
            e.run("unit")
        clean = not A.refused
        A.armed = False
        assert np.array_equal(e.read("path").cols, want), at
        e.close()
        assert not A.live
    assert at > 12  # the run made at least that many requests


HOPS = "hop(x,y,1) :- edge(x,y).\nhop(x,z,d + 1) :- hop(x,y,d), edge(y,z), d < 4.\n"


def _tagged(kind):
    s = W.stream(7600)
    if kind == "kinship":  # masked last steps
        n, r, a, b, p = W.kinship_instance(s)
        return W.KIN_PROGRAM, {"fact": ((r, a, b), p), "comp": (W.composition_table(),)}, "kin", "fact"
    if kind == "grid":  # a linear component
        g = W.grid_reach_instance(9, sub=761)
        return W.REACH_PROGRAM, {"edge": (g["edge"][:2], g["edge"][2]), "start": (g["start"],)}, "reach", "edge"
    src, dst = W.erdos_renyi(40, 90, seed_index=762)  # a computed column of few bits
    return HOPS, {"edge": ((src, dst), s.prob(90))}, "hop", "edge"


@pytest.mark.parametrize("kind,semiring,options", [
    ("kinship", "max_min", {"driver": 0}), ("kinship", "diff_add_mult", {"driver": 0}), ("kinship", "diff_max_min", {"driver": 2}),
    ("grid", "max_min", {"driver": 2}), ("grid", "diff_add_mult", {"driver": 2}),
    ("grid", "diff_top1_proofs", {"driver": 2, "proof_arena_words": 256}), ("hops", "max_min", {"driver": 0})])
def test_tagged_runs_with_a_request_refused(kind, semiring, options):
    """Every single request of a run refused in turn.  Once the run has a use for
    memory that it could do without, the refusal costs it only that; before, it is an
    LOB_E_OOM after which the engine runs again.  Tags are compared with those of a
    run that lost nothing (add-mult: FP64 sums in another order, rounded once)."""
    from paper_2503_21937_gb300 import LobsterError
    program, inputs, rel, _ = _tagged(kind)
    want, lost, kept, at = None, [], [], 0
    while True:
        A = Refusing()
        e = loaded_engine(program, inputs, options, A)
        A.arm(at)
        try:
            e.run(semiring)
            if A.refused:
                kept.append(at)
        except LobsterError as x:
            assert x.code == -5
            lost.append(at)
            A.armed = False
            e.run(semiring)
        refused, A.armed = A.refused, False
        r = e.read(rel)
        e.close()
        assert not A.live
        if want is None:  # the first run loses nothing
            assert not refused
            want = r
        assert np.array_equal(r.cols, want.cols), at
        np.testing.assert_allclose(r.tags, want.tags, rtol=3e-7 if "add" in semiring else 0, atol=0)
        if at and not refused:
            break
        at += 1
    assert len(kept) > 5 and (not lost or max(lost) < min(kept)), (lost, kept)
    if kind != "grid":
        assert not lost


@pytest.mark.parametrize("kind", ["kinship", "grid"])
def test_backward_with_a_request_refused(kind):
    """Every single request of an add-mult backward pass refused in turn: the pass
    ends without what it could do without, or with LOB_E_OOM and the gradients as
    they were.  Gradients within the order of their FP64 sums, rounded to f32."""
    from paper_2503_21937_gb300 import LobsterError
    program, inputs, rel, grad = _tagged(kind)
    A = Refusing()
    e = loaded_engine(program, inputs, {"driver": 2}, A)
    e.run("diff_add_mult")
    seed = np.linspace(-1, 1, e.size(rel)).astype(np.float32)
    want, lost, kept, at = None, [], [], 0
    while True:
        g = np.zeros(len(inputs[grad][1]), np.float32)
        A.arm(at)
        try:
            e.backward(rel, seed, {grad: g})
            if A.refused:
                kept.append(at)
        except LobsterError as x:
            assert x.code == -5 and not g.any()
            lost.append(at)
            A.armed = False
            e.backward(rel, seed, {grad: g})
        refused, A.armed = A.refused, False
        want = g if want is None else want
        np.testing.assert_allclose(g, want, rtol=1e-6, atol=1e-6 * float(np.abs(want).max()))
        if at and not refused:
            break
        at += 1
    e.close()
    assert not A.live
    assert len(kept) > 2 and max(lost) < min(kept), (lost, kept)
