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
