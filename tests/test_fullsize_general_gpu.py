"""The unit semiring's general path (option bit_matrix = 0, every other option at its
default) at the benchmark's full sizes: relations equal to those of the bit matrices,
which tests/test_fullsize_gpu.py checks against closed forms and textbook
computations, and the same-generation count against its closed form."""
import numpy as np
import pytest

from paper_2503_21937_gb300 import workloads as W
from tests import pins

pytestmark = pytest.mark.gpu


def _run(program, inputs, on):
    import torch
    from paper_2503_21937_gb300 import Engine
    e = Engine()
    e.program(program)
    e.set_option("bit_matrix", on)
    for name, cols in inputs.items():
        e.load(name, torch.from_numpy(np.stack(cols).astype(np.int32)).cuda())
    return e, e.run("unit")


@pytest.mark.parametrize("name", ["same_generation", "closure", "points_to"])
def test_general_path_at_full_size(name):
    import torch
    if name == "same_generation":
        parent, child, depth = W.random_tree(50_000)
        program, inputs, rel = W.SG_PROGRAM, {"parent": (parent, child)}, "sg"
    elif name == "closure":
        program, inputs, rel = W.TC_PROGRAM, {"edge": W.chung_lu_power_law(20_000, 100_000)}, "path"
    else:
        A = W.andersen_program(200_000, 400_000)
        program, inputs, rel = W.ANDERSEN_PROGRAM, {k: (v[0], v[1]) for k, v in A.items()}, "pt"
    e, st = _run(program, inputs, 0)
    general = e.read(rel, device=True).cols.clone()
    e.close()
    if name == "same_generation":
        assert general.shape[1] == pins.same_generation_closed_form(depth)
    e, sb = _run(program, inputs, 1)
    assert torch.equal(e.read(rel, device=True).cols, general)
    for k in ("iterations", "derived", "candidates", "new_facts"):
        assert st[k] == sb[k], k
    e.close()
