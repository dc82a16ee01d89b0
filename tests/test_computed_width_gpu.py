"""Key widths of computed columns: bounded by the rules' comparisons, whatever
their form, and any u32 where nothing bounds them or arithmetic can wrap."""
import numpy as np
import pytest

from paper_2503_21937_gb300 import workloads as W
from tests.common import compare

pytestmark = pytest.mark.gpu

HOP = "hop(x,y,1) :- edge(x,y).\nhop(x,z,d + 1) :- hop(x,y,d), edge(y,z), {}.\n"
PROGRAMS = {
    "below_1": (HOP.format("d < 1"), "hop"), "below_3": (HOP.format("d < 3"), "hop"), "below_4": (HOP.format("d < 4"), "hop"),
    "at_most": (HOP.format("d <= 6"), "hop"), "above": (HOP.format("7 > d"), "hop"), "at_least": (HOP.format("7 >= d"), "hop"),
    "computed": (HOP.format("d * 2 < 11"), "hop"),  # a bound that is not taken: any u32
    "twice": ("n(x,y) :- edge(x,y).\nn(x,d * 2 + 1) :- n(x,d), d < 100.\n", "n"),
    "down": ("n(x,y) :- edge(x,y).\nn(x,d - 1) :- n(x,d), d > 2.\n", "n"),
    "wraps": ("n(x,y) :- edge(x,y).\nn(x,d - 3) :- n(x,d), d < 9.\n", "n"),  # 2 - 3 is 2^32 - 1 and dropped
    "divides": ("n(x,y) :- edge(x,y).\nn(x,100 / d) :- n(x,d), d < 50.\n", "n"),  # 100 / 0 drops the row
    "onwards": ("a(x,d + 1) :- edge(x,d), d < 5.\nn(x,d * d) :- a(x,d).\nn(d,x + 1) :- n(x,d), x < 20.\n", "n"),
}


@pytest.mark.parametrize("semiring", ["unit", "max_min", "diff_add_mult"])
@pytest.mark.parametrize("name", list(PROGRAMS))
def test_bounds_of_computed_columns(name, semiring):
    s = W.stream(970)
    edge = (s.below(90, 30), s.below(90, 30))
    p = (s.prob(90) * 0.3).astype(np.float32)
    text, rel = PROGRAMS[name]
    compare(text, {"edge": (edge, p if semiring != "unit" else None)}, semiring, rels=[rel])


@pytest.mark.parametrize("bitmap_delta", [1, 2])
def test_rows_a_filter_drops_set_no_bit(bitmap_delta):
    """One-atom rules with a comparison under the unit semiring: the dropped rows'
    all-ones keys are not keys of the membership bitmap."""
    s = W.stream(971)
    edge = (s.below(200, 60), s.below(200, 60))
    text = "p(x,y) :- edge(x,y), x < 40.\np(y,x) :- p(x,y), y < 30.\n"
    compare(text, {"edge": (edge, None)}, "unit", options={"bitmap_delta": bitmap_delta, "emit_filter": 2})
