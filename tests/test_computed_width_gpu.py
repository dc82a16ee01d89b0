"""Rules with comparisons over one atom under the unit semiring."""
import pytest

from paper_2503_21937_gb300 import workloads as W
from tests.common import compare

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bitmap_delta", [1, 2])
def test_rows_a_filter_drops_set_no_bit(bitmap_delta):
    """One-atom rules with a comparison under the unit semiring: the dropped rows'
    all-ones keys are not keys of the membership bitmap."""
    s = W.stream(971)
    edge = (s.below(200, 60), s.below(200, 60))
    text = "p(x,y) :- edge(x,y), x < 40.\np(y,x) :- p(x,y), y < 30.\n"
    compare(text, {"edge": (edge, None)}, "unit", options={"bitmap_delta": bitmap_delta, "emit_filter": 2})
