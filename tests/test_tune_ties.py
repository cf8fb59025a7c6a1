"""Which timings the tile tuner takes as ties (no GPU)."""

import pytest

from paper_1712_07973_gb300 import tune


# (ms per call by tile edge, choice): the fastest wherever a call's time is told
# apart from the scatter of its launches, however small the share; else the larger
@pytest.mark.parametrize("timings,best", [
    ({6: 28.6, 8: 31.2}, 6), ({6: 31.2, 8: 31.3}, 6), ({4: 4.49, 8: 4.50}, 4), ({2: 0.9, 6: 0.300, 8: 0.310}, 6),
    ({6: 0.0425, 8: 0.0426}, 8), ({6: 0.0414, 8: 0.0449}, 8), ({4: 0.050, 6: 0.0425, 8: 0.0500}, 6),
    ({6: 1.0, 8: 1.005}, 8), ({6: 1.0, 8: 1.007}, 6),
])
def test_ties_are_the_scatter_of_short_calls(timings, best):
    assert tune.select(timings) == best
