"""The tuner can reach what it is said to have found."""
import pytest

from paper_2505_15771_gb300 import tune


@pytest.mark.parametrize("arith", sorted(tune.TABLE))
def test_committed_entries_lie_on_the_axes(arith):
    tables = tune.read_tables(open(tune.HEADER).read())
    for field in tune.FIELDS:
        assert set(tables[arith][field]) <= set(tune.AXES[field]), field
