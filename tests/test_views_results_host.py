"""Results of a batch as tensors (CPU): no views give an empty list."""
from paper_2511_16298_gb300 import tdgs


def test_no_views():
    assert tdgs.Context._results(None, (tdgs._ViewResult * 0)(), 0, False) == []
    assert tdgs.Context._results(None, (tdgs._ViewResult * 0)(), 0, True) == []
