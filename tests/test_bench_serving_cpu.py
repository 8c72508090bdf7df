"""bench.py ends with an error when serving gave other residues than the same
matrices one per launch, and only then."""
import sys

import pytest

from conftest import ROOT

sys.path.insert(0, ROOT)


@pytest.mark.parametrize("line,status", [
    (None, 0), ({}, 0), ({"extra": {}}, 0), ({"extra": {"serve": {"jobs": 3}}}, 0),
    ({"extra": {"serve": {"results_identical": True}}}, 0),
    ({"extra": {"serve": {"results_identical": False}}}, 1)])
def test_exit_status_says_whether_serving_was_right(line, status, capsys):
    import bench
    assert bench.served_wrong(line) == status
    assert bool(capsys.readouterr().err) == bool(status)
