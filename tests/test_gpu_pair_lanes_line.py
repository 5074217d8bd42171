"""The lanes that share a particle's walk around the line between 8 and 32 (the
particles over the candidates expected in a stencil row) and where counts keep
one: the checks and tolerances of tests/test_gpu_pair_lanes.py on sizes to both
sides (GPU, C ABI)."""
import pytest

import test_gpu_pair_lanes as lanes
from test_gpu_pair_lanes import ab  # noqa: F401

pytestmark = pytest.mark.gpu

# dim, n, mean neighbours, periodic, blobs
CASES = {
    "below_2d": (2, 14001, 180.0, (1, 1), 0),
    "above_2d": (2, 20001, 180.0, (1, 0), 0),
    "below_3d": (3, 12001, 260.0, (1, 1, 1), 0),
    "above_3d": (3, 30011, 220.0, (1, 0, 1), 0),
    "counts_below": (2, 196608, 20.0, (1, 1), 0),
    "counts_above": (2, 196609, 20.0, (1, 1), 0),
}


@pytest.mark.parametrize("name", list(CASES))
def test_values_and_adjoints(ab, cuda, monkeypatch, name):  # noqa: F811
    monkeypatch.setitem(lanes.CASES, name, CASES[name])
    lanes.test_values_and_adjoints(ab, cuda, name)
