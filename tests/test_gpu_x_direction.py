"""Maps whose lines move more than two columns per k row (every row differenced along x0), with one
count per cell and with two: rows beside a tile's, lines wider than a tile apart, both signs of k.  Every
map cell, candidate and statistic equals the oracle's (whole numbers: no tolerance)."""
import pytest

torch = pytest.importorskip("torch")

from test_gpu_hough_events import fields_of
from test_gpu_sparse import check

pytestmark = pytest.mark.gpu

CASES = {
    "sparse": fields_of(5.0, 150, 300, 24, 37, dk_cols=5.0),
    "dense": fields_of(5.0, 200, 150, 500, 61, dk_cols=5.0),
    "just_over": fields_of(4.0, 200, 150, 200, 16, dk_cols=2.1),
    "far": fields_of(5.0, 200, 100, 60, 9, dk_cols=700.0),
    "both_signs": fields_of(0.0, 300, 90, 150, 50, dk_cols=3.0, k_min_rows=-25.0),
    "one_row": fields_of(5.0, 200, 100, 60, 1, dk_cols=5.0, k_min_rows=40.0),
}


@pytest.mark.parametrize("tile", [None, (4, 1024, 256), (32, 1024, 1024)], ids=str)
@pytest.mark.parametrize("name", sorted(CASES))
def test_maps_equal_the_oracle(built_lib, gpu_ctx, name, tile):
    check(built_lib, gpu_ctx, [CASES[name]], tile)


def test_both_forms_in_one_plan(built_lib, gpu_ctx):
    check(built_lib, gpu_ctx, [dict(CASES["dense"], list=0), dict(fields_of(5.0, 200, 150, 200, 60), list=1),
                               dict(CASES["sparse"], list=2)], None)
