"""Arena sizes: a budget that held a problem before its diagonals and reciprocals were stored still does."""
import pytest

from paper_1312_2880_gb300 import hz

# Bytes of the arena with k h alone stored (no diagonals, no reciprocals), per options and grid.
WITHOUT_STORED = [
    ({"precision": "fp64"}, {8: 1133312, 24: 1094144, 64: 2180608, 240: 16821248, 512: 59866368, 992: 267872256,
                             4096: 3681026560, 32768: 234882660096}),
    ({"precision": "fp32"}, {8: 1079808, 24: 1054208, 64: 2021120, 240: 15465216, 512: 55790848, 992: 245916928,
                             4096: 3452963072, 32768: 220531455232}),
    ({"precision": "fp64", "batch": 16}, {16: 14100224, 240: 211806464, 1024: 3554169600}),
    ({"precision": "fp64", "levels": 2}, {4: 822016, 8: 865536, 24: 2329088, 64: 58726912}),
    ({"precision": "fp64", "gs_smoother": "jacobi"}, {24: 1106944, 240: 17808384, 512: 64331520, 4096: 3951625216}),
]


@pytest.mark.parametrize("opts,sizes", WITHOUT_STORED)
def test_stored_diagonals_cost_no_arena(opts, sizes):
    for n, before in sizes.items():
        assert 0 < hz.footprint_bytes(n, **opts) <= before, n


def test_two_elimination_fronts_cost_no_ray_arena():
    for n, k, m, before in ((64, 20.0, 0, 5074432), (512, 160.0, 0, 1723697408), (1024, 320.0, 0, 13334409472),
                            (16, 20.0, 8, 210432), (2, 1.0, 1, 174592)):
        assert 0 < hz.lib().hz_ray_footprint_bytes(n, k, m) <= before, n
