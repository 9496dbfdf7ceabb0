"""Projections on both sides of the rule that takes the fused pass or the mode products: every
entry, the norm, the error and the reconstruction within the rounding bounds of the sums that form
them, against the oracle."""

import pytest

import test_gpu_projection as base
from paper_2201_06958_gb300 import tdb

pytestmark = pytest.mark.gpu

DOUBLE = [
    ((51, 40), (6, 6), 0), ((52, 40), (6, 6), 0), ((53, 31), (17, 17), 1),         # two modes
    ((30, 20, 64), (5, 4, 6), 0), ((30, 20, 65), (5, 4, 6), 0),                    # the last of three
    ((40, 256, 65), (9, 17, 5), 0), ((47, 257, 65), (9, 17, 5), 0), ((48, 257, 65), (9, 17, 5), 0),   # the middle
    ((896, 4, 66), (7, 4, 5), 0), ((897, 4, 66), (7, 4, 5), 0),                    # a long first
    ((8, 33, 70), (3, 9, 5), 0), ((9, 9, 70), (3, 9, 5), 0), ((3, 9, 70), (3, 9, 5), 1),   # padding of 30 times
    ((131, 65, 66), (8, 3, 4), 0), ((128, 128, 65), (5, 5, 5), 0), ((128, 250, 66), (4, 4, 4), 1),
    ((130, 129, 65), (9, 17, 5), 0), ((19076, 28), (6, 6), 1),
    ((120, 64, 5, 3), (6, 5, 4, 3), 0), ((120, 60, 5, 3), (6, 5, 4, 3), 0), ((85, 64, 5, 3), (6, 5, 4, 3), 0),
]
FLOAT = [
    ((7, 20, 4096), (3, 4, 5), 0), ((7, 20, 4097), (3, 4, 5), 0), ((7, 21, 4097), (3, 4, 5), 1),
    ((40, 20, 9, 7), (6, 5, 4, 3), 0), ((40, 21, 9, 7), (6, 5, 4, 3), 0), ((5, 3, 4, 90), (3, 3, 3, 6), 1),
]


@pytest.mark.parametrize("precision,dims,ranks,shift", [("fp64", *c) for c in DOUBLE] + [("fp32", *c) for c in FLOAT])
def test_both_routes_within_rounding(precision, dims, ranks, shift):
    base.test_projection_and_error_within_rounding(precision, dims, ranks, shift)


@pytest.mark.parametrize("precision,dims,ranks,route", [
    ("bf16", (40, 30, 20), (4, 4, 4), "tensor cores"), ("fp32", (40, 30, 20), (4, 4, 4), "fused pass"),
    ("fp32", (16, 21, 16, 16), (6, 6, 11, 11), "fused pass"), ("fp32", (16, 21, 16, 16), (6, 6, 12, 12), "mode products"),
    ("fp64", (52, 40), (6, 6), "fused pass"), ("fp64", (51, 40), (6, 6), "mode products"),
    ("fp64", (30, 20, 65), (4, 4, 4), "fused pass"), ("fp64", (30, 20, 64), (4, 4, 4), "mode products"),
])
def test_route_by_shape(precision, dims, ranks, route):
    w, U, T, V0, _ = base._case(dims, ranks, 3, precision != "fp64")
    c = tdb.TDB(dims, ranks, weights=w, precision=precision)
    c.init_from_factors(T, U, base._device(V0, c.dtype, 0))
    assert c.projection_route() == route
    c.close()
