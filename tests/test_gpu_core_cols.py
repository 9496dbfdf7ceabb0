"""The column factors H = T x_2 U_2 ... x_p U_p formed in one launch, through the
reconstruction U_1 H, at the edges of its groups: entries of a core slice over and under one
warp's lanes and one CTA's warps, column blocks with a remainder, four modes, and a case large
enough to take the chain of mode products.

A float sum of n terms is off by at most n u times the sum of their magnitudes (u = 2^-24), so
the reconstruction by (r_1 + r_2 + J + a few) u |T| x |U|, J the product of the other ranks.
"""

import numpy as np
import pytest
import torch

import oracle as O
from paper_2201_06958_gb300 import synth, tdb

pytestmark = pytest.mark.gpu

CASES = [
    ((20, 300, 3), (11, 21, 3)),         # 231 entries a slice: eight warps, no split over j
    ((24, 40, 12), (11, 11, 7)),         # 121 entries: two runs of j
    ((6, 700, 5), (3, 2, 2)),            # 6 entries; mode 2 in several column blocks
    ((9, 17, 5, 4), (5, 6, 5, 4)),       # four modes, 20 products
    ((40, 33, 4, 3), (32, 32, 4, 3)),    # 1024 entries a slice
    ((32, 40, 600), (32, 32, 32)),       # above the limit: the chain of mode products
]


@pytest.mark.parametrize("dims,ranks", CASES)
def test_reconstruction_within_rounding(dims, ranks):
    rng = np.random.default_rng(77)
    U = [np.linalg.qr(rng.standard_normal((n, r)))[0] * np.sqrt(n) for n, r in zip(dims, ranks)]
    T = rng.standard_normal(ranks)
    V0 = synth.from_logical(rng.standard_normal(dims), dtype=torch.float32, device="cuda")
    c = tdb.TDB(dims, ranks, precision="fp32", error_mode="exact")
    c.init_from_factors(T, U, V0)
    Tg, Ug = c.factors()
    rec = synth.to_logical(c.reconstruct())
    terms = ranks[0] + ranks[1] + int(np.prod(ranks[2:])) + 8 * len(dims)
    big = O.reconstruct(np.abs(Tg), [np.abs(x) for x in Ug])
    assert np.all(np.abs(rec - O.reconstruct(Tg, Ug)) <= terms * 2.0 ** -24 * big)
    c.close()
