"""HOSVDs of data whose spectrum hardly decays (Gaussian noise, one
mode far longer than the other): the kept subspaces are the leading singular subspaces, also where a subspace iteration would take hundreds of rounds to find them.

The Gram's rounding E moves the subspace by |E| / gap, gap the difference of the squared singular
values at the cut.  In double |E| <= N_2 u |V|_F^2 (a sum of N_2 products), and the eigensolver adds a few
n u |V|_F^2; in float the products of 32 columns are summed in float, |E| <= 32 2^-24 |V|_F^2, and
everything after that in double.  The vectors of the other mode follow from these.
"""

import numpy as np
import pytest
import torch

from paper_2201_06958_gb300 import synth, tdb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,dims,r", [
    ("fp64", (64, 5000), 10),
    ("fp64", (64, 2000), 30),
    ("fp64", (51, 3000), 4),      # one more point than the widest block
    ("fp64", (95, 4000), 10),     # odd: a padded row
    ("fp64", (96, 3000), 32),     # the largest mode that is solved whole
    ("fp64", (25, 4000), 6),      # one more point than this block
    ("fp64", (40, 45), 14),       # settles
    ("fp32", (48, 3000), 10),
    ("fp32", (95, 4000), 10),
])
def test_subspaces_of_noise(precision, dims, r):
    rng = np.random.default_rng(sum(dims))
    V = rng.standard_normal(dims)
    if precision == "fp32":
        V = V.astype(np.float32).astype(np.float64)
    dtype = torch.float64 if precision == "fp64" else torch.float32
    c = tdb.TDB(dims, [r, r], [r, r], precision=precision, error_mode="exact")
    c.init(synth.from_logical(V, dtype=dtype, device="cuda"))
    _, U = c.factors()
    c.close()
    X, s, Y = np.linalg.svd(V)
    F, gap = (s ** 2).sum(), s[r - 1] ** 2 - s[r] ** 2
    n = max(dims)
    bound = ((n + 16 * n) * 2.0 ** -53 if precision == "fp64" else 32 * 2.0 ** -24) * F / gap
    for u, full in zip(U, (X, Y.T)):
        lead = full[:, :r]
        sine = np.linalg.norm(u - lead @ (lead.T @ u), 2)
        assert sine <= bound, (sine, bound)
