"""The HOSVD's eigensolver on matrices of prescribed spectra: by Eckart and Young the
projection of a two-mode tensor on the leading r vectors of one mode leaves exactly the
discarded singular values (also where the cut splits a degenerate space, whose bases in the
two modes need not match).

A kept subspace off by an angle a_j at singular value s_j raises the error by at most
sum (a_j s_j)^2 under the root.  Rounding of the Gram (relative to its largest entry: a few n
u in double, 1e-9 in float) moves the j-th eigenvector by that over the gap, at most 1e4 for
the spectra below (every kept s_j at least 1e-2 of the largest, degenerate or separated), so
a_j s_j stays below 1e-10 and 1e-5 of ||V||.
"""

import numpy as np
import pytest
import torch

from paper_2201_06958_gb300 import synth, tdb

pytestmark = pytest.mark.gpu


def _spectrum(kind, n):
    j = np.arange(n)
    return {"flat": np.ones(n), "slow": 0.97 ** j, "steep": 10.0 ** (-0.4 * j),
            "clustered": 0.5 ** (j // 3), "deficient": np.where(j < 9, 0.8 ** j, 0.0)}[kind]


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("kind", ["flat", "slow", "steep", "clustered", "deficient"])
@pytest.mark.parametrize("dims,r", [
    ((7, 9), 3),            # every vector kept (fewer points than the block's columns)
    ((24, 25), 6),          # the block's size (6 + 2 + 16) and one more
    ((50, 51), 32),         # the largest block and one more
    ((97, 300), 6),         # iterated modes, ragged rows
    ((1024, 33), 5),        # the longest direct mode
    ((3000, 40), 6),        # a long mode from its short side
])
def test_truncation_error_is_the_discarded_spectrum(precision, kind, dims, r):
    rng = np.random.default_rng(3)
    n = min(dims)
    s = _spectrum(kind, n)
    r = min(r, int((s >= 1e-2).sum()), 9 if kind == "deficient" else n)
    Q = [np.linalg.qr(rng.standard_normal((d, n)))[0] for d in dims]
    V = (Q[0] * s) @ Q[1].T
    dtype = torch.float64 if precision == "fp64" else torch.float32
    c = tdb.TDB(dims, [r, r], [r, r], precision=precision, error_mode="exact")
    c.init(synth.from_logical(V, dtype=dtype, device="cuda"))
    _, U = c.factors()
    tail = np.linalg.norm(s[r:])
    slack = (1e-10 if precision == "fp64" else 1e-5) * np.linalg.norm(s)
    for u, X in zip(U, (V, V.T)):
        err = np.linalg.norm(X - u @ (u.T @ X))
        assert tail - slack <= err <= np.hypot(tail, slack) + slack, (err, tail)
        assert np.abs(u.T @ u - np.eye(r)).max() <= 1e-12
    c.close()
