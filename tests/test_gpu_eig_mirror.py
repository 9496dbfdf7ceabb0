"""The HOSVD of data whose Gram is exactly rank deficient: rows that repeat bit for bit make the
product of the Gram with any block repeat them too, so that no rounding fills the block up.
The truncation error is the discarded spectrum all the same (Eckart and Young).

Rounding of the Gram (1e-9 of its largest entry in float, a few n u in double) over the gaps of
the kept spectrum (at least 1e-2 of the largest value squared) leaves 1e-5 and 1e-10 of ||V||.
"""

import numpy as np
import pytest
import torch

from paper_2201_06958_gb300 import synth, tdb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("copies,dims,r", [
    (2, (32, 300), 6),         # rank 16 under a block of 24
    (4, (64, 90), 5),          # rank 16 of 64
    (32, (64, 70), 2),         # rank 2: the kept vectors only
    (2, (200, 27), 3),         # rank 27 in mode 1, full in mode 2
])
def test_repeated_rows(precision, copies, dims, r):
    dtype = torch.float64 if precision == "fp64" else torch.float32
    rng = np.random.default_rng(8)
    base = dims[0] // copies
    n = min(base, dims[1])
    s = 0.7 ** np.arange(n)
    Q = [np.linalg.qr(rng.standard_normal((d, n)))[0] for d in (base, dims[1])]
    V = np.tile((Q[0] * s) @ Q[1].T, (copies, 1))
    if precision == "fp32":
        V = V.astype(np.float32).astype(np.float64)
    c = tdb.TDB(dims, [r, r], [r, r], precision=precision, error_mode="exact")
    c.init(synth.from_logical(V, dtype=dtype, device="cuda"))
    _, U = c.factors()
    sv = np.linalg.svd(V, compute_uv=False)
    tail = np.linalg.norm(sv[r:])
    slack = (1e-10 if precision == "fp64" else 1e-5) * np.linalg.norm(sv)
    for u, X in zip(U, (V, V.T)):
        err = np.linalg.norm(X - u @ (u.T @ X))
        assert tail - slack <= err <= np.hypot(tail, slack) + slack, (err, tail)
        assert np.abs(u.T @ u - np.eye(r)).max() <= 1e-12
    c.close()
