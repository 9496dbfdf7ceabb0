"""HOSVDs of mode sizes whose eigenproblems share the SMs unevenly (a mode of a hundred points
beside one of a thousand), at the default rank caps, from init and from reinit.

The data is sum_j s_j a_j o b_j o ... with orthonormal vectors a_j per mode, so every unfolding has
the singular values s_j and the vectors a_j.  The part of an unfolding outside a kept subspace of r
vectors is then |(I - U U^T) A diag(s)|_F, at least the tail of s (Eckart and Young).  Rounding of the
Gram (a few n u in double, 1e-9 of its largest entry in float) over the gaps of the kept spectrum
(at least 4e-4 of the largest value squared) leaves 1e-10 and 1e-5 of ||V||.
"""

import numpy as np
import pytest
import torch

from paper_2201_06958_gb300 import tdb

pytestmark = pytest.mark.gpu

TERMS, RANK = 40, 20


def _data(dims, dtype, seed):
    g = torch.Generator().manual_seed(seed)
    k = min(TERMS, *dims)
    s = 0.85 ** torch.arange(k, dtype=torch.float64)
    A = [torch.linalg.qr(torch.randn(d, k, generator=g, dtype=torch.float64))[0] for d in dims]
    # storage order: the last mode slowest, the first fastest
    rest = torch.ones(1, k, dtype=torch.float64, device="cuda")
    for a in A[1:]:
        rest = (a.cuda()[:, None, :] * rest).reshape(-1, k)
    V = rest @ (A[0] * s).T.cuda()
    return A, s, V.reshape(tuple(reversed(dims))).to(dtype)


def _check(c, A, s, precision):
    _, U = c.factors()
    r, S = RANK, s.numpy()
    slack = (1e-10 if precision == "fp64" else 1e-5) * np.linalg.norm(S)
    tail = np.linalg.norm(S[r:])
    for u, a in zip(U, A):
        X = a.numpy() * S
        err = np.linalg.norm(X - u @ (u.T @ X))
        assert tail - slack <= err <= np.hypot(tail, slack) + slack, (err, tail)
        assert np.abs(u.T @ u - np.eye(r)).max() <= 1e-12


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("dims", [(1024, 119), (1024, 112), (1024, 160, 40), (127, 768, 892), (160, 1024, 24, 24)])
def test_init_and_reinit(precision, dims):
    dtype = torch.float64 if precision == "fp64" else torch.float32
    c = tdb.TDB(dims, [RANK] * len(dims), precision=precision, error_mode="exact")     # rank_max: the default
    for seed in (0, 1):
        A, s, V = _data(dims, dtype, seed)
        c.init(V) if seed == 0 else c.reinit(V)
        _check(c, A, s, precision)
    c.close()
