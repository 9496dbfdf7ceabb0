"""The exact error and the reconstruction at the edges of their chunks of columns: ranks at and
one past every size of the register rows, chunks of 32 and of 16 (double above rank 16), fewer
columns than a chunk and a remainder, one row block and several.

A sum of n terms is off by at most n u times the sum of their magnitudes; V itself and the
factors are exact in the compute type or read back from it.
"""

import numpy as np
import pytest
import torch

import oracle as O
from paper_2201_06958_gb300 import synth, tdb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("dims,ranks", [
    ((300, 9, 7), (8, 4, 3)),          # 63 columns
    ((130, 12, 11), (12, 6, 4)),       # 132
    ((33, 40, 2), (13, 8, 2)),
    ((257, 17, 9), (16, 6, 4)),        # 153
    ((70, 19, 25), (17, 6, 5)),
    ((129, 31, 8), (32, 8, 4)),
    ((40, 37), (32, 32)),
    ((5, 3, 4), (5, 2, 3)),            # 12 columns
])
def test_error_and_reconstruction_within_rounding(precision, dims, ranks):
    f64 = precision == "fp64"
    dtype, u = (torch.float64, 2.0 ** -53) if f64 else (torch.float32, 2.0 ** -24)
    rng = np.random.default_rng(21)
    w, U = [], []
    for N, r in zip(dims, ranks):
        x = rng.uniform(0.5, 1.5, N)
        w.append(x / x.sum())
        U.append(np.linalg.qr(rng.standard_normal((N, r)))[0] / np.sqrt(w[-1])[:, None])
    V = [synth.from_logical(v, dtype=dtype, device="cuda")
         for v in (lambda a: (a, a + 1e-2 * rng.standard_normal(dims)))(rng.standard_normal(dims))]
    c = tdb.TDB(dims, ranks, weights=w, precision=precision, error_mode="exact")
    c.init_from_factors(rng.standard_normal(ranks), U, V[0])
    info = c.push(V[1])
    T, Ug = c.factors()
    V1 = synth.to_logical(V[1]).astype(np.float64)
    big = O.reconstruct(np.abs(T), [np.abs(x) for x in Ug])
    off = (sum(ranks) + int(np.prod(ranks[2:])) + 8 * len(dims)) * u * big
    assert np.all(np.abs(synth.to_logical(c.reconstruct()) - O.reconstruct(T, Ug)) <= off)
    ww = np.ones(())
    for n, x in enumerate(w):
        ww = ww * x.reshape([-1 if m == n else 1 for m in range(len(dims))])
    e = O.error_exact(V1, T, Ug, w)
    slack = np.sqrt(np.sum(ww * (off + 8 * u * np.abs(V1)) ** 2)) + (sum(dims) + 16) * u * e
    assert abs(info["eps"] - e) <= slack
    c.close()
