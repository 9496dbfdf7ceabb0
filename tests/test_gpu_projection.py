"""The float and double projection pass, the exact error and the reconstruction at the edges
of their tiles.

Every entry of dS and Y_n against the oracle's, within the rounding bound of the sums that
form it: a chain of products contracting N_1, ..., N_p terms in arithmetic of unit roundoff u
is off by at most (sum of the contracted lengths + a few) u times the same chain over
absolute values.
"""

import numpy as np
import pytest
import torch

import oracle as O
from paper_2201_06958_gb300 import synth, tdb

pytestmark = pytest.mark.gpu


def _case(dims, ranks, seed, f32):
    rng = np.random.default_rng(seed)
    w, U = [], []
    for N, r in zip(dims, ranks):
        x = rng.uniform(0.5, 1.5, N)
        w.append(x / x.sum())
        Q, _ = np.linalg.qr(rng.standard_normal((N, r)))
        U.append(Q / np.sqrt(w[-1])[:, None])
    T = rng.standard_normal(ranks)
    V0 = rng.standard_normal(dims)
    V1 = V0 + 1e-2 * rng.standard_normal(dims)
    if f32:
        V0, V1 = (v.astype(np.float32).astype(np.float64) for v in (V0, V1))
    return w, U, T, V0, V1


def _device(a, dtype, shift):
    """The storage tensor of `a`, its first element `shift` elements past an aligned address."""
    t = synth.from_logical(a, dtype=dtype, device="cuda")
    buf = torch.empty(t.numel() + 8, dtype=dtype, device="cuda")
    out = buf[shift:shift + t.numel()].view(t.shape)
    out.copy_(t)
    return out


FLOAT = [
    ((128, 128, 5), (4, 4, 3), 0),            # whole tiles, smallest rank block
    ((132, 33, 7), (5, 9, 4), 0),             # remainders of both tiles
    ((127, 129, 3), (8, 8, 2), 0),            # rows off 16 bytes, one row past a tile
    ((260, 300, 2), (17, 31, 2), 0),          # two rank blocks; mode 2 above one finish column
    ((64, 31), (12, 12), 0),                  # two modes
    ((3, 5, 4), (2, 3, 2), 0),                # smaller than one warp's lanes
    ((40, 24, 9, 3), (13, 4, 6, 3), 0),       # four modes
    ((128, 64, 6), (11, 7, 3), 1),            # aligned rows at an unaligned address
    ((2100, 20), (6, 6), 0),                  # more tiles of mode 1 than the finish loads at once
]
DOUBLE = [
    ((128, 128, 32), (5, 5, 5), 0),           # 2^19 points: the smallest the pass takes
    ((131, 65, 63), (8, 3, 4), 0),            # rows off 16 bytes, remainders
    ((130, 129, 32), (9, 17, 5), 0),          # several rank blocks
    ((96, 74, 26, 3), (6, 5, 7, 3), 0),       # four modes
    ((128, 256, 17), (4, 4, 4), 1),           # aligned rows at an unaligned address
    ((19076, 28), (6, 6), 0),                 # two modes, a long first
]


@pytest.mark.parametrize("precision,dims,ranks,shift",
                         [("fp32", *c) for c in FLOAT] + [("fp64", *c) for c in DOUBLE])
def test_projection_and_error_within_rounding(precision, dims, ranks, shift):
    f64 = precision == "fp64"
    dtype, u = (torch.float64, 2.0 ** -53) if f64 else (torch.float32, 2.0 ** -24)
    w, U, T, V0, V1 = _case(dims, ranks, 11, not f64)
    c = tdb.TDB(dims, ranks, weights=w, precision=precision, error_mode="exact")
    v0, v1 = _device(V0, dtype, shift), _device(V1, dtype, shift)
    c.init_from_factors(T, U, v0)
    info = c.push(v1)
    dS, Y = c.projection()
    dV = V1 - V0
    dSo, Yo = O.project(dV, U, w)
    p = len(dims)
    A = [np.abs(w[n][:, None] * U[n]) for n in range(p)]
    wide = np.abs(V1) + np.abs(V0)            # dV itself is rounded relative to |dV| only

    def bound(keep):
        X = np.abs(dV)
        for m in range(p):
            if m != keep:
                X = O.mode_product(X, A[m].T, m)
        return (sum(dims) + 8 * p) * u * X

    assert np.all(np.abs(dS - dSo) <= bound(-1))
    for n in range(p):
        sh = list(ranks)
        sh[n] = dims[n]
        assert np.all(np.abs(Y[n] - O.fold(Yo[n], n, sh)) <= bound(n)), n
    dv = np.sqrt(np.sum(_weights(w) * dV ** 2))
    # a sum of positive terms: relative error of at most its length in roundoffs
    assert abs(info["dv_norm"] - dv) <= (sum(dims) + 16) * u * dv
    # the error of the state that was reached; the reconstruction is off by at most
    # (sum of ranks + a few) u of |T| x |U|, plus the rounding of V's own float factors
    Tg, Ug = c.factors()
    e = O.error_exact(V1, Tg, Ug, w)
    big = O.reconstruct(np.abs(Tg), [np.abs(x) for x in Ug])
    slack = np.sqrt(np.sum(_weights(w) * ((sum(ranks) + 8 * p) * u * (big + wide)) ** 2))
    assert abs(info["eps"] - e) <= slack + (sum(dims) + 16) * u * e
    out = torch.empty(v0.numel() + 8, dtype=dtype, device="cuda")[shift:shift + v0.numel()].view(v0.shape)
    rec = synth.to_logical(c.reconstruct(out))
    assert np.all(np.abs(rec - O.reconstruct(Tg, Ug)) <= (sum(ranks) + 8 * p) * u * big)
    c.close()


def _weights(w):
    p = len(w)
    out = 1.0
    for n in range(p):
        out = out * w[n].reshape([-1 if m == n else 1 for m in range(p)])
    return out


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("value", [np.inf, np.nan])
def test_non_finite_difference_is_refused(precision, value):
    dims, ranks = ((130, 129, 32), (4, 4, 4))
    w, U, T, V0, V1 = _case(dims, ranks, 5, precision == "fp32")
    V1[129, 128, 31] = value
    dtype = torch.float64 if precision == "fp64" else torch.float32
    c = tdb.TDB(dims, ranks, weights=w, precision=precision, error_mode="none")
    c.init_from_factors(T, U, _device(V0, dtype, 0))
    with pytest.raises(tdb.TDBError) as e:
        c.push(_device(V1, dtype, 0))
    assert e.value.status == 5
    c.close()
