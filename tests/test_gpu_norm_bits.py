"""||dV||_W of the float contexts: single products may be float, their sum and the weights of the
modes after the first are double (or hold as many bits)."""

import numpy as np
import pytest
import torch

from paper_2201_06958_gb300 import tdb

pytestmark = pytest.mark.gpu

# dims, ranks: the fused pass with its tallest tile (32 rows a warp), with rows off 16 bytes, and
# four modes of more outputs than it takes (mode products)
SHAPES = [((4, 128, 1824), (2, 3, 3)), ((5, 128, 1824), (2, 3, 3)), ((260, 40, 30), (3, 3, 3)),
          ((1024, 6, 16, 16), (12, 6, 12, 12))]


def _norm(dims, ranks, d, w):
    rng = np.random.default_rng(1)
    U = [np.linalg.qr(rng.standard_normal((n, r)))[0] / np.sqrt(x)[:, None] for n, r, x in zip(dims, ranks, w)]
    V0 = torch.zeros(tuple(reversed(dims)), device="cuda")
    V1 = torch.from_numpy(np.ascontiguousarray(d.T).astype(np.float32)).cuda()
    c = tdb.TDB(dims, ranks, ranks, weights=w, precision="fp32", error_mode="none")
    c.init_from_factors(rng.standard_normal(ranks), U, V0)
    got = c.push(V1)["dv_norm"]
    c.close()
    x = d.astype(np.float64) ** 2
    for n, wn in enumerate(w):
        x = x * wn.reshape([-1 if m == n else 1 for m in range(len(dims))])
    return got, np.sqrt(x.sum())


@pytest.mark.parametrize("dims,ranks", SHAPES)
def test_small_squares_beside_large_ones(dims, ranks):
    """One entry of 1 to 31 whose squares are 2^-25 along modes 1 and 2: a float sum from the large
    one on loses them all, 31 2^-26 of the norm.  The first mode's weight, a product and a sum of
    four in float leave 3 2^-24."""
    i = np.indices(dims, sparse=True)
    large = (i[1] % 32 == 0) & (i[0] < 32) if dims[0] > 32 else (i[1] % 32 == 0) | (i[0] < 0)
    d = np.where(np.broadcast_to(large, dims), 1.0, 2.0 ** -12.5)
    got, want = _norm(dims, ranks, d, [np.ones(n) for n in dims])
    assert abs(got - want) <= 3 * 2.0 ** -24 * want


@pytest.mark.parametrize("dims,ranks", SHAPES)
def test_weights_after_the_first_mode(dims, ranks):
    """Differences of one and a first mode of unit weights are exact in float: what is left is the
    product of the other weights in double and the order of its sum."""
    rng = np.random.default_rng(2)
    w = [np.ones(dims[0])] + [rng.uniform(0.5, 1.5, n) for n in dims[1:]]
    got, want = _norm(dims, ranks, np.ones(dims), w)
    assert abs(got - want) <= 2.0 ** -44 * want
