"""Reconstructions on both sides of the rule that takes mode 1 last or the modes in order, and at
the ends of a warp's rows and columns: within (sum of ranks + a few) u of |T| x |U|, from the state
as it is read back."""

import numpy as np
import pytest
import torch

import oracle as O
from paper_2201_06958_gb300 import synth, tdb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("dims,ranks", [
    ((64, 48), (6, 6)), ((200, 9), (5, 5)),                       # two modes
    ((76, 20, 11), (5, 4, 3)), ((77, 20, 11), (5, 4, 3)),         # the rows of float, one block
    ((153, 20, 11), (5, 4, 3)), ((154, 20, 11), (5, 4, 3)),       # ... two blocks
    ((31, 20, 4), (5, 4, 3)), ((32, 20, 4), (5, 4, 3)),           # ... beside a last mode kept whole
    ((127, 9, 4), (9, 5, 3)), ((128, 9, 4), (9, 5, 3)),           # the rows of double
    ((128, 9, 5), (9, 5, 3)),                                     # a last mode that is shortened
    ((130, 7, 3), (17, 6, 3)), ((129, 3, 5, 3), (20, 3, 5, 3)),   # a ragged block, ranks above sixteen
    ((5, 40, 300), (3, 4, 5)), ((6, 5, 4, 400), (3, 3, 3, 6)),    # a short first mode
    ((7, 20000), (7, 7)), ((16, 8, 700), (4, 4, 9)), ((127, 640), (6, 6)), ((129, 640), (6, 6)),   # outputs a thread
    ((260, 1, 9), (3, 1, 3)), ((1, 30, 20), (1, 4, 4)),
])
def test_reconstruction_within_rounding(precision, dims, ranks, shift):
    f64 = precision == "fp64"
    dtype, u = (torch.float64, 2.0 ** -53) if f64 else (torch.float32, 2.0 ** -24)
    rng = np.random.default_rng(4)
    U = [np.linalg.qr(rng.standard_normal((d, r)))[0] for d, r in zip(dims, ranks)]
    c = tdb.TDB(dims, ranks, precision=precision)
    c.init_from_factors(rng.standard_normal(ranks), U, torch.zeros(tuple(reversed(dims)), dtype=dtype, device="cuda"))
    T, W = c.factors()
    n = int(np.prod(dims))
    out = torch.empty(n + 8, dtype=dtype, device="cuda")[shift:shift + n].view(tuple(reversed(dims)))
    rec = synth.to_logical(c.reconstruct(out))
    c.close()
    big = O.reconstruct(np.abs(T), [np.abs(x) for x in W])
    assert np.all(np.abs(rec - O.reconstruct(T, W)) <= (sum(ranks) + 8 * len(dims)) * u * big)
