"""A non-finite entry in the field of an init or a reinit, for modes of every kind (solved whole,
iterated, from the short side of a long one): the next push is refused, and a re-initialisation from
a finite field gives a finite state again."""

import numpy as np
import pytest
import torch

from paper_2201_06958_gb300 import tdb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("dims,ranks", [((3000, 20), (5, 5)), ((1100, 4, 2), (3, 3, 2)), ((40, 30), (4, 4)),
                                        ((120, 100, 9), (4, 4, 3)), ((60, 20, 16, 5), (4, 4, 3, 2))])
def test_non_finite_field(precision, value, dims, ranks):
    dtype = torch.float64 if precision == "fp64" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(0)
    good = torch.randn(tuple(reversed(dims)), generator=g, device="cuda", dtype=dtype)
    bad = good.clone()
    bad.view(-1)[7] = value
    c = tdb.TDB(dims, ranks, ranks, precision=precision)
    c.init(bad)
    with pytest.raises(tdb.TDBError):
        c.push(good)
    c.reinit(good)
    assert all(np.isfinite(u).all() for u in c.factors()[1])
    c.reinit(bad)
    c.reinit(good)
    assert all(np.isfinite(u).all() for u in c.factors()[1])
    assert np.isfinite(c.push(good + 1e-3)["eps"])
    c.close()
