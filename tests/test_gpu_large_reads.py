"""Reads of the factors on both sides of the size up to which they leave the device packed: the
state that was loaded, bit for bit, and without a packing kernel for a large one."""

import numpy as np
import pytest
import torch

from paper_2201_06958_gb300 import tdb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,ranks", [((40, 30), (4, 4)), ((4086, 6), (4, 4)), ((4087, 6), (4, 4)),
                                        ((5000, 12, 2), (8, 5, 2))])       # 16384 values, four more
def test_factors_are_the_state(dims, ranks):
    rng = np.random.default_rng(0)
    core = rng.standard_normal(ranks)
    U = [np.linalg.qr(rng.standard_normal((d, r)))[0] for d, r in zip(dims, ranks)]
    total = core.size + sum(u.size for u in U)
    c = tdb.TDB(dims, ranks, ranks, precision="fp32")
    c.init_from_factors(core, U, torch.zeros(tuple(reversed(dims)), device="cuda"))
    c.factors()
    l0 = c.lib.tdb_kernel_launches()
    T, W = c.factors()
    assert c.lib.tdb_kernel_launches() - l0 == (1 if total <= 16384 else 0)
    c.close()
    assert np.array_equal(T, core)
    for u, v in zip(U, W):
        assert np.array_equal(u, v)
