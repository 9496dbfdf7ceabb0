"""The profile's update phases are those that the update kernel times, for any number of modes."""

import numpy as np
import pytest
import torch

from paper_2201_06958_gb300 import tdb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(40, 30), (40, 30, 20), (20, 16, 12, 10)])
def test_seven_phases(dims):
    ranks = [4] * len(dims)
    rng = np.random.default_rng(0)
    g = torch.Generator(device="cuda").manual_seed(0)
    V = [torch.randn(tuple(reversed(dims)), generator=g, device="cuda") for _ in range(2)]
    V[1] = V[0] + 1e-3 * V[1]
    c = tdb.TDB(dims, ranks, ranks, precision="fp32", error_mode="exact")
    c.init_from_factors(rng.standard_normal(ranks), [np.linalg.qr(rng.standard_normal((d, 4)))[0] for d in dims], V[0])
    c.set_profiling(True)
    for k in range(4):
        c.push(V[(k + 1) % 2])
    us = c.profile()["us_update_phase"]
    c.close()
    # rows, rows, factors with rows, core products (two), Gram partials, Gram finish (its own launch
    # beside the error); two modes have no product in the second set
    assert len(us) == 7
    timed = [0, 1, 2, 3, 5] + ([4] if len(dims) > 2 else [])
    assert all(us[k] > 0 for k in timed), us
