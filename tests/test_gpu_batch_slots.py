"""A batch's recorded steps read its members' input slots: a member that gets new slots between two
pushes is stepped on those, as by its own pushes, bit for bit."""

import numpy as np
import pytest
import torch

from paper_2201_06958_gb300 import tdb

pytestmark = pytest.mark.gpu


def _member(precision, seed):
    dims, ranks = (40, 24, 12), (5, 4, 3)
    dtype = torch.float64 if precision == "fp64" else torch.float32
    g = torch.Generator().manual_seed(seed)
    shape = tuple(reversed(dims))
    first = torch.randn(shape, generator=g, dtype=dtype).cuda()
    slots = [[first + 1e-3 * torch.randn(shape, generator=g, dtype=dtype).cuda() for _ in range(2)] for _ in range(2)]
    rng = np.random.default_rng(seed)
    U = [np.linalg.qr(rng.standard_normal((d, r)))[0] for d, r in zip(dims, ranks)]
    c = tdb.TDB(dims, ranks, ranks, precision=precision, error_mode="exact")
    c.init_from_factors(rng.standard_normal(ranks), U, slots[0][0])
    c.set_input_slots(*slots[0])
    return c, slots


@pytest.mark.parametrize("precision", ["bf16", "fp32", "fp64"])
def test_new_slots_of_one_member(precision):
    own = [_member(precision, i) for i in range(3)]
    together = [_member(precision, i) for i in range(3)]
    batch = tdb.Batch([c for c, _ in together], nstreams=2)

    def push(parity):
        a = [c.push_slot(parity) for c, _ in own]
        b = batch.push(parity)
        for x, y in zip(a, b):
            for key in ("eps", "dv_norm", "sigma_min"):
                assert np.array_equal(x[key], y[key]), (key, x, y)

    for parity in (1, 0, 1, 0):
        push(parity)
    for c, slots in (own[1], together[1]):          # the stream goes on in other buffers
        c.load_state(c.save_state(), slots[1][0])
        c.set_input_slots(*slots[1])
    for parity in (1, 0):
        push(parity)
    for (c, _), (d, _) in zip(own, together):
        (T, U), (S, W) = c.factors(), d.factors()
        assert np.array_equal(T, S) and all(np.array_equal(u, v) for u, v in zip(U, W))
    batch.close()
    for c, _ in own + together:
        c.close()
