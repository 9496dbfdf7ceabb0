"""A batch of float contexts runs its members' updates phase by phase in common launches; every
member's state and step record must be those of its own steps, bit for bit."""

import numpy as np
import pytest
import torch

from paper_2201_06958_gb300 import tdb

pytestmark = pytest.mark.gpu

# dims, ranks, precision, error mode
MEMBERS = [
    ((64, 48, 40), (24, 24, 24), "bf16", "exact"),      # more core slabs than CTAs take at once
    ((33, 70, 36), (5, 7, 4), "bf16", "every_k"),       # odd first mode
    ((40, 36), (6, 6), "fp32", "exact"),                # two modes
    ((36, 20, 18, 3), (6, 5, 7, 3), "fp32", "none"),    # four modes
    ((36, 20, 18, 3), (6, 5, 7, 3), "bf16", "exact"),
    ((1500, 12), (5, 5), "bf16", "exact"),              # more row tiles than are summed in one go
    ((8, 6, 5), (1, 1, 1), "fp32", "exact"),            # rank one
    ((32, 32, 32), (32, 32, 32), "fp32", "exact"),      # every vector kept
]


def _member(dims, ranks, precision, mode, seed):
    g = torch.Generator().manual_seed(seed)
    shape = tuple(reversed(dims))
    V = [torch.randn(shape, generator=g).cuda() for _ in range(2)]
    V[1] = V[0] + 1e-3 * V[1]
    rng = np.random.default_rng(seed)
    w = [np.asarray(x / x.sum()) for x in (rng.uniform(0.5, 1.5, d) for d in dims)]
    U = [np.linalg.qr(rng.standard_normal((d, r)))[0] / np.sqrt(wn)[:, None] for d, r, wn in zip(dims, ranks, w)]
    core = rng.standard_normal(ranks)
    c = tdb.TDB(dims, ranks, ranks, weights=w, precision=precision, error_mode=mode, error_every=3)
    c.init_from_factors(core, U, V[0])
    c.set_input_slots(*V)
    return c


@pytest.mark.parametrize("count,nstreams", [(len(MEMBERS), 3), (2 * len(MEMBERS) + 1, 8), (35, 1)])
def test_batch_equals_own_steps(count, nstreams):
    spec = [MEMBERS[i % len(MEMBERS)] + (i,) for i in range(count)]
    own, together = ([_member(*s) for s in spec] for _ in range(2))
    batch = tdb.Batch(together, nstreams=nstreams)
    for k in range(4):
        a = [c.push_slot((k + 1) % 2) for c in own]
        b = batch.push((k + 1) % 2)
        for x, y in zip(a, b):
            for key in ("eps", "dv_norm", "ds_norm", "gamma", "sigma_min"):
                assert np.array_equal(x[key], y[key], equal_nan=True), (k, key, x, y)
    for i, (c, d) in enumerate(zip(own, together)):
        (T, U), (S, W) = c.factors(), d.factors()
        assert np.array_equal(T, S) and all(np.array_equal(u, v) for u, v in zip(U, W)), i
    assert batch.counters()["graph_replays"] >= 2
    batch.close()
    for c in own + together:
        c.close()
