"""Calls between pushes share scratch with the pushes (the packed state, reconstruction, HOSVD):
a stream with such calls in it goes on as one without, bit for bit."""

import numpy as np
import pytest
import torch

from paper_2201_06958_gb300 import tdb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,dims,ranks,integrator", [
    ("fp32", (96, 40, 33), (6, 5, 4), "euler"),
    ("fp32", (96, 40, 33), (6, 5, 4), "heun"),
    ("fp32", (40, 24, 16, 14), (6, 5, 12, 11), "euler"),      # 132 outputs: mode products
    ("fp64", (96, 90, 64), (6, 5, 4), "euler"),               # the fused pass
    ("fp64", (96, 90, 64), (6, 5, 4), "rk2_central"),
    ("fp64", (40, 24, 16), (6, 5, 4), "euler"),               # mode products
    ("bf16", (96, 40, 33), (6, 5, 4), "euler"),
    ("bf16", (40, 24, 16, 5), (6, 5, 4, 3), "euler"),
])
def test_calls_between_pushes(precision, dims, ranks, integrator):
    dtype = torch.float64 if precision == "fp64" else torch.float32
    g = torch.Generator().manual_seed(7)
    shape = tuple(reversed(dims))
    V = [torch.randn(shape, generator=g, dtype=dtype).cuda()]
    for _ in range(6):
        V.append(V[-1] + 1e-2 * torch.randn(shape, generator=g, dtype=dtype).cuda())
    rng = np.random.default_rng(7)
    U = [np.linalg.qr(rng.standard_normal((d, r)))[0] for d, r in zip(dims, ranks)]
    core = rng.standard_normal(ranks)
    plain, mixed = (tdb.TDB(dims, ranks, ranks, precision=precision, error_mode="exact", integrator=integrator)
                    for _ in range(2))
    infos = []
    for c in (plain, mixed):
        c.init_from_factors(core, U, V[0])
        out = []
        for k, v in enumerate(V[1:]):
            out.append(c.push(v))
            if c is mixed:
                c.factors()
                c.reconstruct()
                c.save_state()
                if k == 1 and integrator != "rk2_central":
                    c.load_state(c.save_state(), v)
            elif k == 1 and integrator != "rk2_central":
                c.load_state(c.save_state(), v)           # (a load restarts the warm eigenvectors)
            if k == 3:
                c.reinit(v)
        infos.append(out)
    for a, b in zip(*infos):
        for key in ("eps", "dv_norm", "sigma_min", "gamma"):
            assert np.array_equal(a[key], b[key]), (key, a, b)
    (T, W), (S, X) = plain.factors(), mixed.factors()
    assert np.array_equal(T, S) and all(np.array_equal(u, v) for u, v in zip(W, X))
    dS, Y = plain.projection()
    dQ, Z = mixed.projection()
    assert np.array_equal(dS, dQ) and all(np.array_equal(u, v) for u, v in zip(Y, Z))
    plain.close()
    mixed.close()
