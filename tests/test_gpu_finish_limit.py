"""The finishing launch of a projection needs up to 58 KB of dynamic shared memory in float and 116
KB in double, by the ranks and N_2: every need launches, and contexts of different needs on
several host threads do not take each other's limit away."""

import threading

import numpy as np
import pytest
import torch

from paper_2201_06958_gb300 import tdb

pytestmark = pytest.mark.gpu


def _context(dims, ranks, precision, seed, stream=None):
    rng = np.random.default_rng(seed)
    dtype = torch.float64 if precision == "fp64" else torch.float32
    U = [np.linalg.qr(rng.standard_normal((d, r)))[0] for d, r in zip(dims, ranks)]
    g = torch.Generator(device="cuda").manual_seed(seed)
    V = [torch.randn(tuple(reversed(dims)), generator=g, device="cuda", dtype=dtype) for _ in range(2)]
    V[1] = V[0] + 1e-3 * V[1]
    torch.cuda.synchronize()
    c = tdb.TDB(dims, ranks, ranks, precision=precision, error_mode="none", stream=stream)
    c.init_from_factors(rng.standard_normal(ranks), U, V[0])
    return c, U, V


@pytest.mark.parametrize("precision,dims,ranks", [
    ("fp32", (64, 256, 24), (6, 31, 6)),       # 256 bytes below 48 KB, and 256 bytes of static memory
    ("bf16", (64, 256, 24), (6, 31, 8)),
    ("fp32", (32, 229, 40), (7, 31, 5)),
    ("fp32", (64, 256, 40), (32, 32, 32)),     # the most of three modes
    ("fp64", (160, 256, 16), (8, 32, 16)),
])
def test_every_need_launches(precision, dims, ranks):
    c, U, V = _context(dims, ranks, precision, 1)
    c.push(V[1])
    dS, Y = c.projection()
    # off by at most (contracted lengths + 8) u times the same sums over absolute values; BF16
    # operands are rounded to 9 bits each besides
    d = (V[1].double() - V[0].double()).cpu().numpy().transpose(2, 1, 0)
    rel = (sum(dims) + 8) * (2.0 ** -53 if precision == "fp64" else 2.0 ** -24) + (2.0 ** -8 if precision == "bf16" else 0)
    Y3, aY3 = (np.einsum("ijk,ia,jb->abk", f(d), f(U[0]), f(U[1])) for f in (np.asarray, np.abs))
    assert (np.abs(Y[2] - Y3) <= rel * aY3).all()
    assert (np.abs(dS - np.einsum("abk,kc->abc", Y3, U[2])) <= rel * np.einsum("abk,kc->abc", aY3, np.abs(U[2]))).all()
    c.close()


def test_two_threads_of_different_needs():
    specs = [((8, 256, 32), (4, 32, 32), "fp32"), ((8, 256, 32), (4, 32, 20), "fp32")]
    streams = [torch.cuda.Stream() for _ in specs]
    made = [_context(*s, seed=i, stream=q) for i, (s, q) in enumerate(zip(specs, streams))]
    # a ring of more snapshots than a context remembers: every push is launched, none replayed
    rings = [[v[0].clone() for _ in range(67)] for _, _, v in made]
    torch.cuda.synchronize()
    errors = []

    def work(i):
        try:
            for k in range(3000):
                made[i][0].push(rings[i][k % 67])
        except Exception as e:                 # noqa: BLE001 (the thread's error, for the assert)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(specs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for c, _, _ in made:
        c.close()
