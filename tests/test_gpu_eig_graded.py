"""HOSVDs of many small double modes with graded and clustered spectra, for which a cyclic Jacobi
takes most sweeps: every kept subspace is the leading singular subspace.

Rounding of the Gram and of the eigensolver, E <= (N_2 + 16 n) u |V|_F^2 (a sum of N_2 products and a few
operations an entry), moves it by |E| / gap, gap the difference of the squared singular values at
the cut.
"""

import numpy as np
import pytest
import torch

from paper_2201_06958_gb300 import synth, tdb

pytestmark = pytest.mark.gpu


def _squares(kind, n, rng):
    j = np.arange(n)
    return {"halves": 0.5 ** j, "tenths": 0.1 ** np.minimum(j, 12.0), "clusters": 0.1 ** (j // 5) * rng.uniform(0.9, 1.1, n),
            "pairs": 0.3 ** (j // 2) * rng.uniform(0.95, 1.05, n), "spread": 10.0 ** rng.uniform(-8, 0, n),
            "noise below": np.where(j < 6, 0.3 ** j, 1e-5 * rng.uniform(0.5, 1.5, n))}[kind]


@pytest.mark.parametrize("kind", ["halves", "tenths", "clusters", "pairs", "spread", "noise below"])
def test_leading_subspaces(kind):
    rng = np.random.default_rng(len(kind))
    for k in range(60):
        n, m = int(rng.integers(7, 51)), int(rng.integers(60, 200))
        s = np.sqrt(np.sort(_squares(kind, n, rng))[::-1])
        Q, P = (np.linalg.qr(rng.standard_normal((d, n)))[0] for d in (n, m))
        V = (Q * s) @ P.T
        r = 2 + int(np.argmax(s[1:6] / s[2:7]))            # the clearest cut among the first
        c = tdb.TDB((n, m), [r, r], precision="fp64", error_mode="exact")       # rank_max 32: solved whole
        c.init(synth.from_logical(V, dtype=torch.float64, device="cuda"))
        _, U = c.factors()
        c.close()
        X, sv, Y = np.linalg.svd(V, full_matrices=False)
        bound = (m + 16 * n) * 2.0 ** -53 * (sv ** 2).sum() / (sv[r - 1] ** 2 - sv[r] ** 2)
        for u, full in zip(U, (X, Y.T)):
            lead = full[:, :r]
            sine = np.linalg.norm(u - lead @ (lead.T @ u), 2)
            assert sine <= bound, (k, n, m, r, sine, bound)
