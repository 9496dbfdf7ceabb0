"""The HOSVD's Jacobi ends with the off-diagonal mass below 1e-15 of the diagonal's in every compute
type.  Small integers have an exact Gram C in float too, so the kept vectors of a two-point mode
diagonalise C itself: u_1^T C u_2 is at most 1e-15 |C|_F and a few roundings (sixteen u for the
rotations, the scaling and the orthonormalisation)."""

from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2201_06958_gb300 import synth, tdb

pytestmark = pytest.mark.gpu

ROWS = [([9, -1, 9, 0], [5, -5, 8, 3]), ([9, -9, 9, -1], [9, -6, 9, 0]), ([6, 4, 8, -8], [1, 1, 9, -6]),
        ([-9, 3, -8, -8], [7, -5, 5, 8]), ([9, -9, -4, 6], [7, -9, -5, -3]), ([1, 0, 0, 1], [1, 1, 0, 0]),
        ([9, 0, 1, 0], [1, 0, 0, 9]), ([1, 2, 3, 4], [1, -1, 1, 0])]


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("x,y", ROWS)
def test_two_point_mode(precision, x, y):
    V = np.array([x, y], dtype=np.float64)
    dtype = torch.float64 if precision == "fp64" else torch.float32
    c = tdb.TDB((2, 4), [2, 2], [2, 2], precision=precision, error_mode="exact")
    c.init(synth.from_logical(V, dtype=dtype, device="cuda"))
    _, U = c.factors()
    c.close()
    u = [[Fraction(float(v)) for v in U[0][:, j]] for j in range(2)]
    C = [[sum(Fraction(int(p)) * int(q) for p, q in zip(a, b)) for b in (x, y)] for a in (x, y)]
    off = abs(float(sum(u[0][i] * C[i][j] * u[1][j] for i in range(2) for j in range(2))))
    assert off <= (1e-15 + 16 * 2.0 ** -53) * np.linalg.norm(V @ V.T), off / np.linalg.norm(V @ V.T)
