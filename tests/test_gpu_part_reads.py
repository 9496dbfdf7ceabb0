"""tdb_get_factors with part of its outputs: the values of a full read, and no kernel to pack what
was not asked for."""

import ctypes as C

import numpy as np
import pytest
import torch

from paper_2201_06958_gb300 import tdb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("with_core,which", [(True, None), (True, ()), (False, (0, 1, 2)), (False, (1,)), (True, (0, 2)),
                                             (False, None)])
def test_part_of_the_factors(precision, with_core, which):
    dims, ranks = (50, 30, 20), (5, 4, 3)
    rng = np.random.default_rng(0)
    dtype = torch.float64 if precision == "fp64" else torch.float32
    V0 = torch.zeros(tuple(reversed(dims)), dtype=dtype, device="cuda")
    c = tdb.TDB(dims, ranks, ranks, precision=precision)
    c.init_from_factors(rng.standard_normal(ranks), [np.linalg.qr(rng.standard_normal((d, r)))[0]
                                                     for d, r in zip(dims, ranks)], V0)
    T, U = c.factors()
    core = np.full(T.size, np.nan)
    out = [np.full(u.size, np.nan) for u in U]
    dp = C.POINTER(C.c_double)
    ptr = None if which is None else (dp * 3)(*(o.ctypes.data_as(dp) if n in which else dp() for n, o in enumerate(out)))
    l0 = c.lib.tdb_kernel_launches()
    assert c.lib.tdb_get_factors(c.ctx, core.ctypes.data_as(dp) if with_core else None, ptr, None) == 0
    assert c.lib.tdb_kernel_launches() == l0
    c.close()
    assert np.array_equal(core, T.ravel(order="F")) if with_core else np.isnan(core).all()
    for n, (o, u) in enumerate(zip(out, U)):
        assert np.array_equal(o, u.ravel(order="F")) if which and n in which else np.isnan(o).all()
