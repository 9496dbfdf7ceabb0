"""tdb_workspace_bytes stays near what a context needs: at most a quarter above what it was when
every projection in float and double went through mode products (bytes noted then).  The fused
pass keeps its partials where the HOSVD and the mode products have their scratch.  No GPU calls."""

import ctypes as C

import pytest

from paper_2201_06958_gb300 import build_lib, tdb


@pytest.mark.parametrize("precision,dims,cap,then", [
    ("fp64", (20, 20, 20, 20), 20, 25982976),
    ("fp32", (32, 32, 32, 32), 32, 82985216),
    ("fp64", (48, 48, 48, 48), 32, 237332992),
    ("fp32", (192, 129, 192, 3), 30, 254664448),
    ("fp32", (256, 128, 512), 20, 182198016),
    ("fp64", (126, 126, 126), 7, 44819712),
    ("fp64", (64, 64, 64), 12, 15541504),
    ("bf16", (256, 128, 512), 20, 210081024),
    ("bf16", (512, 256, 12), 20, 57536000),
    ("bf16", (192, 129, 192, 3), 30, 330722560),
    ("fp64", (19076, 23), 23, 71302912),
    ("fp64", (1024, 1024), 32, 80551936),
])
def test_workspace_is_near_the_need(precision, dims, cap, then):
    build_lib.build()
    cfg, _ = tdb.make_config(dims, [0] * len(dims), [cap] * len(dims), precision=precision)
    assert 0 < tdb.load().tdb_workspace_bytes(C.byref(cfg)) <= 1.25 * then
