"""The HOSVD's eigensolver finds CTAs for mode Grams of every size that a context takes (modes of
up to 1024 points, or the short side of a longer one), within the SMs and the shared memory of a
GB300: 152 SMs, 227 KB a CTA less the 2 KB left for the kernel's static part.  No GPU calls."""

import ctypes as C
import random

import pytest

from paper_2201_06958_gb300 import build_lib, tdb

SMS, SMEM = 152, 227 * 1024 - 2048


@pytest.fixture(scope="module")
def lib():
    build_lib.build()
    return tdb.load()


def _split(lib, sizes, caps, sms=SMS, smem=SMEM):
    p = len(sizes)
    n, k = (C.c_int * p)(*sizes), (C.c_int * p)(*(min(s, c + 2) for s, c in zip(sizes, caps)))
    ctas, need = (C.c_int * p)(), C.c_int64()
    st = lib.tdb_selftest_eig_split(p, n, k, sms, smem, ctas, C.byref(need))
    return st, list(ctas), need.value


def _fits(lib, sizes, caps):
    st, ctas, need = _split(lib, sizes, caps)
    return st == 0 and sum(ctas) <= SMS and min(ctas) >= 2 and need <= SMEM and \
        all(c - 1 <= max(1, s) for c, s in zip(ctas, sizes))


@pytest.mark.parametrize("cap", [32, 24, 5])
def test_every_two_mode_size(lib, cap):
    bad = [(a, b) for a in range(1, 1025) for b in range(1, a + 1) if not _fits(lib, (a, b), (cap, cap))]
    assert not bad, bad[:5]


@pytest.mark.parametrize("sizes", [(127, 768, 892), (114, 359, 928), (1024, 160, 1024), (1024, 119, 3),
                                   (1024, 1024, 170, 1), (768, 768, 127)])
def test_short_modes_beside_long_ones(lib, sizes):
    assert _fits(lib, sizes, (32,) * len(sizes))


@pytest.mark.parametrize("p", [1, 3, 4])
def test_sampled_sizes(lib, p):
    rng = random.Random(p)
    for _ in range(20000):
        sizes = [int(2 ** rng.uniform(0, 10)) for _ in range(p)]
        caps = [rng.randint(1, 32) for _ in range(p)]
        assert _fits(lib, sizes, caps), (sizes, caps)


def test_too_small_a_device_is_refused(lib):
    unsupported = 11
    assert lib.tdb_status_string(unsupported) == b"TDB_ERR_UNSUPPORTED"
    assert _split(lib, (1024, 1024), (32, 32), sms=8)[0] == unsupported      # 20 CTAs for the rows
    assert _split(lib, (64,), (32,), smem=64 * 1024)[0] == unsupported       # not one row
