"""The run lengths that gsstv_autotune times and reports: of at least 8 bands, or
all of fewer, and no longer than the cube (the host-side plan; no GPU needed)."""
import ctypes

import pytest

from paper_2510_00562_gb300 import binding as B
from paper_2510_00562_gb300 import build


class Geom(ctypes.Structure):
    _fields_ = [("n1", ctypes.c_int), ("n2", ctypes.c_int), ("n3", ctypes.c_int), ("p2", ctypes.c_int),
                ("cube", ctypes.c_longlong)]


@pytest.mark.parametrize("shape", [(64, 64, 32), (70, 100, 40), (24, 40, 10), (30, 19, 6), (16, 32, 1), (16, 32, 9),
                                   (512, 512, 224), (157, 203, 61), (1, 1, 65536), (2048, 2048, 7)])
def test_candidates(shape):
    build.build()
    n1, n2, n3 = shape
    p2 = (n2 + 7) // 8 * 8
    g = Geom(n1, n2, n3, p2, n1 * n3 * p2)
    out = (ctypes.c_int * 6)()
    fn = B.load()._ZN5gsstv23k1_tma_chunk_candidatesERKNS_4GeomEPii
    n = fn(ctypes.byref(g), out, 6)
    runs = list(out[:n])
    assert 1 <= n <= 6 and len(set(runs)) == n
    assert all(min(8, n3) <= r <= n3 for r in runs), runs
