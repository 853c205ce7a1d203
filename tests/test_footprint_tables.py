"""The device bytes a context asks for count its tables, which on small boxes are most of it: the
phase matrix and its three split images, the lattice offsets and the sweep's displacements."""
import ctypes

import paper_2105_01028_gb300 as T
from paper_2105_01028_gb300 import _lib


def _bytes(nx, ny, nz, nside, boundary=0, precision=0):
    d = _lib.GridDesc(nx, ny, nz, 1.0, nside, 0.5, 1.4, boundary, precision, 1e-6, 2000)
    return T.lib().trinity_footprint_bytes(ctypes.byref(d))


def test_tables_are_counted():
    for nside, images in ((1, 0), (2, 3 * 48 * 64 * 2), (4, 3 * 3 * 192 * 64 * 2)):
        na = 12 * nside ** 2
        for shape in ((2, 2, 2), (64, 2, 2)):
            nv, nmax = shape[0] * 4, shape[0]
            fields = 11 * na * nv * 4
            tables = na * na * 6 + images + na * nmax * (2 + 8)
            for precision in (0, 1) if nside > 1 else (0,):
                assert _bytes(*shape, nside, 0, precision) >= fields + tables
            # mirror faces keep the sweep without displacements
            assert _bytes(*shape, nside, 0) - _bytes(*shape, nside, 2) >= na * nmax * 8
