"""Level counts beyond what an int nlon can be halved to are refused on the host (the
shift that checks the divisibility has no meaning there)."""
import ctypes

import pytest


@pytest.mark.parametrize("levels", [30, 31, 32, 33, 34, 40, 64, 1000])
def test_too_many_levels(levels):
    from paper_2307_04528_gb300 import _lib as L
    lib = L.load()
    g, p, n = L.mg_grid(64, 32, 4), L.default_params(levels=levels), ctypes.c_size_t(0)
    assert lib.mg_workspace_bytes(ctypes.byref(g), ctypes.byref(p),
                                  ctypes.byref(n)) == L.MG_ERR_ARG


def test_most_levels():
    from paper_2307_04528_gb300 import _lib as L
    lib = L.load()
    g, p, n = L.mg_grid(64, 32, 4), L.default_params(levels=6), ctypes.c_size_t(0)
    assert lib.mg_workspace_bytes(ctypes.byref(g), ctypes.byref(p), ctypes.byref(n)) == 0
