"""Workspace queries (host only): a buffer sized for the largest grid serves every smaller
one, also across the grid sizes at which kernels change their blocks."""
import ctypes as C

import pytest

from paper_2105_14782_gb300 import _build


@pytest.fixture(scope="module")
def lib():
    return C.CDLL(_build.build())


def test_response_workspace_grows_with_the_grid(lib):
    f = lib.response_workspace_bytes
    f.restype, f.argtypes = C.c_size_t, [C.c_int64]
    sizes = [f(n) for n in range(1, 40000)]
    assert all(a <= b for a, b in zip(sizes, sizes[1:]))


def test_emission_workspace_grows_with_the_grid_and_the_layers(lib):
    f = lib.emission_workspace_bytes
    f.restype, f.argtypes = C.c_size_t, [C.c_int32, C.c_int64]
    for L in (1, 5, 100):
        sizes = [f(L, n) for n in range(1, 40000)]
        assert all(a <= b for a, b in zip(sizes, sizes[1:]))
    for n in (500, 9727, 20000):
        sizes = [f(L, n) for L in range(1, 200)]
        assert all(a <= b for a, b in zip(sizes, sizes[1:]))
