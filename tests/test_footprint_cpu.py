"""The bound by which the server admits a job (csrc/footprint.h, compiled for
the host) against the bytes that a build can take: window streams of the worst
windows of either width, adjacency at fixed places and of exact lengths, and the
buffers of every step of the build."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1502_00355_gb300", "csrc")

SHIM = r"""
#include "footprint.h"
using namespace sls;
extern "C" unsigned long long stream_bound(long long n, long long m) { return window_stream_bound(n, m); }
extern "C" unsigned long long admission(long long n, long long m) { return admission_bound(n, m, 32); }
// bytes of a window as window_build.cu lays it out: d, l: degree and step
// number of each of its four subtiles
extern "C" unsigned long long window_bytes(const unsigned *d, const unsigned *l, unsigned halo, unsigned bits) {
    unsigned long long rows = win::halo_rows(halo) + win::kColdRows;
    for (int k = 0; k < 4; ++k) rows += win::subtile_rows(d[k], l[k], bits);
    return rows * 128 + 4 * win::kHeaderWords;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("footprint")
    (d / "shim.cpp").write_text(SHIM)
    so = d / "libfoot.so"
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp"), "-o", str(so)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = C.CDLL(str(so))
    for f in (L.stream_bound, L.admission, L.window_bytes):
        f.restype = C.c_ulonglong
    L.stream_bound.argtypes = L.admission.argtypes = [C.c_longlong, C.c_longlong]
    return L


SIZES = [3, 31, 64, 65, 127, 128, 129, 1000, 4096, 9999, 65536, 100001]


@pytest.mark.parametrize("width", [64, 128])
@pytest.mark.parametrize("n", SIZES)
def test_streams_of_the_worst_windows(lib, width, n):
    # rings of 15 in every subtile that has a node, every neighbour in the halo;
    # a node of degree 15 has 15 corners, so n nodes mean at least 5 n triangles
    total = 0
    for first in range(0, n, width):
        count = min(width, n - first)
        used = (count + 31) // 32
        d = (C.c_uint * 4)(*[15 if k < used else 0 for k in range(4)])
        total += lib.window_bytes(d, d, min(15 * count, 1920), 16)
    assert lib.stream_bound(n, 5 * n) >= total


@pytest.mark.parametrize("seed", range(5))
def test_streams_of_random_windows(lib, seed):
    rng = np.random.default_rng(seed)
    for n in SIZES:
        for width, bits in ((128, 8), (128, 16), (64, 16)):
            total, corners = 0, 0
            for first in range(0, n, width):
                count = min(width, n - first)
                used = (count + 31) // 32
                deg = [int(rng.integers(2, 16)) if k < used else 0 for k in range(4)]
                corners += sum(x * min(32, max(0, count - 32 * k)) for k, x in enumerate(deg))
                total += lib.window_bytes((C.c_uint * 4)(*deg), (C.c_uint * 4)(*deg),
                                          int(rng.integers(0, 1 + sum(deg) * 32)), bits)
            assert lib.stream_bound(n, (corners + 2) // 3) >= total


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("ratio", [0.0, 0.1, 0.33, 1.0, 1.9, 5.0])
def test_every_step_fits(lib, n, ratio):
    m = max(1, int(n * ratio))
    bound = lib.admission(n, m)
    held = 32 * n + 32 + 12 * m  # both coordinate arrays, statistics, triangles
    bits = 1
    while bits < 13 and 4 ** bits <= n:
        bits += 1
    cells = 4 ** bits
    scan = 8 * (cells // 4096 + 2)
    assert bound >= held + 4 * cells + 4 * (cells + 1) + 8 * n + 16 * n + scan  # the spatial numbering
    maps, counts = 8 * n, 2 * 4 * (n + 1) + 12 * m + n
    assert bound >= held + maps + counts + 4 * (n + 1) + 4 * (2 * n + 6 * m)  # records at fixed places
    exact = 24 * m + 4 * (n + 1) + n + 4 * n
    assert bound >= held + maps + counts + exact + 4 * (n + 1) + 4 * (n + 9 * m)  # of exact lengths
    for words in (2 * n + 6 * m, n + 9 * m):  # the stream (the triangles and one map are gone)
        assert bound >= 32 * n + 32 + 4 * n + 4 * (n + 1) + 4 * words + lib.stream_bound(n, m)


def test_no_more_than_the_largest_step(lib):
    # a planar mesh (m = 2 n): what it may hold, not the sum over its steps
    n = 1 << 20
    assert lib.admission(n, 2 * n) <= 262 * n + 65536
