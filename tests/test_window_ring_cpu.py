"""The ring order of a node's triangles (csrc/window.cuh: order_ring), which
the screened pass walks instead of the adjacency record's triangle list.  The
header compiles for the host; every ring is expanded back and must give
exactly the node's triangles, each with its slot and the stored order of its
other two vertices, whatever the link looks like: closed rings, fans with an
open end, several fans or rings at one node, triangles stored in either
direction, the same triangle twice."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import meshgen
import oracle

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1502_00355_gb300", "csrc")

SHIM = r"""
#include "window.cuh"
extern "C" int ring(const uint32_t *codes, uint32_t deg, uint32_t ntri, uint64_t *seq, uint32_t *out) {
    const sls::win::Ring r = sls::win::order_ring(codes, deg, ntri);
    *seq = r.seq;
    out[0] = r.steps; out[1] = r.slots; out[2] = r.rev; out[3] = r.regular; out[4] = r.ok;
    return 0;
}
"""


@pytest.fixture(scope="module")
def ring(tmp_path_factory):
    d = tmp_path_factory.mktemp("ring")
    (d / "shim.cpp").write_text(SHIM)
    so = d / "libring.so"
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp"), "-o", str(so)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = C.CDLL(str(so))

    def order(codes, deg):
        a = np.ascontiguousarray(codes, np.uint32)
        seq, out = C.c_uint64(), (C.c_uint32 * 5)()
        L.ring(a.ctypes.data_as(C.c_void_p), deg, len(a), C.byref(seq), out)
        return seq.value, list(out)

    return order


def _expand(seq, out):
    """(slot, first, second) of every step with a triangle, positions in stored order."""
    steps, slots, rev = out[0], out[1], out[2]
    got = []
    for t in range(steps):
        slot = (slots >> (2 * t)) & 3
        if slot == 3:
            continue
        p, q = (seq >> (4 * t)) & 15, (seq >> (4 * t + 4)) & 15
        swap = bool((rev >> t) & 1) != (slot == 1)
        got.append((slot, q, p) if swap else (slot, p, q))
    return got


def _codes(tris, node, nbrs):
    pos = {v: k for k, v in enumerate(nbrs)}
    out = []
    for t in tris:
        slot = list(t).index(node)
        a, b = [pos[v] for v in t if v != node]
        out.append((slot << 30) | (a << 15) | b)
    return out


def _check(ring, codes, deg):
    seq, out = ring(codes, deg)
    if not out[4]:
        return False, False
    want = sorted(((c >> 30), (c >> 15) & 0x7FFF, c & 0x7FFF) for c in codes)
    assert sorted(_expand(seq, out)) == want
    assert out[0] <= 15
    visited = {(seq >> (4 * t)) & 15 for t in range(out[0] + 1)}
    assert visited == set(range(deg))
    return True, bool(out[3])


@pytest.mark.parametrize("flip", [0.0, 0.3, 1.0])
@pytest.mark.parametrize("name", ["grid", "delaunay"])
def test_mesh_rings(ring, name, flip):
    mesh = meshgen.jittered_grid(23, 19, 0.35, 5) if name == "grid" else meshgen.delaunay_random(700, 6)
    rng = np.random.default_rng(8)
    tri = mesh.tri.copy()
    turned = rng.random(len(tri)) < flip
    tri[turned] = tri[turned][:, [0, 2, 1]]
    spin = rng.integers(0, 3, len(tri))
    tri = np.stack([tri[np.arange(len(tri)), (spin + k) % 3] for k in range(3)], 1)
    regular = 0
    for node in range(mesh.n):   # boundary nodes too: their fans are open
        tris = [tuple(t) for t in tri[(tri == node).any(1)]]
        nbrs = sorted({v for t in tris for v in t} - {node}, key=lambda v: tuple(mesh.xy[v]))
        ok, reg = _check(ring, _codes(tris, node, nbrs), len(nbrs))
        assert ok == (len(nbrs) <= 15 and len(tris) <= 15)
        regular += reg
    inner = int((mesh.boundary == 0).sum())
    if flip in (0.0, 1.0):
        assert regular >= 0.98 * inner   # closed rings stored one way round are the regular case
    else:
        assert regular < inner


def test_links_of_several_pieces(ring):
    # node 0; fans and rings over disjoint neighbour sets, a doubled triangle
    cases = {
        "two_rings": [(0, 1, 2), (0, 2, 3), (0, 3, 1), (0, 4, 5), (0, 5, 6), (0, 6, 4)],
        "ring_and_fan": [(0, 1, 2), (0, 2, 3), (0, 3, 1), (0, 4, 5), (5, 6, 0)],
        "three_fans": [(0, 1, 2), (0, 3, 4), (4, 5, 0), (6, 0, 7)],
        "doubled": [(0, 1, 2), (0, 1, 2)],
        "pillow": [(0, 1, 2), (0, 2, 1)],
        "one": [(1, 0, 2)],
    }
    for name, tris in cases.items():
        nbrs = sorted({v for t in tris for v in t} - {0})
        ok, _ = _check(ring, _codes(tris, 0, nbrs), len(nbrs))
        assert ok, name


def test_longest_rings(ring):
    # 15 neighbours fit, closed or open; 16 do not; nor do links whose steps
    # and breaks together exceed 15
    for deg, closed, fits in ((15, True, True), (15, False, True), (14, True, True), (16, True, False)):
        tris = [(0, 1 + k, 1 + (k + 1) % deg) for k in range(deg if closed else deg - 1)]
        ok, _ = _check(ring, _codes(tris, 0, list(range(1, deg + 1))), deg)
        assert ok == fits
    tris = [(0, 1 + 2 * k, 2 + 2 * k) for k in range(7)]          # seven fans: 7 + 6 steps
    assert _check(ring, _codes(tris, 0, list(range(1, 15))), 14)[0]
    rings = [[(0, b, b + 1), (0, b + 1, b + 2), (0, b + 2, b)] for b in (1, 4, 7, 10, 13)]
    assert _check(ring, _codes(sum(rings[:4], []), 0, list(range(1, 13))), 12)[0]      # 12 + 3 steps
    assert not _check(ring, _codes(sum(rings, []), 0, list(range(1, 16))), 15)[0]      # 15 + 4 steps


def test_same_triangles_as_the_oracle(ring):
    mesh = meshgen.delaunay_random(300, 9)
    nbr_ptr, nbr, tri_ptr, tri_of, _ = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary).adjacency()
    for node in range(mesh.n):
        nbrs = list(nbr[nbr_ptr[node]:nbr_ptr[node + 1]])
        tris = [tuple(mesh.tri[t]) for t in tri_of[tri_ptr[node]:tri_ptr[node + 1]]]
        if 0 < len(nbrs) <= 15 and len(tris) <= 15:
            assert _check(ring, _codes(tris, node, nbrs), len(nbrs))[0]
