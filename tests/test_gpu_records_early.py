"""Rounds of the batched and served forms start while the round before still
runs; nodes decided by their records (more than 15 neighbours, coordinates
outside the splits' range) read coordinates that this round has just written.
Meshes of many windows with such nodes all over, their neighbours moving and in
other windows, many rounds, bit-identical to the oracle."""
import numpy as np
import pytest

import meshgen
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sls():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1502_00355_gb300 as mod
    mod.build()
    mod.lib()
    return mod


def _hubs(side, ring, seed):
    """side x side free nodes of degree `ring` or so, each in a ring of free
    nodes, in a Delaunay triangulation numbered at random."""
    from scipy.spatial import Delaunay
    rng = np.random.default_rng(seed)
    pts = []
    for i in range(side):
        for j in range(side):
            ang = 2 * np.pi * (np.arange(ring) + 0.2 * rng.random(ring)) / ring
            pts += [np.array([[i, j]]), np.c_[i + 0.4 * np.cos(ang), j + 0.4 * np.sin(ang)] * 1.0]
    pts = np.vstack(pts)[rng.permutation(side * side * (ring + 1))]
    dt = Delaunay(pts)
    bnd = np.zeros(len(pts), np.uint8)
    bnd[np.unique(dt.convex_hull)] = 1
    return meshgen.Mesh(xy=pts, tri=np.ascontiguousarray(dt.simplices, np.int32), boundary=bnd)


def _meshes():
    tiny = meshgen.jittered_grid(61, 53, 0.35, 41, numbering="random")
    tiny = meshgen.Mesh(xy=tiny.xy * 2.0 ** -100, tri=tiny.tri, boundary=tiny.boundary)  # all nodes by their records
    return [_hubs(14, 21, 42), tiny, meshgen.jittered_grid(120, 90, 0.35, 43), _hubs(9, 33, 44), _hubs(11, 17, 45)]


ITERS = [60, 45, 60, 37, 50]


@pytest.fixture(scope="module")
def wanted():
    out = []
    for m, it in zip(_meshes(), ITERS):
        out.append(oracle.OracleMesh(m.xy, m.tri, m.boundary).smooth(m.xy, it))
    return out


def test_the_meshes_hold_such_nodes():
    for m in (_meshes()[0], _meshes()[3]):
        deg = np.bincount(m.tri.reshape(-1), minlength=m.n)
        assert (deg[m.boundary == 0] > 15).sum() > 50 and m.n > 20 * 128


@pytest.mark.parametrize("layout", ["aos", "soa"])
@pytest.mark.parametrize("chunk", [0, 1, 8, -2])
def test_batched(sls, wanted, layout, chunk):
    meshes = _meshes()
    handles = [sls.Mesh(m.xy, m.tri, m.boundary, layout=layout, numbering="given", record_accept=True) for m in meshes]
    try:
        with sls.Batch(handles, ITERS, layout=layout) as b:
            b.set_shape(128, chunk)
            for _ in range(3):
                b.reset()
                infos = b.smooth()
                for j, (xy, info, acc) in enumerate(wanted):
                    assert np.array_equal(b.coords(j), xy), j
                    assert np.array_equal(handles[j].accept_mask(), acc), j
                    assert infos[j]["accepted_last"] == info["accepted_last"]
    finally:
        for h in handles:
            h.close()


def test_served(sls, wanted):
    srv = sls.Server(numbering="given")
    try:
        for _ in range(3):
            ids = [srv.submit(m.xy, m.tri, m.boundary, max_iter=it) for m, it in zip(_meshes(), ITERS)]
            for jid, (want, winfo, _) in zip(ids, wanted):
                xy, info = srv.wait(jid, timeout=120.0)
                assert np.array_equal(xy, want)
                assert info["accepted_last"] == winfo["accepted_last"]
    finally:
        srv.close()
