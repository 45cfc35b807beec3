"""Meshes most of whose accept tests the screen of the pass leaves open (flat
triangles, graded rows, coordinates far from the origin): the closer screen, the
queue and the qualities that warps evaluate 32 at a time when the queue has no
room, bit-identical to the oracle in every form that shares them."""
import numpy as np
import pytest

import meshgen
import oracle
from test_gpu_windows import _fans, _split_thrice, _turned, _with_free_rim

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


def _moved(mesh, scale=(1.0, 1.0), shift=0.0, graded=0.0):
    xy = mesh.xy.copy()
    if graded:
        t = (xy[:, 1] - xy[:, 1].min()) / (xy[:, 1].max() - xy[:, 1].min())
        xy[:, 1] = np.expm1(np.log(graded) * t) / np.expm1(np.log(graded))
    return meshgen.Mesh(xy=xy * scale + shift, tri=mesh.tri, boundary=mesh.boundary)


def _grid(**k):
    return meshgen.jittered_grid(103, 87, 0.35, 91, pull_fraction=0.05, pull_centres=16, **k)


MESHES = {
    "flat 1e-2": lambda: _moved(_grid(), (1.0, 1e-2)),
    "flat 1e-3": lambda: _moved(_grid(), (1.0, 1e-3)),
    "flat 1e-5": lambda: _moved(_grid(), (1e-5, 1.0)),
    "flat 1e-9": lambda: _moved(_grid(), (1.0, 1e-9)),
    "graded": lambda: _moved(_grid(), graded=1e6),
    "graded rows": lambda: _moved(_grid(numbering="natural"), graded=1e4),
    "far": lambda: _moved(_grid(), shift=1e5),
    "far and flat": lambda: _moved(_grid(), (1.0, 1e-3), shift=300.0),
    "turned": lambda: _turned(_moved(_grid(), (1.0, 1e-3)), 0.4, 92),
    "open fans": lambda: _turned(_with_free_rim(_moved(_grid(), (1.0, 1e-4))), 0.2, 93),
    "delaunay": lambda: _moved(meshgen.delaunay_random(7000, 94), (1.0, 1e-3)),
    "long rings": lambda: _moved(_fans(list(range(3, 16)) * 24, 95), (1.0, 1e-4)),
    "rings of 12": lambda: _moved(_split_thrice(23, 19, 96), (1.0, 1e-3)),
}
KEYS = ("iterations", "converged", "accepted_last", "maxd2_last")


@pytest.mark.parametrize("name", sorted(MESHES))
@pytest.mark.parametrize("opts", [dict(), dict(copy_back=True, layout="soa"), dict(strict=True, numbering="given"),
                                  dict(skip_unchanged=True), dict(form="B"), dict(block_size=32, layout="soa")], ids=str)
def test_same_bits(sls, name, opts):
    mesh = MESHES[name]()
    kw = dict(strict=opts.get("strict", False), form=opts.get("form", "A"))
    want, winfo, wacc = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary).smooth(mesh.xy, 9, **kw)
    with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary, record_accept=True, **opts) as g:
        info = g.smooth(9)
        assert np.array_equal(g.coords(), want)
        assert np.array_equal(g.accept_mask(), wacc)
    for k in KEYS:
        assert info[k] == winfo[k], k


@pytest.mark.parametrize("name", ["flat 1e-3", "flat 1e-5", "graded", "far"])
def test_the_same_counts_every_time(sls, name):
    # which nodes find the queue full depends on the order of the warps; what a
    # call reports does not
    mesh = MESHES[name]()
    infos = []
    with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary, copy_back=True) as g:
        for _ in range(6):
            g.set_coords(mesh.xy)
            infos.append(g.smooth(20))
    assert infos[0]["fp64_fallbacks"] > mesh.n
    assert all(i == infos[0] for i in infos)


@pytest.mark.parametrize("layout", ["aos", "soa"])
def test_in_a_batch(sls, layout):
    names = sorted(MESHES)
    meshes = [MESHES[k]() for k in names]
    handles = [sls.Mesh(m.xy, m.tri, m.boundary, layout=layout, record_accept=True) for m in meshes]
    iters = [5 + j for j in range(len(meshes))]
    try:
        with sls.Batch(handles, iters, layout=layout) as b:
            infos = b.smooth()
            for j, m in enumerate(meshes):
                want, winfo, wacc = oracle.OracleMesh(m.xy, m.tri, m.boundary).smooth(m.xy, iters[j])
                assert np.array_equal(b.coords(j), want), names[j]
                assert np.array_equal(handles[j].accept_mask(), wacc), names[j]
                assert all(infos[j][k] == winfo[k] for k in KEYS), names[j]
    finally:
        for h in handles:
            h.close()
