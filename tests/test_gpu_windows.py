"""The window stream of the screened pass: meshes at the edges of its forms
(8- and 16-bit lists, 64-node windows, open and irregular rings, rings around
the longest that fit, spatial renumbering, all passes in one launch or one
launch each, full queues), every one bit-identical to the oracle."""
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


def _check(sls, mesh, iters, tol=0.0, strict=False, **opts):
    rxy, rinfo, racc = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary).smooth(mesh.xy, iters, tol=tol, strict=strict)
    with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary, strict=strict, record_accept=True, **opts) as g:
        info = g.smooth(iters, tol)
        xy, acc = g.coords(), g.accept_mask()
    assert np.array_equal(xy, rxy)
    assert np.array_equal(acc, racc)
    for k in ("iterations", "converged", "accepted_last", "maxd2_last"):
        assert info[k] == rinfo[k], k
    return info


def _turned(mesh, share, seed):
    """Some triangles stored the other way round, all of them rotated."""
    rng = np.random.default_rng(seed)
    tri = mesh.tri.copy()
    t = rng.random(len(tri)) < share
    tri[t] = tri[t][:, [0, 2, 1]]
    spin = rng.integers(0, 3, len(tri))
    tri = np.stack([tri[np.arange(len(tri)), (spin + k) % 3] for k in range(3)], 1)
    return meshgen.Mesh(xy=mesh.xy, tri=np.ascontiguousarray(tri, np.int32), boundary=mesh.boundary)


def _with_free_rim(mesh):
    """Boundary nodes free but for the four corners: open fans."""
    b = np.zeros(mesh.n, np.uint8)
    corners = [np.argmin(mesh.xy @ np.array(d)) for d in ((1, 1), (1, -1), (-1, 1), (-1, -1))]
    b[corners] = 1
    return meshgen.Mesh(xy=mesh.xy, tri=mesh.tri, boundary=b)


def _split_thrice(nx, ny, seed):
    """Every triangle of a grid cut into six around its centre and edge
    midpoints, the grid's nodes (degree 12 inside) numbered first and at
    random: windows whose neighbours are all different."""
    g = meshgen.jittered_grid(nx, ny, 0.2, seed, numbering="random")
    mid, xy, tri, bnd = {}, list(map(tuple, g.xy)), [], list(g.boundary)
    uses = {}
    for a, b, c in g.tri:
        for u, v in ((a, b), (b, c), (c, a)):
            uses[(min(u, v), max(u, v))] = uses.get((min(u, v), max(u, v)), 0) + 1
    def m(u, v):
        k = (min(u, v), max(u, v))
        if k not in mid:
            mid[k] = len(xy)
            xy.append(tuple(0.5 * (np.array(xy[u]) + np.array(xy[v])) + 1e-3 * np.sin([u + 2.0 * v, 3.0 * u - v]) / nx))
            bnd.append(1 if uses[k] == 1 else 0)
        return mid[k]
    for a, b, c in g.tri:
        ab, bc, ca = m(a, b), m(b, c), m(c, a)
        z = len(xy)
        xy.append(tuple((np.array(xy[a]) + np.array(xy[b]) + np.array(xy[c])) / 3.0))
        bnd.append(0)
        tri += [(a, ab, z), (ab, b, z), (b, bc, z), (bc, c, z), (c, ca, z), (ca, a, z)]
    return meshgen.Mesh(xy=np.array(xy), tri=np.array(tri, np.int32), boundary=np.array(bnd, np.uint8))


def _fans(degrees, seed):
    """One free node inside a ring of each given length, side by side."""
    rng = np.random.default_rng(seed)
    xy, tri, bnd = [], [], []
    for j, k in enumerate(degrees):
        ang = 2 * np.pi * (np.arange(k) + 0.3 * rng.random(k)) / k
        at = len(xy)
        xy += list(np.c_[3.0 * j + np.cos(ang), np.sin(ang)]) + [np.array([3.0 * j + 0.1, -0.05])]
        bnd += [1] * k + [0]
        tri += [(at + k, at + t, at + (t + 1) % k) for t in range(k)]
    return meshgen.Mesh(xy=np.array(xy), tri=np.array(tri, np.int32), boundary=np.array(bnd, np.uint8))


FORMS = {"resident": {}, "launches": dict(copy_back=True), "soa": dict(layout="soa"), "given": dict(numbering="given")}


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("share", [0.3, 1.0])
def test_turned_triangles(sls, form, share):
    _check(sls, _turned(meshgen.jittered_grid(61, 47, 0.35, 7, pull_fraction=0.05, pull_centres=16), share, 1), 30, 1e-9,
           **FORMS[form])
    _check(sls, _turned(meshgen.delaunay_random(3000, 8), share, 2), 12, **FORMS[form])


@pytest.mark.parametrize("form", sorted(FORMS))
def test_open_fans(sls, form):
    _check(sls, _with_free_rim(meshgen.jittered_grid(45, 33, 0.3, 9)), 25, **FORMS[form])
    _check(sls, _turned(_with_free_rim(meshgen.jittered_grid(45, 33, 0.3, 9)), 0.4, 3), 25, strict=True, **FORMS[form])


@pytest.mark.parametrize("form", sorted(FORMS))
def test_rings_around_the_longest(sls, form):
    _check(sls, _fans(list(range(3, 34)), 4), 4, **FORMS[form])


@pytest.mark.parametrize("form", sorted(FORMS))
def test_windows_of_64_nodes(sls, form):
    _check(sls, _split_thrice(31, 29, 5), 10, **FORMS[form])


@pytest.mark.parametrize("numbering", ["natural", "random"])
@pytest.mark.parametrize("n", [(89, 91), (181, 131)])
def test_numberings_that_are_not_local(sls, numbering, n):
    # below and above the size from which such a mesh is renumbered
    mesh = meshgen.jittered_grid(n[0], n[1], 0.35, 10, numbering=numbering)
    for opts in ({}, dict(layout="soa"), dict(numbering="given"), dict(copy_back=True)):
        _check(sls, mesh, 20, 1e-9, **opts)


def test_renumbered_duplicate_points(sls):
    # equal coordinates among a node's neighbours: the caller's ids decide the
    # summation order, also in a renumbered mesh
    mesh = meshgen.jittered_grid(120, 97, 0.3, 11, numbering="random")
    rng = np.random.default_rng(12)
    for t in rng.choice(mesh.m, 300, replace=False):
        a, b, _ = mesh.tri[t]
        if not mesh.boundary[a]:
            mesh.xy[a] = mesh.xy[b]
    _check(sls, mesh, 8)


def test_renumbered_then_host_build(sls):
    # a node in more triangles than the device build handles, in a mesh whose
    # numbering would be changed
    mesh = meshgen.jittered_grid(120, 97, 0.3, 13, numbering="random")
    fan = _fans([40], 14)
    m = meshgen.Mesh(xy=np.vstack([mesh.xy, fan.xy + 5.0]), tri=np.vstack([mesh.tri, fan.tri + mesh.n]).astype(np.int32),
                     boundary=np.concatenate([mesh.boundary, fan.boundary]))
    _check(sls, m, 6)


def test_many_passes_of_one_launch(sls):
    mesh = meshgen.jittered_grid(8, 7, 0.3, 15)
    _check(sls, mesh, 4100)
    info = _check(sls, mesh, 9000, 1e-7)
    assert info["converged"] == 1


@pytest.mark.parametrize("layout", ["aos", "soa"])
def test_full_queue(sls, layout):
    # far from the origin no local frame holds: every node's every quality is
    # evaluated in FP64, more of them than the queue takes
    mesh = meshgen.jittered_grid(40, 37, 0.3, 16)
    mesh.xy = mesh.xy + 3.0e7
    info = _check(sls, mesh, 5, layout=layout)
    assert info["fp64_fallbacks"] > 1000
    _check(sls, mesh, 5, layout=layout, copy_back=True)


def test_block_sizes(sls):
    mesh = meshgen.jittered_grid(75, 63, 0.35, 17, pull_fraction=0.05, pull_centres=16)
    for block in (32, 64, 96, 128, 256):
        for cb in (False, True):
            _check(sls, mesh, 9, block_size=block, copy_back=cb)


def test_mixed_list_widths_in_a_batch(sls):
    meshes = [meshgen.jittered_grid(90, 80, 0.3, 18), meshgen.jittered_grid(70, 75, 0.3, 19, numbering="random"),
              _split_thrice(11, 13, 20), _fans([5, 16, 20], 21)]
    iters = [12, 7, 9, 3]
    handles = [sls.Mesh(m.xy, m.tri, m.boundary, numbering="given", kernel="fp64" if k == 1 else "auto")
               for k, m in enumerate(meshes)]
    try:
        with sls.Batch(handles, iters) as b:
            b.smooth()
            for k, m in enumerate(meshes):
                want, _, _ = oracle.OracleMesh(m.xy, m.tri, m.boundary).smooth(m.xy, iters[k])
                assert np.array_equal(b.coords(k), want), k
    finally:
        for h in handles:
            h.close()


def test_served_random_numbering(sls):
    mesh = meshgen.jittered_grid(150, 120, 0.35, 22, numbering="random")
    srv = sls.Server()
    try:
        jid = srv.submit(mesh.xy, mesh.tri, mesh.boundary, max_iter=15, tol=1e-9)
        xy, info = srv.wait(jid, timeout=60.0)
    finally:
        srv.close()
    want, rinfo, _ = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary).smooth(mesh.xy, 15, tol=1e-9)
    assert np.array_equal(xy, want) and info["maxd2_last"] == rinfo["maxd2_last"]


def _check32(sls, mesh, iters, tol=0.0, strict=False, form="A", **opts):
    rxy, rinfo, racc = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary).smooth(
        mesh.xy, iters, tol=tol, strict=strict, form=form, precision=32)
    with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary, strict=strict, record_accept=True, form=form, precision=32,
                  **opts) as g:
        info = g.smooth(iters, tol)
        xy, acc = g.coords(), g.accept_mask()
    assert np.array_equal(xy, rxy)
    assert np.array_equal(acc, racc)
    for k in ("iterations", "accepted_last", "maxd2_last"):
        assert info[k] == rinfo[k], k


@pytest.mark.parametrize("form", ["A", "B"])
@pytest.mark.parametrize("layout", ["aos", "soa"])
def test_binary32_forms(sls, form, layout):
    opts = dict(form=form, layout=layout)
    grid = meshgen.jittered_grid(61, 47, 0.35, 7, pull_fraction=0.05, pull_centres=16)
    _check32(sls, grid, 60, 1e-9, **opts)                       # down to rounding-level ties
    _check32(sls, grid, 20, strict=True, **opts)
    _check32(sls, _turned(grid, 0.3, 1), 20, **opts)
    _check32(sls, _turned(grid, 1.0, 2), 20, **opts)
    _check32(sls, _with_free_rim(meshgen.jittered_grid(45, 33, 0.3, 9)), 15, **opts)
    _check32(sls, _fans(list(range(3, 34)), 4), 4, **opts)
    _check32(sls, _split_thrice(31, 29, 5), 10, **opts)
    _check32(sls, meshgen.delaunay_random(5000, 6, numbering="random"), 15, **opts)
    _check32(sls, meshgen.jittered_grid(120, 97, 0.3, 11, numbering="random"), 10, **opts)
    _check32(sls, meshgen.jittered_grid(33, 33, 0.0, 3, h=2.0 ** -5, diagonals="uniform"), 3, **opts)


@pytest.mark.parametrize("scale", [1e-17, 1e-21, 1e14, 1e18, 1e30])
def test_binary32_range(sls, scale):
    # sums of squares below and above the quick quotients' range, and infinite
    mesh = meshgen.jittered_grid(31, 29, 0.35, 23)
    mesh.xy = mesh.xy * scale
    with np.errstate(all="ignore"):
        for opts in ({}, dict(block_size=32)):
            rxy, rinfo, _ = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary).smooth(mesh.xy, 4, precision=32)
            with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary, precision=32, **opts) as g:
                info = g.smooth(4)
                assert np.array_equal(g.coords(), rxy, equal_nan=True)
            assert info["accepted_last"] == rinfo["accepted_last"]


def test_binary32_far_from_the_origin(sls):
    mesh = meshgen.jittered_grid(40, 37, 0.3, 16)
    mesh.xy = mesh.xy + 3.0e3
    _check32(sls, mesh, 12)
    _check32(sls, mesh, 12, strict=True, form="B")


def _pinched(fans, seed):
    """A free node where `fans` separate groups of three triangles meet."""
    rng = np.random.default_rng(seed)
    xy, tri = [np.array([0.03, -0.02])], []
    for f in range(fans):
        ang = 2 * np.pi * (f + np.array([0.1, 0.3, 0.5, 0.8]) + 0.05 * rng.random(4)) / fans
        at = len(xy)
        xy += list(np.c_[np.cos(ang), np.sin(ang)])
        tri += [(0, at + k, at + k + 1) for k in range(3)]
    bnd = np.ones(len(xy), np.uint8)
    bnd[0] = 0
    return meshgen.Mesh(xy=np.array(xy), tri=np.array(tri, np.int32), boundary=bnd)


@pytest.mark.parametrize("share", [0.0, 0.5, 1.0])
@pytest.mark.parametrize("rounded", [False, True])
def test_records_built_on_the_device(sls, share, rounded):
    # rings up to and beyond what the build keeps in registers (at most 32, so
    # the host build does not take over), all orientations, coordinates that tie
    fans = _fans(list(range(3, 33)), 16)
    grid = meshgen.jittered_grid(23, 19, 0.3, 17)
    for mesh in (fans, _with_free_rim(grid)):
        m = _turned(mesh, share, 18)
        if rounded:
            m = meshgen.Mesh(xy=np.round(m.xy * 8) / 8, tri=m.tri, boundary=m.boundary)  # also -0.0
        _check(sls, m, 3)
        _check(sls, m, 3, numbering="given")


@pytest.mark.parametrize("fans", [1, 2, 3, 5, 10])
def test_records_longer_than_their_place(sls, fans):
    # separate fans at a free node have more neighbours than its triangles
    # leave room for: the whole mesh is built with exact lengths
    mesh = _turned(_pinched(fans, 19), 0.5, 20)
    rest = meshgen.jittered_grid(31, 17, 0.3, 21)
    _check(sls, mesh, 3)
    both = meshgen.Mesh(xy=np.vstack([rest.xy, mesh.xy + 4.0]), tri=np.vstack([rest.tri, mesh.tri + rest.n]).astype(np.int32),
                        boundary=np.concatenate([rest.boundary, mesh.boundary]))
    _check(sls, both, 5)
