"""Binary32 passes where the quick quotients of the accept test are not to be
trusted: qualities below the normal range (coordinates of subnormal extent in
one direction) and coordinates that are not finite, against the oracle's
binary32 definition, bit for bit."""
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


UNIT = 2.0 ** -149  # the least binary32 number


def _check(sls, mesh, start, iters, strict, **opts):
    with np.errstate(all="ignore"):
        rxy, rinfo, racc = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary).smooth(start, iters, strict=strict,
                                                                                      precision=32)
    import torch
    with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary, strict=strict, record_accept=True, precision=32, **opts) as g:
        g.set_coords(torch.from_numpy(start).cuda())  # (device input may hold anything)
        info = g.smooth(iters)
        xy, acc = g.coords(), g.accept_mask()
    assert np.array_equal(acc, racc)
    assert np.array_equal(xy, rxy, equal_nan=True)
    for k in ("iterations", "accepted_last"):
        assert info[k] == rinfo[k], k


def test_one_ring_of_subnormal_width(sls):
    # both minima are 22 units of 2^-149 exactly; a product with a reciprocal
    # makes one of them 23
    ring = np.array([(47, 1), (24, 2), (-55, -1), (-39, -2), (-2, -2), (-16, -1)], float) * [UNIT, 1.0]
    tri = np.array([(5, k, (k + 1) % 5) for k in range(5)], np.int32)
    mesh = meshgen.Mesh(xy=ring, tri=tri, boundary=np.array([1, 1, 1, 1, 1, 0], np.uint8))
    for strict in (False, True):
        _check(sls, mesh, mesh.xy, 1, strict)


@pytest.mark.parametrize("units", [60.0, 3e3, 1e6, 1e9, 1e13, 1e18])
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("opts", [dict(), dict(layout="soa", block_size=32), dict(form="B")], ids=["aos", "soa", "b"])
def test_meshes_of_subnormal_width(sls, units, axis, opts):
    # one direction about `units` least numbers wide per cell, the other one
    # of order 1: edge sums of order 1, qualities from 0 to beyond the normal range
    mesh = meshgen.jittered_grid(41, 37, 0.4, 31, pull_fraction=0.1, pull_centres=16, h=1.0)
    scale = np.ones(2)
    scale[axis] = units * UNIT
    mesh = meshgen.Mesh(xy=np.float32(mesh.xy * scale).astype(np.float64), tri=mesh.tri, boundary=mesh.boundary)
    opts = dict(opts)
    form = opts.pop("form", None)
    if form:
        with np.errstate(all="ignore"):
            rxy, rinfo, racc = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary).smooth(mesh.xy, 6, form="B",
                                                                                          precision=32)
        with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary, record_accept=True, precision=32, form="B") as g:
            info = g.smooth(6)
            assert np.array_equal(g.accept_mask(), racc)
            assert np.array_equal(g.coords(), rxy)
        assert info["accepted_last"] == rinfo["accepted_last"]
        return
    for strict in (False, True):
        _check(sls, mesh, mesh.xy, 6, strict, **opts)


@pytest.mark.parametrize("opts", [dict(), dict(layout="soa", block_size=32)], ids=["aos", "soa"])
@pytest.mark.parametrize("strict", [False, True])
def test_coordinates_that_are_not_numbers(sls, opts, strict):
    # a quality with a NaN in its edge sum is 0 by definition; NaN nodes among
    # finite ones, NaN in one coordinate only, and the infinity that a double
    # beyond the binary32 range becomes
    grid = meshgen.jittered_grid(41, 37, 0.35, 32)
    rng = np.random.default_rng(33)
    for bad in ((np.nan, np.nan), (np.nan, None), (None, np.nan), (1e300, 0.5)):
        start = grid.xy.copy()
        for i in rng.choice(grid.n, 40, replace=False):
            for c in range(2):
                if bad[c] is not None:
                    start[i, c] = bad[c]
        for iters in (1, 2, 5):
            _check(sls, grid, start, iters, strict, **opts)
