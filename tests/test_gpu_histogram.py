"""The quality histogram where its fast evaluation could differ from the
definition: bin edges that qualities fall on, ranges far from or much wider
than the qualities, coordinates whose products under- or overflow, degenerate
triangles, equal qualities.  Counts and minimum equal the oracle's; the mean,
a sum in another order, within 1e-12."""
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


def _scaled(factor, shift=0.0):
    m = meshgen.jittered_grid(40, 37, 0.3, 5)
    m.xy = m.xy * factor + shift
    return m


MESHES = {
    "grid": lambda: meshgen.jittered_grid(300, 257, 0.35, 3, pull_fraction=0.1, pull_centres=32),
    "delaunay": lambda: meshgen.delaunay_random(20000, 4),
    "uniform": lambda: meshgen.jittered_grid(65, 65, 0.0, 3, h=2.0 ** -6, diagonals="uniform"),
    "one": lambda: meshgen.edge_case_meshes()[0],
    "degenerate": lambda: meshgen.edge_case_meshes()[1],
    "overflowing": lambda: _scaled(1e200),
    "underflowing": lambda: _scaled(1e-170),
    "far": lambda: _scaled(1.0, 1e6),
}
RANGES = [(20, -1.0, 1.0), (1, -1.0, 1.0), (4096, -1.0, 1.0), (256, 0.0, 1.0), (10, 0.8660254037844386, 1.0),
          (7, -1e300, 1e300), (33, 0.5, 0.5000001), (16, 1e6, 2e6)]


@pytest.mark.parametrize("layout", ["aos", "soa"])
@pytest.mark.parametrize("name", sorted(MESHES))
def test_histogram_equals_the_definition(sls, name, layout):
    mesh = MESHES[name]()
    om = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary)
    with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary, layout=layout) as g:
        for nbins, lo, hi in RANGES:
            counts, qmin, qmean = g.histogram(nbins, lo, hi)
            rcounts, rmin, rmean = om.histogram(mesh.xy, nbins, lo, hi)
            assert np.array_equal(counts, rcounts), (nbins, lo, hi)
            assert qmin == rmin or (qmin != qmin and rmin != rmin)
            assert rmean != rmean or abs(qmean - rmean) <= 1e-12 * max(abs(rmean), 1e-300)
