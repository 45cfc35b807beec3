"""skip_unchanged on meshes whose numbering lets no tile be skipped, or only the
tiles of one part: the results of the plain passes, and the skipped nodes counted
where there are any."""
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


def _side_by_side(a, b):
    """Two meshes in one, the second's ids after the first's."""
    return meshgen.Mesh(xy=np.vstack([a.xy, b.xy + [5.0, 0.0]]), tri=np.vstack([a.tri, b.tri + a.n]).astype(np.int32),
                        boundary=np.concatenate([a.boundary, b.boundary]))


RANDOM = meshgen.jittered_grid(97, 89, 0.35, 111, numbering="random")
LOCAL = meshgen.jittered_grid(65, 61, 0.3, 112)


@pytest.mark.parametrize("layout", ["aos", "soa"])
@pytest.mark.parametrize("mesh, skips", [(RANDOM, False), (_side_by_side(RANDOM, LOCAL), True)], ids=["none", "some"])
def test_results_and_counts(sls, layout, mesh, skips):
    want, winfo, wacc = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary).smooth(mesh.xy, 400, tol=1e-9)
    with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary, layout=layout, skip_unchanged=True, record_accept=True) as g:
        for _ in range(2):
            g.set_coords(mesh.xy)
            info = g.smooth(400, 1e-9)
            assert np.array_equal(g.coords(), want) and np.array_equal(g.accept_mask(), wacc)
            for k in ("iterations", "converged", "accepted_last", "maxd2_last"):
                assert info[k] == winfo[k], k
            assert (info["nodes_skipped"] > 0) == skips
