"""The form that runs all passes of a small mesh in one launch: a wait between
its blocks that runs out is reported whichever launch of the call it was in."""
import ctypes as C

import numpy as np
import pytest

import meshgen
import oracle

pytestmark = pytest.mark.gpu

TIMEOUT = 5


@pytest.fixture(scope="module")
def sls():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1502_00355_gb300 as mod
    mod.build()
    f = mod.lib().sls_test_resident
    f.restype, f.argtypes = C.c_int, [C.c_void_p, C.c_uint32]
    return mod


@pytest.mark.parametrize("layout", ["aos", "soa"])
@pytest.mark.parametrize("passes, tol", [(10, 0.0), (200, 1e-9), (4097, 0.0), (9000, 0.0), (9000, 1e-300)])
def test_a_wait_that_runs_out(sls, layout, passes, tol):
    # one poll, in the call's first launch only (4,096 passes a launch): blocks
    # that are not the last to arrive give up, and later launches find that out
    mesh = meshgen.jittered_grid(101, 97, 0.35, 61)
    with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary, layout=layout) as g:
        assert sls.lib().sls_test_resident(g.handle, 1) == 0
        with pytest.raises(sls.SlsError) as e:
            g.smooth(passes, tol)
        assert e.value.code == TIMEOUT
        # the handle is as good as before once it has its coordinates again
        g.set_coords(mesh.xy)
        info = g.smooth(20)
        want, winfo, _ = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary).smooth(mesh.xy, 20)
        assert np.array_equal(g.coords(), want) and info["accepted_last"] == winfo["accepted_last"]
        assert info["launches"] == 1
