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


@pytest.mark.parametrize("numbering", ["morton", "random"])
@pytest.mark.parametrize("passes, tol", [(37, 0.0), (200, 1e-4)])
def test_a_refused_launch_falls_back(sls, numbering, passes, tol):
    # more windows than blocks can be resident together: the driver refuses the
    # cooperative launch, and the passes are launched one by one
    mesh = meshgen.jittered_grid(601, 457, 0.35, 62, numbering=numbering)
    want, winfo, wacc = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary, openmp=True).smooth(mesh.xy, passes, tol=tol)
    with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary, record_accept=True) as g:
        assert sls.lib().sls_test_resident(g.handle, 0) == 0
        for _ in range(2):
            g.set_coords(mesh.xy)
            info = g.smooth(passes, tol)
            assert np.array_equal(g.coords(), want) and np.array_equal(g.accept_mask(), wacc)
            for key in ("iterations", "converged", "accepted_last", "maxd2_last"):
                assert info[key] == winfo[key], key
            assert info["launches"] >= winfo["iterations"]


def test_two_such_meshes_at_once(sls):
    # two threads, each with a mesh that fills the GPU's resident blocks: the
    # launches cannot run side by side and must not wait for each other's blocks
    import threading
    mesh = meshgen.jittered_grid(421, 311, 0.35, 63)
    want, _, _ = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary, openmp=True).smooth(mesh.xy, 25)
    bad = []

    def work():
        try:
            with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary) as g:
                for _ in range(20):
                    g.set_coords(mesh.xy)
                    info = g.smooth(25)
                    if info["launches"] != 1 or not np.array_equal(g.coords(), want):
                        bad.append(info)
        except Exception as e:  # noqa: BLE001 (reported by the main thread)
            bad.append(e)

    threads = [threading.Thread(target=work) for _ in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(120.0)
    assert not bad and not any(t.is_alive() for t in threads)
