"""sls_smooth_noalloc on a mesh that the library renumbered inside: the same
bits as sls_smooth, on either stream and either buffer, and no device memory
taken by a process's first call, loading of code included."""
import os
import subprocess
import sys

import numpy as np
import pytest

import meshgen
import oracle

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1502_00355_gb300 as sls
    sls.build()
    sls.lib()
    return sls, torch


FIRST_CALL = """
import numpy as np, torch
import meshgen, paper_1502_00355_gb300 as sls
mesh = meshgen.jittered_grid(128, 96, 0.35, 71, numbering="random")
xy = torch.from_numpy(mesh.xy).cuda()
a, b = xy * 1.0, xy * 0.0
torch.cuda.synchronize()
g = sls.Mesh(mesh.xy, mesh.tri, mesh.boundary)
torch.cuda.synchronize()
free0 = torch.cuda.mem_get_info()[0]
info = g.smooth_noalloc(a, b, 25)
torch.cuda.synchronize()
free1 = torch.cuda.mem_get_info()[0]
assert free0 == free1, (free0, free1)
assert info["iterations"] == 25
g.set_coords(mesh.xy)
g.smooth(25)
assert np.array_equal(b.cpu().numpy(), g.coords())
"""


def test_first_call_of_a_process(env):
    r = subprocess.run([sys.executable, "-c", FIRST_CALL], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env={**os.environ, "CUDA_MODULE_LOADING": "LAZY"})
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("passes, tol", [(0, 0.0), (30, 0.0), (31, 0.0), (300, 1e-6)])
def test_same_bits(env, passes, tol):
    sls, torch = env
    mesh = meshgen.jittered_grid(131, 97, 0.35, 72, numbering="random")
    want, winfo, _ = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary).smooth(mesh.xy, passes, tol=tol)
    side = torch.cuda.Stream()
    with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary) as g:
        for stream in (None, side.cuda_stream):
            a = torch.from_numpy(mesh.xy.copy()).cuda()
            b = torch.empty_like(a)
            torch.cuda.synchronize()
            info = g.smooth_noalloc(a, b, passes, tol, stream=stream)
            assert np.array_equal(b.cpu().numpy(), want)
            for key in ("iterations", "converged", "accepted_last", "maxd2_last"):
                assert info[key] == winfo[key], key
