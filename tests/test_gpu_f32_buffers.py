"""The binary32 pass with one buffer of window data and with two: wide windows
(random ids kept as they are, colour classes) of meshes with more and with fewer
windows than the GPU's blocks, a ragged number of windows a block, both layouts,
against the oracle."""
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


MESHES = {
    "one window a block": lambda: meshgen.jittered_grid(261, 187, 0.35, 101, numbering="random"),
    "two windows and a part": lambda: meshgen.jittered_grid(701, 609, 0.35, 102, numbering="random"),
    "rows": lambda: meshgen.jittered_grid(901, 403, 0.35, 103, numbering="natural"),
    "local": lambda: meshgen.jittered_grid(701, 467, 0.35, 104),
}


@pytest.mark.parametrize("name", sorted(MESHES))
@pytest.mark.parametrize("opts", [dict(numbering="given"), dict(numbering="given", layout="soa"), dict(form="B"),
                                  dict(form="B", layout="soa"), dict(numbering="given", copy_back=True),
                                  dict(numbering="given", block_size=32)], ids=str)
def test_same_bits(sls, name, opts):
    mesh = MESHES[name]()
    form = opts.get("form", "A")
    om = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary, openmp=True)
    want, winfo, wacc = om.smooth(mesh.xy, 7, form=form, precision=32)
    with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary, precision=32, record_accept=True, **opts) as g:
        info = g.smooth(7)
        assert np.array_equal(g.coords(), want) and np.array_equal(g.accept_mask(), wacc)
        for k in ("iterations", "accepted_last", "maxd2_last"):
            assert info[k] == winfo[k], k
        g.set_coords(mesh.xy)
        want, winfo, _ = om.smooth(mesh.xy, 60, tol=1e-4, form=form, precision=32)
        info = g.smooth(60, 1e-4)
        assert np.array_equal(g.coords(), want) and info["iterations"] == winfo["iterations"]
