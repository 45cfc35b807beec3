"""Form-A meshes that the library renumbers inside (8,192 nodes or more, a
numbering that is not local): every entry point that takes or gives node ids,
coordinates or decisions works in the caller's numbering, against the oracle
and against the same mesh in the caller's order (numbering = given)."""
import numpy as np
import pytest

import meshgen
import oracle
from test_gpu_domain import _run_split  # (the tests folder is on the path)

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
    "grid": lambda: meshgen.jittered_grid(163, 101, 0.35, 81, numbering="random", pull_fraction=0.05, pull_centres=32),
    "delaunay": lambda: meshgen.delaunay_random(12000, 82, numbering="random"),
    "rows": lambda: meshgen.jittered_grid(191, 67, 0.35, 83, numbering="natural"),
}
KEYS = ("iterations", "converged", "accepted_last", "maxd2_last")


@pytest.mark.parametrize("name", sorted(MESHES))
@pytest.mark.parametrize("opts", [dict(), dict(layout="soa"), dict(copy_back=True), dict(passes_per_check=3),
                                  dict(l2_window=True)], ids=str)
def test_coordinates_and_exchange(sls, name, opts):
    import torch
    mesh = MESHES[name]()
    assert mesh.n >= 8192
    rng = np.random.default_rng(84)
    start = mesh.xy + np.where(mesh.boundary[:, None] == 0, rng.uniform(-1e-4, 1e-4, mesh.xy.shape), 0.0)
    om = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary)
    ids = rng.choice(mesh.n, 300, replace=False).astype(np.int32)
    idx = torch.from_numpy(ids).cuda()
    with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary, record_accept=True, **opts) as g:
        for device in (False, True):
            g.set_coords(torch.from_numpy(start).cuda() if device else start)
            assert np.array_equal(g.coords(), start)
            info = g.smooth(7)
            want, winfo, wacc = om.smooth(start, 7)
            assert np.array_equal(g.coords(), want)
            assert np.array_equal(g.coords_device().cpu().numpy(), want)
            assert np.array_equal(g.coords(), want)  # (a download leaves the arrays as they were)
            assert np.array_equal(g.accept_mask(), wacc)
            assert all(info[k] == winfo[k] for k in KEYS)
            counts, qmin, qmean = g.histogram(16)
            wc, wmin, wmean = om.histogram(want, 16)
            assert np.array_equal(counts, wc) and qmin == wmin and abs(qmean - wmean) <= 1e-12 * abs(wmean)
            # go on from a scatter: some nodes, fixed ones among them, elsewhere
            got = torch.empty((len(ids), 2), dtype=torch.float64, device="cuda")
            g.gather(idx, got)
            assert np.array_equal(got.cpu().numpy(), want[ids])
            g.scatter(idx, got + 1e-5)
            want[ids] += 1e-5
            assert np.array_equal(g.coords(), want)
            g.smooth(5)
            want, _, wacc = om.smooth(want, 5)
            assert np.array_equal(g.coords(), want) and np.array_equal(g.accept_mask(), wacc)
        bad = torch.tensor([0, mesh.n], dtype=torch.int32, device="cuda")
        with pytest.raises(sls.SlsError):
            g.gather(bad, got[:2])


@pytest.mark.parametrize("name", sorted(MESHES))
def test_binary32_round_trip(sls, name):
    import torch
    mesh = MESHES[name]()
    start = mesh.xy + 1e-4 * np.random.default_rng(85).standard_normal(mesh.xy.shape)
    om = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary)
    with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary, record_accept=True, precision=32) as g:
        for device in (False, True):
            g.set_coords(torch.from_numpy(start).cuda() if device else start)
            want, winfo, wacc = om.smooth(start, 6, precision=32)
            info = g.smooth(6)
            assert np.array_equal(g.coords(), want) and np.array_equal(g.coords_device().cpu().numpy(), want)
            assert np.array_equal(g.accept_mask(), wacc) and info["accepted_last"] == winfo["accepted_last"]


@pytest.mark.parametrize("layout", ["aos", "soa"])
def test_batch(sls, layout):
    meshes = [MESHES[k]() for k in sorted(MESHES)]
    iters, tols = [31, 12, 300], [0.0, 0.0, 1e-6]
    handles = [sls.Mesh(m.xy, m.tri, m.boundary, layout=layout, record_accept=True) for m in meshes]
    try:
        with sls.Batch(handles, iters, tols, layout=layout) as b:
            infos = b.smooth()
            for j, m in enumerate(meshes):
                want, winfo, wacc = oracle.OracleMesh(m.xy, m.tri, m.boundary).smooth(m.xy, iters[j], tol=tols[j])
                assert np.array_equal(b.coords(j), want), j
                assert np.array_equal(handles[j].coords_device().cpu().numpy(), want), j
                assert np.array_equal(handles[j].accept_mask(), wacc), j
                assert all(infos[j][k] == winfo[k] for k in KEYS), j
            b.reset()
            for j, m in enumerate(meshes):
                assert np.array_equal(b.coords(j), m.xy), j
    finally:
        for h in handles:
            h.close()


@pytest.mark.parametrize("layout", ["aos", "soa"])
def test_subdomains(sls, layout):
    mesh = meshgen.jittered_grid(211, 151, 0.35, 86, numbering="random")
    xy, info = _run_split(mesh, 2, 12, 0.0, layout=layout)
    want, winfo, _ = oracle.OracleMesh(mesh.xy, mesh.tri, mesh.boundary).smooth(mesh.xy, 12)
    assert np.array_equal(xy, want)
    assert info["accepted_last"] == winfo["accepted_last"] and info["maxd2_last"] == winfo["maxd2_last"]


def test_alive_and_destroyed_out_of_order(sls):
    meshes = [meshgen.jittered_grid(100 + 11 * k, 90 + 5 * k, 0.3, 87 + k, numbering="random") for k in range(5)]
    handles = [sls.Mesh(m.xy, m.tri, m.boundary, numbering="given" if k == 2 else "auto") for k, m in enumerate(meshes)]
    for k in (3, 0, 4, 2, 1):
        handles[k].smooth(6)
        want, _, _ = oracle.OracleMesh(meshes[k].xy, meshes[k].tri, meshes[k].boundary).smooth(meshes[k].xy, 6)
        assert np.array_equal(handles[k].coords(), want)
        handles[k].close()
