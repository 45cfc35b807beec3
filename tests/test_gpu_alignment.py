"""Device coordinates at an odd float64 offset (8-byte aligned, not 16): a
contiguous view into a larger tensor.  Every entry point that takes them gives
what it gives for an aligned buffer, except sls_smooth_noalloc, which refuses."""
import numpy as np
import pytest

import meshgen

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


def _odd(values):
    """The values in a device tensor that starts 8 bytes off a 16-byte boundary."""
    import torch
    t = torch.empty(values.size + 1, dtype=torch.float64, device="cuda")[1:].view(values.shape)
    t.copy_(torch.from_numpy(np.ascontiguousarray(values)))
    assert t.data_ptr() % 16 == 8 and t.is_contiguous()
    return t


@pytest.mark.parametrize("numbering", ["morton", "random"])
@pytest.mark.parametrize("opts", [dict(), dict(layout="soa"), dict(form="B"), dict(form="B", layout="soa"),
                                  dict(precision=32), dict(precision=32, layout="soa"), dict(numbering="given"),
                                  dict(skip_unchanged=True)], ids=str)
def test_odd_offsets(sls, numbering, opts):
    import torch
    mesh = meshgen.jittered_grid(113, 97, 0.3, 51, numbering=numbering)  # random ids: renumbered inside
    start = mesh.xy + 1e-4 * np.random.default_rng(52).standard_normal(mesh.xy.shape)
    with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary, **opts) as g:
        g.set_coords(_odd(start))
        want = start.astype(np.float32).astype(np.float64) if opts.get("precision") == 32 else start
        assert np.array_equal(g.coords(), want)
        g.smooth(3)
        want = g.coords()
        assert np.array_equal(g.coords_device(_odd(np.zeros_like(start))).cpu().numpy(), want)
        assert np.array_equal(g.coords_device().cpu().numpy(), want)
        if "form" in opts or "precision" in opts:
            return
        ids = np.array([5, 0, mesh.n - 1, 77, 4096], np.int32)
        idx = torch.from_numpy(ids).cuda()
        got = g.gather(idx, _odd(np.zeros((len(ids), 2))))
        assert np.array_equal(got.cpu().numpy(), want[ids])
        g.scatter(idx, _odd(want[ids] + 0.5))
        want[ids] += 0.5
        assert np.array_equal(g.coords(), want)


def test_noalloc_refuses_odd_offsets(sls):
    mesh = meshgen.jittered_grid(33, 21, 0.3, 53)
    import torch
    with sls.Mesh(mesh.xy, mesh.tri, mesh.boundary) as g:
        even = torch.from_numpy(mesh.xy).cuda()
        for a, b in ((_odd(mesh.xy), even), (even, _odd(mesh.xy))):
            with pytest.raises(sls.SlsError) as e:
                g.smooth_noalloc(a, b, 2)
            assert e.value.code == 1
            assert g.smooth_noalloc(a, b, 0)["iterations"] == 0  # (a copy)
        assert g.smooth_noalloc(even, torch.empty_like(even), 2)["iterations"] == 2
