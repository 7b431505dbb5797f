"""An image width that gives the pair engine's candidate pass no tile (wider than the rays, up to the largest a caller can
pass) leaves every answer as it is, in every call that takes one."""
import numpy as np
import pytest

from paper_1811_03510_gb300 import ccs, scenegen as sg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_03510_gb300 import build_ext
    build_ext.build()
    torch.cuda.set_device(0)


def same(a, b, what):
    for k in ("t", "u", "v", "pid"):
        assert np.array_equal(a[k], b[k]), (what, k, int((a[k] != b[k]).sum()))


@pytest.mark.parametrize("n", [31, 3001])
def test_widths_beyond_the_rays(n):
    s = sg.make_scene(4, 0.06, 3, 1)
    sc = ccs.Scene(s.P, s.types, local=True)
    r = sg.random_rays(n, seed=n)
    rays = ccs.rays_to_device(r.soa())
    ref = ccs.hits_to_numpy(ccs.intersect(sc, rays, ccs.make_opts(chunk=32)))
    assert (ref["pid"] != 0xFFFFFFFF).sum() > n // 4
    planes = [np.ascontiguousarray(a) for a in r.soa()]
    for w in (n // 8 * 8 + 8, 1 << 20, 1 << 29, 1 << 30, 3 << 30, 1 << 31, 2 ** 32 - 8):
        for kw in ({}, dict(pairs=True)):
            opts = ccs.make_opts(image_width=w, **kw)
            hits = [torch.full((n,), -7.0, device="cuda") for _ in range(3)] + \
                [torch.full((n,), 0x5A5A5A5A, dtype=torch.int32, device="cuda")]
            ccs.ccs_intersect(sc.handle, rays, n, hits, opts)
            same(ccs.hits_to_numpy(hits), ref, (w, kw))
            occ = ccs.occluded(sc, rays, opts)
            assert np.array_equal(occ.cpu().numpy().astype(bool), ref["pid"] != 0xFFFFFFFF), (w, kw)
            out = [np.empty(n, np.float32) for _ in range(3)] + [np.empty(n, np.uint32)]
            ccs.ccs_intersect_host(sc.handle, [a.ctypes.data for a in planes], n, [a.ctypes.data for a in out], opts)
            same(dict(t=out[0], u=out[1], v=out[2], pid=out[3]), ref, ("host", w, kw))
    b = ccs.ccs_batch_create([sc, sc], [rays, rays], [ccs.alloc_hits(n), hits])
    ccs.ccs_batch_run(b, ccs.CCS_BATCH_INTERSECT, ccs.make_opts(pairs=True, image_width=1 << 30))
    torch.cuda.synchronize()
    same(ccs.hits_to_numpy(hits), ref, "batch")
    ccs.ccs_batch_destroy(b)
    sc.close()
