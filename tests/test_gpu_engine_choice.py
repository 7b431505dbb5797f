"""A launch whose options leave the engine to the library: the same hits as the ray-persistent kernel (asked for by an
option that only it has) over every form of call that may take the pair engine, and on the streams where it may not."""
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


def trace(sc, rays, n, opts):
    hits = ccs.alloc_hits(max(n, 1))
    ccs.ccs_intersect(sc.handle, rays, n, hits, opts)
    torch.cuda.synchronize()
    assert ccs.ccs_scene_sync_status(sc.handle) == ccs.CCS_OK
    return ccs.hits_to_numpy(hits)


@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("width", [2, 4, "both"])
@pytest.mark.parametrize("n", [1, 33, 4097, 70001])
def test_library_choice_equals_the_ray_kernel(n, width, local):
    s = sg.make_scene(4, 0.06, 3, n, gregory_ring=True)
    sc = ccs.Scene(s.P, s.types, local=local, bvh_width=width)
    r = sg.random_rays(n, seed=n, target=1.1)
    r.tmax[::3] = 2.5
    rays = ccs.rays_to_device(r.soa())
    ref = trace(sc, rays, n, ccs.make_opts(chunk=32))
    for opts in (None, ccs.make_opts(), ccs.make_opts(refill=3), ccs.make_opts(cache_slots=0), ccs.make_opts(cache_slots=2),
                 ccs.make_opts(image_width=64)):
        same(trace(sc, rays, n, opts), ref, "device")
    for depth in (1, 5, 11):
        same(trace(sc, rays, n, ccs.make_opts(leaf_depth=depth)), trace(sc, rays, n, ccs.make_opts(leaf_depth=depth, chunk=32)),
             depth)
    occ = ccs.occluded(sc, rays)
    torch.cuda.synchronize()
    assert np.array_equal(occ.cpu().numpy().astype(bool), ref["pid"] != 0xFFFFFFFF)
    planes = [np.ascontiguousarray(a) for a in r.soa()]
    out = [np.empty(n, np.float32) for _ in range(3)] + [np.empty(n, np.uint32)]
    ccs.ccs_intersect_host(sc.handle, [a.ctypes.data for a in planes], n, [a.ctypes.data for a in out])
    same(dict(t=out[0], u=out[1], v=out[2], pid=out[3]), {k: v[:n] for k, v in ref.items()}, "host")
    sc.close()


def test_default_launch_is_capturable():
    """Under stream capture the ray-persistent kernel runs, which allocates nothing; replays follow the inputs."""
    s = sg.make_scene(4, 0.06, 3, 1)
    sc = ccs.Scene(s.P, s.types, local=True)
    a, b = sg.random_rays(5000, seed=1), sg.random_rays(5000, seed=2)
    rays = ccs.rays_to_device(a.soa())
    hits = ccs.alloc_hits(5000)
    ccs.ccs_intersect(sc.handle, rays, 5000, hits, ccs.make_opts(chunk=32))   # the kernel's attributes are set
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        ccs.ccs_intersect(sc.handle, rays, 5000, hits)
    for q in (a, b):
        for dst, src in zip(rays, ccs.rays_to_device(q.soa())):
            dst.copy_(src)
        g.replay()
        torch.cuda.synchronize()
        same(ccs.hits_to_numpy(hits), trace(sc, rays, 5000, None), "replay")
    sc.close()


def test_default_launches_on_two_streams_and_threads():
    from concurrent.futures import ThreadPoolExecutor
    s = sg.make_scene(6, 0.06, 3, 1)
    sc = ccs.Scene(s.P, s.types, local=True)
    sets = [ccs.rays_to_device(sg.random_rays(40000 + 1000 * k, seed=k).soa()) for k in range(4)]
    ref = [trace(sc, r, int(r[0].numel()), ccs.make_opts(chunk=32)) for r in sets]

    def work(k):
        st = torch.cuda.Stream()
        n = int(sets[k][0].numel())
        out = []
        with torch.cuda.stream(st):
            for _ in range(6):
                h = ccs.alloc_hits(n)
                ccs.ccs_intersect(sc.handle, sets[k], n, h, None, st)
                out.append(h)
        st.synchronize()
        return [ccs.hits_to_numpy(h) for h in out]

    with ThreadPoolExecutor(4) as ex:
        for k, got in enumerate(ex.map(work, range(4))):
            for g in got:
                same(g, ref[k], k)
    sc.close()
