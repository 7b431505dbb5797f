"""After an update of the points the Gregory box tables hold as many levels as the bound of an update leaves them, down to
none (32,856 patches): the pair engine's hits stay bit-identical to the ray-persistent kernel's (asked for by a launch option
that only it has) and to a scene made of the new points, for one scene and for a batch of scenes of very different size."""
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


def trace(sc, rays, n, **kw):
    hits = ccs.alloc_hits(n)
    ccs.ccs_intersect(sc.handle, rays, n, hits, ccs.make_opts(**kw))
    torch.cuda.synchronize()
    assert ccs.ccs_scene_sync_status(sc.handle) == ccs.CCS_OK
    return ccs.hits_to_numpy(hits)


def same(a, b, what):
    for k in ("t", "u", "v", "pid"):
        assert np.array_equal(a[k], b[k]), (what, k, int((a[k] != b[k]).sum()))


def gregory_scene(n):
    V, F = sg.cube_sphere(n, 0.05, 3, 1)
    P, types = sg.patches_from_mesh(*sg.catmull_clark(V, F), gregory_everywhere=True)
    return P.astype(np.float32), types


def planes_of(P):
    return [torch.from_numpy(np.ascontiguousarray(P[..., c]).reshape(-1)).cuda() for c in range(3)]


@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("n", [2, 8, 37])
def test_hits_after_an_update(n, local):
    P, types = gregory_scene(n)
    moved = sg.deform(P, 1, 4, 3, amp=0.05)
    r = sg.random_rays(6001, seed=n, target=1.05)
    rays = ccs.rays_to_device(r.soa())
    sc, fresh = ccs.Scene(P, types, local=local), ccs.Scene(moved, types, local=local)
    before = trace(sc, rays, r.n)
    ccs.ccs_scene_update_points(sc.handle, *planes_of(moved))
    ccs.ccs_bvh_refit(sc.handle)
    got = trace(sc, rays, r.n)
    assert (got["t"] != before["t"]).sum() > 1000
    for depth in (3, 8):
        ref = trace(sc, rays, r.n, leaf_depth=depth, chunk=32)
        same(trace(sc, rays, r.n, leaf_depth=depth, pairs=True), ref, depth)
        same(trace(fresh, rays, r.n, leaf_depth=depth, pairs=True), ref, (depth, "fresh"))
    sc.close()
    fresh.close()


# (a batch of more than 2^17 patches refits in a launch of its own)
@pytest.mark.parametrize("large", [37, 75])
@pytest.mark.parametrize("moves", ["all", "small", "large"])
def test_batch_of_scenes_of_very_different_size(moves, large):
    parts = [gregory_scene(large), sg.make_scene(4, 0.03, 3, 2), gregory_scene(2), gregory_scene(8),
             sg.make_scene(3, 0.03, 3, 4)]
    parts = [q if isinstance(q, tuple) else (q.P, q.types) for q in parts]
    parts[4] = (parts[4][0], np.zeros_like(parts[4][1]))   # without a Gregory patch
    scenes = [ccs.Scene(P, t, local=True) for P, t in parts]
    rays, hits = [], []
    for k in range(len(parts)):
        rays.append(ccs.rays_to_device(sg.random_rays(2001 + k, seed=k, target=1.05).soa()))
        hits.append(ccs.alloc_hits(2001 + k))
    b = ccs.ccs_batch_create(scenes, rays, hits)
    stages = ccs.CCS_BATCH_UPDATE | ccs.CCS_BATCH_REFIT | ccs.CCS_BATCH_INTERSECT
    ccs.ccs_batch_capture(b, stages, ccs.make_opts(pairs=True, cache_slots=1))
    now = [P for P, _ in parts]
    planes = []
    for frame in (1, 2):
        for k, (P, _) in enumerate(parts):
            if moves == "all" or (k == 0) == (moves == "large"):
                now[k] = sg.deform(P, frame, 4, 3, amp=0.05)
                planes.append(planes_of(now[k]))
                ccs.ccs_batch_set_points(b, k, *planes[-1])
        ccs.ccs_batch_launch(b)
        assert ccs.ccs_batch_sync_status(b) == ccs.CCS_OK
        for k, (_, types) in enumerate(parts):
            fresh = ccs.Scene(now[k], types, local=True)
            same(ccs.hits_to_numpy(hits[k]), trace(fresh, rays[k], 2001 + k, chunk=32), (frame, k))
            fresh.close()
    ccs.ccs_batch_destroy(b)
    for sc in scenes:
        sc.close()
