"""The box table of Gregory patches: the pair engine takes the child boxes of the upper levels of a Gregory
patch's subdivision from a table stored with the scene, the ray-persistent kernel computes them anew.  The stored
boxes are the computed ones, so every hit is bit-identical, whatever the leaf depth is to the table's depth (above
it, at it, below it), after updates of the points (a shallower table), and in batches."""
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


# 96 patches hold 15 levels, 1536 patches 11 (256 MiB): leaf depths 1..9 lie above, at and below them
@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("n,depth", [(2, 1), (2, 3), (2, 7), (2, 8), (2, 9), (8, 4), (8, 5), (8, 6)])
def test_table_hits_equal_the_ray_kernel(n, depth, local):
    P, types = gregory_scene(n)
    r = sg.random_rays(6001, seed=90 + depth, target=1.05)
    rays = ccs.rays_to_device(r.soa())
    sc = ccs.Scene(P, types, local=local)
    ref = trace(sc, rays, r.n, leaf_depth=depth, chunk=32)   # an option that only that kernel has
    assert (ref["pid"] != 0xFFFFFFFF).sum() > 1000
    for K in (0, 1):
        same(trace(sc, rays, r.n, leaf_depth=depth, pairs=True, cache_slots=K), ref, K)
    occ = ccs.occluded(sc, rays, ccs.make_opts(leaf_depth=depth, pairs=True))
    torch.cuda.synchronize()
    assert np.array_equal(occ.cpu().numpy().astype(bool), ref["pid"] != 0xFFFFFFFF)
    sc.close()


def test_table_follows_updates_of_the_points():
    s = sg.make_scene(3, 0.03, 3, 2, gregory_ring=True)
    r = sg.random_rays(6001, seed=99, target=1.05)
    rays = ccs.rays_to_device(r.soa())
    sc = ccs.Scene(s.P, s.types, local=True)
    before = trace(sc, rays, r.n, pairs=True)
    moved = sg.deform(s.P, 1, 4, 3, amp=0.05)
    planes = [torch.from_numpy(np.ascontiguousarray(moved[..., c]).reshape(-1)).cuda() for c in range(3)]
    ccs.ccs_scene_update_points(sc.handle, *planes)
    ccs.ccs_bvh_refit(sc.handle)
    got = trace(sc, rays, r.n, pairs=True)
    assert (got["t"] != before["t"]).sum() > 1000
    same(got, trace(sc, rays, r.n, chunk=32), "updated")
    sc.close()
    # the same through a batch of two scenes, one of them without a Gregory patch and one with new points
    flat = ccs.Scene(s.P, np.zeros_like(s.types), local=True)
    sc = ccs.Scene(s.P, s.types, local=True)
    hits = [ccs.alloc_hits(r.n) for _ in range(2)]
    b = ccs.ccs_batch_create([flat, sc], [rays, rays], hits)
    ccs.ccs_batch_set_points(b, 1, *planes)
    stages = ccs.CCS_BATCH_UPDATE | ccs.CCS_BATCH_REFIT | ccs.CCS_BATCH_INTERSECT
    ccs.ccs_batch_run(b, stages, ccs.make_opts(pairs=True))
    assert ccs.ccs_batch_sync_status(b) == ccs.CCS_OK
    same(ccs.hits_to_numpy(hits[1]), got, "batch")
    same(ccs.hits_to_numpy(hits[0]), trace(flat, rays, r.n, chunk=32), "batch, no table")
    ccs.ccs_batch_destroy(b)
    flat.close()
    sc.close()


@pytest.mark.parametrize("depth", [3, 7, 8, 9])
def test_learned_traversal_with_the_table(depth):
    """The directed descent and the skipped subtree of the learned order, over table nodes (15 levels) and below."""
    P, types = gregory_scene(2)
    r = sg.random_rays(6001, seed=70 + depth, target=1.05)
    rays = ccs.rays_to_device(r.soa())
    sc = ccs.Scene(P, types, local=True)
    ref = trace(sc, rays, r.n, leaf_depth=depth, chunk=32)
    p = ccs.ccs_proposal_create(seed=6)   # untrained: its cells are arbitrary
    hits = ccs.alloc_hits(r.n)
    ccs.ccs_intersect_learned(sc.handle, p, rays, r.n, hits, ccs.make_opts(leaf_depth=depth), 0.0)
    torch.cuda.synchronize()
    same(ccs.hits_to_numpy(hits), ref, depth)
    ccs.ccs_proposal_destroy(p)
    sc.close()
