"""The two closest-hit engines against each other and against the FP64 oracle, each asked for by name: the pair engine by its
flag, the ray-persistent kernel by a launch option that only it has (chunk).  A launch without options takes the pair engine,
so it is no reference for it."""
import numpy as np
import pytest

import oracle
from paper_1811_03510_gb300 import ccs, scenegen as sg
from parity import MISS, compare
from test_gpu_pairs import tunnel_rays, tunnel_scene

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

RAY = dict(chunk=32)


@pytest.fixture(scope="module", autouse=True)
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_03510_gb300 import build_ext
    build_ext.build()
    oracle.build()
    torch.cuda.set_device(0)


def run(sc, r, counters=None, **kw):
    """Hits of rays r, the hit planes filled with a pattern first so that an unwritten record shows."""
    rays = ccs.rays_to_device(r.soa())
    hits = [torch.full((r.n,), -7.0, device="cuda") for _ in range(3)] + \
        [torch.full((r.n,), 0x5A5A5A5A, dtype=torch.int32, device="cuda")]
    ccs.ccs_intersect(sc.handle, rays, r.n, hits, ccs.make_opts(counters=counters, **kw))
    torch.cuda.synchronize()
    assert ccs.ccs_scene_sync_status(sc.handle) == ccs.CCS_OK
    return ccs.hits_to_numpy(hits)


def occluded(sc, r, **kw):
    occ = ccs.occluded(sc, ccs.rays_to_device(r.soa()), ccs.make_opts(**kw))
    torch.cuda.synchronize()
    return occ.cpu().numpy()


def same(a, b, what):
    for k in ("t", "u", "v", "pid"):
        assert np.array_equal(a[k], b[k]), (what, k, int((a[k] != b[k]).sum()))


@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("width", [2, 4])
@pytest.mark.parametrize("engine", [RAY, dict(pairs=True)], ids=["ray", "pairs"])
def test_each_engine_against_the_oracle(engine, width, local):
    for s, r, depth in ((sg.config_scene(1), sg.pinhole_rays(96, 64), 8),
                        (sg.make_scene(6, 0.05, 3, 4, gregory_ring=True), sg.random_rays(4000, seed=31), 6)):
        sc = ccs.Scene(s.P, s.types, local=local, bvh_width=width)
        got = run(sc, r, leaf_depth=depth, **engine)
        rep = compare(got, oracle.intersect(s.P, s.types, r.soa(), L=depth, flags=True, local=local), depth,
                      max_flagged_frac=0.05)
        assert rep["hits"] > 500
        assert np.array_equal(occluded(sc, r, leaf_depth=depth, **engine).astype(bool), got["pid"] != MISS)
        sc.close()


@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("width", [2, 4])
def test_options_of_the_pair_engine(local, width):
    s = sg.make_scene(8, 0.05, 3, 1, gregory_ring=True)
    sc = ccs.Scene(s.P, s.types, local=local, bvh_width=width)
    for r in (sg.random_rays(30000, seed=71), sg.random_rays(3000, seed=75, target=1.05)):   # (the second hands subtrees over)
        ref = run(sc, r, **RAY)
        assert (ref["pid"] != MISS).sum() > 1000
        for kw in (dict(cache_slots=0), dict(cache_slots=1), dict(cache_slots=2, refill=1), dict(refill=24),
                   dict(refill=32, cache_slots=1)):
            same(run(sc, r, pairs=True, **kw), ref, kw)
        cnt = torch.zeros(ccs.CCS_NUM_COUNTERS, dtype=torch.int64, device="cuda")
        same(run(sc, r, counters=cnt, pairs=True), ref, "counting")
    assert int(cnt[11]) > 100
    sc.close()


def test_image_tiles_and_host_chunks():
    s = sg.config_scene(2)
    r = sg.pinhole_rays(336, 211)
    sc = ccs.Scene(s.P, s.types, local=True)
    ref = run(sc, r, **RAY)
    assert (ref["pid"] != MISS).sum() > 10000
    for w in (336, 8, 333, 0):
        same(run(sc, r, pairs=True, cache_slots=1, image_width=w), ref, w)
        assert np.array_equal(occluded(sc, r, pairs=True, image_width=w).astype(bool), ref["pid"] != MISS)
    planes = [np.ascontiguousarray(a) for a in r.soa()]
    for kw in (dict(pairs=True, image_width=336, host_chunk=20000), dict(pairs=True), dict(chunk=32, host_chunk=20000)):
        out = [np.empty(r.n, np.float32) for _ in range(3)] + [np.empty(r.n, np.uint32)]
        ccs.ccs_intersect_host(sc.handle, [a.ctypes.data for a in planes], r.n, [a.ctypes.data for a in out],
                               ccs.make_opts(**kw))
        same(dict(t=out[0], u=out[1], v=out[2], pid=out[3]), ref, kw)
    sc.close()


@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("gregory_every", [0, 3])
@pytest.mark.parametrize("width", [2, 4])
def test_rays_that_drop_candidates(gregory_every, width, local):
    P, types = tunnel_scene(40, gregory_every)
    r = tunnel_rays(40)
    sc = ccs.Scene(P, types, bvh_width=width, local=local)
    ref = run(sc, r, **RAY)
    assert (ref["pid"][:84] == 40).all()
    for kw in (dict(), dict(cache_slots=0), dict(cache_slots=1, refill=1)):
        same(run(sc, r, pairs=True, **kw), ref, kw)
    r.tmax[:] = 100.0
    assert np.array_equal(occluded(sc, r, pairs=True), occluded(sc, r, **RAY))
    sc.close()


def test_any_hit_with_bounded_intervals():
    s = sg.make_scene(8, 0.05, 3, 1, gregory_ring=True)
    r = sg.random_rays(20000, seed=72)
    r.tmax[:] = np.random.default_rng(3).uniform(0.5, 6.0, r.n).astype(np.float32)
    for local in (False, True):
        sc = ccs.Scene(s.P, s.types, local=local)
        ref = occluded(sc, r, **RAY)
        assert np.array_equal(occluded(sc, r, pairs=True), ref)
        assert np.array_equal(run(sc, r, **RAY)["pid"] != MISS, ref.astype(bool))
        assert 1000 < ref.sum() < r.n - 1000
        sc.close()


def test_invalid_rays_one_patch_and_after_the_cap():
    s = sg.config_scene(1)
    r = sg.random_rays(4000, seed=73, radius=2.0)
    r.o[::7, 0] = np.nan
    r.tmin[1::11] = 5.0
    r.tmax[1::11] = 1.0
    for P, types in ((s.P, s.types), (s.P[:1], s.types[:1])):
        sc = ccs.Scene(P, types)
        ref = run(sc, r, **RAY)
        same(run(sc, r, pairs=True), ref, len(P))
        ccs.intersect(sc, ccs.rays_to_device(r.soa()), ccs.make_opts(pairs=True, iter_cap=2))
        torch.cuda.synchronize()
        assert ccs.ccs_scene_sync_status(sc.handle) == ccs.CCS_ERR_TRAVERSAL_LIMIT
        same(run(sc, r, pairs=True), ref, (len(P), "after the cap"))
        sc.close()


def test_batches():
    scenes = [sg.make_scene(n, 0.02 * k, 3, k + 1, gregory_ring=k == 1) for k, n in enumerate([2, 5, 3, 4])]
    rays = [sg.pinhole_rays(64, 48), sg.random_rays(4001, seed=3), sg.random_rays(517, seed=4), sg.random_rays(0, seed=5)]
    for order in ((0, 1, 2, 3), (1, 3, 0, 2)):   # a scene with local frames first, or one without
        handles = [ccs.Scene(scenes[k].P, scenes[k].types, local=k % 2 == 0) for k in order]
        rs = [rays[k] for k in order]
        ref = [run(h, r, **RAY) if r.n else None for h, r in zip(handles, rs)]
        hits = [ccs.alloc_hits(max(r.n, 1)) for r in rs]
        for kw in (dict(pairs=True), dict(pairs=True, image_width=64), dict(chunk=32)):
            ccs.ccs_intersect_batched(handles, [ccs.rays_to_device(r.soa()) for r in rs], hits, ccs.make_opts(**kw))
            torch.cuda.synchronize()
            for h, rf, r in zip(hits, ref, rs):
                if r.n:
                    same({k: v[:r.n] for k, v in ccs.hits_to_numpy(h).items()}, rf, (order, kw))
        for h in handles:
            h.close()


@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("width", [2, 4])
def test_grazing_rays_keep_every_hit(width, local):
    """Rays just above the surface and nearly tangent, which a too-tight test of a patch's root box would lose, with the boxes
    in the patches' own frames (counter 17) and in world axes (counter 18)."""
    s = sg.config_scene(2)
    cam = sg.pinhole_rays(160, 90)
    sc = ccs.Scene(s.P, s.types, local=local, bvh_width=width)
    h = run(sc, cam, **RAY)
    hit = h["pid"] != MISS
    p = cam.o[hit].astype(np.float64) + cam.d[hit].astype(np.float64) * h["t"][hit][:, None]
    rng = np.random.default_rng(17)
    nrm = p / np.linalg.norm(p, axis=1, keepdims=True)
    tan = np.cross(nrm, rng.normal(size=p.shape))
    tan /= np.linalg.norm(tan, axis=1, keepdims=True)
    oo, dd = [], []
    for lift in (1e-6, 1e-5, 1e-4, 1e-3, 1e-2):
        for reach in (0.3, 2.0, 200.0):
            tilt = rng.uniform(-2.0, 2.0, (len(p), 1)) * lift
            dv = tan - tilt * nrm
            dv /= np.linalg.norm(dv, axis=1, keepdims=True)
            oo.append(p * (1.0 + lift) - reach * dv)
            dd.append(dv)
    oo, dd = np.concatenate(oo).astype(np.float32), np.concatenate(dd).astype(np.float32)
    n = len(oo)
    r = sg.Rays(oo, dd, np.zeros(n, np.float32), np.full(n, np.inf, np.float32))
    for depth in (3, 8):
        ref = run(sc, r, leaf_depth=depth, **RAY)
        assert 0.2 * n < (ref["pid"] != MISS).sum() < n
        cnt = torch.zeros(ccs.CCS_NUM_COUNTERS, dtype=torch.int64, device="cuda")
        same(run(sc, r, counters=cnt, leaf_depth=depth, pairs=True), ref, depth)
        same(run(sc, r, leaf_depth=depth, pairs=True, cache_slots=1), ref, depth)
    assert int(cnt[17 if local else 18]) > n // 10 and int(cnt[18 if local else 17]) == 0
    same(run(sc, cam, pairs=True), h, "primary")
    sc.close()
