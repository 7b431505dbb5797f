"""In scenes without local frames the candidate pass drops Bezier patches whose root box in the patch's own frame, padded
by the size of a leaf's box, the ray does not come near.  Rays that graze the surface are the ones a too-tight pad would
lose: their hits are bit-identical to the ray-persistent kernel's, which never culls, at every leaf depth, for patches
that are flat, degenerate, far from the origin or large."""
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


def grazing(points, normals, sizes, seed):
    """Rays nearly tangent to the surface at the points, above and below it by fractions of the given sizes."""
    rng = np.random.default_rng(seed)
    tan = np.cross(normals, rng.normal(size=points.shape))
    tan /= np.linalg.norm(tan, axis=1, keepdims=True)
    oo, dd = [], []
    for lift in (0.0, 1e-5, 1e-3, 1e-2, 5e-2, 0.2):
        for side in (-1.0, 1.0):
            tilt = rng.uniform(-2.0, 2.0, (len(points), 1)) * lift
            d = tan - tilt * normals
            d /= np.linalg.norm(d, axis=1, keepdims=True)
            oo.append(points + side * lift * sizes * normals - 3.0 * sizes * d)
            dd.append(d)
    o, d = np.concatenate(oo).astype(np.float32), np.concatenate(dd).astype(np.float32)
    n = len(o)
    return sg.Rays(o, d, np.zeros(n, np.float32), np.full(n, np.inf, np.float32))


def check(P, types, r, depths, least_culled):
    sc = ccs.Scene(P, types, local=False)
    rays = ccs.rays_to_device(r.soa())
    cnt = torch.zeros(ccs.CCS_NUM_COUNTERS, dtype=torch.int64, device="cuda")
    for depth in depths:
        ref = trace(sc, rays, r.n, leaf_depth=depth, chunk=32)
        assert (ref["pid"] != 0xFFFFFFFF).sum() > r.n // 50
        same(trace(sc, rays, r.n, leaf_depth=depth, pairs=True, cache_slots=1), ref, depth)
    cnt.zero_()
    same(trace(sc, rays, r.n, leaf_depth=depths[-1], pairs=True, counters=cnt), ref, "counting")
    assert int(cnt[18]) >= least_culled
    sc.close()


@pytest.mark.parametrize("n,scale,shift", [(2, 1.0, 0.0), (8, 1.0, 0.0), (8, 300.0, 1000.0), (8, 1e-3, 0.5)])
def test_grazing_rays_on_cube_spheres(n, scale, shift):
    s = sg.make_scene(n, 0.05, 3, 2)
    rng = np.random.default_rng(n)
    pid = rng.integers(0, s.n, 900)
    q = s.P[pid][:, [0, 3, 12, 15]].astype(np.float64)   # a point near the surface: a mean of corners
    w = rng.dirichlet(np.ones(4), 900)
    p = np.einsum("nk,nkc->nc", w, q)
    nrm = np.cross(q[:, 3] - q[:, 0], q[:, 2] - q[:, 1])
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    size = np.linalg.norm(q[:, 3] - q[:, 0], axis=1, keepdims=True)
    r = grazing(p * scale + shift, nrm, size * scale, n)
    check((s.P * scale + shift).astype(np.float32), s.types, r, (1, 3, 6, 8), r.n // 4 if scale >= 1 else 0)


def test_grazing_rays_on_flat_twisted_and_collapsed_patches():
    rng = np.random.default_rng(3)
    P = np.zeros((60, 20, 3), np.float32)
    w = np.linspace(0.0, 1.0, 4)
    for k in range(60):
        A = np.linalg.qr(rng.normal(size=(3, 3)))[0]
        for j in range(4):
            for i in range(4):
                z = 0.0 if k % 3 == 0 else rng.normal() * (0.02 if k % 3 == 1 else 0.5)
                x, y = (w[i], w[j]) if k % 5 else (w[i], w[j] * (1 - w[i]))   # an edge collapsed to a point
                P[k, 4 * j + i] = A @ np.array([x - 0.5, y - 0.5, z]) + (k % 8, k // 8, 0)
        P[k, 16:20] = P[k, [5, 6, 9, 10]]
    q = P[:, [0, 3, 12, 15]].astype(np.float64)
    pid = np.repeat(np.arange(60), 12)
    p = np.einsum("nk,nkc->nc", rng.dirichlet(np.ones(4), len(pid)), q[pid])
    nrm = np.cross(q[pid, 3] - q[pid, 0], q[pid, 2] - q[pid, 1])
    nrm /= np.maximum(np.linalg.norm(nrm, axis=1, keepdims=True), 1e-9)
    r = grazing(p, nrm, np.ones((len(pid), 1)), 8)
    check(P, np.zeros(60, np.uint8), r, (2, 5, 8), 1)
