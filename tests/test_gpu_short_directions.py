"""Directions of any length, also those whose components the ray kernel moves to 1e-20: the pair engine's hits are
bit-identical to the ray-persistent kernel's (asked for by a launch option that only it has), which culls no patch by its
root box."""
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


# 2^-40 and 2^100 are the ends of the range that is culled
LENGTHS = [0.0, 1e-38, 1e-24, 1e-20, 3e-20, 1e-19, 1e-18, 1e-16, 2.0 ** -40, 1e-11, 1.0, 1e20, 2.0 ** 100, 1e31, 1e37, 3e38]


@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("width", [2, 4])
def test_hits_of_short_and_long_directions(width, local):
    s = sg.make_scene(6, 0.06, 3, 2, gregory_ring=True)
    sc = ccs.Scene(s.P, s.types, local=local, bvh_width=width)
    spread, cam = sg.random_rays(6000, seed=5), sg.pinhole_rays(72, 48)
    ax = sg.random_rays(900, seed=6, target=0.9)   # along the axes: components of exactly zero
    ax.d[:] = np.eye(3, dtype=np.float32)[np.arange(900) % 3] * np.where(np.arange(900) % 2, 1.0, -1.0)[:, None]
    ax.o[:] = ax.o / 3.0 - 3.0 * ax.d
    hits = 0
    for r in (spread, cam, ax):
        for length in LENGTHS:
            q = sg.Rays(r.o, (r.d.astype(np.float64) * length).astype(np.float32), r.tmin, r.tmax)
            rays = ccs.rays_to_device(q.soa())
            ref = trace(sc, rays, q.n, chunk=32)
            same(trace(sc, rays, q.n), ref, length)
            same(trace(sc, rays, q.n, pairs=True, image_width=8), ref, (length, "tiles"))
            occ = ccs.occluded(sc, rays)
            torch.cuda.synchronize()
            assert np.array_equal(occ.cpu().numpy().astype(bool), ref["pid"] != 0xFFFFFFFF), length
            hits += int((ref["pid"] != 0xFFFFFFFF).sum()) if 1e-20 < length < 1e-12 else 0
    assert hits > 1000
    sc.close()


def test_dropped_candidates_of_short_directions():
    """More patches along a ray than its list holds: the walks for the dropped ones do not cull either."""
    n = 40
    P = np.zeros((n, 20, 3), np.float32)
    w = np.array([-1.0, -1.0 / 3.0, 1.0 / 3.0, 1.0])
    for k in range(n):
        for j in range(4):
            for i in range(4):
                P[k, 4 * j + i] = (w[i], w[j], -0.1 * k + 0.6 * w[i] * w[j])
        P[k, 16:20] = P[k, [5, 6, 9, 10]]
    g = np.stack(np.meshgrid(np.linspace(-1.1, 1.1, 37), np.linspace(-1.1, 1.1, 21)), -1).reshape(-1, 2)
    o = np.concatenate([g, np.full((len(g), 1), 2.0)], 1).astype(np.float32)
    for local in (False, True):
        sc = ccs.Scene(P, np.zeros(n, np.uint8), local=local)
        for length in (1e-19, 1e-16, 1.0):
            d = np.repeat(np.array([[0.3, 0.2, -1.0]]) * length, len(o), 0).astype(np.float32)
            r = sg.Rays(o, d, np.zeros(len(o), np.float32), np.full(len(o), np.inf, np.float32))
            rays = ccs.rays_to_device(r.soa())
            same(trace(sc, rays, r.n), trace(sc, rays, r.n, chunk=32), (local, length))
        sc.close()
