"""The candidate pass walks the BVH once for a warp whose rays are coherent, as a beam, and once per ray otherwise.
Rays that make a beam, just miss making one, or overflow its buffers get bit-identical hits from the ray-persistent
kernel (asked for by a launch option that only it has), which walks every ray on its own."""
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


def trace(sc, r, **kw):
    hits = ccs.alloc_hits(r.n)
    ccs.ccs_intersect(sc.handle, ccs.rays_to_device(r.soa()), r.n, hits, ccs.make_opts(**kw))
    torch.cuda.synchronize()
    assert ccs.ccs_scene_sync_status(sc.handle) == ccs.CCS_OK
    return ccs.hits_to_numpy(hits)


def same(a, b, what):
    for k in ("t", "u", "v", "pid"):
        assert np.array_equal(a[k], b[k]), (what, k, int((a[k] != b[k]).sum()))


def make(o, d, tmin=0.0, tmax=np.inf):
    o, d = np.broadcast_arrays(np.asarray(o, np.float32), np.asarray(d, np.float32))
    n = len(o)
    return sg.Rays(np.ascontiguousarray(o), np.ascontiguousarray(d), np.full(n, tmin, np.float32), np.full(n, tmax, np.float32))


def ray_sets():
    rng = np.random.default_rng(5)
    g = np.stack(np.meshgrid(np.linspace(-1.2, 1.2, 71), np.linspace(-1.2, 1.2, 53)), -1).reshape(-1, 2)
    flat = np.concatenate([g, np.full((len(g), 1), 3.0)], 1)
    one = np.repeat(np.array([[0.1, 0.2, 3.0]]), 64, 0)
    yield "pinhole, directions change sign inside warps", sg.pinhole_rays(70, 50)
    yield "pinhole from inside the surface", sg.pinhole_rays(64, 37, eye=(0.1, -0.2, 0.05))
    yield "parallel, oblique: wide beams of one direction", make(flat, (0.21, -0.13, -1.0))
    yield "parallel to an axis: zero components of either sign", make(flat, (0.0, -0.0, -1.0))
    yield "one ray 64 times", make(one, (-0.02, -0.05, -1.0))
    yield "bounded intervals, unnormalised directions", make(flat, (0.4, -0.3, -2.0), 0.6, 1.3)
    r = make(flat, (0.21, -0.13, -1.0))
    r.o[5::32] = np.inf                       # a lane in every warp whose origin is not finite
    r.d[40::64] = np.nan                      # and lanes without a ray
    r.tmin[9::96], r.tmax[9::96] = 2.0, 1.0
    yield "rays that are not finite among others", r
    jit = make(flat + rng.normal(size=flat.shape) * 0.4, rng.normal(size=flat.shape) * 0.2 + (0.5, 0.6, -1.0))
    yield "origins and directions of wide spread", jit


@pytest.mark.parametrize("local", [False, True])
@pytest.mark.parametrize("width", [2, 4])
def test_beam_hits_equal_the_ray_kernel(width, local):
    s = sg.make_scene(5, 0.08, 3, 3, gregory_ring=True)
    sc = ccs.Scene(s.P, s.types, local=local, bvh_width=width)
    for name, r in ray_sets():
        ref = trace(sc, r, chunk=32)
        got = trace(sc, r, pairs=True, cache_slots=1)
        same(got, ref, name)
        occ = ccs.occluded(sc, ccs.rays_to_device(r.soa()), ccs.make_opts(pairs=True))
        torch.cuda.synchronize()
        assert np.array_equal(occ.cpu().numpy().astype(bool), ref["pid"] != 0xFFFFFFFF), name
    sc.close()


@pytest.mark.parametrize("n", [1, 2, 60, 140])
@pytest.mark.parametrize("width", [2, 4])
def test_beam_over_stacked_patches(n, width):
    """n patches one behind another, each with a hole where its box is but its surface is not: more than the list's 8
    and, at 140, more than the beam's buffers."""
    P = np.zeros((n, 20, 3), np.float32)
    w = np.array([-1.0, -1.0 / 3.0, 1.0 / 3.0, 1.0])
    for k in range(n):
        for j in range(4):
            for i in range(4):
                P[k, 4 * j + i] = (w[i], w[j], -0.1 * k + 0.6 * w[i] * w[j])
        P[k, 16:20] = P[k, [5, 6, 9, 10]]
    sc = ccs.Scene(P, np.zeros(n, np.uint8), bvh_width=width)
    g = np.stack(np.meshgrid(np.linspace(-1.1, 1.1, 37), np.linspace(-1.1, 1.1, 21)), -1).reshape(-1, 2)
    r = make(np.concatenate([g, np.full((len(g), 1), 2.0)], 1), (0.3, 0.2, -1.0))
    ref = trace(sc, r, chunk=32)
    assert (ref["pid"] != 0xFFFFFFFF).sum() > 100
    same(trace(sc, r, pairs=True), ref, n)
    sc.close()
