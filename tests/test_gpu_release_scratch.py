"""Scratch of launches that leave the engine open: the library's pool keeps no more of it than it says, and gives it back when
asked, while other launches go on.  In a process of its own, whose device memory nothing else moves."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = r'''
import numpy as np
import torch
from paper_1811_03510_gb300 import ccs, scenegen as sg

torch.cuda.set_device(0)
s = sg.make_scene(4, 0.06, 3, 1)
sc = ccs.Scene(s.P, s.types, local=True)
small = sg.random_rays(1 << 16, seed=1)
n = 1 << 23   # the largest launch that takes the pair engine by itself: 164 bytes of scratch a ray and more
rays = [p.repeat(n // small.n) for p in ccs.rays_to_device(small.soa())]
hits = [ccs.alloc_hits(n) for _ in range(3)]
ref = ccs.hits_to_numpy(ccs.intersect(sc, ccs.rays_to_device(small.soa()), ccs.make_opts(chunk=32)))
streams = [torch.cuda.Stream() for _ in range(3)]
ccs.ccs_release_scratch()   # nothing held yet


def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


# the kernels are loaded and the ray-persistent one has run: only scratch moves from here on
for st in (None, *streams):
    ccs.ccs_intersect(sc.handle, ccs.rays_to_device(small.soa()), small.n, hits[0], None, st)
    ccs.ccs_occluded(sc.handle, ccs.rays_to_device(small.soa()), small.n, torch.empty(small.n, dtype=torch.uint8, device="cuda"))
torch.cuda.synchronize()
ccs.ccs_release_scratch()
base = free()
ccs.ccs_intersect(sc.handle, rays, n, hits[0])
held = base - free()
assert 164 * n <= held <= 200 * n + (64 << 20), held
ccs.ccs_release_scratch()
assert base - free() <= 64 << 20, base - free()
# three streams: with the bound, and a release between launches that are still queued
for _ in range(4):
    for st, h in zip(streams, hits):
        ccs.ccs_intersect(sc.handle, rays, n, h, None, st)
    ccs.ccs_release_scratch()
assert base - free() <= (4 << 30) + (64 << 20), base - free()
ccs.ccs_release_scratch()
assert base - free() <= 64 << 20, base - free()
for h in hits:
    for k, p in zip(("t", "u", "v", "pid"), h):
        q = p.view(n // small.n, small.n)
        assert bool((q[0].view(torch.int32) == q.view(torch.int32)).all())
        a = q[0].cpu().numpy()
        assert np.array_equal(a.view(np.uint32) if k == "pid" else a, ref[k]), k
print("OK")
'''


def test_scratch_is_bounded_and_given_back():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_03510_gb300 import build_ext
    build_ext.build()
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=300, cwd=ROOT)
    assert r.returncode == 0 and r.stdout.split()[-1:] == ["OK"], r.stdout + r.stderr
