"""The first launches of a process, in a process of their own: several threads whose first calls have leaf depths (shared
memory sizes) of their own, and a capture whose warm-up was the same call outside of it, which takes another engine."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = r'''
import threading
import numpy as np
import torch
from paper_1811_03510_gb300 import ccs, scenegen as sg

ccs.lib()
torch.cuda.set_device(0)
s = sg.make_scene(4, 0.06, 3, 1)
sc = ccs.Scene(s.P, s.types, local=True)
n = 5000
rays = ccs.rays_to_device(sg.random_rays(n, seed=1).soa())


def same(a, b):
    return all(np.array_equal(a[k], b[k]) for k in ("t", "u", "v", "pid"))
'''

THREADS = HEAD + r'''
DEPTHS = (15, 1, 8, 12, 3, 10)
hits = [ccs.alloc_hits(n) for _ in DEPTHS]
streams = [torch.cuda.Stream() for _ in DEPTHS]
torch.cuda.synchronize()
gate, errors = threading.Barrier(len(DEPTHS)), []


def work(k):
    try:
        torch.cuda.set_device(0)
        gate.wait()
        for _ in range(20):
            ccs.ccs_intersect(sc.handle, rays, n, hits[k], ccs.make_opts(leaf_depth=DEPTHS[k]), streams[k])
    except Exception as e:
        errors.append((DEPTHS[k], repr(e)))


pool = [threading.Thread(target=work, args=(k,)) for k in range(len(DEPTHS))]
for p in pool:
    p.start()
for p in pool:
    p.join()
torch.cuda.synchronize()
assert not errors, errors
for k, L in enumerate(DEPTHS):
    ref = ccs.hits_to_numpy(ccs.intersect(sc, rays, ccs.make_opts(leaf_depth=L, chunk=32)))
    assert same(ccs.hits_to_numpy(hits[k]), ref), L
print("OK")
'''

CAPTURE = HEAD + r'''
hits, occ = ccs.alloc_hits(n), torch.zeros(n, dtype=torch.uint8, device="cuda")


def step():
    ccs.ccs_intersect(sc.handle, rays, n, hits)
    ccs.ccs_occluded(sc.handle, rays, n, occ)


side = torch.cuda.Stream()
side.wait_stream(torch.cuda.current_stream())
with torch.cuda.stream(side):   # the warm-up: the pair engine
    for _ in range(3):
        step()
torch.cuda.current_stream().wait_stream(side)
torch.cuda.synchronize()
ref = ccs.hits_to_numpy(hits)
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g):       # the ray-persistent kernel, for the first time in this process
    step()
for p in hits:
    p.fill_(-3)
occ.fill_(7)
g.replay()
torch.cuda.synchronize()
assert same(ccs.hits_to_numpy(hits), ref)
assert np.array_equal(occ.cpu().numpy().astype(bool), ref["pid"] != 0xFFFFFFFF) and int(occ.max()) == 1
print("OK")
'''


@pytest.fixture(scope="module", autouse=True)
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1811_03510_gb300 import build_ext
    build_ext.build()


def run_alone(code):
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300, cwd=ROOT)
    assert r.returncode == 0 and r.stdout.split()[-1:] == ["OK"], r.stdout + r.stderr


def test_first_calls_of_threads_with_their_own_leaf_depths():
    run_alone(THREADS)


def test_capture_after_a_warm_up_with_the_same_call():
    run_alone(CAPTURE)
