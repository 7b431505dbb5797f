"""Options that leave the engine to the library, as bench.py closes them before it times and counts: the counting launch, whose
flag would send open options to the ray-persistent kernel, runs the same engine, and the screen-space workload's arms both run
the ray-persistent kernel."""
import pytest

import bench
from paper_1811_03510_gb300 import ccs


@pytest.mark.parametrize("kw,n,patches,local,engine", [
    ({}, 2073600, 1536, True, "pairs"), (dict(refill=32), 2073600, 1536, False, "pairs"), ({}, 31, 96, True, "ray"),
    ({}, (1 << 23) + 1, 96, True, "ray"), (dict(leaf_depth=2), 4096, 1536, False, "ray"),
    (dict(leaf_depth=2), 4096, 1536, True, "pairs"), (dict(leaf_depth=2), 4096, 96, False, "pairs"),
    (dict(chunk=64), 2073600, 1536, True, "ray"), (dict(order=True), 2073600, 1536, True, "ray+order"),
    (dict(pairs=True, cache_slots=0), 100, 96, True, "pairs"), (dict(lanes_per_ray=3), 2073600, 1536, True, "ray")])
def test_closed_options_hold_the_engine_with_and_without_counters(kw, n, patches, local, engine):
    o = bench.closed_opts(ccs.make_opts(**kw), n, patches, local)
    assert not bench.leaves_engine_open(o) and bench.engine_of(o) == engine
    counting = ccs.make_opts(**ccs.opts_dict(o), counters=1)
    assert bench.engine_of(counting) == engine
    assert (counting.flags & ccs.CCS_TRACE_PAIRS) == (o.flags & ccs.CCS_TRACE_PAIRS)
    if engine == "pairs":
        assert o.cache_slots == kw.get("cache_slots", 1) and o.refill <= 24
    assert o.leaf_depth == kw.get("leaf_depth", 8)


@pytest.mark.parametrize("kw", [{}, dict(pairs=True, image_width=1920), dict(chunk=64), dict(refill=16)])
def test_screen_space_arms_ask_for_the_ray_kernel(kw):
    for spread in (0.0, 0.001):
        o = ccs.make_opts(**bench.ray_kernel_opts(ccs.make_opts(**kw)), pixel_spread=spread)
        assert not bench.leaves_engine_open(o) and bench.engine_of(o) == "ray" and o.chunk == kw.get("chunk", 32)


def test_options_tuned_for_the_pair_engine_do_not_reach_the_ray_kernel():
    d = bench.ray_kernel_opts(ccs.make_opts(pairs=True, min_blocks=4, vote=12, block_threads=96, cache_slots=0, refill=24,
                                            bvh_width=4, image_width=1920, leaf_depth=7))
    assert (d["min_blocks"], d["vote"], d["block_threads"], d["refill"], d["cache_slots"]) == (0, 0, 0, 0, ccs.CCS_CACHE_DEFAULT)
    assert (d["bvh_width"], d["image_width"], d["leaf_depth"], d["chunk"]) == (4, 1920, 7, 32)
    assert bench.ray_kernel_opts(ccs.make_opts(min_blocks=4, vote=12, chunk=64))["min_blocks"] == 4   # its own stay
