// Device routines of the Gregory box tables (described in table.cu), shared by its kernels and the batch's refit.
#pragma once

#include "table_plan.h"
#include "traverse.cuh"

namespace ccs {

// Node m of 2^D - 1 (level by level) of the Gregory patch of the given rank.
CCS_DEV void greg_table_node(const GregTabStore &t, const float4 *__restrict__ rec, uint32_t rank, uint32_t m)
{
    const int level = 31 - __clz(m + 1u);
    const uint32_t path = m + 1u - (1u << level);
    float u0, u1, v0, v1, g[48], d[3];
    Grp G;
    G.c = 0;
    node_domain(path, level, kMaxLeafDepth, u0, u1, v0, v1);   // (exact on any grid that holds the node)
    gregory_node<3>(rec + (size_t)t.list[rank] * kRecF4, u0, u1, v0, v1, level, G, g, d);
    SplitPts<3> S;
    float lmin[3], lmax[3], rmin[3], rmax[3];
    split_boxes<3>(g, d, S, lmin, lmax, rmin, rmax);
    float4 *nd = t.node + 4 * (((size_t)rank << t.stride) + table_index(level, path));
#pragma unroll
    for (int k = 0; k < 3; ++k) nd[k] = make_float4(lmin[k], lmax[k], rmin[k], rmax[k]);
}

// Thread i of the build over a batch's scenes that have new points: 2^levels threads per Gregory patch (the prefix
// counts the patches of scenes with a table).
CCS_DEV void batch_greg_node(const BatchEntry *__restrict__ entries, const uint32_t *__restrict__ prefix,
                             uint32_t n_scenes, uint32_t n, uint32_t levels, size_t i)
{
    const uint32_t p = (uint32_t)(i >> levels), m = (uint32_t)i & ((1u << levels) - 1u);
    if (p >= n) return;
    uint32_t lo = 0, hi = n_scenes;   // largest s with prefix[s] <= p
    while (hi - lo > 1) {
        const uint32_t h = (lo + hi) >> 1;
        if (__ldg(prefix + h) <= p) lo = h; else hi = h;
    }
    const BatchEntry &e = entries[lo];
    const uint32_t rank = p - prefix[lo], D = greg_update_levels(e.tab.n, e.tab.stride);
    if (!e.px) return;
    if (rank == 0 && m == 0) *e.tab.depth = D;
    if (m + 1u >= (1u << D)) return;
    greg_table_node(e.tab, e.rec, rank, m);
}

}  // namespace ccs
