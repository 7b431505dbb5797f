// Device routines of the Gregory box tables (described in table.cu), shared by its kernel and the batch's.
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

}  // namespace ccs
