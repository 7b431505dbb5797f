// Gregory box tables: the boxes of the sub-domains of a scene's Gregory patches, stored once per scene (and again
// after an update of its points) instead of computed by every ray that visits them.  A node's bound (Algorithm 2
// with the crop of Algorithm 1, about 1130 operations, then a split of 360) does not depend on the ray: the
// extension of local frames and the clipping to the parent's interval come where a ray tests the boxes.  The
// stored boxes are bit for bit those that gregory_node and split_step give, by the same code.
//
// Why: a Gregory step takes a lone warp about 7,000 cycles, a Bezier step 1,600, and a ray that grazes a Gregory patch
// takes dozens of them one after another, so launches ended on such rays.  A table step (48 bytes, two slab tests)
// is bound by the latency of its load, so two siblings share a line and each step asks for the lines of the nodes two
// levels down.  Measured, before and after (us per pair-engine call): 64 x 64 rays on 96 patches 165 -> 115, 330 k
// diffuse rays on 1,632 patches 250 -> 191, 1.2 M mirror rays on 98,400 patches 665 -> 525; 1080p primary rays, which
// rarely meet one, unchanged.  (The prefetches and the siblings' shared lines: 214 -> 202 us on the diffuse rays.)
// Levels: meshes have few irregular faces, so their tables may be deep; 16 levels, all of leaf depth 8 (4.2 MB), per
// patch while they fit in 256 MB (14 levels: 149 us instead of 132 on 96 patches of another seed).  After an update of
// the points at most 10 levels and 2^16 nodes (table_plan.h), built beside a batch's refit.
#include "table_dev.cuh"

namespace ccs {

namespace {

__global__ void __launch_bounds__(kGregBlock) k_greg_table(GregTabStore t, const float4 *__restrict__ rec, uint32_t D)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) *t.depth = D;
    if (i >= (size_t)t.n << D) return;
    const uint32_t m = (uint32_t)i & ((1u << D) - 1u);
    if (m + 1u < (1u << D)) greg_table_node(t, rec, (uint32_t)(i >> D), m);
}

}  // namespace

cudaError_t launch_greg_table(const GregTabStore &t, const float4 *rec, bool update, cudaStream_t s)
{
    if (!t.stride) return cudaSuccess;
    const uint32_t D = update ? greg_update_levels(t.n, t.stride) : t.stride;
    const uint32_t blocks = update ? greg_update_blocks(t.n, t.stride) : (uint32_t)((((size_t)t.n << D) + kGregBlock - 1) / kGregBlock);
    k_greg_table<<<blocks, kGregBlock, 0, s>>>(t, rec, D);
    return cudaGetLastError();
}

}  // namespace ccs
