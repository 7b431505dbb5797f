// Sizes of the Gregory box tables (table.cu), plain host/device C++ so that they can be tested on the host.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define CCS_TABLE_HD __host__ __device__ inline
#else
#define CCS_TABLE_HD inline
#endif

namespace ccs {

constexpr uint32_t kGregLevels = 16;                   // levels stored
constexpr uint64_t kGregBytes = (uint64_t)256 << 20;   // bytes of nodes stored

// Levels that `bytes`, at most kGregBytes, hold for n patches.
inline uint32_t greg_table_levels(uint32_t n, uint64_t bytes)
{
    const uint64_t most = bytes < kGregBytes ? bytes : kGregBytes;
    uint32_t D = n ? kGregLevels : 0;
    while (D > 0 && ((uint64_t)n << D) * 64 > most) --D;
    return D;
}

// Levels built after an update of the points, which an animated scene pays for every frame, whoever traces it: at most 10,
// and 2^16 nodes in all.  An update takes 11 us without a table, 17 with up to 2^16 nodes (29 to 31 on 64,896 patches,
// where the repack itself is as long); with 10 levels of every patch it took 80 us on 1,536 Gregory patches, 188 on 4,056
// and 237 on 64,896.  An update, a refit and a pair-engine call on 230,400 rays, us without a table / 10 levels / 2^16
// nodes: 24 patches 280 / 166 / 169, 384 300 / 269 / 257, 1,536 324 / 331 / 289, 4,056 339 / 454 / 305, 64,896 626 / 828 /
// 626; with 2^15 nodes 168 / 265 / 291 / 312 / 617, with 2^18 167 / 255 / 281 / 305 / 623.
constexpr uint32_t kGregUpdateLevels = 10;
constexpr uint64_t kGregUpdateNodes = 1u << 16;
CCS_TABLE_HD uint32_t greg_update_levels(uint32_t n, uint32_t stored)
{
    uint32_t D = stored < kGregUpdateLevels ? stored : kGregUpdateLevels;
    while (D > 0 && ((uint64_t)n << D) > kGregUpdateNodes) --D;
    return D;
}

// Blocks of kGregBlock threads that build those levels, one thread per node (one block for the depth word where no level is
// built, none for a scene without a table).
constexpr uint32_t kGregBlock = 128;
inline uint32_t greg_update_blocks(uint32_t n, uint32_t stored)
{
    if (n == 0 || stored == 0) return 0;
    const uint32_t D = greg_update_levels(n, stored);
    return D ? (uint32_t)((((uint64_t)n << D) + kGregBlock - 1) / kGregBlock) : 1;
}

}  // namespace ccs
