// The engine of a launch whose options leave it open, plain host C++ so that it can be tested on its own.
#pragma once
#include <stdint.h>

namespace ccs {

// Whether n rays on a scene of n_patches take the pair engine.  Both engines' times (us, ray-persistent / pair engine, on
// 96 to 98,304 patches; rays from one pixel to 1283 x 717 images, and the diffuse and mirror rays that leave them):
//
//  - In general it is 1.05 to 9.4 times faster: 1283 x 717 image of 1,536 patches 523 / 239 with local frames, 1338 / 433 in
//    world axes, of 98,304 patches 735 / 398 and 2410 / 671; 6,144 bounce rays there 160 / 106 and 480 / 191.
//  - Not below 32 rays, less than a warp: its three launches and the pool take longer than such rays (one pixel 25 / 33, 12
//    pixels 26 / 36 on 1,536 patches; bounce rays, which mostly miss, 13 / 21 to 31 / 38 on 96).  Few bounce rays on many
//    patches pay for that line (12 on 98,304 patches, world axes: 31 / 28 to 97 / 32).
//  - Not in world axes at leaf depths to 3, unless the rays are many for the patches: leaves are then so large (the cull
//    pads a root box by a leaf) that nearly every patch box is a candidate, and a pair's few steps do not repay its start
//    (4,096 rays at depth 2: 1,536 patches 73 / 98, 24,576 106 / 127, 98,304 109 / 146; 230,400 rays at depth 1 161 / 189
//    and 167 / 208).  With more rays than 16 a patch it wins there too (4,096 on 96 patches 55 / 39, 230,400 on 1,536
//    174 / 115, 919,911 on 24,576 420 / 347).
//  - Not above 2^23 rays (an 8.3 M pixel image fits), whose scratch of 1.6 GB the library's pool would keep.
inline bool pairs_by_default(uint32_t n, uint32_t n_patches, bool local, uint32_t leaf_depth)
{
    if (n < 32u || n > 1u << 23) return false;
    return local || leaf_depth > 3u || n > 16ull * n_patches;
}

// The refill threshold it runs with there: at 32 a warp waits for its slowest ray before it takes more (1283 x 717 image of
// 1,536 patches in world axes 1488 us, at 24 and below 433 to 440, the ray-persistent kernel 1187).
inline uint32_t default_pairs_refill(uint32_t refill) { return refill < 24u ? refill : 24u; }

}  // namespace ccs
