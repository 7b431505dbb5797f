// Which ray a thread of the pair engine's candidate pass takes (pairs.cuh), plain host/device C++ so that it can be tested
// on the host.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define CCS_CAND_HD __host__ __device__ __forceinline__
#else
#define CCS_CAND_HD inline
#endif

namespace ccs {

// The width in whose 8 x 4 pixel tiles the pass takes n rays, or 0: 32 consecutive rays per warp.  An image width that is
// a multiple of 8 and has at least one whole row; a wider one makes no tiles but up to 4 rows of threads without a ray
// (1,000 rays at a width of 2^24: 329 us, 98 in their own order).  The padded threads and the blocks' rounding fit in 32
// bits.
inline uint32_t cand_tile_width(uint32_t n, uint32_t image_width)
{
    if (image_width == 0 || (image_width & 7u) || image_width > n) return 0;
    return (uint64_t)n + 4ull * image_width <= 0xFFFFF000ull ? image_width : 0;
}

// The ray of candidate-pass thread t.  With img_w > 0 (from cand_tile_width) the rays are an image of that width,
// ray y * img_w + x, and each warp takes a tile of 8 x 4 pixels, whose rays walk more of the same BVH nodes
// than a row of 32; the threads then cover whole bands of 4 rows (cand_threads), and those past the last ray
// have none.  A bijection of [0, cand_threads) onto the same range either way.
CCS_CAND_HD uint32_t cand_ray(uint32_t t, uint32_t img_w)
{
    if (img_w == 0u) return t;
    const uint32_t w = t >> 5, l = t & 31u, tiles_x = img_w >> 3;
    const uint32_t ty = w / tiles_x, tx = w - ty * tiles_x;
    return (ty * 4u + (l >> 3)) * img_w + tx * 8u + (l & 7u);
}
inline uint32_t cand_threads(uint32_t n, uint32_t img_w)
{
    if (img_w == 0u) return n;
    const uint64_t band = 4ull * img_w;
    return (uint32_t)((n + band - 1) / band * band);
}

}  // namespace ccs
