// The pair engine's launch sequence (CCS_TRACE_PAIRS): counters zeroed, the candidate pass (which also
// lists each task under its cost class), then the subdivision pass.  One scene takes its scratch from the
// library's stream-ordered memory pool on the launch's stream; a batch brings its own, allocated with the
// batch, so that its run stays capturable in a CUDA graph.
#include <mutex>

#include "engine_plan.h"
#include "pairs_launch.cuh"

namespace ccs {

bool use_pairs(const LaunchCfg &cfg)
{
    return (cfg.flags & CCS_TRACE_PAIRS) && (cfg.mode == kModePlain || cfg.mode == kModeAnyHit) &&
           cfg.lanes_per_ray == 1;
}

// The engine of a launch that leaves it open: by its size (engine_plan.h), with the 1-slot sibling cache, the pair engine's
// fastest on images.  Not while the stream is captured, where the ray-persistent kernel needs no allocation; that kernel
// also takes the launch when the scratch cannot be had (launch_intersect).
void choose_engine(LaunchCfg &cfg, const ccs_scene *sc, uint32_t n, cudaStream_t s)
{
    if (!cfg.auto_engine || !pairs_by_default(n, sc->n, sc->local, cfg.leaf_depth)) return;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) {
        (void)cudaGetLastError();
        return;
    }
    if (cap != cudaStreamCaptureStatusNone) return;
    cfg.flags |= CCS_TRACE_PAIRS;
    cfg.refill = default_pairs_refill(cfg.refill);
    if (cfg.auto_cache) cfg.cache_slots = 1;
}

size_t pairs_scratch_bytes(uint32_t n) { return pair_scratch_bytes(n); }

namespace {

// The library's memory pools, one per device, created on first use.  Freed memory stays in a pool for reuse, as mapping it
// again would cost a launch more than it takes, up to kPoolKeep, which two of the largest launches that the library gives
// the pair engine by itself fit in (1.6 GB each), or the largest launch's scratch where that is more; the driver takes the
// rest back at the next synchronisation, and ccs_release_scratch all that no launch uses.
constexpr uint64_t kPoolKeep = (uint64_t)4 << 30;
struct ScratchPool {
    cudaMemPool_t pool = nullptr;
    uint64_t keep = 0;   // the release threshold set
};
std::mutex g_pool_mu;   // of the table
ScratchPool *current_pool()
{
    constexpr int kMaxDevices = 64;
    static ScratchPool pools[kMaxDevices];
    int dev = 0;
    return cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kMaxDevices ? &pools[dev] : nullptr;
}

// The pool of the current device for a launch that takes `bytes` of it.
cudaError_t pool_for(uint64_t bytes, cudaMemPool_t *out)
{
    std::lock_guard<std::mutex> lock(g_pool_mu);
    ScratchPool *p = current_pool();
    if (!p) return cudaErrorInvalidDevice;
    cudaError_t e;
    if (!p->pool) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        if ((e = cudaGetDevice(&props.location.id)) != cudaSuccess) return e;
        if ((e = cudaMemPoolCreate(&p->pool, &props)) != cudaSuccess) {
            p->pool = nullptr;
            return e;
        }
    }
    uint64_t keep = bytes > kPoolKeep ? bytes : kPoolKeep;
    if (keep > p->keep) {
        if ((e = cudaMemPoolSetAttribute(p->pool, cudaMemPoolAttrReleaseThreshold, &keep)) != cudaSuccess) return e;
        p->keep = keep;
    }
    *out = p->pool;
    return cudaSuccess;
}

template <bool STATS, int MODE, class Src, int BW>
cudaError_t launch_cand(const Src &src, const PairBufs &pb, const LaunchCfg &cfg, uint32_t n, uint32_t *status,
                        cudaStream_t s)
{
    const uint32_t img_w = cand_tile_width(n, cfg.image_width);
    const uint32_t t = cand_threads(n, img_w);
    k_cand<STATS, MODE, Src, BW><<<t / kCandBlock + (t % kCandBlock != 0), kCandBlock, 0, s>>>(
        src, pb, img_w, (int)cfg.leaf_depth, cfg.iter_cap, status, cfg.counters, cfg.mc.occluded);
    return cudaGetLastError();
}

template <int MODE, class Src>
cudaError_t cand_pass(const Src &src, const PairBufs &pb, const LaunchCfg &cfg, uint32_t n, uint32_t width,
                      uint32_t *status, cudaStream_t s)
{
    const bool stats = (cfg.flags & CCS_TRACE_COUNT) != 0;
    if (width == 4)
        return stats ? launch_cand<true, MODE, Src, 4>(src, pb, cfg, n, status, s)
                     : launch_cand<false, MODE, Src, 4>(src, pb, cfg, n, status, s);
    return stats ? launch_cand<true, MODE, Src, 2>(src, pb, cfg, n, status, s)
                 : launch_cand<false, MODE, Src, 2>(src, pb, cfg, n, status, s);
}

}  // namespace

cudaError_t pool_alloc(void **p, size_t bytes, cudaStream_t s)
{
    cudaMemPool_t pool = nullptr;
    const cudaError_t e = pool_for(bytes, &pool);
    if (e != cudaSuccess) return e;
    return cudaMallocFromPoolAsync(p, bytes, pool, s);
}

cudaError_t pool_free(void *p, cudaStream_t s) { return cudaFreeAsync(p, s); }

cudaError_t pool_trim()
{
    std::lock_guard<std::mutex> lock(g_pool_mu);
    ScratchPool *p = current_pool();
    if (!p) return cudaErrorInvalidDevice;
    return p->pool ? cudaMemPoolTrimTo(p->pool, 0) : cudaSuccess;
}

cudaError_t launch_pairs_single(const DevScene &sc, const DevRays &r, const DevHits &h, uint32_t n,
                                const LaunchCfg &cfg, uint32_t *status, int num_sms, cudaStream_t s)
{
    if (n == 0) return cudaSuccess;
    void *base = nullptr;
    cudaError_t e = pool_alloc(&base, pair_scratch_bytes(n), s);
    if (e != cudaSuccess) return e;
    const PairBufs pb = pair_bufs_at(base, n);
    const DirectSource src{{sc, r, h, n, nullptr}};
    e = cudaMemsetAsync(pb.ctr, 0, kPairCtrWords * sizeof(uint32_t), s);
    if (e == cudaSuccess) {
        if (cfg.mode == kModeAnyHit) {
            e = cand_pass<kModeAnyHit>(src, pb, cfg, n, sc.width, status, s);
            if (e == cudaSuccess) e = pair_passes_single_anyhit(src, pb, cfg, n, status, num_sms, s);
        } else {
            e = cand_pass<kModePlain>(src, pb, cfg, n, sc.width, status, s);
            if (e == cudaSuccess) e = pair_passes_single_plain(src, pb, cfg, n, status, num_sms, s);
        }
    }
    const cudaError_t e2 = pool_free(base, s);
    return e != cudaSuccess ? e : e2;
}

cudaError_t launch_pairs_batch(const BatchEntry *entries, const uint32_t *ray_prefix, uint32_t n_scenes,
                               uint32_t n_total, const LaunchCfg &cfg, void *scratch,
                               uint32_t *status, int num_sms, cudaStream_t s, uint32_t width)
{
    if (n_total == 0) return cudaSuccess;
    const PairBufs pb = pair_bufs_at(scratch, n_total);
    const BatchSource src{entries, ray_prefix, n_scenes, n_total};
    cudaError_t e = cudaMemsetAsync(pb.ctr, 0, kPairCtrWords * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    if ((e = cand_pass<kModePlain>(src, pb, cfg, n_total, width, status, s)) != cudaSuccess) return e;
    return pair_passes_batch(src, pb, cfg, n_total, status, num_sms, s);
}

}  // namespace ccs
