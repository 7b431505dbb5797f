// Closest hit in passes that each keep a warp on one kind of work (the pair engine, CCS_TRACE_PAIRS).
//
//  1. k_cand: one thread per ray walks the BVH (Sec. 4) and keeps the ray's kPairCands nearest candidate
//     patches, ordered by (entry distance of the patch box, patch id).  Before the list is full nothing
//     is pruned but [tmin, tmax]; once it is full, subtrees that enter beyond its last entry are skipped
//     and the smallest entry distance dropped that way is kept (t_evict).  A Bezier patch whose root box in its
//     own frame the ray does not come near is no candidate (root_box_near: its pair would record no leaf).  A ray with
//     candidates becomes a task with a cost class (the highest when a candidate is a Gregory patch, else its number of
//     candidates); rays with no candidate are written as misses here.
//  2. Each task's index goes to the list of its cost class (the candidate pass counts the classes' places),
//     and the subdivision pass's queue takes the classes costliest first, so that the long rays start
//     early and the launch does not end on a few of them.
//  3. k_pairs: persistent warps take tasks in that order.  A lane runs Algorithm 3 on one (ray, patch) pair
//     at a time, taking the ray's candidates in entry order and stopping at the first one that enters
//     beyond the ray's best hit.  Every warp iteration is one or two subdivision steps (Algorithm 3's loop
//     body) of up to 32 pairs: the BVH walk, whose step count differs from ray to ray, is not in the loop.
//  4. A ray whose dropped candidates could still hold the answer (best hit not before t_evict) has its lane
//     collect the next ones, those after the last listed, by a BVH walk of its own (collect_more), and goes
//     on with them.
//
// The answer is the smallest leaf key over all nested intervals (readings A14/A15), which does not depend
// on the order in which pairs are searched, so every pass reuses the arithmetic of traverse.cuh and the
// hits are bit-identical to k_intersect's.
#pragma once

#include "cand_plan.h"
#include "intersect_impl.cuh"

namespace ccs {

constexpr int kPairCands = 8;            // candidates kept per ray (nearest entries)
constexpr int kCandBlock = 128;          // threads of a candidate-pass block (its warps work independently)
constexpr int kStepsPerIter = 2;         // subdivision steps per warp iteration of the subdivision pass
constexpr int kCostClasses = 16;
// counter words of a launch: the queue head, the tasks of each cost class
constexpr int kCtrQueue = 3, kCtrHist = 16, kPairCtrWords = 64;
// Ray i's task and candidates have fixed places (task i, candidates from i kPairCands), so the candidate
// pass needs no atomic counter for them.  A task is 4 uint4 (64 bytes), everything a lane needs to start
// the ray:
//   (ray, first candidate, z, t_evict bits), (first candidate's patch id, its entry distance, tmin, tmax),
//   (ox, oy, oz, dx), (dy, dz, 0, 0) as float bits;
// z = candidates (bits 0..7) | cost class (bits 8..11) | candidates were dropped (bit 30).
constexpr uint32_t kTaskEvicted = 0x40000000u;

struct PairBufs {
    uint32_t *ctr;            // kPairCtrWords words, zeroed before the candidate pass
    uint4 *task;              // task of ray i at 4 i (rays with candidates only)
    uint32_t *cls;            // per cost class c, from c * n: the rays of its tasks
    uint2 *cand;              // (patch id, entry distance bits), ray i's from i kPairCands
    uint32_t n;               // rays of the launch (the stride of cls)
};

// Bytes of the pair engine's scratch for n rays, and its layout (every part 256-byte aligned).
__host__ __device__ inline size_t pair_align(size_t b) { return (b + 255) & ~(size_t)255; }
inline size_t pair_scratch_bytes(uint32_t n)
{
    return pair_align(kPairCtrWords * 4) + pair_align((size_t)n * 64) + pair_align((size_t)n * 4 * kCostClasses) +
           pair_align((size_t)n * kPairCands * 8);
}
inline PairBufs pair_bufs_at(void *base, uint32_t n)
{
    char *p = static_cast<char *>(base);
    PairBufs b;
    b.ctr = reinterpret_cast<uint32_t *>(p);
    p += pair_align(kPairCtrWords * 4);
    b.task = reinterpret_cast<uint4 *>(p);
    p += pair_align((size_t)n * 64);
    b.cls = reinterpret_cast<uint32_t *>(p);
    p += pair_align((size_t)n * 4 * kCostClasses);
    b.cand = reinterpret_cast<uint2 *>(p);
    b.n = n;
    return b;
}

// Shared memory of a k_pairs thread after its traversal scratch: the world ray of its task (origin,
// 1 / direction, tmin, tmax), t_evict and the direction, read when a pair starts and when the ray ends, and
// the first and end places of the task's candidates (kept here, not in registers, so that the 1-slot sibling
// cache variant does not spill); then the thread's mailbox for the subtrees it handed to other lanes (the smallest (t, cell) key they found,
// 64 bits), the number of them still running, and a flag for one that reached the iteration cap.
constexpr int kRaySlotFloats = 14, kHelpFloats = 4;
// the per-thread helper area must hold the mailbox and the two counters k_pairs places there
static_assert(kHelpFloats * sizeof(float) >= sizeof(unsigned long long) + 2 * sizeof(int),
              "the helper area of a k_pairs thread is smaller than its mailbox and counters");
// A subtree is handed to an idle lane when it has at least this many levels below its root.
constexpr int kMinDonateLevels = 4;

// Order-preserving map of a float's bits to an unsigned integer, and back (the mailbox key).
CCS_DEV uint32_t ord_bits(float t)
{
    const uint32_t u = __float_as_uint(t);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
CCS_DEV float unord_bits(uint32_t k) { return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k); }

// The scene of a lane's pair, handed from lane `from` to the lanes that take one of its subtrees (a batch
// lane carries its scene's index; one scene is the launch's).
template <class Src>
CCS_DEV void share_scene(typename Src::LaneScene &l, int from)
{
    if constexpr (std::is_same<Src, BatchSource>::value) l.s = __shfl_sync(0xffffffffu, l.s, from);
}

template <class Src>
CCS_DEV bool same_scene(const typename Src::LaneScene &a, const typename Src::LaneScene &b)
{
    if constexpr (std::is_same<Src, BatchSource>::value) return a.s == b.s;
    else return true;
}

CCS_DEV bool cand_less(float ta, uint32_t pa, float tb, uint32_t pb) { return ta < tb || (ta == tb && pa < pb); }

// The ray as k_intersect's begin_ray reads it (false: a ray that is a miss by definition).
CCS_DEV bool load_world_ray(const DevRays &rr, uint32_t j, float (&o)[3], float (&d)[3], float (&inv)[3], float &tmin,
                            float &tmax)
{
    o[0] = __ldg(rr.ox + j);
    o[1] = __ldg(rr.oy + j);
    o[2] = __ldg(rr.oz + j);
    d[0] = __ldg(rr.dx + j);
    d[1] = __ldg(rr.dy + j);
    d[2] = __ldg(rr.dz + j);
    tmin = __ldg(rr.tmin + j);
    tmax = __ldg(rr.tmax + j);
#pragma unroll
    for (int k = 0; k < 3; ++k) inv[k] = safe_inv(d[k]);
    return !(!(tmin <= tmax) || isnan(o[0]) || isnan(o[1]) || isnan(o[2]) || isnan(d[0]) || isnan(d[1]) ||
             isnan(d[2]));
}

template <int MODE, class Src>
CCS_DEV void write_miss(const Src &src, uint32_t scene, uint32_t j, uint8_t *occluded)
{
    if (MODE == kModeAnyHit) {
        occluded[j] = 0;
    } else {
        const DevHits &hh = src.hits_of(scene);
        hh.t[j] = __int_as_float(0x7f800000);
        hh.u[j] = 0.0f;
        hh.v[j] = 0.0f;
        hh.pid[j] = kMissId;
    }
}

// Cull test of a candidate: does the ray pass near the patch's root box in the patch's own frame (Sec. 3.4)?  With
// local frames every box of a Bezier pair's subdivision lies in that box (de Casteljau midpoints stay between their
// operands), widened by the box extension by at most tau / 2.  Without them the boxes are world boxes, but what a pair
// records are leaves, and a leaf's box reaches at most its own size beyond the points inside the root box
// (leaf = 2^-L: at most leaf times the bound in slot 19).  A pair's FP32 slab tests report a hit only within about
// 1e-6 (|o - anchor| + box diagonal) of a box; the test pads the box by 2^-16 (1 + |o - anchor|_1 + |hi - lo|_1),
// far more than that and far less than a patch, and by the leaf's size, so a culled pair holds no leaf that its
// subdivision would record.  Gregory patches are kept (their boxes come from the bounds of Algorithm 2, not from the
// control points).
// Without local frames this measured (1283 x 717 images, binary BVH): candidates 699 k -> 385 k and rays with more than
// the list holds 15,090 -> 2 on 1,536 patches, so that no lane ends the launch walking the BVH again; call 813 -> 628 us,
// on 24,576 patches 1714 -> 1131 us, 153 k bounce rays there 746 -> 310 us.
CCS_DEV bool root_box_near(const float4 *__restrict__ rec, const float (&o)[3], const float (&d)[3], float tmin,
                           bool local, float leaf, const Grp &G)
{
    const float4 an = __ldg(rec + 15);
    if (an.w != 0.0f) return true;
    const float4 R[3] = {__ldg(rec + 16), __ldg(rec + 17), __ldg(rec + 18)};
    const float4 hb = __ldg(rec + 19);
    const float o3[3] = {__fsub_rn(o[0], an.x), __fsub_rn(o[1], an.y), __fsub_rn(o[2], an.z)};
    const float diag1 = local ? hb.w : 1.0f + ((hb.x - R[0].w) + (hb.y - R[1].w) + (hb.z - R[2].w));
    float pad = __fmul_rn(__int_as_float((127 - 16) << 23),
                          __fadd_rn(diag1, __fadd_rn(__fadd_rn(fabsf(o3[0]), fabsf(o3[1])), fabsf(o3[2]))));
    if (!local) pad = fmaf(leaf, hb.w, pad);
    RayG<3> r;
    float lo[3], hi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        r.org[k] = fmaf(R[k].x, o3[0], fmaf(R[k].y, o3[1], R[k].z * o3[2]));
        r.inv[k] = safe_inv(fmaf(R[k].x, d[0], fmaf(R[k].y, d[1], R[k].z * d[2])));
        lo[k] = __fsub_rn(R[k].w, pad);
        hi[k] = __fadd_rn(pick(k, hb.x, hb.y, hb.z), pad);
    }
    float t0, t1;
    slab<3>(r, lo, hi, tmin, __int_as_float(0x7f800000), G, t0, t1);
    return t0 <= t1;
}

// ------------------------------------------------------------------------------------------------
// Pass 1: BVH walk with the sorted candidate list.
// ------------------------------------------------------------------------------------------------
// Whether root_box_near can tell for a ray with direction d.  safe_inv moves components below 1e-20 to that size, along the
// world axes for the BVH's boxes and along the frame's axes here, so the two rays agree only where that is nothing: with a
// largest component of 2^-40 or more it is less than the rounding of the rotated direction.  Up to 2^100 the rotated
// components and their inverses are finite and normal.
CCS_DEV bool cullable(const float (&d)[3])
{
    const float m = max3f(fabsf(d[0]), fabsf(d[1]), fabsf(d[2]));
    return m >= __int_as_float((127 - 40) << 23) && m <= __int_as_float((127 + 100) << 23);
}

// A patch whose box the ray enters at n0: into the sorted list, unless the ray does not come near its root box; the last
// entry of a full list, or the patch itself, is dropped.
template <bool STATS>
CCS_DEV void list_patch(const DevScene &sc, uint32_t p, float n0, const float (&ro)[3], const float (&rd)[3], float tmin,
                        float leaf, float (&kt)[kPairCands], uint32_t (&kp)[kPairCands], int &cnt, float &t_evict, bool &evicted,
                        unsigned long long &culled, const Grp &G)
{
    constexpr int C = kPairCands;
    if (!root_box_near(rec_of(sc, p), ro, rd, tmin, sc.local != 0, leaf, G)) {
        if (STATS) ++culled;
        return;
    }
    if (cnt == C) {
        evicted = true;
        if (!cand_less(n0, p, kt[C - 1], kp[C - 1])) {
            t_evict = fminf(t_evict, n0);
            return;
        }
        t_evict = fminf(t_evict, kt[C - 1]);
    } else {
        ++cnt;
    }
    int m = 0;
#pragma unroll
    for (int j = 0; j < C; ++j) m += cand_less(kt[j], kp[j], n0, p) ? 1 : 0;
#pragma unroll
    for (int j = C - 1; j >= 1; --j) {
        kt[j] = j > m ? kt[j - 1] : (j == m ? n0 : kt[j]);
        kp[j] = j > m ? kp[j - 1] : (j == m ? p : kp[j]);
    }
    kt[0] = m == 0 ? n0 : kt[0];
    kp[0] = m == 0 ? p : kp[0];
}

// A BVH walk of one ray (Sec. 4): the C candidates of the ray with the smallest keys (entry distance of the patch box,
// patch id) above (lb_t, lb_p), sorted in kt / kp: those that an earlier walk did not list (all its dropped keys are
// above its last listed one).  Before the list is full nothing is pruned but [tmin, tmax]; once it is full, subtrees
// entered beyond its last entry are skipped and the smallest entry distance dropped that way is kept (t_evict).  Bezier
// patches whose root box the ray does not come near are no candidates (root_box_near).  Returns false when the
// iteration budget it ran out.
template <int BW>
CCS_DEV bool walk_candidates(const DevScene &sc, const RayG<3> &r, const float (&ro)[3], const float (&rd)[3],
                             float tmin, float tmax, float leaf, float lb_t, uint32_t lb_p, uint32_t &it,
                             float (&kt)[kPairCands], uint32_t (&kp)[kPairCands], int &cnt, float &t_evict,
                             bool &evicted, const Grp &G)
{
    constexpr int C = kPairCands;
    const float kInf = __int_as_float(0x7f800000);
    int2 stk[kBvhStack];
    int sp = 0, node = 0;
    float n0 = tmin;
    unsigned long long none = 0;   // (its culls are not counted)
    for (;;) {
        if (node == kDone) break;
        if (it == 0) return false;
        --it;
        if (node < 0) {   // a patch: into the list (the leaf's box is the patch box)
            const uint32_t p = (uint32_t)(~node);
            // (not one that an earlier walk listed)
            if (cand_less(lb_t, lb_p, n0, p))
                list_patch<false>(sc, p, n0, ro, rd, tmin, leaf, kt, kp, cnt, t_evict, evicted, none, G);
        } else {
            // once the list is full, a subtree entered beyond its last entry only holds dropped patches
            const float bound = cnt == C ? kt[C - 1] : tmax;
            if constexpr (BW == 4) {
                const float4 *nd = sc.nodes + (size_t)node * kNode4F4;
                float4 lo4[3], hi4[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    lo4[k] = __ldg(nd + 2 * k);
                    hi4[k] = __ldg(nd + 2 * k + 1);
                }
                const int4 ch = __ldg(reinterpret_cast<const int4 *>(nd + 6));
                int c[4] = {ch.x, ch.y, ch.z, ch.w};
                float key[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float lo[3], hi[3];
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        lo[k] = j == 0 ? lo4[k].x : j == 1 ? lo4[k].y : j == 2 ? lo4[k].z : lo4[k].w;
                        hi[k] = j == 0 ? hi4[k].x : j == 1 ? hi4[k].y : j == 2 ? hi4[k].z : hi4[k].w;
                    }
                    float t0, t1;
                    slab<3>(r, lo, hi, tmin, tmax, G, t0, t1);
                    bool h = t0 <= t1 && c[j] != kEmptyChild;
                    if (h && t0 > bound) {
                        h = false;
                        evicted = true;
                        t_evict = fminf(t_evict, t0);
                    }
                    key[j] = h ? t0 : kInf;
                }
                cx4(key, c, 0, 1);
                cx4(key, c, 2, 3);
                cx4(key, c, 0, 2);
                cx4(key, c, 1, 3);
                cx4(key, c, 1, 2);
                if (key[0] < kInf) {
#pragma unroll
                    for (int j = 3; j >= 1; --j) {
                        if (key[j] < kInf && sp < kBvhStack) {
                            stk[sp] = make_int2(c[j], __float_as_int(key[j]));
                            ++sp;
                        }
                    }
                    node = c[0];
                    n0 = key[0];
                    continue;
                }
            } else {
                const float4 *nd = sc.nodes + (size_t)node * kNodeF4;
                float4 q[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) q[k] = __ldg(nd + k);
                const int2 ch = __ldg(reinterpret_cast<const int2 *>(nd + 3));
                float a0, a1, b0, b1;
                node_child_boxes<3>(q, r, tmin, tmax, G, a0, a1, b0, b1);
                bool ha = a0 <= a1 && ch.x != kEmptyChild;
                bool hb = b0 <= b1 && ch.y != kEmptyChild;
                if (ha && a0 > bound) {
                    ha = false;
                    evicted = true;
                    t_evict = fminf(t_evict, a0);
                }
                if (hb && b0 > bound) {
                    hb = false;
                    evicted = true;
                    t_evict = fminf(t_evict, b0);
                }
                if (ha && hb) {
                    const bool bfirst = b0 < a0;
                    if (sp < kBvhStack) {
                        stk[sp] = make_int2(bfirst ? ch.x : ch.y, __float_as_int(bfirst ? a0 : b0));
                        ++sp;
                    }
                    node = bfirst ? ch.y : ch.x;
                    n0 = bfirst ? b0 : a0;
                    continue;
                }
                if (ha || hb) {
                    node = ha ? ch.x : ch.y;
                    n0 = ha ? a0 : b0;
                    continue;
                }
            }
        }
        // pop the nearest pending subtree that can still add to the list
        node = kDone;
        while (sp > 0) {
            --sp;
            const int2 e = stk[sp];
            const float t0 = __int_as_float(e.y);
            if (cnt == C && t0 > kt[C - 1]) {
                evicted = true;
                t_evict = fminf(t_evict, t0);
                continue;
            }
            node = e.x;
            n0 = t0;
            break;
        }
    }
    return true;
}

// The walk of one ray in the candidate pass: the kPairCands nearest of all its candidates.  Patches go to a buffer of the
// lane in shared memory (buf, strided), and are looked at together once a lane's buffer is full or its walk done: the
// lanes of a warp, out of step in the tree, then share the expensive part (the cull, 5 loads, and the insertion), and the
// node loop holds nothing else.  The children are not sorted, but the nearest is entered first: the order only decides
// what a full list drops.
// Measured (us per call, walking node by node and patch by patch before): 1.2 M mirror rays on 98,400 patches 527 -> 492,
// 330 k diffuse rays on 1,632 patches 190 -> 177, 4K image of 98,304 patches (warps without a beam) 1761 -> 1753; with a
// buffer of 4 patches 569 / 185 / 1866, of 8 506 / 179 / 1775, of 16 490 / 176 / 1750 but 1410 instead of 1376 us for an
// animated batch (shared memory).
constexpr int kLeafBuf = 12;
template <bool STATS, int BW>
CCS_DEV bool walk_buffered(const DevScene &sc, const RayG<3> &r, const float (&ro)[3], const float (&rd)[3], float tmin,
                           float tmax, float leaf, uint32_t &it, float (&kt)[kPairCands], uint32_t (&kp)[kPairCands],
                           int &cnt, float &t_evict, bool &evicted, unsigned long long &nodes, unsigned long long &culled,
                           uint2 *buf, int stride, const Grp &G)
{
    constexpr int C = kPairCands;
    int stk[kBvhStack];
    int sp = 0, node = 0, nb = 0;
    for (;;) {
        while (node != kDone && nb <= kLeafBuf - BW) {
            if (it == 0) return false;
            --it;
            ++nodes;
            // once the list is full, a subtree entered beyond its last entry only holds dropped patches
            const float bound = cnt == C ? kt[C - 1] : __int_as_float(0x7f800000);
            int next = kDone;
            float next_t = 0.0f;
            auto child = [&](int c, float t0, float t1) {
                if (!(t0 <= t1) || c == kEmptyChild) return;
                if (t0 > bound) {
                    evicted = true;
                    t_evict = fminf(t_evict, t0);
                } else if (c < 0) {
                    buf[nb * stride] = make_uint2((uint32_t)(~c), __float_as_uint(t0));
                    ++nb;
                } else {
                    int far = c;
                    if (next == kDone || t0 < next_t) {
                        far = next;
                        next = c;
                        next_t = t0;
                    }
                    if (far != kDone && sp < kBvhStack) stk[sp++] = far;
                }
            };
            if constexpr (BW == 4) {
                const float4 *nd = sc.nodes + (size_t)node * kNode4F4;
                float4 lo4[3], hi4[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    lo4[k] = __ldg(nd + 2 * k);
                    hi4[k] = __ldg(nd + 2 * k + 1);
                }
                const int4 ch = __ldg(reinterpret_cast<const int4 *>(nd + 6));
                const int c[4] = {ch.x, ch.y, ch.z, ch.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float lo[3], hi[3];
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        lo[k] = j == 0 ? lo4[k].x : j == 1 ? lo4[k].y : j == 2 ? lo4[k].z : lo4[k].w;
                        hi[k] = j == 0 ? hi4[k].x : j == 1 ? hi4[k].y : j == 2 ? hi4[k].z : hi4[k].w;
                    }
                    float t0, t1;
                    slab<3>(r, lo, hi, tmin, tmax, G, t0, t1);
                    child(c[j], t0, t1);
                }
            } else {
                const float4 *nd = sc.nodes + (size_t)node * kNodeF4;
                float4 q[3];
#pragma unroll
                for (int k = 0; k < 3; ++k) q[k] = __ldg(nd + k);
                const int2 ch = __ldg(reinterpret_cast<const int2 *>(nd + 3));
                float a0, a1, b0, b1;
                node_child_boxes<3>(q, r, tmin, tmax, G, a0, a1, b0, b1);
                child(ch.x, a0, a1);
                child(ch.y, b0, b1);
            }
            node = next != kDone ? next : sp > 0 ? stk[--sp] : kDone;
        }
#pragma unroll 1
        for (int q = 0; q < nb; ++q) {
            if (it == 0) return false;
            --it;
            const uint2 e = buf[q * stride];
            list_patch<STATS>(sc, e.x, __uint_as_float(e.y), ro, rd, tmin, leaf, kt, kp, cnt, t_evict, evicted, culled, G);
        }
        nb = 0;
        if (node == kDone) return true;
    }
}

// ------------------------------------------------------------------------------------------------
// The walk of a warp whose rays are coherent: the BVH once for all of them, as a beam.  Per axis the beam is the
// interval of the rays' origins and the interval of their inverse directions, all of one sign; rounded subtraction
// and multiplication are monotone, so the products of the interval ends bound every ray's own slab distances, and a
// box that the beam misses is missed by every ray (whose entry into a leaf box implies its entry into the boxes
// above).  Each round 8 nodes (16 binary ones) are taken from a stack in shared memory and each lane tests one child;
// then every ray is tested against the boxes of the patches found, with the arithmetic of the rays' own walk.
//
// Why: rays of an image tile (32 pixels) walk the same nodes, but one after the other and out of step: a warp took
// as many iterations as its slowest ray has nodes and patches, both branches in each.  The beam needs one round of
// about 60 instructions per level.  Measured (this pass, before and after): 1080p image of 1,536 patches 150 -> 76 us,
// 4K image of 98,304 patches 1000 -> 545 us; bounce rays, which make no beam, unchanged (the test costs them about
// 20 reductions per warp).
// ------------------------------------------------------------------------------------------------
constexpr int kBeamStack = 64, kBeamLeaves = 96;
constexpr int kBeamWords = kBeamStack + kBeamLeaves;   // shared-memory words per warp
// below this iteration cap every ray walks on its own, as the cap counts its steps
constexpr uint32_t kBeamMinCap = 1u << 16;

CCS_DEV float warp_min(float v)
{
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}
CCS_DEV float warp_max(float v)
{
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

// Patches whose boxes the warp's beam meets, in `leaves`; their number, or -1 when the rays make no beam (directions
// of both signs along an axis, a value that is not finite) or a buffer is full.  Lanes with ok = false have no ray.
// Called by all lanes with one scene.
template <bool STATS, int BW>
CCS_DEV int beam_walk(const DevScene &sc, bool ok, const RayG<3> &r, float tmin, float tmax, int *stack,
                      uint32_t *leaves, int lane, unsigned long long &nodes)
{
    const unsigned FULL = 0xffffffffu;
    const float kInf = __int_as_float(0x7f800000);
    float on[3], of[3], imin[3], imax[3];   // origins to take for the near and the far plane; inverse directions
    bool pos[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        imin[k] = warp_min(ok ? r.inv[k] : kInf);
        imax[k] = warp_max(ok ? r.inv[k] : -kInf);
        const float omin = warp_min(ok ? r.org[k] : kInf), omax = warp_max(ok ? r.org[k] : -kInf);
        pos[k] = imin[k] > 0.0f;
        if (!(imin[k] > 0.0f || imax[k] < 0.0f) || !(omin > -kInf) || !(omax < kInf)) return -1;
        on[k] = pos[k] ? omax : omin;
        of[k] = pos[k] ? omin : omax;
    }
    const float t_lo = warp_min(ok ? tmin : kInf), t_hi = warp_max(ok ? tmax : -kInf);
    constexpr int kShift = BW == 4 ? 2 : 1;   // lanes of a node: its children
    const int c = lane & (BW - 1);
    int sp = 1, nl = 0;
    if (lane == 0) stack[0] = 0;
    __syncwarp();
    while (sp > 0) {
        const int take = min(sp, 32 >> kShift);
        sp -= take;
        bool keep = (lane >> kShift) < take;
        int child = kEmptyChild;
        if (keep) {
            const int node = stack[sp + (lane >> kShift)];
            float lo[3], hi[3];
            if constexpr (BW == 4) {   // [8 k + c] lo, [8 k + 4 + c] hi, [24 + c] the child word
                const float *nd = reinterpret_cast<const float *>(sc.nodes + (size_t)node * kNode4F4) + c;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    lo[k] = __ldg(nd + 8 * k);
                    hi[k] = __ldg(nd + 8 * k + 4);
                }
                child = __ldg(reinterpret_cast<const int *>(nd) + 24);
            } else {   // [4 k + 2 c] lo, hi, [12 + c] the child word
                const float2 *nd = reinterpret_cast<const float2 *>(sc.nodes + (size_t)node * kNodeF4) + c;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const float2 q = __ldg(nd + 2 * k);
                    lo[k] = q.x;
                    hi[k] = q.y;
                }
                child = __ldg(reinterpret_cast<const int *>(sc.nodes + (size_t)node * kNodeF4 + 3) + c);
            }
            if (STATS && c == 0) ++nodes;
            float tn[3], tf[3];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float a = __fsub_rn(pos[k] ? lo[k] : hi[k], on[k]), b = __fsub_rn(pos[k] ? hi[k] : lo[k], of[k]);
                tn[k] = __fmul_rn(a, a >= 0.0f ? imin[k] : imax[k]);
                tf[k] = __fmul_rn(b, b >= 0.0f ? imax[k] : imin[k]);
            }
            const float t0 = fmaxf(max3f(tn[0], tn[1], tn[2]), t_lo);
            const float t1 = fminf(__fmul_rn(min3f(tf[0], tf[1], tf[2]), kFarScale), t_hi);
            keep = t0 <= t1 && child != kEmptyChild;
        }
        const unsigned mi = __ballot_sync(FULL, keep && child >= 0), ml = __ballot_sync(FULL, keep && child < 0);
        if (sp + __popc(mi) > kBeamStack || nl + __popc(ml) > kBeamLeaves) return -1;
        const unsigned lt = (1u << lane) - 1u;
        if (keep && child >= 0) stack[sp + __popc(mi & lt)] = child;
        if (keep && child < 0) leaves[nl + __popc(ml & lt)] = (uint32_t)(~child);
        sp += __popc(mi);
        nl += __popc(ml);
        __syncwarp();
    }
    return nl;
}

template <bool STATS, int MODE, class Src, int BW>
__global__ void __launch_bounds__(kCandBlock) k_cand(Src src, PairBufs pb, uint32_t img_w, int L, uint32_t iter_cap,
                                              uint32_t *status, unsigned long long *counters, uint8_t *occluded)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const uint32_t n = src.total();
    const uint32_t i = cand_ray(blockIdx.x * blockDim.x + threadIdx.x, img_w);
    constexpr int C = kPairCands;
    const float kInf = __int_as_float(0x7f800000), leaf = __int_as_float((127 - L) << 23);
    float kt[C];
    uint32_t kp[C];
#pragma unroll
    for (int j = 0; j < C; ++j) {
        kt[j] = kInf;
        kp[j] = kMissId;
    }
    int cnt = 0;
    float t_evict = kInf;
    bool evicted = false, live = false, capped = false;
    uint32_t ray_scene = 0, ray_local = 0;
    typename Src::LaneScene lsc;
    unsigned long long nodes = 0, culled = 0;
    Grp G;
    G.c = 0;
    G.mask = FULL;
    G.l0 = G.l1 = G.l2 = lane;
    float ro[3] = {0.0f, 0.0f, 0.0f}, rd[3] = {0.0f, 0.0f, 0.0f}, tmin = 0.0f, tmax = 0.0f;
    __shared__ int beam[kCandBlock / 32 * kBeamWords];
    __shared__ uint2 leaf_buf[kLeafBuf * kCandBlock];
    RayG<3> r;
    bool ok = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) r.org[k] = r.inv[k] = 0.0f;
    if (i < n) {
        live = true;
        src.locate(i, lsc, ray_scene, ray_local);
        ok = load_world_ray(src.rays_of(ray_scene), ray_local, r.org, rd, r.inv, tmin, tmax) &&
             src.scene(lsc).n_nodes != 0;
        ro[0] = r.org[0];
        ro[1] = r.org[1];
        ro[2] = r.org[2];
    }
    // (a register less than a flag: with a NaN component root_box_near keeps every patch)
    if (!cullable(rd)) rd[0] = __int_as_float(0x7fffffff);
    const unsigned rays = __ballot_sync(FULL, ok);
    if (rays != 0u) {
        // one walk for the warp, when its rays make a beam (of one scene)
        int nl = -1;
        int *stack = beam + (threadIdx.x >> 5) * kBeamWords;
        uint32_t *leaves = reinterpret_cast<uint32_t *>(stack + kBeamStack);
        typename Src::LaneScene wsc = lsc;
        share_scene<Src>(wsc, __ffs(rays) - 1);
        if (iter_cap >= kBeamMinCap && __all_sync(FULL, !ok || same_scene<Src>(lsc, wsc)))
            nl = beam_walk<STATS, BW>(src.scene(wsc), ok, r, tmin, tmax, stack, leaves, lane, nodes);
        const DevScene &sc = src.scene(lsc);
        if (nl >= 0) {
#pragma unroll 1
            for (int q = 0; q < nl; ++q) {
                const uint32_t p = leaves[q];
                if (!ok) continue;
                const float4 blo = __ldg(sc.leaf_box + 2 * (size_t)p), bhi = __ldg(sc.leaf_box + 2 * (size_t)p + 1);
                const float lo[3] = {blo.x, blo.y, blo.z}, hi[3] = {bhi.x, bhi.y, bhi.z};
                float t0, t1;
                slab<3>(r, lo, hi, tmin, tmax, G, t0, t1);
                if (t0 <= t1) list_patch<STATS>(sc, p, t0, ro, rd, tmin, leaf, kt, kp, cnt, t_evict, evicted, culled, G);
            }
        } else if (ok) {
            uint32_t it = iter_cap;
            capped = !walk_buffered<STATS, BW>(sc, r, ro, rd, tmin, tmax, leaf, it, kt, kp, cnt, t_evict, evicted, nodes,
                                               culled, leaf_buf + threadIdx.x, kCandBlock, G);
        }
    }
    // the task: the candidates in list order in one run of the buffer; its cost class
    const bool has = live && !capped && cnt > 0;
    int key = -1;
    if (has) {
        const DevScene &sc = src.scene(lsc);
        int ng = 0;
#pragma unroll
        for (int j = 0; j < C; ++j)
            if (j < cnt && __ldg(sc.types + kp[j]) != 0) ++ng;
        // rays with a Gregory candidate first: their pairs then share warps, so fewer warp iterations pay
        // for the bound of Algorithm 2 with a single Gregory lane; the others by their number of candidates
        key = ng > 0 ? kCostClasses - 1 : min(kCostClasses - 2, cnt);
    }
    const uint32_t want = has ? (uint32_t)cnt : 0u;
    const unsigned lt = (1u << lane) - 1u;
    if (has) {
        const size_t off = (size_t)i * C;
        uint2 *dst = pb.cand + off;
#pragma unroll
        for (int j = 0; j < C; ++j)
            if (j < cnt) dst[j] = make_uint2(kp[j], __float_as_uint(kt[j]));
        uint4 *tk = pb.task + 4 * (size_t)i;
        if (isnan(rd[0])) rd[0] = __ldg(src.rays_of(ray_scene).dx + ray_local);
        tk[0] = make_uint4(i, (uint32_t)off, (uint32_t)cnt | ((uint32_t)key << 8) | (evicted ? kTaskEvicted : 0u),
                           __float_as_uint(t_evict));
        tk[1] = make_uint4(kp[0], __float_as_uint(kt[0]), __float_as_uint(tmin), __float_as_uint(tmax));
        tk[2] = make_uint4(__float_as_uint(ro[0]), __float_as_uint(ro[1]), __float_as_uint(ro[2]), __float_as_uint(rd[0]));
        tk[3] = make_uint4(__float_as_uint(rd[1]), __float_as_uint(rd[2]), 0u, 0u);
    }
    // the task's place in the list of its class
    const int hkey = has ? key : -1;
    const unsigned same = __match_any_sync(FULL, hkey);
    const int leader = __ffs(same) - 1;
    uint32_t cb = 0;
    if (has && lane == leader) cb = atomicAdd(pb.ctr + kCtrHist + key, (uint32_t)__popc(same));
    cb = __shfl_sync(FULL, cb, leader);
    if (has) pb.cls[(size_t)key * pb.n + cb + __popc(same & lt)] = i;
    if (live && !has) {
        if (capped) atomicOr(status, 1u);
        write_miss<MODE>(src, ray_scene, ray_local, occluded);
    }
    if (STATS) {   // BVH nodes; diagnostics in the schedule slots: candidates listed, rays that dropped some,
                   // candidates culled by their root box
        // (those culled where the boxes are world boxes in a slot of their own)
        const bool world = live && src.scene(lsc).local == 0;
        unsigned long long v[5] = {nodes, want, (unsigned long long)(has && evicted), world ? 0ull : culled,
                                   world ? culled : 0ull};
#pragma unroll
        for (int k = 0; k < 5; ++k)
            for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(FULL, v[k], o);
        if (lane == 0) {
            if (v[0]) atomicAdd(counters + 0, v[0]);
            if (v[1]) atomicAdd(counters + 8, v[1]);
            if (v[2]) atomicAdd(counters + 9, v[2]);
            if (v[3]) atomicAdd(counters + 17, v[3]);
            if (v[4]) atomicAdd(counters + 18, v[4]);
        }
    }
}

// The next candidates of a ray whose best hit may lie among those the candidate pass dropped: a walk of the
// BVH by one lane for the kPairCands smallest keys above (lb_t, lb_p), the last listed, written to the ray's
// candidate places.  The ray comes from the lane's task slot in shared memory (rs, strided).  Rare: rays
// with more candidates than the list holds, whose best hit is not before the first dropped one.
struct MoreCands {
    int cnt;          // candidates written (0: none left)
    float t_evict;    // smallest entry distance this walk dropped
    bool evicted, capped;
};
template <int BW>
__device__ __forceinline__ MoreCands collect_more(const DevScene sc, const float *rs, int stride, float leaf, float lb_t,
                                               uint32_t lb_p, uint32_t iter_cap, uint2 *dst)
{
    constexpr int C = kPairCands;
    RayG<3> r;
    float ro[3], rd[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        ro[k] = r.org[k] = rs[k * stride];
        r.inv[k] = rs[(3 + k) * stride];
        rd[k] = rs[(9 + k) * stride];
    }
    if (!cullable(rd)) rd[0] = __int_as_float(0x7fffffff);
    float kt[C];
    uint32_t kp[C];
#pragma unroll
    for (int j = 0; j < C; ++j) {
        kt[j] = __int_as_float(0x7f800000);
        kp[j] = kMissId;
    }
    MoreCands out;
    out.cnt = 0;
    out.t_evict = __int_as_float(0x7f800000);
    out.evicted = false;
    Grp G;
    G.c = 0;
    G.mask = 0xffffffffu;
    G.l0 = G.l1 = G.l2 = threadIdx.x & 31;
    uint32_t it = iter_cap;
    out.capped = !walk_candidates<BW>(sc, r, ro, rd, rs[6 * stride], rs[7 * stride], leaf, lb_t, lb_p, it, kt, kp, out.cnt,
                                      out.t_evict, out.evicted, G);
    if (!out.capped)
        for (int j = 0; j < out.cnt; ++j) dst[j] = make_uint2(kp[j], __float_as_uint(kt[j]));
    return out;
}

// ------------------------------------------------------------------------------------------------
// Pass 3: Algorithm 3 over (ray, patch) pairs, one pair per lane.
// ------------------------------------------------------------------------------------------------
template <bool STATS, int K, int MODE, class Src>
__global__ void __launch_bounds__(128, 3) k_pairs(Src src, PairBufs pb, int L, uint32_t refill, uint32_t iter_cap,
                                                  uint32_t *status, unsigned long long *counters, uint8_t *occluded)
{
    extern __shared__ __align__(16) float smem[];
    const int stride = blockDim.x;
    Scratch scr;
    scr.stride = stride;
    scr.cstride = cache_floats(K, 3);
    scr.cache = smem + threadIdx.x * scr.cstride;
    scr.tag = reinterpret_cast<int *>(scr.cache + 48 * K);
    scr.sib = reinterpret_cast<float2 *>(smem + cache_floats(K, 3) * stride) + threadIdx.x;
    scr.node = nullptr;
    float *rs = smem + scratch_floats(L, K, 3) * stride + threadIdx.x;   // [k * stride], k < kRaySlotFloats
    // mailboxes, helper counts and cap flags of the block's threads (indexed by thread)
    unsigned long long *mbox =
        reinterpret_cast<unsigned long long *>(smem + (scratch_floats(L, K, 3) + kRaySlotFloats) * stride);
    int *hcount = reinterpret_cast<int *>(mbox + stride);
    int *hcap = hcount + stride;
    const int wbase = threadIdx.x & ~31;
    mbox[threadIdx.x] = ~0ull;
    hcount[threadIdx.x] = 0;
    hcap[threadIdx.x] = 0;
    // the queue hands out the tasks class by class, costliest first: cstart[c] = first place of class c
    __shared__ uint32_t cstart[kCostClasses + 1], share[2];
    if (threadIdx.x < kCostClasses) {
        uint32_t a = 0;
        for (int c = kCostClasses - 1; c > (int)threadIdx.x; --c) a += pb.ctr[kCtrHist + c];
        cstart[threadIdx.x] = a;
        if (threadIdx.x == 0) {
            const uint32_t all = a + pb.ctr[kCtrHist], warps = gridDim.x * (blockDim.x >> 5);
            cstart[kCostClasses] = all;
            // A refill takes at most share[0] tasks, so that a short queue is spread over all warps, whose other lanes
            // help (64 x 64 image: 128 -> 90 us).  Without local frames the first shares of all warps, the costliest
            // tasks, are dealt out like cards, every share[1]-th task to one warp: neighbours in the list are
            // neighbours on the surface, grazing rays among them many times longer than the others, and one warp would
            // hold 32 of them (1283 x 717 image of 1,536 patches 625 -> 477 us).  With local frames no ray is that long,
            // and what counts is that the rays of a warp share patches (1080p image 422 us, dealt out 443).
            share[0] = min(32u, max(1u, (all + warps - 1u) / warps));
            share[1] = src.world_boxes() ? min(warps, all / share[0]) : 0u;
        }
    }
    __syncthreads();
    Counters cnt;
#pragma unroll
    for (int k = 0; k < kNumSumCounters; ++k) cnt.v[k] = 0;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    Grp G;
    G.c = 0;
    G.mask = FULL;
    G.l0 = G.l1 = G.l2 = lane;
    const float kInf = __int_as_float(0x7f800000);
    const float cellw = __int_as_float((127 - L) << 23);
    uint32_t *queue = pb.ctr + kCtrQueue;
    if (STATS && lane == 0) atomicMax(counters + 20, ~global_ns());   // first warp start

    // levels of Gregory pairs in the table: one scene's are the same for every lane
    int tab_d = 0;
    if constexpr (!std::is_same<Src, BatchSource>::value) tab_d = src.sc.n_nodes ? table_levels(src.sc, L) : 0;
    auto tab_levels = [&](const typename Src::LaneScene &l) {
        if constexpr (std::is_same<Src, BatchSource>::value) return table_levels(src.scene(l), L);
        else return tab_d;
    };
    // the lane's ray (task)
    bool has_task = false, exhausted = false, evicted = false;
    uint32_t ray = 0, cur = 0, ray_scene = 0, ray_local = 0, iters = 0;
    uint2 nxt = make_uint2(0u, 0u);   // the ray's candidate at cur, loaded ahead
    typename Src::LaneScene lsc;
    Best best;
    best.t = 0.0f;
    best.pid = best.cell = kMissId;
    best.lvl = 0;
    // the lane's pair
    bool in_pair = false, want_root = false, start = false, gpend = false, greg = false;
    bool helper = false, waiting = false;   // a subtree of lane `owner`'s pair; waiting for helpers
    int owner = lane;
    uint32_t pid = 0, start_pid = 0, path = 0, trail = 0;
    RayG<3> pr;
    float tau = 0.0f, c0 = 0.0f, c1 = 0.0f, te = 0.0f;   // intervals are distances from the anchored origin
    int level = 0, rd_target = -1, ctop = 0, cvalid = 0;
    float g[48];

    for (;;) {
        // (1) a lane whose pair has ended takes its ray's next candidate (collecting more when dropped
        //     candidates may still hold the answer), or writes the ray's answer; idle lanes take new rays
        //     from the queue, then their first candidate
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            if (has_task && !in_pair && !start) {
                if (cur < __float_as_uint(rs[13 * stride]) && __uint_as_float(nxt.y) <= best.t) {
                    start = true;
                    start_pid = nxt.x;
                    ++cur;
                } else {   // entries are sorted: the rest enter later still
                    // the answer may lie among the candidates the walk dropped (entries from t_evict on): this
                    // lane collects the next ones, after the last listed, by a walk of its own
                    bool finish = true;
                    if (evicted && (MODE == kModeAnyHit ? best.pid == kMissId : !(best.t < rs[8 * stride]))) {
                        const uint2 last = pb.cand[__float_as_uint(rs[13 * stride]) - 1];
                        const uint32_t cbase = __float_as_uint(rs[12 * stride]);
                        const DevScene &sc = src.scene(lsc);
                        const MoreCands mc =
                            sc.width == 4
                                ? collect_more<4>(sc, rs, stride, cellw, __uint_as_float(last.y), last.x, iter_cap, pb.cand + cbase)
                                : collect_more<2>(sc, rs, stride, cellw, __uint_as_float(last.y), last.x, iter_cap, pb.cand + cbase);
                        if (STATS) cnt.v[10]++;
                        evicted = mc.evicted;
                        if (mc.capped) {   // iteration cap of the walk: a miss, status latched
                            finish = false;
                            has_task = false;
                            atomicOr(status, 1u);
                            write_miss<MODE>(src, ray_scene, ray_local, occluded);
                        } else if (mc.cnt > 0) {
                            finish = false;
                            cur = cbase;
                            rs[13 * stride] = __uint_as_float(cbase + (uint32_t)mc.cnt);
                            nxt = pb.cand[cbase];
                            rs[8 * stride] = mc.t_evict;
                        }
                    }
                    if (finish) {   // the ray's answer
                        has_task = false;
                        if (MODE == kModeAnyHit) {
                            occluded[ray_local] = best.pid != kMissId ? 1 : 0;
                        } else {
                            const DevHits &hh = src.hits_of(ray_scene);
                            const uint32_t j = ray_local;
                            if (best.pid != kMissId) {
                                const uint32_t cu = best.cell & ((1u << L) - 1u), cv = best.cell >> L;
                                hh.t[j] = best.t;
                                hh.u[j] = ((float)cu + 0.5f) * cellw;
                                hh.v[j] = ((float)cv + 0.5f) * cellw;
                                hh.pid[j] = best.pid;
                            } else {
                                hh.t[j] = kInf;
                                hh.u[j] = 0.0f;
                                hh.v[j] = 0.0f;
                                hh.pid[j] = kMissId;
                            }
                        }
                    }
                }
            }
            if (pass == 1 || exhausted) break;
            const unsigned idle = __ballot_sync(FULL, !has_task);
            if (idle == 0u || ((uint32_t)__popc(idle) < refill && idle != FULL)) break;
            uint32_t qb = 0;
            const uint32_t take = min(share[0], (uint32_t)__popc(idle));
            if (lane == 0) qb = atomicAdd(queue, take);
            qb = __shfl_sync(FULL, qb, 0);
            if (qb + take >= cstart[kCostClasses]) {
                exhausted = true;
                if (STATS && lane == 0) atomicMax(counters + 21, ~global_ns());   // queue found empty
            }
            const uint32_t rank = (uint32_t)__popc(idle & lt);
            uint32_t k = qb + rank;
            if (!has_task && rank < take && k < cstart[kCostClasses]) {
                if (k < share[0] * share[1]) k = k % share[0] * share[1] + k / share[0];
                int c = kCostClasses - 1;
                while (c > 0 && k >= cstart[c - 1]) --c;
                const uint4 *tp = pb.task + 4 * (size_t)__ldg(pb.cls + (size_t)c * pb.n + (k - cstart[c]));
                const uint4 w0 = tp[0], w1 = tp[1], w2 = tp[2], w3 = tp[3];
                has_task = true;
                ray = w0.x;
                cur = w0.y;
                rs[12 * stride] = __uint_as_float(w0.y);
                rs[13 * stride] = __uint_as_float(w0.y + (w0.z & 255u));
                evicted = (w0.z & kTaskEvicted) != 0u;
                nxt = make_uint2(w1.x, w1.y);
                rs[0 * stride] = __uint_as_float(w2.x);
                rs[1 * stride] = __uint_as_float(w2.y);
                rs[2 * stride] = __uint_as_float(w2.z);
                rs[3 * stride] = safe_inv(__uint_as_float(w2.w));
                rs[4 * stride] = safe_inv(__uint_as_float(w3.x));
                rs[5 * stride] = safe_inv(__uint_as_float(w3.y));
                rs[6 * stride] = __uint_as_float(w1.z);
                rs[7 * stride] = __uint_as_float(w1.w);
                rs[8 * stride] = __uint_as_float(w0.w);
                rs[9 * stride] = __uint_as_float(w2.w);
                rs[10 * stride] = __uint_as_float(w3.x);
                rs[11 * stride] = __uint_as_float(w3.y);
                src.locate(ray, lsc, ray_scene, ray_local);
                iters = iter_cap;
                best.t = __uint_as_float(w1.w);
                best.pid = best.cell = kMissId;
            }
        }
        // (2) the lanes that start a pair: the next candidate ahead, root interval, the ray in the patch
        //     frame, and (Bezier) the root grid
        if (start) {
            start = false;
            if (cur < __float_as_uint(rs[13 * stride])) nxt = pb.cand[cur];
            const DevScene &sc = src.scene(lsc);
            pid = start_pid;
            const float4 *rec = rec_of(sc, pid);
            const float4 an = __ldg(rec + 15);
            in_pair = true;
            greg = an.w != 0.0f;
            if (STATS) cnt.v[7]++;
            RayG<3> wr;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                wr.org[k] = rs[k * stride];
                wr.inv[k] = rs[(3 + k) * stride];
            }
            const float tmin = rs[6 * stride];
            {   // the root interval: the slab of the patch box from tmin (as k_intersect computes it)
                const float4 blo = __ldg(sc.leaf_box + 2 * (size_t)pid), bhi = __ldg(sc.leaf_box + 2 * (size_t)pid + 1);
                const float lo[3] = {blo.x, blo.y, blo.z}, hi[3] = {bhi.x, bhi.y, bhi.z};
                slab<3>(wr, lo, hi, tmin, kInf, G, c0, c1);
            }
            {
                const float dw[3] = {rs[9 * stride], rs[10 * stride], rs[11 * stride]};
                te = c0;
                anchored_ray<3>(rec, an, sc.local != 0, wr.org, dw, wr.inv, c0, G, pr);
                c1 = __fsub_rn(c1, c0);
                c0 = 0.0f;
            }
            tau = 0.0f;
            if (sc.local) {   // box extension (Sec. 3.4)
                float o3[3];
#pragma unroll
                for (int c = 0; c < 3; ++c) o3[c] = wr.org[c] - pick(c, an.x, an.y, an.z);
                tau = pair_tau(o3);
            }
            level = 0;
            rd_target = -1;
            path = trail = 0u;
            ctop = cvalid = 0;
            gpend = greg;
            want_root = !greg;
        }
        if (want_root) {   // a Bezier pair's start or a re-descent: the root grid
            want_root = false;
            load_grid<3>(rec_of(src.scene(lsc), pid), G, g);
        }
        if (STATS) {   // schedule of this warp iteration, in lanes (slots 12..16)
            const unsigned ks = __ballot_sync(FULL, in_pair && !waiting), kh = __ballot_sync(FULL, helper);
            const unsigned kw = __ballot_sync(FULL, waiting), ki = __ballot_sync(FULL, !in_pair && !has_task);
            if (lane == 0) {
                cnt.v[12] += 1;
                cnt.v[13] += __popc(ks);
                cnt.v[14] += __popc(kh);
                cnt.v[15] += __popc(kw);
                cnt.v[16] += __popc(ki);
            }
        }
        // (3) subdivision steps of every lane's pair: the iteration cap first
        if (in_pair && !waiting && iters == 0) {
            if (helper) {   // iteration cap in a subtree: the owner's ray becomes a capped miss
                atomicOr(status, 1u);
                hcap[wbase + owner] = 1;
                __threadfence_block();
                atomicSub(hcount + wbase + owner, 1);
                helper = false;
                in_pair = false;
            } else if (hcount[threadIdx.x] > 0) {   // wait for the subtrees, then the cap
                hcap[threadIdx.x] = 1;
                waiting = true;
            } else {   // iteration cap: a miss, status latched
                has_task = false;
                in_pair = false;
                atomicOr(status, 1u);
                if (MODE == kModeAnyHit) {
                    occluded[ray_local] = 0;
                } else {
                    const DevHits &hh = src.hits_of(ray_scene);
                    hh.t[ray_local] = kInf;
                    hh.u[ray_local] = 0.0f;
                    hh.v[ray_local] = 0.0f;
                    hh.pid[ray_local] = kMissId;
                }
            }
        }
        // up to kStepsPerIter steps (Algorithm 3's loop body) per warp iteration: after the first, the lanes
        // whose pair keeps descending (no leaf, no backtrack, no Gregory bound due) step again, so that the
        // divergent rest of the iteration is paid once for more steps
        bool stepping = in_pair && !waiting && iters > 0, back = false;
#pragma unroll 1
        for (int pass = 0; pass < kStepsPerIter; ++pass) {
            if (pass > 0 && !__any_sync(FULL, stepping)) break;
            if (stepping) {
                --iters;
                const bool redesc = rd_target >= 0;
                int slot = -1;
                StepOut so;
                if (gpend && level < tab_levels(lsc)) {
                    // a Gregory node in the scene's table: the lane goes down through the table at once, a load
                    // and two slab tests per level, while the others split
                    const float4 *nodes = table_nodes(src.scene(lsc), pid);
                    const int last = tab_levels(lsc) - 1;
                    uint32_t h = table_index(level, path);
                    // a step takes less time than a load: each step asks for the lines of the nodes two levels
                    // down (four nodes, two lines), the first one also for those of one level down
                    if (level < last) prefetch_l1(nodes + 8 * (size_t)h);
                    for (;;) {
                        if (level + 1 < last) {
                            prefetch_l1(nodes + 16 * (size_t)h);
                            prefetch_l1(nodes + 16 * (size_t)h + 8);
                        }
                        if (STATS) cnt.v[2]++;
                        so = table_step(nodes + 4 * (size_t)h, pr, c0, c1, te, best.t, true,
                                        true, -1, G, tau);
                        if (level == last || iters == 0 || !(so.hitL || so.hitR)) break;
                        --iters;
                        const uint32_t bit = 1u << level;
                        if (so.hitL && so.hitR) {
                            trail |= bit;
                            scr.sib[level * stride] = so.goR ? make_float2(so.l0, so.l1) : make_float2(so.r0, so.r1);
                        }
                        path = so.goR ? (path | bit) : path;
                        c0 = so.goR ? so.r0 : so.l0;
                        c1 = so.goR ? so.r1 : so.l1;
                        h = 2 * h + (so.goR ? 1u : 0u);
                        ++level;
                    }
                } else {
                    float d[3] = {0.0f, 0.0f, 0.0f};   // displacement of the upper bound (Gregory)
                    if (gpend) {   // Algorithm 2 with the crop of Algorithm 1 for the Gregory node (path, level)
                        float u0, u1, v0, v1;
                        node_domain(path, level, L, u0, u1, v0, v1);
                        gregory_node<3>(rec_of(src.scene(lsc), pid), u0, u1, v0, v1, level, G, g, d);
                    }
                    const bool leafkids = !redesc && level + 1 == 2 * L;
                    const int force = redesc ? (int)((path >> level) & 1u) : -1;
                    slot = (!redesc && !leafkids && K > 0 && !greg) ? (ctop % (K > 0 ? K : 1)) : -1;
                    if (STATS && !redesc) cnt.v[greg ? 2 : 1]++;
                    so = split_step<K, 3>(g, pr, d, c0, c1, te, best.t, redesc || (!greg && !leafkids), scr, slot, true,
                                          true, force, G, tau);
                }
                gpend = false;
                const bool leafkids = !redesc && level + 1 == 2 * L;
                if (redesc) {
                    if (++level == rd_target) rd_target = -1;
                } else if (so.hitL || so.hitR) {
                    const uint32_t bit = 1u << level;
                    if (leafkids) {   // both children are leaves: record them here (key order, A14/A15)
                        uint32_t cu, cv;
                        if (so.hitL) {
                            path_cells(path, L, cu, cv);
                            const uint32_t cell = (cv << L) | cu;
                            const float tk = __fadd_rn(te, so.l0);
                            if (key_less(tk, pid, cell, best)) {
                                best.t = tk;
                                best.pid = pid;
                                best.cell = cell;
                            }
                        }
                        if (so.hitR) {
                            path_cells(path | bit, L, cu, cv);
                            const uint32_t cell = (cv << L) | cu;
                            const float tk = __fadd_rn(te, so.r0);
                            if (key_less(tk, pid, cell, best)) {
                                best.t = tk;
                                best.pid = pid;
                                best.cell = cell;
                            }
                        }
                        if (STATS) cnt.v[3] += (so.hitL ? 1 : 0) + (so.hitR ? 1 : 0);
                        back = true;
                    } else {
                        if (so.hitL && so.hitR) {
                            trail |= bit;
                            scr.sib[level * stride] = so.goR ? make_float2(so.l0, so.l1) : make_float2(so.r0, so.r1);
                            if (K > 0 && slot >= 0) {
                                scr.tag[slot] = level;
                                ++ctop;
                                cvalid = cvalid < K ? cvalid + 1 : K;
                            }
                        }
                        path = so.goR ? (path | bit) : path;
                        c0 = so.goR ? so.r0 : so.l0;
                        c1 = so.goR ? so.r1 : so.l1;
                        ++level;
                        gpend = greg;
                    }
                } else {
                    back = true;
                }
                stepping = !back && !gpend && iters > 0;
            }
        }
        if (back) {   // the deepest pending sibling that may still hold a closer leaf, or the pair ends
            bool found = false;
            if (!(MODE == kModeAnyHit && best.pid != kMissId)) {
                while (trail != 0u) {
                    const int l = 31 - __clz(trail);
                    const uint32_t bit = 1u << l;
                    trail ^= bit;
                    bool cached = false;
                    int cslot = 0;
                    if (K > 0 && !greg && cvalid > 0) {
                        cslot = (ctop - 1) % (K > 0 ? K : 1);
                        if (scr.tag[cslot] == l) {
                            cached = true;
                            --ctop;
                            --cvalid;
                        }
                    }
                    const float2 sb = scr.sib[l * stride];
                    if (__fadd_rn(te, sb.x) > best.t) {
                        if (STATS) cnt.v[6]++;
                        continue;
                    }
                    path = (path & (bit - 1u)) | (~path & bit);
                    c0 = sb.x;
                    c1 = sb.y;
                    if (STATS) cnt.v[4]++;
                    if (greg) {
                        level = l + 1;
                        gpend = true;
                    } else if (cached) {
                        level = l + 1;
                        load_cached<3>(scr.cache + cslot * 48, g);
                    } else {
                        if (STATS) cnt.v[5] += l + 1;
                        level = 0;
                        rd_target = l + 1;
                        want_root = true;
                    }
                    found = true;
                    break;
                }
            } else {
                cur = __float_as_uint(rs[13 * stride]);   // any hit: the ray is answered
            }
            if (!found) {
                if (helper) {   // the subtree is searched: its best leaf to the owner's mailbox
                    if (best.pid == pid)
                        atomicMin(mbox + wbase + owner, ((unsigned long long)ord_bits(best.t) << 32) | best.cell);
                    __threadfence_block();
                    atomicSub(hcount + wbase + owner, 1);
                    helper = false;
                    in_pair = false;
                } else {
                    waiting = true;   // merged when every subtree handed out is searched
                }
            }
        }
        // a lane whose search has ended takes the best leaf of the subtrees it handed out, once every one of
        // them is searched (until then it waits)
        __syncwarp();
        if (waiting && hcount[threadIdx.x] == 0) {
            __threadfence_block();
            const unsigned long long mk = mbox[threadIdx.x];
            if (mk != ~0ull) {
                const float mt = unord_bits((uint32_t)(mk >> 32));
                const uint32_t mc = (uint32_t)mk;
                if (key_less(mt, pid, mc, best)) {
                    best.t = mt;
                    best.pid = pid;
                    best.cell = mc;
                }
                mbox[threadIdx.x] = ~0ull;
            }
            waiting = false;
            in_pair = false;
            if (MODE == kModeAnyHit && best.pid != kMissId) cur = __float_as_uint(rs[13 * stride]);   // answered
            if (hcap[threadIdx.x]) {   // a subtree reached the iteration cap: answered as a capped ray
                hcap[threadIdx.x] = 0;
                iters = 0;
                in_pair = true;
            }
        }
        // (4) once the queue is empty, idle lanes take a pending subtree of a busy lane of the warp: the
        //     deepest one when its grid is in the busy lane's sibling cache or the patch is a Gregory patch
        //     (no re-descent), else the shallowest one of at least kMinDonateLevels levels (re-descended); the
        //     key of a pair's best leaf is the minimum over its subtrees.  (In the any-hit query too: a ray
        //     that meets nothing searches as much as a closest-hit ray; 300 k shadow rays on 1,632 patches 350 ->
        //     266 us.)
        if (exhausted) {
            const bool idle_l = !has_task && !in_pair;
            const int lmin = trail != 0u ? __ffs(trail) - 1 : 2 * L;
            const int ldeep = trail != 0u ? 31 - __clz(trail) : 2 * L;
            int cslot = -1;
            if (K > 0 && !greg && cvalid > 0 && trail != 0u) {
                const int c = (ctop - 1) % (K > 0 ? K : 1);
                if (scr.tag[c] == ldeep) cslot = c;
            }
            const bool deep = trail != 0u && (greg || cslot >= 0);
            const int lgive = deep ? ldeep : lmin;
            const bool can_give = in_pair && !waiting && (deep || 2 * L - (lmin + 1) >= kMinDonateLevels);
            const unsigned T = __ballot_sync(FULL, idle_l), D = __ballot_sync(FULL, can_give);
            if (T != 0u && D != 0u) {
                const int m = min(__popc(T), __popc(D));
                int from = lane;
                if (idle_l && __popc(T & lt) < m) from = (int)__fns(D, 0, __popc(T & lt) + 1);
                const bool gives = can_give && __popc(D & lt) < m;
                uint32_t sp = 0u;
                float sx = 0.0f, sy = 0.0f;
                int gslot = -1;   // the donor's cache slot holding the subtree root's grid
                if (gives) {   // the sibling's path and interval, as a backtrack to it would set them
                    const uint32_t bit = 1u << lgive;
                    sp = (path & (bit - 1u)) | (~path & bit);
                    const float2 sb = scr.sib[lgive * stride];
                    sx = sb.x;
                    sy = sb.y;
                    trail ^= bit;
                    if (deep && cslot >= 0) {
                        gslot = cslot;
                        --ctop;
                        --cvalid;
                    }
                }
                const int x_gslot = __shfl_sync(FULL, gslot, from);
                const uint32_t x_pid = __shfl_sync(FULL, pid, from);
                const int x_greg = __shfl_sync(FULL, greg ? 1 : 0, from);
                float x_pr[6];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    x_pr[k] = __shfl_sync(FULL, pr.org[k], from);
                    x_pr[3 + k] = __shfl_sync(FULL, pr.inv[k], from);
                }
                const float x_tau = __shfl_sync(FULL, tau, from);
                const float x_te = __shfl_sync(FULL, te, from);
                const float x_bt = __shfl_sync(FULL, best.t, from);
                const uint32_t x_bp = __shfl_sync(FULL, best.pid, from);
                const uint32_t x_bc = __shfl_sync(FULL, best.cell, from);
                const uint32_t x_sp = __shfl_sync(FULL, sp, from);
                const int x_sl = __shfl_sync(FULL, lgive, from);
                const float x_sx = __shfl_sync(FULL, sx, from);
                const float x_sy = __shfl_sync(FULL, sy, from);
                const int x_owner = __shfl_sync(FULL, helper ? owner : lane, from);
                share_scene<Src>(lsc, from);
                if (idle_l && from != lane) {   // a helper on the subtree below the sibling
                    helper = true;
                    in_pair = true;
                    owner = x_owner;
                    pid = x_pid;
                    greg = x_greg != 0;
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        pr.org[k] = x_pr[k];
                        pr.inv[k] = x_pr[3 + k];
                    }
                    tau = x_tau;
                    te = x_te;
                    best.t = x_bt;
                    best.pid = x_bp;
                    best.cell = x_bc;
                    path = x_sp;
                    trail = 0u;
                    c0 = x_sx;
                    c1 = x_sy;
                    ctop = cvalid = 0;
                    iters = iter_cap;
                    if (greg) {
                        level = x_sl + 1;
                        rd_target = -1;
                        gpend = true;
                    } else if (x_gslot >= 0) {   // the grid from the donor's cache slot
                        level = x_sl + 1;
                        rd_target = -1;
                        gpend = false;
                        load_cached<3>(scr.cache + (from - lane) * scr.cstride + x_gslot * 48, g);
                    } else {
                        level = 0;
                        rd_target = x_sl + 1;
                        gpend = false;
                        want_root = true;
                    }
                    atomicAdd(hcount + wbase + owner, 1);
                    if (STATS) cnt.v[11]++;
                }
            }
            __syncwarp();
        }
        if (exhausted && !__any_sync(FULL, has_task)) break;
    }
    if (STATS) {
#pragma unroll
        for (int k = 0; k < kNumSumCounters; ++k) {
            unsigned long long v = cnt.v[k];
            for (int o2 = 16; o2 > 0; o2 >>= 1) v += __shfl_xor_sync(FULL, v, o2);
            if (lane == 0 && v) atomicAdd(counters + k, v);
        }
        if (lane == 0) atomicMax(counters + 22, global_ns());   // last warp exit
    }
}

}  // namespace ccs
