// APRIL intermediate filter on sm_103a: context, device upload, and the
// filter kernels behind april_filter_pairs.
//
// Every kernel computes, per candidate pair (r, s), Algorithm 2 of the paper
// (Sec. 4.2): IntervalJoin(A(r), A(s)); if it finds no overlap the pair is a
// true negative; else IntervalJoin(A(r), F(s)) or IntervalJoin(F(r), A(s))
// finding an overlap makes it a true hit; else it is inconclusive.
//
// Interval convention: [st, end) with end stored mod 2^32; all comparisons
// use last = end - 1 (uint32), so an interval that reaches cell 2^32-1 works.
//   X_i overlaps Y_j   <=>  X_i.st <= Y_j.last  and  Y_j.st <= X_i.last
//   merge step         :    advance X if X_i.last <= Y_j.last, else Y.
//
// Parallel joins.  "Does any interval of X overlap one of Y" has one answer
// however the merge is split.  The sequential merge visits the states
// (i, j) of the merge path of X and Y ordered by `last` (ties: X first) and
// at each state tests X_i against Y_j; the element emitted at that state is
// the smaller of the two.  So the set of tests the merge performs is
//   { (X_i, Y_rank_Y(X_i)) }  u  { (X_rank_X(Y_j), Y_j) }
// where rank_Y(X_i) = #{ j : Y_j.last < X_i.last } and
//       rank_X(Y_j) = #{ i : X_i.last <= Y_j.last }.
// A group of lanes loads a window of both lists, computes these ranks inside
// the window by binary search over registers (shuffles), runs the tests of
// the first W merge positions at once, and advances by the number of X and Y
// elements those W positions consumed.  The default shape of the batched
// filter gives each pair to one lane instead (K2, join_device.cuh).

#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cstdio>
#include <mutex>
#include <string>
#include <vector>

#include "april_internal.h"
#include "join_device.cuh"

using namespace april_dev;

namespace {

// status bits in the context's device status block
constexpr uint32_t ST_BAD_ID = 1u;
constexpr uint32_t ST_TIMEOUT = 2u;
static_assert(kMbarSpinLimit == APRIL_WAIT_LIMIT_DEFAULT, "the documented default wait limit");

constexpr uint32_t kBlock = 256;                 // threads per CTA for K1/K3
constexpr uint32_t kWarpsPerBlock = kBlock / 32;
constexpr uint32_t kWarpWMax = 256;              // largest warp window per list
constexpr uint32_t kCtaWMax = 2048;              // largest CTA window per list
// cta_threshold value meaning "no long pairs": every pair goes to the lane
// groups, whatever its length, and the binning kernel is not launched
constexpr uint32_t kNoLongPairs = 0xffffffffu;
// join_order value meaning AF, AA, FA: most pairs are true hits, which AF settles
constexpr uint32_t kJoinOrderAuto = 2;
static inline uint32_t join_order_of(uint32_t jo) { return jo == kJoinOrderAuto ? 0u : jo; }
constexpr uint32_t kWarpFirstWindow = 64;        // first window of a join in APRIL_MODE_WARP
constexpr uint32_t kWarpBuf = kWarpWMax + 2;     // staging buffer per list (odd start + rounding)
constexpr uint32_t kCtaBuf = kCtaWMax + 2;
// Compile-time knobs (defaults are the shipped configuration):
//   APRIL_MIN_BLOCKS  minimum resident CTAs per SM requested for k_persistent
//   APRIL_GROUP_PER   diagonals each lane walks per window in the group engine
//   APRIL_GENERAL_MIN_BLOCKS  minimum resident CTAs per SM requested for k_general
//   APRIL_STAGE2      1: a lane group's two windows are copied by two lanes (mbarrier count 2)
#ifdef APRIL_MIN_BLOCKS
#define APRIL_PERSISTENT_BOUNDS __launch_bounds__(256, APRIL_MIN_BLOCKS)
#else
// the lane-group instances over raw lists run five CTAs per SM (at most 51
// registers a thread: their warps wait on memory, more of them hide more);
// the others leave the register count to the compiler
#define APRIL_PERSISTENT_BOUNDS __launch_bounds__(256, (G < 32 && !SetsT::kPacked) ? 5 : 0)
#endif
#ifndef APRIL_STAGE2
#define APRIL_STAGE2 1
#endif
constexpr bool kStage2 = APRIL_STAGE2 != 0;  // lane groups stage their two windows from two lanes
#ifndef APRIL_GROUP_PER
#define APRIL_GROUP_PER 8
#endif
constexpr uint32_t kGroupPer = APRIL_GROUP_PER;
// intervals of shared staging per warp for kernels with whole-warp joins only
// (K1, K7): two windows of a warp, and a CTA's two windows across its warps
constexpr uint32_t kWarpShare = 2 * (kWarpWMax + 2);
constexpr uint32_t kSharedIv = kWarpsPerBlock * kWarpShare > 2 * kCtaBuf ? kWarpsPerBlock * kWarpShare : 2 * kCtaBuf;
static_assert(kWarpBuf % 2 == 0 && kCtaBuf % 2 == 0, "buffers must stay 16-byte aligned");

// scratch of the batched mode: counters, the list of long pairs, the routed
// entries of partitioned sets, then the queue of joins handed from the lane
// groups to whole warps (one uint4 {pair, step, i0, j0} each, room for a
// quarter of the pairs; when it is full a group finishes its join itself)
constexpr uint32_t C_BIG_COUNT = 0, C_BIG_HEAD = 1, C_CHUNK_HEAD = 2, C_ESC_COUNT = 3, C_ESC_HEAD = 4,
                   C_REST_COUNT = 5;
constexpr uint32_t C_LANE_HEAD = 8;  // the first pass's chunk counters, one per chunk of the host pipeline (up to 8)
static inline uint64_t esc_capacity(uint64_t n) { return (n + 3) / 4; }
constexpr uint32_t kMaxEscalateWindows = 64;
constexpr size_t kCounterBytes = 256;

__device__ __forceinline__ uint4 shfl4(const uint4 &v, uint32_t src) {
    return make_uint4(__shfl_sync(kFull, v.x, src), __shfl_sync(kFull, v.y, src), __shfl_sync(kFull, v.z, src),
                      __shfl_sync(kFull, v.w, src));
}

// Entry-level views of a set for the warp and CTA joins.  RawSets reads the
// interval lists; PackedSets reads the compressed lists of Sec. 5.1.
struct RawSets {
    static constexpr bool kPacked = false;
    DevSet s;
    using Desc = uint4;  // {a_off, a_len, f_off, f_len}
    __device__ __forceinline__ uint32_t n() const { return s.n; }
    __device__ __forceinline__ Desc load(uint32_t e) const { return __ldg(s.desc + e); }
    static __device__ __forceinline__ uint32_t a_len(const Desc &d) { return d.y; }
    static __device__ __forceinline__ Desc shfl(const Desc &d, uint32_t src) { return shfl4(d, src); }
    __device__ __forceinline__ RawList list(const Desc &d, bool f) const {
        const uint32_t off = f ? d.z : d.x;
        return RawList{s.iv + off, f ? d.w : d.y, s.posts + off / 16};
    }
};

struct PackedSets {
    static constexpr bool kPacked = true;
    const uint4 *pdesc;    // per entry {a_block, a_len, f_block, f_len}
    const uint2 *blocks;   // block table {anchor, gap_off64 | wide << 31}
    const uint8_t *gaps;
    uint32_t nent;
    using Desc = uint4;
    __device__ __forceinline__ uint32_t n() const { return nent; }
    __device__ __forceinline__ Desc load(uint32_t e) const { return __ldg(pdesc + e); }
    static __device__ __forceinline__ uint32_t a_len(const Desc &d) { return d.y; }
    static __device__ __forceinline__ Desc shfl(const Desc &d, uint32_t src) { return shfl4(d, src); }
    __device__ __forceinline__ PackedList list(const Desc &d, bool f) const {
        return f ? PackedList{blocks + d.z, gaps, d.w} : PackedList{blocks + d.x, gaps, d.y};
    }
};

// ------------------------------------------------------- K0: thread/pair
__global__ void __launch_bounds__(256) k_plain(DevSet R, DevSet S, const uint32_t *__restrict__ pr,
                                               const uint32_t *__restrict__ ps, uint64_t n,
                                               uint8_t *__restrict__ out, uint32_t *status) {
    for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
         k += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t r = __ldg(pr + k), s = __ldg(ps + k);
        if (r >= R.n || s >= S.n) {
            out[k] = APRIL_VERDICT_ERROR;
            atomicOr(status, ST_BAD_ID);
            continue;
        }
        const uint4 dr = __ldg(R.desc + r), ds = __ldg(S.desc + s);
        uint8_t v;
        if (!seq_join(R.iv + dr.x, dr.y, S.iv + ds.x, ds.y)) v = APRIL_TRUE_NEGATIVE;
        else if (seq_join(R.iv + dr.x, dr.y, S.iv + ds.z, ds.w)) v = APRIL_TRUE_HIT;
        else if (seq_join(R.iv + dr.z, dr.w, S.iv + ds.x, ds.y)) v = APRIL_TRUE_HIT;
        else v = APRIL_INCONCLUSIVE;
        out[k] = v;
    }
}

// Algorithm 2 for one pair by one warp: AA; if no overlap, a true negative;
// else AF, then FA.
// Shared-memory synchronisation state of a warp or CTA join: the mbarrier the
// window copies complete on, its phase bit, and a timeout flag.
struct JoinSync;

// The order of a pair's joins in the batched kernels (april_tune.join_order).
// The verdicts of Sec. 4.2 do not depend on it (F is a subset of A, so an AF
// or FA overlap implies an AA overlap).
//   order 0, AF AA FA: AF first settles most true hits in one join; a pair
//     without an AF overlap takes AA (none: true negative), then FA.
//   order 1, AA AF FA (Algorithm 2's): a true negative takes one join.
// Step s joins X = F(r) when s == 2 (else A(r)) with Y = F(s) when s is the
// AF step (else A(s)).  A join with an empty list has no overlap.
__device__ __forceinline__ bool step_x_f(uint32_t s, uint32_t jo) { return s == 2; }
__device__ __forceinline__ bool step_y_f(uint32_t s, uint32_t jo) { return s == (jo ? 1u : 0u); }
// The verdict after step s found `overlap` (>= 0), or -1 with s advanced.
__device__ __forceinline__ int step_outcome(uint32_t &s, bool overlap, uint32_t jo) {
    if (s == 2) return overlap ? APRIL_TRUE_HIT : APRIL_INCONCLUSIVE;
    const bool aa = (s == 0) == (jo != 0);  // this step is AA
    if (aa && !overlap) return APRIL_TRUE_NEGATIVE;
    if (!aa && overlap) return APRIL_TRUE_HIT;
    ++s;
    return -1;
}

struct JoinSync {
    uint32_t bar;
    uint32_t phase;
    bool timeout;
};

// With resume, the pair's join step st0 continues from merge position
// (ri, rj), where the lane groups left it (see k_long).
template <class SetsT>
__device__ __forceinline__ uint8_t warp_verdict(const SetsT &R, const SetsT &S, const typename SetsT::Desc &dr,
                                                const typename SetsT::Desc &ds, uint2 *xs, uint2 *ys, uint32_t lane,
                                                uint32_t w0, JoinSync &js, uint32_t jo, uint32_t st0 = 0,
                                                bool resume = false, uint32_t ri = 0, uint32_t rj = 0) {
    uint32_t st = st0;
    for (;;) {
        const bool ov = tile_join<WarpScope, 32, kWarpWMax>(R.list(dr, step_x_f(st, jo)), S.list(ds, step_y_f(st, jo)),
                                                            xs, ys, nullptr, lane, w0, js.bar, &js.phase, &js.timeout,
                                                            0, 0, resume, ri, rj);
        if (js.timeout) return APRIL_VERDICT_ERROR;
        resume = false;
        const int v = step_outcome(st, ov, jo);
        if (v >= 0) return (uint8_t)v;
    }
}

// The same for one pair by the whole CTA.
template <class SetsT>
__device__ __forceinline__ uint8_t cta_verdict(const SetsT &R, const SetsT &S, const typename SetsT::Desc &dr,
                                               const typename SetsT::Desc &ds, uint2 *xs, uint2 *ys, uint32_t *slot,
                                               uint32_t tid, uint32_t w0, JoinSync &js, uint32_t jo) {
    uint32_t st = 0;
    for (;;) {
        const bool ov = tile_join<CtaScope, kBlock, kCtaWMax>(R.list(dr, step_x_f(st, jo)), S.list(ds, step_y_f(st, jo)),
                                                              xs, ys, slot, tid, w0, js.bar, &js.phase, &js.timeout);
        if (js.timeout) return APRIL_VERDICT_ERROR;
        const int v = step_outcome(st, ov, jo);
        if (v >= 0) return (uint8_t)v;
    }
}

// One warp filters the 32 pairs starting at `base`: every lane fetches the
// ids and descriptors of its own pair at once (coalesced ids, 32 descriptor
// gathers in flight), then the warp joins the pairs one after another.  Pairs
// whose cost |A(r)| + |A(s)| exceeds cta_threshold are left to the CTA phase
// (pass UINT32_MAX to take every pair).
template <class SetsT>
__device__ __forceinline__ bool warp_chunk(const SetsT &R, const SetsT &S, const uint32_t *__restrict__ pr,
                                           const uint32_t *__restrict__ ps, uint64_t n, uint64_t base,
                                           uint8_t *__restrict__ out, uint32_t *status, uint2 *xs, uint2 *ys,
                                           uint32_t lane, uint32_t w0, uint32_t cta_threshold, bool flag_bad,
                                           JoinSync &js, uint32_t jo) {
    const uint64_t k = base + lane;
    typename SetsT::Desc dr{}, ds{};
    bool take = false;
    if (k < n) {
        const uint32_t r = __ldg(pr + k), s = __ldg(ps + k);
        if (r < R.n() && s < S.n()) {
            dr = R.load(r);
            ds = S.load(s);
            take = cta_threshold == kNoLongPairs ||
                   (uint64_t)SetsT::a_len(dr) + SetsT::a_len(ds) <= (uint64_t)cta_threshold;
        } else if (flag_bad) {
            out[k] = APRIL_VERDICT_ERROR;
            atomicOr(status, ST_BAD_ID);
        }
    }
    uint32_t todo = __ballot_sync(kFull, take);
    uint8_t mine = 0;
    while (todo) {
        const uint32_t t = __ffs(todo) - 1;
        todo &= todo - 1;
        const typename SetsT::Desc a = SetsT::shfl(dr, t), b = SetsT::shfl(ds, t);
        const uint8_t v = warp_verdict(R, S, a, b, xs, ys, lane, w0, js, jo);
        if (lane == t) mine = v;
        if (js.timeout) {  // the pairs of the chunk not decided yet read as errors
            if (lane == 0) atomicOr(status, ST_TIMEOUT);
            if (take) out[k] = (lane == t || ((todo >> lane) & 1u)) ? (uint8_t)APRIL_VERDICT_ERROR : mine;
            return false;
        }
    }
    if (take) out[k] = mine;
    return true;
}

// Initialises `count` mbarriers (8 bytes each, 8-byte aligned) at bars;
// every thread of the block must call it.
__device__ __forceinline__ void init_barriers(uint64_t *bars, uint32_t count) {
    for (uint32_t i = threadIdx.x; i < count; i += blockDim.x) mbar_init(smem_addr(bars + i), 1);
    if (threadIdx.x == 0) mbar_init_fence();
    __syncthreads();
}

// ------------------------------------------------------- K1: warp/pair
__global__ void __launch_bounds__(kBlock) k_warp(DevSet R, DevSet S, const uint32_t *__restrict__ pr,
                                                 const uint32_t *__restrict__ ps, uint64_t n,
                                                 uint8_t *__restrict__ out, uint32_t *status, uint32_t w0,
                                                 uint32_t jo) {
    __shared__ __align__(16) uint2 sm[kWarpsPerBlock][2][kWarpBuf];
    __shared__ uint64_t bars[kWarpsPerBlock];
    init_barriers(bars, kWarpsPerBlock);
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    JoinSync js{smem_addr(&bars[warp]), 0u, false};
    const uint64_t stride = (uint64_t)gridDim.x * kWarpsPerBlock * 32;
    for (uint64_t base = ((uint64_t)blockIdx.x * kWarpsPerBlock + warp) * 32; base < n; base += stride)
        if (!warp_chunk(RawSets{R}, RawSets{S}, pr, ps, n, base, out, status, sm[warp][0], sm[warp][1], lane, w0,
                        0xffffffffu, true, js, jo))
            return;
}

// --------------------------------------------- K4: length binning (batched)
// Validates ids (error verdicts), and appends every pair whose cost
// |A(r)| + |A(s)| exceeds the threshold to the long-pair list (warp-
// aggregated atomics).  Not launched when the threshold is kNoLongPairs: the
// lane groups then take every pair and report bad ids themselves.
template <class SetsT>
__global__ void __launch_bounds__(256) k_bin(SetsT R, SetsT S, const uint32_t *__restrict__ pr,
                                             const uint32_t *__restrict__ ps, uint64_t n, uint8_t *__restrict__ out,
                                             uint32_t *status, uint32_t cta_threshold, uint32_t *big_list,
                                             uint32_t *counters) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t kb = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); kb < n; kb += stride) {
        const uint64_t k = kb + lane;
        bool big = false;
        if (k < n) {
            const uint32_t r = __ldg(pr + k), s = __ldg(ps + k);
            if (r < R.n() && s < S.n()) {
                big = (uint64_t)SetsT::a_len(R.load(r)) + SetsT::a_len(S.load(s)) > (uint64_t)cta_threshold;
            } else {
                out[k] = APRIL_VERDICT_ERROR;
                atomicOr(status, ST_BAD_ID);
            }
        }
        const uint32_t mask = __ballot_sync(kFull, big);
        if (mask) {
            const uint32_t leader = __ffs(mask) - 1;
            uint32_t pos = 0;
            if (lane == leader) pos = atomicAdd(&counters[C_BIG_COUNT], __popc(mask));
            pos = __shfl_sync(kFull, pos, leader) + __popc(mask & ((1u << lane) - 1u));
            if (big) big_list[pos] = (uint32_t)k;
        }
    }
}

// ------------------------------------------ K3: persistent filter (batched)
// Group engine.  A warp is split into 32/G groups of G lanes; each group
// filters one pair at a time (its joins in the tuned order, see
// step_outcome), with its own window of at most 8*G intervals per list
// staged in shared memory.
// One pass of the loop below advances every group's current join by one
// window, so the fixed cost of a window step (staging, the per-thread merge-
// path search, the vote) is shared by 32/G joins.  When a group finishes its
// pair it takes the next one from the warp's current chunk of 32 pairs, whose
// eligible pairs are listed compacted in shared memory (a group takes the
// entry at the list's cursor plus its rank among the groups asking); the warp
// pops a new chunk from a global counter when the list is used up.  Pairs
// above a CTA threshold, when one is set, are skipped here (phase 1 did
// them).
template <uint32_t G>
struct GroupCfg {
    static constexpr uint32_t NG = 32 / G;
    static constexpr uint32_t WMAX = kGroupPer * G;
    static constexpr uint32_t BUF = WMAX + 2;
    static constexpr uint32_t LEADS = G == 32 ? 1u : G == 16 ? 0x00010001u : G == 8 ? 0x01010101u : 0x11111111u;
    // intervals of shared staging per warp: the groups' buffers, or two warp
    // windows for the long pairs joined by the warp
    static constexpr uint32_t SHARE = NG * 2 * BUF > 2 * kWarpBuf ? NG * 2 * BUF : 2 * kWarpBuf;
    // mbarriers: [0] the CTA phase, [1 + warp * NG + group] the group engine,
    // [1 + kWarpsPerBlock * NG + warp] long pairs joined by warps
    static constexpr uint32_t BARS = 1 + kWarpsPerBlock * (NG + 1);
    static __device__ __forceinline__ uint32_t group_bar(uint32_t warp, uint32_t g) { return 1 + warp * NG + g; }
    static __device__ __forceinline__ uint32_t warp_bar(uint32_t warp) { return 1 + kWarpsPerBlock * NG + warp; }
};
static_assert(2 * kCtaBuf <= kWarpsPerBlock * GroupCfg<32>::SHARE, "CTA windows must fit in the warps' buffers");
static_assert(GroupCfg<4>::SHARE % 2 == 0 && GroupCfg<8>::SHARE % 2 == 0 && GroupCfg<16>::SHARE % 2 == 0,
              "warp shares keep 16-byte alignment");

// Lists of join step `stage` of a pair (in join order jo, see step_outcome);
// false when one of them is empty (the join then has no overlap).
template <class SetsT, class ListT>
__device__ __forceinline__ bool join_lists(const SetsT &R, const SetsT &S, const uint4 &dr, const uint4 &ds,
                                           uint32_t stage, ListT &X, ListT &Y, uint32_t jo) {
    X = R.list(dr, step_x_f(stage, jo));
    Y = S.list(ds, step_y_f(stage, jo));
    return X.n != 0 && Y.n != 0;
}

// The start searches of every group of a warp at once (warp-collective;
// `need` names a group's lists to search, bit 0 X and bit 1 Y, 0 for none).
// A fresh join searches each list longer than a first window for its first
// interval whose last cell reaches the other list's first start; a galloping
// search (a window advanced one list only) searches that list, from its
// merge position, against the target `gt` (the other list's current start).
// Both lists are searched in the same rounds over their search keys (the skip
// index's posts for raw lists, block anchors for compressed lists; see
// RawList / PackedList).  Each probing round every lane probes P evenly spaced
// keys per list (fan-out G*P) and the group counts the probes below the
// target (a prefix, the keys being sorted), which leaves one gap of the
// spacing.  The probing stops once both ranges fit one vector round of
// 4 G kPostVec keys, and that round ends the search.
#ifndef APRIL_SEARCH_MIN
#define APRIL_SEARCH_MIN 0
#endif
constexpr uint32_t kSearchProbes = 1;
constexpr uint32_t kSearchMin = APRIL_SEARCH_MIN;  // lists up to this long are not searched by fresh joins
template <uint32_t G, class ListT>
__device__ __forceinline__ void dual_search(const ListT &X, const ListT &Y, uint32_t need, bool fresh, uint32_t gt,
                                            uint32_t t, uint32_t gbits, uint32_t &i0, uint32_t &j0) {
    constexpr uint32_t P = kSearchProbes, F = G * P;
    // probing stops once a range fits one vector round (post_count) over the
    // skip index (raw lists) or the block anchors (compressed lists)
    constexpr uint32_t PER = 4 / ListT::kKeyStride;  // keys per 16-byte load
    constexpr uint32_t LIMIT = PER * G * kPostVec - (PER - 1);
    const bool sx = need & 1u, sy = need & 2u;
    uint32_t loX = sx ? X.key_lo(i0) : 0, hiX = sx ? X.keys_n() : 0;
    uint32_t loY = sy ? Y.key_lo(j0) : 0, hiY = sy ? Y.keys_n() : 0;
    // the targets: a fresh join's other list's first start, loaded with the
    // first round's probes, whose positions do not depend on them
    const uint32_t kx = sx ? (fresh ? Y.first_start() : gt) : 0u, ky = sy ? (fresh ? X.first_start() : gt) : 0u;
    while (__any_sync(kFull, hiX - loX > LIMIT || hiY - loY > LIMIT)) {  // lo <= hi throughout
        const bool ax = hiX - loX > LIMIT, ay = hiY - loY > LIMIT;
        const uint32_t sX = ax ? (hiX - loX + F - 1) / F : 1, sY = ay ? (hiY - loY + F - 1) / F : 1;
        uint32_t vX[P], vY[P];
#pragma unroll
        for (uint32_t q = 0; q < P; ++q) {
            const uint32_t px = loX + (t * P + q + 1) * sX - 1, py = loY + (t * P + q + 1) * sY - 1;
            vX[q] = (ax && px < hiX) ? X.key(px) : 0u;
            vY[q] = (ay && py < hiY) ? Y.key(py) : 0u;
        }
        uint32_t cX = 0, cY = 0;
#pragma unroll
        for (uint32_t q = 0; q < P; ++q) {
            const uint32_t px = loX + (t * P + q + 1) * sX - 1, py = loY + (t * P + q + 1) * sY - 1;
            cX += __popc(__ballot_sync(kFull, ax && px < hiX && vX[q] < kx) & gbits);
            cY += __popc(__ballot_sync(kFull, ay && py < hiY && vY[q] < ky) & gbits);
        }
        // c below-probes leave the gap after the c-th probe, if that probe
        // exists (c < probes in [lo, hi)), else the tail after the last one
        if (ax) {
            if (loX + (cX + 1) * sX <= hiX) hiX = loX + (cX + 1) * sX - 1;
            loX += cX * sX;
        }
        if (ay) {
            if (loY + (cY + 1) * sY <= hiY) hiY = loY + (cY + 1) * sY - 1;
            loY += cY * sY;
        }
    }
    if (__any_sync(kFull, hiX > loX || hiY > loY)) {
        // the last round: each lane counts its vectors of keys of both lists;
        // the group sums (X in the low half, Y in the high half)
        constexpr uint32_t KS = ListT::kKeyStride;
        uint32_t v = post_count<KS>(X.keys(), loX, hiX, 0, kx, t, G) | (post_count<KS>(Y.keys(), loY, hiY, 0, ky, t, G) << 16);
#pragma unroll
        for (uint32_t m = 1; m < G; m <<= 1) v += __shfl_xor_sync(kFull, v, m);
        loX += v & 0xFFFFu;
        loY += v >> 16;
    }
    if (sx) i0 = max(i0, X.start_of(loX));
    if (sy) j0 = max(j0, Y.start_of(loY));
}

// The pairs are all n, or the n that the single lanes left in a rest list
// (Rest): a pair's index there carries in its two top bits, where `stages` says
// so, the join it has reached.
struct Rest {
    const uint32_t *list;  // nullptr: all pairs
    bool stages;
    __device__ __forceinline__ uint32_t entry(uint64_t q) const { return list ? __ldg(list + q) : (uint32_t)q; }
    __device__ __forceinline__ uint32_t pair(uint32_t e) const { return stages ? e & 0x3fffffffu : e; }
    __device__ __forceinline__ uint32_t stage(uint32_t e) const { return stages ? e >> 30 : 0u; }
};

template <uint32_t G, class SetsT>
__device__ __forceinline__ void group_engine(const SetsT &R, const SetsT &S, const uint32_t *__restrict__ pr,
                                             const uint32_t *__restrict__ ps, uint64_t n, uint8_t *__restrict__ out,
                                             uint32_t *status, uint32_t *counters, uint32_t cta_threshold, uint2 *wbuf,
                                             uint4 *chunk_desc, uint32_t *chunk_k, uint32_t bars,
                                             uint32_t lane, uint32_t w0, uint32_t jo, uint32_t esc_windows, uint4 *esc,
                                             uint32_t esc_cap, const Rest &rest) {
    using C = GroupCfg<G>;
    const bool no_long = cta_threshold == kNoLongPairs;  // every pair is joined here; no binning kernel ran

    const uint32_t g = lane / G, t = lane % G, glead = g * G;
    const uint32_t gbits = (G == 32 ? kFull : ((1u << G) - 1u)) << glead;
    uint2 *xb = wbuf + g * 2 * C::BUF, *yb = xb + C::BUF;
    const uint32_t bar = bars + 8u * g;  // this group's mbarrier
    uint32_t phase = 0;
    // the warp's chunk of 32 pairs (from position `base` of the pair list):
    // the pairs it takes are stored compacted, the pair
    // of entry chunk_k[i] with its two descriptors in chunk_desc[i] and
    // chunk_desc[32 + i]; entries [cur, cur + left) are still to be handed out
    uint32_t base = 0;
    uint32_t cur = 0, left = 0;
    bool exhausted = false;
    // this group's pair and join
    bool active = false;
    uint32_t k = 0;
    uint4 dr = make_uint4(0, 0, 0, 0), ds = make_uint4(0, 0, 0, 0);
    uint32_t stage = 0, i0 = 0, j0 = 0, w = w0;
    uint32_t nwin = 0;   // windows of the current join so far
    bool fresh = false;  // the join has just started: its start has not been searched yet
    uint32_t gal = 0, gt = 0;  // a galloping search due (bit 0: X, bit 1: Y) and its target
    using ListT = decltype(R.list(dr, false));
    ListT X = R.list(dr, false), Y = S.list(ds, false);

    for (;;) {
        // -------- hand pairs to idle groups
        uint32_t needg = __ballot_sync(kFull, !active) & C::LEADS;
        while (needg && !exhausted) {
            if (!left) {
                uint32_t c = 0;
                if (lane == 0) c = atomicAdd(&counters[C_CHUNK_HEAD], 1u);
                c = __shfl_sync(kFull, c, 0);
                if (c >= (n + 31) / 32) {
                    exhausted = true;
                    break;
                }
                base = c * 32;  // n < 2^32 pairs
                const bool on = base + lane < n;
                const uint32_t entry = on ? rest.entry(base + lane) : 0u, kk = rest.pair(entry);
                bool take = false;
                __syncwarp();  // every group has read its descriptors from the previous chunk
                uint4 qdr = make_uint4(0, 0, 0, 0), qds = qdr;
                if (on) {
                    const uint32_t r = __ldg(pr + kk), s2 = __ldg(ps + kk);
                    if (r < R.n() && s2 < S.n()) {
                        qdr = R.load(r);
                        qds = S.load(s2);
                        take = no_long || (uint64_t)qdr.y + qds.y <= (uint64_t)cta_threshold;
                    } else if (no_long) {  // no binning kernel ran to report them
                        out[kk] = APRIL_VERDICT_ERROR;
                        atomicOr(status, ST_BAD_ID);
                    }
                }
                // the pairs this warp takes, compacted in order
                const uint32_t tb = __ballot_sync(kFull, take);
                if (take) {
                    const uint32_t pos = __popc(tb & ((1u << lane) - 1u));
                    chunk_k[pos] = entry;
                    chunk_desc[pos] = qdr;
                    chunk_desc[32 + pos] = qds;
                }
                cur = 0;
                left = __popc(tb);
                __syncwarp();
                continue;
            }
            const uint32_t cnt = min((uint32_t)__popc(needg), left);
            const uint32_t grank = __popc(needg & ((1u << glead) - 1u));
            const bool gets = ((needg >> glead) & 1u) && grank < cnt;
            if (gets) {
                const uint32_t src = cur + grank;
                k = rest.pair(chunk_k[src]);
                dr = chunk_desc[src];
                ds = chunk_desc[32 + src];
                stage = rest.stage(chunk_k[src]);
                i0 = j0 = 0;
                w = w0;
                nwin = 0;
                fresh = true;
                int verdict = -1;  // steps with an empty list have no overlap
                while (!join_lists(R, S, dr, ds, stage, X, Y, jo))
                    if ((verdict = step_outcome(stage, false, jo)) >= 0) break;
                active = verdict < 0;
                if (!active && t == 0) out[k] = (uint8_t)verdict;
            }
            cur += cnt;
            left -= cnt;
            needg = __ballot_sync(kFull, !active) & C::LEADS;
        }
        if (!__any_sync(kFull, active)) break;  // only reachable once the pairs are exhausted

        // -------- a join that has just started skips, in each list longer
        // than a window, the intervals ending before the other list's first
        // start (they meet nothing; the merge would pass over them); a list
        // that the last window advanced alone skips those ending before the
        // other list's current start (galloping, see tile_join)
        if (__any_sync(kFull, active && (fresh || gal))) {
            const uint32_t smin = max(w0, kSearchMin);
            const uint32_t nd = !active ? 0u : fresh ? (uint32_t)(X.n > smin) | ((uint32_t)(Y.n > smin) << 1) : gal;
            dual_search<G>(X, Y, nd, fresh, gt, t, gbits, i0, j0);
        }
        fresh = false;
        gal = 0;
        const uint32_t nX = X.n, nY = Y.n;
        const bool ran_out = active && (i0 >= nX || j0 >= nY);  // the search passed a whole list

        // -------- one window of every active group's join: raw lists arrive
        // by two bulk copies on the group's mbarrier, compressed lists are
        // decoded by the group's lanes (one block each)
        uint32_t nx = 0, ny = 0, xa = 0, ya = 0;
        bool ok = true;
        if (active && !ran_out) {
            nx = min(w, nX - i0);
            ny = min(w, nY - j0);
            if constexpr (ListT::kBulk) {
                if constexpr (kStage2) {
                    // lane 0 copies X's window, lane 1 Y's; each arrives once
                    // with its own bytes on the group's mbarrier (count 2)
                    if (t < 2) {
                        fence_proxy_async();
                        const bool isy = t == 1;
                        const uint2 *src = isy ? Y.p + j0 : X.p + i0;
                        const uint2 *a;
                        uint32_t b, o;
                        bulk_span(src, isy ? ny : nx, a, b, o);
                        mbar_arrive_expect_tx(bar, b);
                        bulk_load(smem_addr(isy ? yb : xb), src - o, b, bar);
                    }
                } else if (t == 0) {
                    fence_proxy_async();
                    const uint2 *a;
                    uint32_t bx, by, ox, oy;
                    bulk_span(X.p + i0, nx, a, bx, ox);
                    bulk_span(Y.p + j0, ny, a, by, oy);
                    mbar_arrive_expect_tx(bar, bx + by);
                    bulk_load(smem_addr(xb), X.p + i0 - ox, bx, bar);
                    bulk_load(smem_addr(yb), Y.p + j0 - oy, by, bar);
                }
                ok = mbar_wait(bar, phase);
                phase ^= 1u;
            } else {
                X.template stage<G>(xb, i0, nx, t, gbits);
                Y.template stage<G>(yb, j0, ny, t, gbits);
            }
            xa = X.window(xb, i0);
            ya = Y.window(yb, j0);
        }
        if constexpr (!ListT::kBulk) __syncwarp();  // the decoded windows are visible to the group
        if (!__all_sync(kFull, ok)) {
            // a bounded wait ran out: once the copies in flight have landed
            // (bounded), mark the pairs this warp holds as errors, report
            // and stop this warp
            if (!ok) mbar_drain(bar, phase ^ 1u);
            if (active && t == 0) out[k] = APRIL_VERDICT_ERROR;
            if (lane < left) out[rest.pair(chunk_k[cur + lane])] = APRIL_VERDICT_ERROR;
            if (lane == 0) atomicOr(status, ST_TIMEOUT);
            return;
        }
        bool found = false;
        uint32_t state = 0xffffffffu, D = 0, owner = 0;
        if (active && !ran_out) {
            D = min(w, nx + ny);
            const uint32_t per = w / G;  // a power of two
            owner = (D - 1) >> (__ffs(per) - 1);
            found = window_walk<C::WMAX / G>(xa, nx, ya, ny, w, D, per, t * per, state);
        }
        const uint32_t fmask = __ballot_sync(kFull, found);  // every read of the windows is done here
        const uint32_t split = __shfl_sync(kFull, state, glead + owner);
        if (active) {
            int res = -1;  // -1: join continues, 0: no overlap, 1: overlap
            if (ran_out) res = 0;
            else if (fmask & gbits) res = 1;
            else if (D == nx + ny || split == 0xffffffffu) res = 0;
            else {
                i0 += split;
                j0 += D - split;
                w = min(w * 2u, C::WMAX);
                // the windows stay intact until the next pass's staging,
                // which follows that pass's first warp vote
                if (split == 0 && nY - j0 > w) {
                    gal = 2u;
                    gt = lds1(xa);  // X's current start
                } else if (split == D && nX - i0 > w) {
                    gal = 1u;
                    gt = lds1(ya);  // Y's current start
                }
                if (esc_windows && ++nwin >= esc_windows) {
                    // a long join: hand it, at the position it reached, to a
                    // whole warp (k_long) and take the next pair, unless the
                    // queue is full
                    uint32_t slot = 0;
                    if (t == 0) slot = atomicAdd(&counters[C_ESC_COUNT], 1u);
                    slot = __shfl_sync(gbits, slot, glead);
                    if (slot < esc_cap) {
                        if (t == 0) esc[slot] = make_uint4(k, stage, i0, j0);
                        active = false;
                    } else {
                        nwin = 0;
                    }
                }
            }
            if (res >= 0) {
                int verdict = step_outcome(stage, res != 0, jo);
                while (verdict < 0) {
                    i0 = j0 = 0;
                    w = w0;
                    nwin = 0;
                    fresh = true;
                    if (join_lists(R, S, dr, ds, stage, X, Y, jo)) break;
                    verdict = step_outcome(stage, false, jo);
                }
                if (verdict >= 0) {
                    if (t == 0) out[k] = (uint8_t)verdict;
                    active = false;
                }
            }
        }
    }
}

// Phase 1 (only with a long-pair threshold): the long pairs, each joined by
// one warp (first window below 256) or by the whole CTA (the merge path of one
// join split over 256 threads).  Phase 2: the group engine on the other pairs
// (whole warps when G = 32).
// Work is handed out by atomic counters; nothing waits on another CTA.
template <uint32_t G, class SetsT>
__global__ void APRIL_PERSISTENT_BOUNDS k_persistent(SetsT R, SetsT S,
                                                                         const uint32_t *__restrict__ pr,
                                                       const uint32_t *__restrict__ ps, uint64_t n,
                                                       uint8_t *__restrict__ out, uint32_t *status,
                                                       uint32_t cta_threshold, const uint32_t *__restrict__ big_list,
                                                       uint32_t *counters, uint32_t w0_group, uint32_t w0_cta,
                                                       uint32_t jo, uint32_t esc_windows, uint4 *esc, uint32_t esc_cap) {
    using C = GroupCfg<G>;
    __shared__ __align__(16) uint2 sm[kWarpsPerBlock * C::SHARE];
    __shared__ uint32_t s_item, s_slot;
    __shared__ uint64_t bars[C::BARS];  // see GroupCfg
    __shared__ uint4 s_chunk[kWarpsPerBlock][64];     // group engine: each warp's chunk descriptors
    __shared__ uint32_t s_chunk_k[kWarpsPerBlock][32];    // and their pairs
    if constexpr (kStage2 && G < 32 && !SetsT::kPacked) {
        // the lane groups' mbarriers take two arrivals a window (see group_engine)
        for (uint32_t i = threadIdx.x; i < C::BARS; i += blockDim.x) {
            const bool grp = i >= 1 && i < 1 + kWarpsPerBlock * C::NG;
            mbar_init(smem_addr(bars + i), grp ? 2u : 1u);
        }
        if (threadIdx.x == 0) mbar_init_fence();
        __syncthreads();
    } else {
        init_barriers(bars, C::BARS);
    }
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t nbig = *((volatile uint32_t *)&counters[C_BIG_COUNT]);
    uint2 *wbuf = sm + warp * C::SHARE;
    if (w0_cta < kBlock) {
        // long pairs one per warp (first window w0_cta): the CTA's warps work
        // on eight long pairs at once
        JoinSync ws{smem_addr(&bars[C::warp_bar(warp)]), 0u, false};
        for (;;) {
            uint32_t it = 0;
            if (lane == 0) it = atomicAdd(&counters[C_BIG_HEAD], 1u);
            it = __shfl_sync(kFull, it, 0);
            if (it >= nbig) break;
            const uint64_t k = big_list[it];
            const typename SetsT::Desc dr = R.load(__ldg(pr + k)), ds = S.load(__ldg(ps + k));
            const uint8_t v = warp_verdict(R, S, dr, ds, wbuf, wbuf + kWarpBuf, lane, w0_cta, ws, jo);
            if (lane == 0) out[k] = v;
            if (ws.timeout) {  // a bounded wait ran out: report and stop this warp
                if (lane == 0) atomicOr(status, ST_TIMEOUT);
                return;
            }
        }
        // no CTA barrier here: the warp's phase-2 buffers and mbarriers are
        // its own, so it starts on short pairs while its CTA's other warps
        // still join long ones
    } else {
        JoinSync cs{smem_addr(&bars[0]), 0u, false};
        for (;;) {
            if (tid == 0) s_item = atomicAdd(&counters[C_BIG_HEAD], 1u);
            __syncthreads();
            const uint32_t it = s_item;
            __syncthreads();
            if (it >= nbig) break;
            const uint64_t k = big_list[it];
            const typename SetsT::Desc dr = R.load(__ldg(pr + k)), ds = S.load(__ldg(ps + k));
            const uint8_t v = cta_verdict(R, S, dr, ds, sm, sm + kCtaBuf, &s_slot, tid, w0_cta, cs, jo);
            if (tid == 0) out[k] = v;
            if (cs.timeout) {  // a bounded wait ran out: report and stop this CTA
                if (tid == 0) atomicOr(status, ST_TIMEOUT);
                return;
            }
        }
        __syncthreads();
    }
    if constexpr (G == 32) {
        JoinSync js{smem_addr(&bars[C::group_bar(warp, 0)]), 0u, false};
        const uint64_t nchunks = (n + 31) / 32;
        for (;;) {
            uint32_t c = 0;
            if (lane == 0) c = atomicAdd(&counters[C_CHUNK_HEAD], 1u);
            c = __shfl_sync(kFull, c, 0);
            if (c >= nchunks) break;
            if (!warp_chunk(R, S, pr, ps, n, (uint64_t)c * 32, out, status, wbuf, wbuf + kWarpBuf, lane, w0_group,
                            cta_threshold, cta_threshold == kNoLongPairs, js, jo))
                return;
        }
    } else {
        group_engine<G>(R, S, pr, ps, n, out, status, counters, cta_threshold, wbuf, s_chunk[warp], s_chunk_k[warp],
                        smem_addr(&bars[C::group_bar(warp, 0)]), lane, w0_group, jo, esc_windows, esc, esc_cap,
                        Rest{nullptr, false});
    }
}

// K3 over the rest list: the group engine in CTAs of two warps.  The list is
// nearly always empty.
constexpr uint32_t kRestWarps = 2;
template <uint32_t G, class SetsT>
__global__ void __launch_bounds__(32 * kRestWarps)
    k_persistent_rest(SetsT R, SetsT S, const uint32_t *__restrict__ pr, const uint32_t *__restrict__ ps,
                      uint8_t *__restrict__ out, uint32_t *status, uint32_t *counters, uint32_t w0, uint32_t jo,
                      uint32_t esc_windows, uint4 *esc, uint32_t esc_cap, Rest rest) {
    using C = GroupCfg<G>;
    const uint32_t n = *((volatile uint32_t *)&counters[C_REST_COUNT]);
    if (n == 0) return;
    __shared__ __align__(16) uint2 sm[kRestWarps * C::SHARE];
    __shared__ uint64_t bars[kRestWarps * C::NG];
    __shared__ uint4 s_chunk[kRestWarps][64];
    __shared__ uint32_t s_chunk_k[kRestWarps][32];
    for (uint32_t i = threadIdx.x; i < kRestWarps * C::NG; i += blockDim.x)
        mbar_init(smem_addr(bars + i), kStage2 ? 2u : 1u);
    if (threadIdx.x == 0) mbar_init_fence();
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    group_engine<G>(R, S, pr, ps, n, out, status, counters, kNoLongPairs, sm + warp * C::SHARE, s_chunk[warp],
                    s_chunk_k[warp], smem_addr(&bars[warp * C::NG]), lane, w0, jo, esc_windows, esc, esc_cap, rest);
}

// ------------------------------ K3b: joins handed over by the lane groups
// Each warp takes the next queued join {pair, step, i0, j0} and finishes the
// pair by whole-warp joins: that step resumes at (i0, j0) with first window
// w0, the later steps of the join order start fresh.
template <class SetsT>
__global__ void __launch_bounds__(kBlock) k_long(SetsT R, SetsT S, const uint32_t *__restrict__ pr,
                                                 const uint32_t *__restrict__ ps, uint8_t *__restrict__ out,
                                                 uint32_t *status, const uint4 *__restrict__ esc, uint32_t *counters,
                                                 uint32_t esc_cap, uint32_t w0, uint32_t jo) {
    __shared__ __align__(16) uint2 sm[kWarpsPerBlock][2][kWarpBuf];
    __shared__ uint64_t bars[kWarpsPerBlock];
    init_barriers(bars, kWarpsPerBlock);
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    JoinSync js{smem_addr(&bars[warp]), 0u, false};
    const uint32_t nesc = min(*((volatile uint32_t *)&counters[C_ESC_COUNT]), esc_cap);
    for (;;) {
        uint32_t it = 0;
        if (lane == 0) it = atomicAdd(&counters[C_ESC_HEAD], 1u);
        it = __shfl_sync(kFull, it, 0);
        if (it >= nesc) break;
        const uint4 rec = esc[it];
        const typename SetsT::Desc dr = R.load(__ldg(pr + rec.x)), ds = S.load(__ldg(ps + rec.x));
        const uint8_t v = warp_verdict(R, S, dr, ds, sm[warp][0], sm[warp][1], lane, w0, js, jo, rec.y, true, rec.z,
                                       rec.w);
        if (lane == 0) out[rec.x] = v;
        if (js.timeout) {  // a bounded wait ran out: report and stop this warp
            if (lane == 0) atomicOr(status, ST_TIMEOUT);
            return;
        }
    }
}

// -------------------------------- K7: filter variants (Sec. 4.3.2, Sec. 5.3)
// With the triage the variants run in lanes too (k_triage and k_persistent
// with VAR); this kernel takes the tunings without it, and the pairs that the
// lanes leave.
// A plan is the decision sequence of one filter variant: each stage joins one
// list of r with one list of s under a predicate and either decides the
// verdict or moves to another stage.  The finer side's lists are coarsened
// on load when the two sets use grids of different order (Sec. 5.3).
struct Plan {
    uint8_t nst;
    uint8_t xf[3], yf[3];       // stage's list: 0 = A-list, 1 = F-list (r, s)
    uint8_t pred[3];            // kOverlap or kContain
    int8_t on_true[3], on_false[3];  // >= 0: next stage; < 0: verdict -(v + 1)
    uint8_t sx, sy;             // coarsening shifts of r's / s's intervals (bits)
};

template <class Scope, uint32_t NT, uint32_t WMAX>
__device__ __forceinline__ uint8_t plan_verdict(const Plan &P, const RawSets &R, const RawSets &S, const uint4 &dr,
                                                const uint4 &ds, uint2 *xs, uint2 *ys, uint32_t *slot, uint32_t tid,
                                                uint32_t w0, JoinSync &js, int st = 0) {
    for (int guard = 0; guard < 3; ++guard) {
        const RawList X = R.list(dr, P.xf[st] != 0), Y = S.list(ds, P.yf[st] != 0);
        const bool res =
            P.pred[st] == kContain
                ? tile_join<Scope, NT, WMAX, RawList, kContain>(X, Y, xs, ys, slot, tid, w0, js.bar, &js.phase,
                                                                &js.timeout, P.sx, P.sy)
                : tile_join<Scope, NT, WMAX, RawList, kOverlap>(X, Y, xs, ys, slot, tid, w0, js.bar, &js.phase,
                                                                &js.timeout, P.sx, P.sy);
        if (js.timeout) return APRIL_VERDICT_ERROR;
        const int nx = res ? P.on_true[st] : P.on_false[st];
        if (nx < 0) return (uint8_t)(-(nx + 1));
        st = nx;
    }
    return APRIL_VERDICT_ERROR;
}

// The pairs by warps taking 32-pair chunks (those above the threshold, when all
// n are taken, are the CTAs').
__device__ __forceinline__ void general_pairs(const Plan &P, const RawSets &R, const RawSets &S,
                                              const uint32_t *__restrict__ pr, const uint32_t *__restrict__ ps,
                                              uint64_t n, uint8_t *__restrict__ out, uint32_t *status,
                                              uint32_t cta_threshold, uint32_t *counters, uint2 *xs, uint2 *ys,
                                              uint32_t lane, JoinSync &js, const Rest &rest) {
    const uint64_t nchunks = (n + 31) / 32;
    for (;;) {
        uint32_t c = 0;
        if (lane == 0) c = atomicAdd(&counters[C_CHUNK_HEAD], 1u);
        c = __shfl_sync(kFull, c, 0);
        if (c >= nchunks) break;
        const bool on = (uint64_t)c * 32 + lane < n;
        const uint32_t entry = on ? rest.entry((uint64_t)c * 32 + lane) : 0u, k = rest.pair(entry);
        uint4 dr = make_uint4(0, 0, 0, 0), ds = make_uint4(0, 0, 0, 0);
        bool take = false;
        if (on) {
            const uint32_t r = __ldg(pr + k), s2 = __ldg(ps + k);
            if (r < R.n() && s2 < S.n()) {
                dr = R.load(r);
                ds = S.load(s2);
                take = rest.list || (uint64_t)dr.y + ds.y <= (uint64_t)cta_threshold;
            }
        }
        uint32_t todo = __ballot_sync(kFull, take);
        uint8_t mine = 0;
        while (todo) {
            const uint32_t t = __ffs(todo) - 1;
            todo &= todo - 1;
            const uint8_t v = plan_verdict<WarpScope, 32, kWarpWMax>(P, R, S, shfl4(dr, t), shfl4(ds, t), xs, ys,
                                                                      nullptr, lane, 64u, js,
                                                                      (int)rest.stage(__shfl_sync(kFull, entry, t)));
            if (lane == t) mine = v;
            if (js.timeout) {  // the pairs of the chunk not decided yet read as errors
                if (lane == 0) atomicOr(status, ST_TIMEOUT);
                if (take) out[k] = (lane == t || ((todo >> lane) & 1u)) ? (uint8_t)APRIL_VERDICT_ERROR : mine;
                return;
            }
        }
        if (take) out[k] = mine;
    }
}

// Same shape as K3 with 32-lane groups: long pairs by whole CTAs, the rest by
// warps taking 32-pair chunks.
// the variant kernel at four CTAs per SM (at most 64 registers a thread)
#ifndef APRIL_GENERAL_MIN_BLOCKS
#define APRIL_GENERAL_MIN_BLOCKS 4
#endif
__global__ void __launch_bounds__(kBlock, APRIL_GENERAL_MIN_BLOCKS) k_general(Plan P, DevSet Rd, DevSet Sd, const uint32_t *__restrict__ pr,
                                                    const uint32_t *__restrict__ ps, uint64_t n,
                                                    uint8_t *__restrict__ out, uint32_t *status,
                                                    uint32_t cta_threshold, const uint32_t *__restrict__ big_list,
                                                    uint32_t *counters, uint32_t long_window) {
    __shared__ __align__(16) uint2 sm[kSharedIv];
    __shared__ uint32_t s_item, s_slot;
    __shared__ uint64_t bars[1 + kWarpsPerBlock];
    init_barriers(bars, 1 + kWarpsPerBlock);
    const RawSets R{Rd}, S{Sd};
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint32_t nbig = *((volatile uint32_t *)&counters[C_BIG_COUNT]);
    uint2 *xs = sm + warp * kWarpShare, *ys = xs + kWarpBuf;
    JoinSync js{smem_addr(&bars[1 + warp]), 0u, false};
    if (long_window < kBlock) {  // long pairs one per warp
        for (;;) {
            uint32_t it = 0;
            if (lane == 0) it = atomicAdd(&counters[C_BIG_HEAD], 1u);
            it = __shfl_sync(kFull, it, 0);
            if (it >= nbig) break;
            const uint64_t k = big_list[it];
            const uint4 dr = R.load(__ldg(pr + k)), ds = S.load(__ldg(ps + k));
            const uint8_t v = plan_verdict<WarpScope, 32, kWarpWMax>(P, R, S, dr, ds, xs, ys, nullptr, lane,
                                                                      long_window, js);
            if (lane == 0) out[k] = v;
            if (js.timeout) break;
        }
        const bool dead = js.timeout;
        if (dead && lane == 0) atomicOr(status, ST_TIMEOUT);
        __syncthreads();
        if (dead) return;  // a bounded wait ran out: this warp stops (after the CTA's only barrier)
    } else {
        JoinSync cs{smem_addr(&bars[0]), 0u, false};
        for (;;) {
            if (tid == 0) s_item = atomicAdd(&counters[C_BIG_HEAD], 1u);
            __syncthreads();
            const uint32_t it = s_item;
            __syncthreads();
            if (it >= nbig) break;
            const uint64_t k = big_list[it];
            const uint4 dr = R.load(__ldg(pr + k)), ds = S.load(__ldg(ps + k));
            const uint8_t v = plan_verdict<CtaScope, kBlock, kCtaWMax>(P, R, S, dr, ds, sm, sm + kCtaBuf, &s_slot,
                                                                        tid, long_window, cs);
            if (tid == 0) out[k] = v;
            if (cs.timeout) {
                if (tid == 0) atomicOr(status, ST_TIMEOUT);
                return;
            }
        }
        __syncthreads();
    }
    general_pairs(P, R, S, pr, ps, n, out, status, cta_threshold, counters, xs, ys, lane, js, Rest{nullptr, false});
}

// K7 over the rest list, in CTAs of two warps (see k_persistent_rest).
__global__ void __launch_bounds__(32 * kRestWarps)
    k_rest_general(Plan P, DevSet Rd, DevSet Sd, const uint32_t *__restrict__ pr, const uint32_t *__restrict__ ps,
                   uint8_t *__restrict__ out, uint32_t *status, uint32_t *counters, Rest rest) {
    const uint32_t n = *((volatile uint32_t *)&counters[C_REST_COUNT]);
    if (n == 0) return;
    __shared__ __align__(16) uint2 sm[kRestWarps * kWarpShare];
    __shared__ uint64_t bars[kRestWarps];
    init_barriers(bars, kRestWarps);
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint2 *xs = sm + warp * kWarpShare;
    JoinSync js{smem_addr(&bars[warp]), 0u, false};
    general_pairs(P, RawSets{Rd}, RawSets{Sd}, pr, ps, n, out, status, 0u, counters, xs, xs + kWarpBuf, lane, js, rest);
}

// ------------------------------------------- K2: one lane per pair (batched)
// The first pass of the batched filter: every lane runs one pair's joins as
// leapfrogs (RawLane / PackedLane) in rounds of one load each, and takes a
// new pair when it is through.  A pair whose join has used up its rounds (a
// finely interleaved one) goes to the rest list: for the merge windows of the
// lane groups (K3) or, of a variant, of warps (K7), or, over compressed lists,
// for eight lanes (K3).  A plan is the decision sequence: per stage the lists
// joined (bit set: the F-list) and, per stage and answer, a nibble of `next`
// (below 8 the next stage, else 8 + the verdict).
struct LanePlan {
    uint32_t xf, yf, contain, next;
    LaneVariant v;
};

template <class SetsT, bool VAR>
struct LaneOf {
    using T = RawLane<VAR>;
};
template <bool VAR>
struct LaneOf<PackedSets, VAR> {
    using T = PackedLane;
};

// Unit rounds a join of lists of xn and yn intervals may take in one lane.
// Where two lists alternate to the end, a round passes one interval, and a merge
// window 32 in the time of about eight rounds: 1M such joins of 500 + 500 took
// 19.8 ms in lanes and 2.7 in groups of four.  Where they alternate in bursts the
// lanes win (100k of 10,000 + 10,000 in bursts of 16: 3.8 ms, 10.4 in groups),
// down to one round for every three intervals.  So a join that has taken a round
// for every sixteen is handed to the windows: 4.0 ms for the former, 2.9 for the
// latter.  Lists of polygons end long before: of the timed cases' pairs none is
// handed over (with a base of 24 and a thirty-second, 10 of 1.2M within pairs).
// With `fixed` only very long joins are: over compressed lists, whose windows
// are decoded before they are merged and never win (5.9 and 7.7 ms for the
// former, 12.5 and 2.4 for bursts of 100), and for requests that share the GPU
// (see april_enqueue_request); eight lanes then take each.
constexpr uint32_t kLaneBase = 64, kLaneShare = 16, kLaneFixed = 512;
__device__ __forceinline__ uint32_t lane_budget(uint32_t xn, uint32_t yn, uint32_t fixed) {
    return fixed ? fixed : kLaneBase + xn / kLaneShare + yn / kLaneShare;
}

__device__ __forceinline__ LaneFirst lane_first(const RawSets &A, uint32_t off) {
    return RawLane<false>::first(A.s.iv, off);
}
__device__ __forceinline__ LaneFirst lane_first(const PackedSets &A, uint32_t off) {
    return PackedLane::first(A.blocks, A.gaps, off);
}

// The stage a pair with descriptors dr and ds goes on with from stage st:
// the first that has two lists (returns -1), or the verdict when the stages
// end before that.
__device__ __forceinline__ int lane_stage(const LanePlan &P, const uint4 &dr, const uint4 &ds, uint32_t &st) {
    for (;;) {
        const uint32_t xn = (P.xf >> st) & 1u ? dr.w : dr.y, yn = (P.yf >> st) & 1u ? ds.w : ds.y;
        if (xn && yn) return -1;
        // no overlap; and nothing contains an interval of r's
        const uint32_t res = ((P.contain >> st) & 1u) && xn ? 1u : 0u;
        const uint32_t c = (P.next >> (4u * (2u * st + res))) & 15u;
        if (c & 8u) return (int)(c & 7u);
        st = c;
    }
}

template <class LaneT, class SetsT>
__device__ __forceinline__ void lane_start(LaneT &L, const LanePlan &P, const SetsT &R, const SetsT &S, const uint4 &dr,
                                           const uint4 &ds, uint32_t st, uint32_t fixed, uint32_t limit) {
    const bool xf = (P.xf >> st) & 1u, yf = (P.yf >> st) & 1u;
    const uint32_t xo = xf ? dr.z : dr.x, yo = yf ? ds.z : ds.x, xn = xf ? dr.w : dr.y, yn = yf ? ds.w : ds.y;
    LaneVariant v = P.v;
    v.contain = (P.contain >> st) & 1u;
    const LaneFirst fx = lane_first(R, xo), fy = lane_first(S, yo);
    L.left = min(limit, lane_budget(xn, yn, fixed));
    L.start(xo, xn, yo, yn, fx, fy, v);
}

// Starts lane t of T on its segment of stage st's join (segments of whole
// UNITs); a lane without one ends with no overlap.
template <uint32_t UNIT, class LaneT, class SetsT>
__device__ __forceinline__ void lane_split(LaneT &L, const LanePlan &P, const SetsT &R, const SetsT &S, const uint4 &dr,
                                           const uint4 &ds, uint32_t st, uint32_t t, uint32_t T) {
    const bool xf = (P.xf >> st) & 1u, yf = (P.yf >> st) & 1u;
    uint32_t xo = xf ? dr.z : dr.x, yo = yf ? ds.z : ds.x, xn = xf ? dr.w : dr.y, yn = yf ? ds.w : ds.y;
    LaneVariant v = P.v;
    v.contain = (P.contain >> st) & 1u;
    const bool sx = v.contain || xn <= yn;
    const uint32_t n = sx ? xn : yn, seg = ((n - 1u) / T / UNIT + 1u) * UNIT;
    const uint64_t a = (uint64_t)t * seg;
    L.left = 0xffffffffu;
    if (a >= n) {
        L.end(0);
        return;
    }
    const uint32_t off = (uint32_t)a / (SetsT::kPacked ? 16u : 1u), cnt = min(seg, n - (uint32_t)a);
    if (sx) xo += off, xn = cnt;
    else yo += off, yn = cnt;
    const LaneFirst fx = lane_first(R, xo), fy = lane_first(S, yo);
    L.start(xo, xn, yo, yn, fx, fy, v);
}

// Rounds of kind `pick` (lane_pick: 1, the index's; 0, the list's), LaneT::kRun
// at a time.
template <class LaneT, class SetsT>
__device__ __forceinline__ void lane_round(LaneT &L, int pick, const LanePlan &P, const SetsT &R, const SetsT &S,
                                           uint32_t st) {
    LaneVariant v = P.v;
    v.contain = (P.contain >> st) & 1u;
    if (pick) {
#pragma unroll 1
        for (int i = 0; i < LaneT::kRun; ++i)
            if (L.mode == kLaneIndex || L.mode == kLaneSeek) L.index_round(R, S, v);
    } else {
#pragma unroll 1
        for (int i = 0; i < LaneT::kRun; ++i)
            if (L.mode == kLaneUnit) L.unit_round(R, S, v);
    }
}

// K2 (k_triage: it settles what single lanes can): one lane per pair.  Bound by
// issue (74 warp instructions a paper-scale pair at 20 active lanes) and, at the
// end, by the last pairs' chains of rounds: 2M paper-scale pairs take 300 us in all (lane groups after a
// centre-cell probe: 567), 8M skewed ones 1.39 ms (2.27), 600k over compressed
// lists 319 us (514), 1.2M within 277 us and 1.2M of different granularity 174
// (a warp per pair: 1,381 and 705).  Five CTAs per SM: four give the compiler
// room, but 3% fewer pairs a second; six spill.
// The pairs come in chunks of 32 from a global counter; a chunk's ids and
// descriptors are fetched by all lanes at once and wait in shared memory,
// compacted to the pairs that are valid.  A rest entry is the pair's index,
// with the stage it has reached in its two top bits where `stages` says so.
#ifndef APRIL_LANE_MIN_BLOCKS
#define APRIL_LANE_MIN_BLOCKS 5
#endif
template <class SetsT, bool VAR>
__global__ void __launch_bounds__(256, APRIL_LANE_MIN_BLOCKS)
    k_triage(SetsT R, SetsT S, LanePlan P, const uint32_t *__restrict__ pr, const uint32_t *__restrict__ ps,
             uint64_t n, uint8_t *__restrict__ out, uint32_t *status, uint32_t *rest, uint32_t *counters,
             uint32_t head, uint32_t k_base, uint32_t chunk, bool stages, uint32_t fixed) {
    __shared__ uint4 s_desc[kWarpsPerBlock][2][32];
    __shared__ uint32_t s_k[kWarpsPerBlock][32];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t below = (1u << lane) - 1u;
    const uint32_t warps = gridDim.x * kWarpsPerBlock;
    uint64_t base = ((uint64_t)blockIdx.x * kWarpsPerBlock + warp) * chunk;  // the next chunk
    uint32_t cur = 0, have = 0;                                             // its pairs still to hand out: [cur, have)
    const uint32_t limit = c_wait_limit;  // a wait limit of 0 leaves every pair to the groups, which wait
    uint32_t k = 0, st = 0;
    uint4 dr = make_uint4(0, 0, 0, 0), ds = dr;
    typename LaneOf<SetsT, VAR>::T L{};
    L.mode = kLaneIdle;
    for (;;) {
        const int pick = lane_pick(L.mode, base < n || cur < have);
        if (pick < 0) break;
        if (pick < 2) {
            lane_round(L, pick, P, R, S, st);
            continue;
        }
        bool begin = false, give_up = false;
        if (L.mode == kLaneDone) {  // the verdict, or the pair's next join
            give_up = L.t == kLaneGiveUp;
            const uint32_t c = give_up ? st : (P.next >> (4u * (2u * st + L.t))) & 15u;
            if (c & 8u) out[k] = (uint8_t)(c & 7u);
            st = c;
            begin = !give_up && !(c & 8u);
            L.mode = kLaneIdle;
        }
        if (cur == have && base < n) {
            const uint64_t q = base + lane;
            bool ok = false;
            uint4 a = make_uint4(0, 0, 0, 0), b = a;
            if (lane < chunk && q < n) {
                const uint32_t r = __ldg(pr + q), s = __ldg(ps + q);
                ok = r < R.n() && s < S.n();
                if (ok) {
                    a = R.load(r);
                    b = S.load(s);
                } else {
                    out[q] = APRIL_VERDICT_ERROR;
                    atomicOr(status, ST_BAD_ID);
                }
            }
            uint32_t c = 0;
            if (lane == 0) c = atomicAdd(&counters[head], 1u);
            const uint32_t oks = __ballot_sync(kFull, ok);
            if (ok) {
                const uint32_t at = __popc(oks & below);
                s_desc[warp][0][at] = a;
                s_desc[warp][1][at] = b;
                s_k[warp][at] = (uint32_t)q;
            }
            cur = 0;
            have = __popc(oks);
            base = ((uint64_t)warps + __shfl_sync(kFull, c, 0)) * chunk;
            __syncwarp();
        }
        const uint32_t idle = __ballot_sync(kFull, L.mode == kLaneIdle && !begin && !give_up);
        const uint32_t at = cur + __popc(idle & below);
        if (((idle >> lane) & 1u) && at < have) {
            dr = s_desc[warp][0][at];
            ds = s_desc[warp][1][at];
            k = s_k[warp][at];
            st = 0;
            begin = true;
        }
        cur = min(have, cur + __popc(idle));
        if (begin) {
            const int v = lane_stage(P, dr, ds, st);
            if (v >= 0) out[k] = (uint8_t)v;
            else if (limit == 0) give_up = true;
            else lane_start(L, P, R, S, dr, ds, st, fixed, limit);
        }
        const uint32_t gm = __ballot_sync(kFull, give_up);
        if (gm) {
            const uint32_t leader = __ffs(gm) - 1;
            uint32_t pos = 0;
            if (lane == leader) pos = atomicAdd(&counters[C_REST_COUNT], __popc(gm));
            pos = __shfl_sync(kFull, pos, leader) + __popc(gm & below);
            if (give_up) rest[pos] = (k + k_base) | (stages ? st << 30 : 0u);
        }
        __syncwarp();  // the chunk's slots handed out have been read
    }
}

// ------------------- K3: several lanes per pair (batched): few or long pairs
// All n pairs of a call that has too few to fill the chip with a lane each, or
// the ones K2 left of compressed lists: each goes to G lanes, which split the
// shorter list (r's, for containment) into equal segments and leapfrog their
// own one against the whole other list; the join's answer is their OR.  A join
// of 150 rounds takes one lane about 70 us, most of it waiting on dependent
// loads, and eight lanes a sixth of that.  A warp starts with `per` pairs, its
// groups' first ones, and takes later ones, four at a time, from the counter;
// where the first ones are all there are the counter is left alone, so that it
// need not be reset for the launch.
constexpr uint32_t kFewLanes = 8;
template <class SetsT, bool VAR, uint32_t G>
__global__ void __launch_bounds__(256, APRIL_LANE_MIN_BLOCKS)
    k_persistent(SetsT R, SetsT S, LanePlan P, const uint32_t *__restrict__ pr, const uint32_t *__restrict__ ps,
                 uint64_t n, uint8_t *__restrict__ out, uint32_t *status, uint32_t *counters, uint32_t per, Rest rest) {
    if (rest.list) n = *((volatile uint32_t *)&counters[C_REST_COUNT]);
    constexpr uint32_t TAKE = 32 / kFewLanes, UNIT = SetsT::kPacked ? 16 : 4;
    const uint32_t lane = threadIdx.x & 31u, g = lane / G, t = lane % G;
    const uint32_t gbits = (0xffffffffu >> (32u - G)) << (g * G);
    const uint32_t leads = G == 32 ? 1u : G == 16 ? 0x00010001u : 0x01010101u;  // the groups' first lanes
    static_assert(G == 8 || G == 16 || G == 32, "the masks are those of groups of 8, 16 and 32 lanes");
    const uint32_t warps = gridDim.x * kWarpsPerBlock, me = blockIdx.x * kWarpsPerBlock + (threadIdx.x >> 5);
    uint64_t cur = (uint64_t)per * me, end = min(n, cur + per);
    bool more = cur < n, mine = false;                   // mine: the group has a pair
    uint32_t k = 0, st = 0;
    uint4 dr = make_uint4(0, 0, 0, 0), ds = dr;
    typename LaneOf<SetsT, VAR>::T L{};
    L.mode = kLaneIdle;
    for (;;) {
        const uint32_t over = __ballot_sync(kFull, L.mode >= kLaneDone),
                       hits = __ballot_sync(kFull, L.mode == kLaneDone && L.t == 1u);
        const bool ended = (hits & gbits) || (over & gbits) == gbits;  // the group's join (or it has none)
        if (!__any_sync(kFull, !ended || mine) && !more) break;
        if (__any_sync(kFull, ended && (mine || more))) {
            bool begin = false;
            if (ended && mine) {
                const uint32_t c = (P.next >> (4u * (2u * st + ((hits & gbits) ? 1u : 0u)))) & 15u;
                if (c & 8u) {
                    if (t == 0) out[k] = (uint8_t)(c & 7u);
                    mine = false;
                } else {
                    st = c;
                    begin = true;
                }
                L.mode = kLaneIdle;
            }
            const uint32_t need = __ballot_sync(kFull, !mine) & leads;
            if (more && need) {
                if (cur >= end) {
                    more = (uint64_t)per * warps < n;
                    if (more) {
                        uint32_t c = 0;
                        if (lane == 0) c = atomicAdd(&counters[C_CHUNK_HEAD], 1u);
                        cur = (uint64_t)per * warps + (uint64_t)TAKE * __shfl_sync(kFull, c, 0);
                        end = min(n, cur + TAKE);
                        more = cur < n;
                    }
                }
                const uint64_t q = cur + __popc(need & ((1u << (g * G)) - 1u));
                if (more && !mine && q < end) {
                    const uint32_t e = rest.entry(q);
                    k = rest.pair(e);
                    st = rest.stage(e);
                    const uint32_t r = __ldg(pr + k), s = __ldg(ps + k);
                    const bool ok = r < R.n() && s < S.n();
                    if (ok) {
                        dr = R.load(r);
                        ds = S.load(s);
                    }
                    mine = begin = ok && c_wait_limit != 0;
                    if (!mine && t == 0) {
                        out[k] = APRIL_VERDICT_ERROR;
                        atomicOr(status, ok ? ST_TIMEOUT : ST_BAD_ID);
                    }
                }
                cur = min(end, cur + __popc(need));
            }
            if (begin) {
                const int v = lane_stage(P, dr, ds, st);
                if (v >= 0) {
                    if (t == 0) out[k] = (uint8_t)v;
                    mine = false;
                } else {
                    lane_split<UNIT>(L, P, R, S, dr, ds, st, t, G);
                }
            }
            continue;
        }
        const uint32_t unit = __popc(__ballot_sync(kFull, L.mode == kLaneUnit)),
                       idx = __popc(__ballot_sync(kFull, L.mode == kLaneIndex || L.mode == kLaneSeek));
        lane_round(L, idx >= unit ? 1 : 0, P, R, S, st);
    }
}

// ----------------------------------------------- skip index of a set
// posts[q] = last cell of interval slot 16 q + 15 (see RawList::key).
__global__ void __launch_bounds__(256) k_posts(const uint2 *__restrict__ iv, uint64_t nposts,
                                               uint32_t *__restrict__ posts) {
    for (uint64_t q = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nposts;
         q += (uint64_t)gridDim.x * blockDim.x)
        posts[q] = __ldg(&iv[16 * q + 15].y) - 1u;
}

// ------------------------------------------- K6: partition routing (a-8)
// Sec. 5.2: a candidate pair is evaluated in the one partition that holds the
// lower-left corner of MBR(r) n MBR(s).  Writes the two entries (object
// approximations on that partition's grid) of every pair; an out-of-range id
// or a missing entry yields UINT32_MAX, which the filter reports as an error.
struct PartView {
    const int2 *ll;
    const uint32_t *obj_entry;
    const uint32_t *entry_pid;
    uint32_t n;
};

__device__ __forceinline__ uint32_t find_entry(const PartView &P, uint32_t obj, uint32_t pid) {
    const uint32_t e1 = __ldg(P.obj_entry + obj + 1);
    for (uint32_t e = __ldg(P.obj_entry + obj); e < e1; ++e)
        if (__ldg(P.entry_pid + e) == pid) return e;
    return 0xffffffffu;
}

__global__ void __launch_bounds__(256) k_route(PartView R, PartView S, uint32_t parts_log2,
                                               const uint32_t *__restrict__ pr, const uint32_t *__restrict__ ps,
                                               uint64_t n, uint32_t *__restrict__ er, uint32_t *__restrict__ es) {
    const uint32_t side_log2 = 24 - parts_log2, pmax = (1u << parts_log2) - 1u;
    for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
         k += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t r = __ldg(pr + k), s = __ldg(ps + k);
        uint32_t a = 0xffffffffu, b = 0xffffffffu;
        if (r < R.n && s < S.n) {
            const int2 lr = __ldg(R.ll + r), ls = __ldg(S.ll + s);
            const uint32_t x = (uint32_t)max(lr.x, ls.x), y = (uint32_t)max(lr.y, ls.y);
            const uint32_t pid = (min(y >> side_log2, pmax) << parts_log2) + min(x >> side_log2, pmax);
            a = find_entry(R, r, pid);
            b = find_entry(S, s, pid);
        }
        er[k] = a;
        es[k] = b;
    }
}

int g_num_sms = 0;

}  // namespace

int april_launch_posts(const uint32_t *iv, uint64_t iv_slots, uint32_t *posts, void *stream) {
    const uint64_t nposts = iv_slots / 16;
    if (nposts == 0) return (int)cudaSuccess;
    const unsigned grid = (unsigned)std::min<uint64_t>((nposts + 255) / 256, 152ull * 8);
    k_posts<<<grid, 256, 0, (cudaStream_t)stream>>>((const uint2 *)iv, nposts, posts);
    return (int)cudaGetLastError();
}

// What the captured launches hold: of each set every address and count that a
// kernel of the batched pipeline gets (a set uploaded again into the same
// buffer may keep some of them and move others), the pairs, verdicts and
// scratch, the tuning and the grids.
using GraphKey = std::array<uint64_t, 2 * 12 + 16>;

static GraphKey graph_key(const april_dev_sets *R, const april_dev_sets *S, const uint32_t *d_r, const uint32_t *d_s,
                          uint64_t n, const uint8_t *out, const void *scratch, bool packed, const april_tune &t,
                          unsigned grid_bin, unsigned grid_main) {
    GraphKey k{};
    size_t i = 0;
    for (const april_dev_sets *d : {R, S})
        for (uint64_t v : {(uint64_t)(uintptr_t)d->desc, (uint64_t)(uintptr_t)d->iv, (uint64_t)(uintptr_t)d->posts,
                           (uint64_t)(uintptr_t)d->pdesc, (uint64_t)(uintptr_t)d->anchors,
                           (uint64_t)(uintptr_t)d->gaps, (uint64_t)(uintptr_t)d->obj_ll,
                           (uint64_t)(uintptr_t)d->obj_entry, (uint64_t)(uintptr_t)d->entry_pid,
                           (uint64_t)d->n_objects, (uint64_t)d->n_entries, (uint64_t)d->parts})
            k[i++] = v;
    for (uint64_t v : {(uint64_t)(uintptr_t)d_r, (uint64_t)(uintptr_t)d_s, n, (uint64_t)(uintptr_t)out,
                       (uint64_t)(uintptr_t)scratch, (uint64_t)packed, (uint64_t)t.cta_threshold,
                       (uint64_t)t.group_lanes, (uint64_t)t.group_window, (uint64_t)t.cta_window,
                       (uint64_t)t.blocks_per_sm, (uint64_t)t.join_order, (uint64_t)t.escalate_windows,
                       (uint64_t)t.triage_off, (uint64_t)grid_bin, (uint64_t)grid_main})
        k[i++] = v;
    return k;
}

struct april_ctx {
    int device = 0;
    uint32_t *d_status = nullptr;  // 256-byte status block (word 0: ST_* bits)
    int num_sms = 0;
    // occupancy of k_persistent<4, 8, 16, 32> over raw lists, then over packed lists
    int persistent_blocks_per_sm[8] = {1, 1, 1, 1, 1, 1, 1, 1};
    int lane_blocks_per_sm[3] = {1, 1, 1};  // of k_triage: raw, packed, variants
    int long_blocks_per_sm = 1;  // occupancy of k_long (the larger of its two instances' limits)
    april_tune tune{};
    cudaStream_t cap_stream = nullptr;  // private stream used only to capture graphs
    // april_filter_pairs_host's pipeline (created on first use): streams for
    // the pair copies, two for the chunks' kernels, one for the verdict
    // copies, and events ordering them (start, end, per chunk: in, kernel)
    cudaStream_t pipe[4] = {nullptr, nullptr, nullptr, nullptr};
    cudaEvent_t pev[2 + 2 * 8] = {};
    cudaGraphExec_t graph = nullptr;    // the batched pipeline, captured once per argument set
    GraphKey key{};
    uint64_t graph_launches = 0;
    uint64_t graph_captures = 0;
};

using april::fail;

static april_status cuda_fail(cudaError_t e, const char *what) {
    return fail(APRIL_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

// index of a group size 4, 8, 16, 32 in the context's occupancy table
static int group_index(uint32_t g) { return g == 4 ? 0 : g == 8 ? 1 : g == 16 ? 2 : 3; }

static april_tune default_tune() {
    april_tune t{};
    // one lane per pair (the triage), then groups of this shape for the pairs it leaves
    t.cta_threshold = 0xffffffffu;
    t.group_lanes = 4;
    t.group_window = 32;
    t.cta_window = 128;      // with a threshold set: long pairs one per warp, first window 128
    t.join_order = kJoinOrderAuto;  // AF first
    t.escalate_windows = 0;  // lane groups finish every join they start
    t.triage_off = 0;        // one lane per pair first
    t.blocks_per_sm = 0;
    t.ms = 0.f;
    return t;
}

static april_status check_tune(const april_tune &t) {
    const uint32_t G = t.group_lanes;
    if (G != 4 && G != 8 && G != 16 && G != 32) return fail(APRIL_ERR_INVALID_ARG, "group_lanes must be 4, 8, 16 or 32");
    const uint32_t gmax = G == 32 ? kWarpWMax : kGroupPer * G;
    if (t.group_window < G || t.group_window > gmax || (t.group_window & (t.group_window - 1)))
        return fail(APRIL_ERR_INVALID_ARG, "group_window must be a power of two in [group_lanes, 8*group_lanes]");
    if (t.cta_window < 32 || t.cta_window > kCtaWMax || (t.cta_window & (t.cta_window - 1)))
        return fail(APRIL_ERR_INVALID_ARG, "cta_window must be a power of two in [32, 2048]");
    if (t.join_order > kJoinOrderAuto)
        return fail(APRIL_ERR_INVALID_ARG, "join_order must be 0 (AF AA FA), 1 (AA AF FA) or 2 (automatic)");
    if (t.escalate_windows > kMaxEscalateWindows) return fail(APRIL_ERR_INVALID_ARG, "escalate_windows must be 0..64");
    if (t.triage_off > 1) return fail(APRIL_ERR_INVALID_ARG, "triage_off must be 0 or 1");
    return APRIL_OK;
}

extern "C" april_status april_ctx_create(int device, april_ctx **out) {
    if (!out) return fail(APRIL_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    cudaError_t e = cudaSetDevice(device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaSetDevice");
    auto *c = new april_ctx();
    c->device = device;
    c->tune = default_tune();
    e = cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, device);
#define APRIL_OCC(I, G, SETS)                                                                                \
    if (e == cudaSuccess)                                                                                      \
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c->persistent_blocks_per_sm[I], k_persistent<G, SETS>, \
                                                          kBlock, 0)
    APRIL_OCC(0, 4, RawSets);
    APRIL_OCC(1, 8, RawSets);
    APRIL_OCC(2, 16, RawSets);
    APRIL_OCC(3, 32, RawSets);
    APRIL_OCC(4, 4, PackedSets);
    APRIL_OCC(5, 8, PackedSets);
    APRIL_OCC(6, 16, PackedSets);
    APRIL_OCC(7, 32, PackedSets);
#undef APRIL_OCC
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c->lane_blocks_per_sm[0], k_triage<RawSets, false>, kBlock, 0);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c->lane_blocks_per_sm[1], k_triage<PackedSets, false>,
                                                          kBlock, 0);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&c->lane_blocks_per_sm[2], k_triage<RawSets, true>, kBlock, 0);
    int occ_long_raw = 1, occ_long_packed = 1;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_long_raw, k_long<RawSets>, kBlock, 0);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ_long_packed, k_long<PackedSets>, kBlock, 0);
    c->long_blocks_per_sm = std::max(1, std::min(occ_long_raw, occ_long_packed));
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaMalloc(&c->d_status, 256);
    if (e == cudaSuccess) e = cudaMemset(c->d_status, 0, 256);
    if (e != cudaSuccess) {
        if (c->d_status) cudaFree(c->d_status);
        if (c->cap_stream) cudaStreamDestroy(c->cap_stream);
        delete c;
        return cuda_fail(e, "april_ctx_create");
    }
    for (int &b : c->persistent_blocks_per_sm) b = b < 1 ? 1 : b;
    for (int &b : c->lane_blocks_per_sm) b = b < 1 ? 1 : b;
    g_num_sms = c->num_sms;
    *out = c;
    return APRIL_OK;
}

extern "C" void april_ctx_destroy(april_ctx *ctx) {
    if (!ctx) return;
    if (ctx->graph) cudaGraphExecDestroy(ctx->graph);
    if (ctx->cap_stream) cudaStreamDestroy(ctx->cap_stream);
    for (cudaStream_t &p : ctx->pipe)
        if (p) cudaStreamDestroy(p);
    for (cudaEvent_t &v : ctx->pev)
        if (v) cudaEventDestroy(v);
    if (ctx->d_status) cudaFree(ctx->d_status);
    delete ctx;
}

extern "C" april_status april_set_tune(april_ctx *ctx, const april_tune *t) {
    if (!ctx || !t) return fail(APRIL_ERR_INVALID_ARG, "NULL argument");
    april_status st = check_tune(*t);
    if (st) return st;
    ctx->tune = *t;
    return APRIL_OK;
}

extern "C" april_status april_ctx_graph_stats(const april_ctx *ctx, uint64_t *captures, uint64_t *launches) {
    if (!ctx) return fail(APRIL_ERR_INVALID_ARG, "NULL context");
    if (captures) *captures = ctx->graph_captures;
    if (launches) *launches = ctx->graph_launches;
    return APRIL_OK;
}

extern "C" april_status april_get_tune(const april_ctx *ctx, april_tune *t) {
    if (!ctx || !t) return fail(APRIL_ERR_INVALID_ARG, "NULL argument");
    *t = ctx->tune;
    return APRIL_OK;
}

extern "C" april_status april_upload(const april_sets *S, void *dev_buf, size_t dev_bytes, void *stream,
                                     april_dev_sets *out) {
    if (!S || !dev_buf || !out) return fail(APRIL_ERR_INVALID_ARG, "NULL argument");
    if (((uintptr_t)dev_buf) & 255u) return fail(APRIL_ERR_INVALID_ARG, "device buffer must be 256-byte aligned");
    const april_image_layout L = april_layout(*S);
    if (dev_bytes < L.total) return fail(APRIL_ERR_INVALID_ARG, "device buffer too small");
    cudaStream_t st = (cudaStream_t)stream;
    char *base = (char *)dev_buf;
    cudaError_t e = cudaSuccess;
    auto put = [&](uint64_t off, const void *src, size_t bytes) {
        if (e == cudaSuccess && bytes) e = cudaMemcpyAsync(base + off, src, bytes, cudaMemcpyHostToDevice, st);
    };
    put(L.desc, S->desc.data(), S->desc.size() * 4);
    put(L.iv, S->iv.data(), S->iv.size() * 4);
    put(L.obj_ll, S->obj_ll.data(), S->obj_ll.size() * 4);
    put(L.obj_entry, S->obj_entry.data(), S->obj_entry.size() * 4);
    put(L.entry_pid, S->entry_pid.data(), S->entry_pid.size() * 4);
    put(L.pdesc, S->pdesc.data(), S->pdesc.size() * 4);
    put(L.anchors, S->anchors.data(), S->anchors.size() * 4);
    put(L.gaps, S->gaps.data(), S->gaps.size());
    put(L.mbr, S->mbr.data(), S->mbr.size() * 4);
    put(L.pgrid, S->part_grid.data(), S->part_grid.size() * 8);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpyAsync(upload)");
    e = (cudaError_t)april_launch_posts((const uint32_t *)(base + L.iv), S->iv.size() / 2,
                                        (uint32_t *)(base + L.posts), stream);
    if (e != cudaSuccess) return cuda_fail(e, "building the skip index (upload)");
    *out = april_dev_sets{};
    out->desc = (const uint32_t *)(base + L.desc);
    out->iv = (const uint32_t *)(base + L.iv);
    out->n_objects = S->n;
    out->order = S->order;
    out->iv_slots = S->iv.size() / 2;
    out->n_entries = S->n_entries;
    out->parts = S->parts;
    out->mbr = S->mbr.empty() ? nullptr : (const int32_t *)(base + L.mbr);
    out->posts = (const uint32_t *)(base + L.posts);
    if (S->grid_known && !S->mbr.empty()) {
        out->grid_ox = S->grid_ox;
        out->grid_oy = S->grid_oy;
        out->grid_log2_cell = S->grid_log2_cell;
        out->grid_known = 1;
        out->grid_id = S->grid_id;
        if (S->parts) out->part_grid = (const int64_t *)(base + L.pgrid);
    }
    if (S->parts) {
        out->obj_ll = (const int32_t *)(base + L.obj_ll);
        out->obj_entry = (const uint32_t *)(base + L.obj_entry);
        out->entry_pid = (const uint32_t *)(base + L.entry_pid);
    }
    if (S->packed) {
        out->pdesc = (const uint32_t *)(base + L.pdesc);
        out->anchors = (const uint32_t *)(base + L.anchors);
        out->gaps = (const uint8_t *)(base + L.gaps);
    }
    return APRIL_OK;
}

static inline uint64_t round256(uint64_t b) { return (b + 255) / 256 * 256; }

extern "C" april_status april_filter_scratch_bytes(int mode, uint64_t n, size_t *bytes) {
    if (!bytes) return fail(APRIL_ERR_INVALID_ARG, "bytes is NULL");
    switch (mode) {
        case APRIL_MODE_PLAIN:
        case APRIL_MODE_WARP: *bytes = 0; return APRIL_OK;
        case APRIL_MODE_BATCHED:
        case APRIL_MODE_BATCHED_PACKED:
            *bytes = (size_t)(kCounterBytes + 3 * round256(4 * n) + round256(16 * esc_capacity(n)));
            return APRIL_OK;
        default: return fail(APRIL_ERR_INVALID_ARG, "unknown mode");
    }
}

// The filter reads sets as april_upload / april_build_sets_device lay them
// out: interval slots 256-byte aligned (a list's place among the skip
// index's 16-slot groups follows from its address) and the skip index.
static april_status check_layout(const april_dev_sets *d) {
    if (!d->desc || !d->iv || !d->posts || (((uintptr_t)d->iv) & 255u))
        return fail(APRIL_ERR_INVALID_ARG, "device sets not laid out by april_upload or april_build_sets_device");
    return APRIL_OK;
}

// The checks april_filter_pairs makes on its sets, size and mode.
static april_status check_filter_args(const april_dev_sets *R, const april_dev_sets *S, uint64_t n, int mode) {
    if (R->order != S->order || R->parts != S->parts)
        return fail(APRIL_ERR_INVALID_ARG, "R and S are on different grids");
    if (check_layout(R) || check_layout(S)) return APRIL_ERR_INVALID_ARG;
    if (n > 0xFFFFFFFFull) return fail(APRIL_ERR_INVALID_ARG, "at most 2^32-1 pairs per call");
    if (R->parts && mode != APRIL_MODE_BATCHED && mode != APRIL_MODE_BATCHED_PACKED)
        return fail(APRIL_ERR_INVALID_ARG, "partitioned sets need APRIL_MODE_BATCHED or APRIL_MODE_BATCHED_PACKED");
    if (mode == APRIL_MODE_BATCHED_PACKED && (!R->pdesc || !S->pdesc))
        return fail(APRIL_ERR_INVALID_ARG, "APRIL_MODE_BATCHED_PACKED needs sets compressed by april_sets_compress");
    return APRIL_OK;
}

static inline DevSet dev_set(const april_dev_sets *d) {
    return DevSet{(const uint4 *)d->desc, (const uint2 *)d->iv, d->n_entries ? d->n_entries : d->n_objects,
                  d->posts};
}

static inline PackedSets packed_set(const april_dev_sets *d) {
    return PackedSets{(const uint4 *)d->pdesc, (const uint2 *)d->anchors, d->gaps,
                      d->n_entries ? d->n_entries : d->n_objects};
}

static inline PartView part_view(const april_dev_sets *d) {
    return PartView{(const int2 *)d->obj_ll, d->obj_entry, d->entry_pid, d->n_objects};
}

// Whether the pairs go to single lanes (K2, then K3 for the ones it leaves)
// instead of lane groups: a tuning with every pair in groups of 4..16 lanes.
static bool triage_applies(const april_tune &t) {
    return !t.triage_off && t.cta_threshold == kNoLongPairs && t.group_lanes < 32;
}

// The same for compressed lists, whose lanes number 16 slots per block of the
// set's block table in 32 bits: tables of 2^28 blocks (134M objects with both
// lists, say) go to the lane groups, which address blocks by pointer.  The
// table reaches up to the gap stream in the device image.
static bool lanes_number(const april_dev_sets *d) {
    return (uint64_t)((uintptr_t)d->gaps - (uintptr_t)d->anchors) / 8 < 1ull << 28;
}
static bool triage_applies(const april_tune &t, const april_dev_sets *R, const april_dev_sets *S, bool packed) {
    return triage_applies(t) && (!packed || (lanes_number(R) && lanes_number(S)));
}

// The plan of Algorithm 2's joins in join order jo (step_outcome's, with the
// automatic order AF AA FA: most pairs are true hits that AF settles).
static LanePlan lane_plan(uint32_t jo) {
    LanePlan P{};
    if (jo == 1) {  // AA, AF, FA
        P.xf = 4, P.yf = 2;
        P.next = 8u | 1u << 4 | 2u << 8 | 9u << 12 | 10u << 16 | 9u << 20;
    } else {  // AF, AA, FA
        P.xf = 4, P.yf = 1;
        P.next = 1u | 9u << 4 | 8u << 8 | 2u << 12 | 10u << 16 | 9u << 20;
    }
    return P;
}

// The first pass's grid: as many CTAs as are resident at once, at most
// APRIL_TRIAGE_GRID_PER_SM per SM.
#ifndef APRIL_TRIAGE_GRID_PER_SM
#define APRIL_TRIAGE_GRID_PER_SM 64
#endif
// Whether rest entries carry the stage: the pairs' indices leave two bits.
static inline bool rest_stages(uint64_t n) { return n <= (1ull << 30); }

// The first pass over pairs [0, n) of the arrays given (a chunk of a longer
// pair array: k_base is its place there, `head` its chunk counter).
template <bool VAR = false, class SetsT>
static void launch_triage(int num_sms, int blocks_per_sm, unsigned max_ctas, const SetsT &R, const SetsT &S,
                          const LanePlan &P, const uint32_t *d_r, const uint32_t *d_s, uint64_t n, uint8_t *out,
                          uint32_t *status, uint32_t *rest, uint32_t *counters, uint32_t head, uint32_t k_base,
                          bool stages, bool windows, cudaStream_t st) {
    const uint64_t warps = (uint64_t)num_sms * std::min(blocks_per_sm, APRIL_TRIAGE_GRID_PER_SM) * kWarpsPerBlock;
    // pairs a warp takes at a time: 32, fewer where that leaves warps without any
    const uint32_t chunk = (uint32_t)std::min<uint64_t>(32, std::max<uint64_t>(4, (n + warps - 1) / warps));
    const uint64_t want = (n + chunk * kWarpsPerBlock - 1) / (chunk * kWarpsPerBlock);
    const unsigned grid = (unsigned)std::min<uint64_t>(std::min<uint64_t>(want, warps / kWarpsPerBlock), max_ctas);
    k_triage<SetsT, VAR><<<std::max(1u, grid), 256, 0, st>>>(R, S, P, d_r, d_s, n, out, status, rest, counters, head,
                                                             k_base, chunk, stages,
                                                             windows ? 0u : kLaneFixed);
}

// The warps of a lane kernel that are resident at once.
static inline uint64_t lane_warps(int num_sms, int blocks_per_sm, unsigned max_ctas) {
    return std::max<uint64_t>(1, std::min<uint64_t>((uint64_t)num_sms * blocks_per_sm, max_ctas)) * kWarpsPerBlock;
}

// Whether a call's n pairs go to K3 at once, without a first pass.  With a
// lane per pair such a call lasts as long as its longest join, and most lanes
// idle: 20k paper-scale pairs take 70 us with a lane each, 48 with eight; 40k
// 71 and 58; 30k skewed ones 84 and 66; 30k over compressed lists 166 and 135.
// From 12 pairs a warp on the chip is full (72k skewed ones: 103 and 109 us).
static inline bool few_pairs(uint64_t n, uint64_t warps) { return n <= 8 * warps; }

// The CTAs a kernel of two warps over the rest list of a call over n pairs
// starts with.  Most calls leave none, so an empty launch must cost nothing (K7
// with sixteen an SM: 2 us of 170) and a full one most of the chip's rate: eight
// K7 CTAs an SM take 5.2 ms for 1M interleaved pairs of 500 + 500, sixteen 4.2;
// K3's sixteen 4.0, eight 4.9.
constexpr unsigned kRestCtas = 16, kRestGeneralCtas = 8;
static inline unsigned rest_grid(uint64_t n, int num_sms, unsigned max_ctas, unsigned per_sm) {
    return (unsigned)std::min<uint64_t>(std::min<uint64_t>((n + 63) / 64, (uint64_t)num_sms * per_sm), 4ull * max_ctas);
}

// K3's lanes over all n pairs of a call of few (rest is null), each warp
// starting with as few as the chip has room for, and with one or two it puts
// all its lanes on them (1,187 pairs of long lists: 44 us with eight lanes each,
// 34 with 32), or over those of its n pairs that the first pass left.
template <bool VAR = false, class SetsT>
static void launch_wide(int num_sms, int blocks_per_sm, unsigned max_ctas, const SetsT &R, const SetsT &S,
                        const LanePlan &P, const uint32_t *d_r, const uint32_t *d_s, uint64_t n, uint8_t *out,
                        uint32_t *status, const uint32_t *rest, uint32_t *counters, cudaStream_t st) {
    const uint64_t warps = lane_warps(num_sms, blocks_per_sm, max_ctas), most = warps / kWarpsPerBlock;
    const uint32_t per = rest ? 32 / kFewLanes : (uint32_t)std::min<uint64_t>(32 / kFewLanes, (n + warps - 1) / warps);
    const uint64_t cta = rest ? 256 : per * kWarpsPerBlock;  // few of a call's pairs are left by the first pass
    const unsigned grid = (unsigned)std::min<uint64_t>((n + cta - 1) / cta, most);
    const auto kernel = per == 1   ? k_persistent<SetsT, VAR, 32>
                        : per == 2 ? k_persistent<SetsT, VAR, 16>
                                   : k_persistent<SetsT, VAR, kFewLanes>;
    kernel<<<grid, 256, 0, st>>>(R, S, P, d_r, d_s, n, out, status, counters, per, Rest{rest, rest && rest_stages(n)});
}

// A call's pairs in lanes: K3 alone, or K2, which may leave some in the rest
// list (*left) for the caller's second pass.
template <bool VAR = false, class SetsT>
static cudaError_t launch_lanes(int num_sms, int blocks_per_sm, unsigned max_ctas, const SetsT &R, const SetsT &S,
                                const LanePlan &P, const uint32_t *d_r, const uint32_t *d_s, uint64_t n, uint8_t *out,
                                uint32_t *status, uint32_t *rest, uint32_t *counters, bool windows, cudaStream_t st,
                                bool *left) {
    const uint64_t warps = lane_warps(num_sms, blocks_per_sm, max_ctas);
    const bool few = few_pairs(n, warps);
    *left = !few;
    if (!few || n > 32 / kFewLanes * warps) {  // else K3 reads no counter
        const cudaError_t e = cudaMemsetAsync(counters, 0, kCounterBytes, st);
        if (e != cudaSuccess) return e;
    }
    if (few)
        launch_wide<VAR>(num_sms, blocks_per_sm, max_ctas, R, S, P, d_r, d_s, n, out, status, nullptr, counters, st);
    else
        launch_triage<VAR>(num_sms, blocks_per_sm, max_ctas, R, S, P, d_r, d_s, n, out, status, rest, counters,
                           C_LANE_HEAD, 0u, rest_stages(n), windows, st);
    return cudaGetLastError();
}

// A tuning's window shapes for joins that escalate to whole warps (k_long).
static inline uint32_t long_window(const april_tune &t) {
    return t.cta_window < kBlock ? std::min<uint32_t>(2 * t.cta_window, kWarpWMax) : 128u;
}

// The second pass over the pairs that the single lanes left (d_r, d_s: routed
// entries for partitioned sets): the lane groups, and K3b when the tuning
// escalates long joins; over compressed lists eight lanes a pair.
static cudaError_t enqueue_rest(april_ctx *ctx, const april_dev_sets *Rd, const april_dev_sets *Sd,
                                const uint32_t *d_r, const uint32_t *d_s, uint64_t n, uint8_t *out, void *scratch,
                                bool packed, unsigned max_ctas, bool windows, cudaStream_t st, uint32_t *status,
                                const uint32_t *rest) {
    uint32_t *counters = (uint32_t *)scratch;
    const april_tune &t = ctx->tune;
    const uint32_t jo = join_order_of(t.join_order);
    const RawSets R{dev_set(Rd)}, S{dev_set(Sd)};
    if (!windows) {
        if (packed)
            launch_wide(ctx->num_sms, ctx->lane_blocks_per_sm[1], max_ctas, packed_set(Rd), packed_set(Sd),
                        lane_plan(jo), d_r, d_s, n, out, status, rest, counters, st);
        else
            launch_wide(ctx->num_sms, ctx->lane_blocks_per_sm[0], max_ctas, R, S, lane_plan(jo), d_r, d_s, n, out,
                        status, rest, counters, st);
        return cudaGetLastError();
    }
    uint4 *esc = (uint4 *)((char *)scratch + kCounterBytes + 3 * round256(4 * n));
    const uint32_t esc_cap = (uint32_t)esc_capacity(n);
    const auto kernel = t.group_lanes == 4   ? k_persistent_rest<4, RawSets>
                        : t.group_lanes == 8 ? k_persistent_rest<8, RawSets>
                                             : k_persistent_rest<16, RawSets>;
    kernel<<<rest_grid(n, ctx->num_sms, max_ctas, kRestCtas), 32 * kRestWarps, 0, st>>>(
        R, S, d_r, d_s, out, status, counters, t.group_window, jo, t.escalate_windows, esc, esc_cap,
        Rest{rest, rest_stages(n)});
    if (t.escalate_windows)
        k_long<<<(unsigned)std::max(1, ctx->num_sms * ctx->long_blocks_per_sm), kBlock, 0, st>>>(
            R, S, d_r, d_s, out, status, esc, counters, esc_cap, long_window(t), jo);
    return cudaGetLastError();
}

static cudaError_t enqueue_groups(april_ctx *ctx, const april_dev_sets *Rd, const april_dev_sets *Sd,
                                  const uint32_t *d_r, const uint32_t *d_s, uint64_t n, uint8_t *out, void *scratch,
                                  bool packed, unsigned grid_main, unsigned max_ctas, cudaStream_t st,
                                  uint32_t *status);

// Enqueues the batched pipeline on `st`: counter reset, partition routing
// (partitioned sets only), then K3 with several lanes per pair of a call of
// few, or K2 with a lane per pair and K3 with lane groups over the pairs it
// left, or K4 binning and K3 with lane groups, and, when the tuning escalates long joins, K3b for
// the joins the lane groups handed over.
static cudaError_t enqueue_batched(april_ctx *ctx, const april_dev_sets *Rd, const april_dev_sets *Sd,
                                   const uint32_t *d_r, const uint32_t *d_s, uint64_t n, uint8_t *out, void *scratch,
                                   bool packed, unsigned grid_bin, unsigned grid_main, unsigned max_ctas,
                                   bool windows, cudaStream_t st, uint32_t *status = nullptr) {
    if (!status) status = ctx->d_status;
    uint32_t *counters = (uint32_t *)scratch;
    uint32_t *big_list = (uint32_t *)((char *)scratch + kCounterBytes);
    const april_tune &t = ctx->tune;
    if (Rd->parts) {
        uint32_t *er = (uint32_t *)((char *)scratch + kCounterBytes + round256(4 * n));
        uint32_t *es = (uint32_t *)((char *)scratch + kCounterBytes + 2 * round256(4 * n));
        uint32_t lg = 0;
        while ((1u << lg) < Rd->parts) ++lg;
        k_route<<<grid_bin, 256, 0, st>>>(part_view(Rd), part_view(Sd), lg, d_r, d_s, n, er, es);
        d_r = er;
        d_s = es;
    }
    if (triage_applies(t, Rd, Sd, packed)) {
        const LanePlan P = lane_plan(join_order_of(t.join_order));
        bool left = false;
        const cudaError_t e =
            packed ? launch_lanes(ctx->num_sms, ctx->lane_blocks_per_sm[1], max_ctas, packed_set(Rd), packed_set(Sd),
                                  P, d_r, d_s, n, out, status, big_list, counters, windows, st, &left)
                   : launch_lanes(ctx->num_sms, ctx->lane_blocks_per_sm[0], max_ctas, RawSets{dev_set(Rd)},
                                  RawSets{dev_set(Sd)}, P, d_r, d_s, n, out, status, big_list, counters, windows, st,
                                  &left);
        if (e != cudaSuccess || !left) return e;
        return enqueue_rest(ctx, Rd, Sd, d_r, d_s, n, out, scratch, packed, max_ctas, windows, st, status, big_list);
    }
    const cudaError_t e = cudaMemsetAsync(counters, 0, kCounterBytes, st);
    if (e != cudaSuccess) return e;
    if (t.cta_threshold != kNoLongPairs) {
        if (packed)
            k_bin<<<grid_bin, 256, 0, st>>>(packed_set(Rd), packed_set(Sd), d_r, d_s, n, out, status, t.cta_threshold,
                                            big_list, counters);
        else
            k_bin<<<grid_bin, 256, 0, st>>>(RawSets{dev_set(Rd)}, RawSets{dev_set(Sd)}, d_r, d_s, n, out, status,
                                            t.cta_threshold, big_list, counters);
    }
    return enqueue_groups(ctx, Rd, Sd, d_r, d_s, n, out, scratch, packed, grid_main, max_ctas, st, status);
}

// The lane groups over all the pairs (d_r, d_s: routed entries for partitioned
// sets), and K3b when the tuning escalates long joins.
static cudaError_t enqueue_groups(april_ctx *ctx, const april_dev_sets *Rd, const april_dev_sets *Sd,
                                  const uint32_t *d_r, const uint32_t *d_s, uint64_t n, uint8_t *out, void *scratch,
                                  bool packed, unsigned grid_main, unsigned max_ctas, cudaStream_t st,
                                  uint32_t *status) {
    uint32_t *counters = (uint32_t *)scratch;
    grid_main = std::min(grid_main, max_ctas);
    uint32_t *big_list = (uint32_t *)((char *)scratch + kCounterBytes);
    uint4 *esc = (uint4 *)((char *)scratch + kCounterBytes + 3 * round256(4 * n));
    const april_tune &t = ctx->tune;
    const uint32_t escw = t.group_lanes < 32 ? t.escalate_windows : 0u;
    const uint32_t w0_long = long_window(t);
    const uint32_t esc_cap = (uint32_t)esc_capacity(n);
    const unsigned grid_long = (unsigned)std::max(1, ctx->num_sms * ctx->long_blocks_per_sm);
    const uint32_t jo = join_order_of(t.join_order);
    if (packed) {
        const PackedSets R = packed_set(Rd), S = packed_set(Sd);
#define APRIL_LAUNCH_PACKED(G)                                                                                  \
    k_persistent<G, PackedSets><<<grid_main, kBlock, 0, st>>>(R, S, d_r, d_s, n, out, status, t.cta_threshold,   \
                                                              big_list, counters, t.group_window, t.cta_window,   \
                                                              jo, escw, esc, esc_cap)
        switch (t.group_lanes) {
            case 4: APRIL_LAUNCH_PACKED(4); break;
            case 8: APRIL_LAUNCH_PACKED(8); break;
            case 16: APRIL_LAUNCH_PACKED(16); break;
            default: APRIL_LAUNCH_PACKED(32); break;
        }
#undef APRIL_LAUNCH_PACKED
        if (escw)
            k_long<<<grid_long, kBlock, 0, st>>>(R, S, d_r, d_s, out, status, esc, counters, esc_cap, w0_long, jo);
        return cudaGetLastError();
    }
    const RawSets R{dev_set(Rd)}, S{dev_set(Sd)};
#define APRIL_LAUNCH_PERSISTENT(G)                                                                            \
    k_persistent<G, RawSets><<<grid_main, kBlock, 0, st>>>(R, S, d_r, d_s, n, out, status, t.cta_threshold,       \
                                                           big_list, counters, t.group_window, t.cta_window,      \
                                                           jo, escw, esc, esc_cap)
    switch (t.group_lanes) {
        case 4: APRIL_LAUNCH_PERSISTENT(4); break;
        case 8: APRIL_LAUNCH_PERSISTENT(8); break;
        case 16: APRIL_LAUNCH_PERSISTENT(16); break;
        default: APRIL_LAUNCH_PERSISTENT(32); break;
    }
#undef APRIL_LAUNCH_PERSISTENT
    if (escw)
        k_long<<<grid_long, kBlock, 0, st>>>(R, S, d_r, d_s, out, status, esc, counters, esc_cap, w0_long, jo);
    return cudaGetLastError();
}

// The most CTAs a lane kernel may run with the context's tuning (april_tune.blocks_per_sm).
static unsigned tuned_ctas(const april_ctx *ctx) {
    const uint64_t b = ctx->tune.blocks_per_sm;
    return b ? (unsigned)std::min<uint64_t>((uint64_t)ctx->num_sms * b, 0xffffffffu) : 0xffffffffu;
}

// The batched pipeline runs as one CUDA graph: captured on the context's
// private stream the first time an argument set is seen, then replayed on the
// caller's stream.
static april_status launch_batched(april_ctx *ctx, const april_dev_sets *R, const april_dev_sets *S,
                                   const uint32_t *d_r, const uint32_t *d_s, uint64_t n, uint8_t *out,
                                   void *scratch, bool packed, cudaStream_t st) {
    const unsigned grid_bin = (unsigned)std::min<uint64_t>((n + 255) / 256, (uint64_t)ctx->num_sms * 8);
    const uint32_t gl = ctx->tune.group_lanes;
    const int occ = ctx->persistent_blocks_per_sm[(packed ? 4 : 0) + group_index(gl)];
    const int bps = ctx->tune.blocks_per_sm ? (int)std::min<uint32_t>(ctx->tune.blocks_per_sm, (uint32_t)occ) : occ;
    const unsigned grid_main = (unsigned)std::max(1, ctx->num_sms * bps);
    const GraphKey key = graph_key(R, S, d_r, d_s, n, out, scratch, packed, ctx->tune, grid_bin, grid_main);
    cudaError_t e;
    if (!ctx->graph || key != ctx->key) {
        if (ctx->graph) {
            cudaGraphExecDestroy(ctx->graph);
            ctx->graph = nullptr;
        }
        cudaGraph_t g = nullptr;
        e = cudaStreamBeginCapture(ctx->cap_stream, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) return cuda_fail(e, "cudaStreamBeginCapture");
        cudaError_t e1 = enqueue_batched(ctx, R, S, d_r, d_s, n, out, scratch, packed, grid_bin, grid_main,
                                         tuned_ctas(ctx), !packed, ctx->cap_stream);
        e = cudaStreamEndCapture(ctx->cap_stream, &g);
        if (e1 != cudaSuccess) e = e1;
        if (e == cudaSuccess) e = cudaGraphInstantiate(&ctx->graph, g, 0);
        if (g) cudaGraphDestroy(g);
        if (e != cudaSuccess) {
            ctx->graph = nullptr;
            return cuda_fail(e, "capturing the batched pipeline");
        }
        ctx->key = key;
        ctx->graph_captures++;
    }
    e = cudaGraphLaunch(ctx->graph, st);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGraphLaunch");
    ctx->graph_launches++;
    return APRIL_OK;
}

// Batched filter of one serving request (see server.cu): plain launches on
// `st` (no graph: every request has its own buffers), at most `max_ctas`
// persistent CTAs so that small requests leave SMs to the requests they
// overlap with, and a per-request status word.  A request that is not `alone`
// on the GPU does without the merge windows: with other requests' lanes on
// every SM, their kernel's launch over an empty list cost 24 overlapping
// requests 3 to 4% (1,215 us, 1,255 with it).
april_status april_enqueue_request(april_ctx *ctx, const april_dev_sets *R, const april_dev_sets *S,
                                   const uint32_t *d_r, const uint32_t *d_s, uint64_t n, uint8_t *d_verdict,
                                   void *d_scratch, uint32_t *d_status, unsigned max_ctas, bool alone, void *stream) {
    if (n == 0) return APRIL_OK;
    if (check_layout(R) || check_layout(S)) return APRIL_ERR_INVALID_ARG;
    const bool packed = false;  // serving reads the raw lists
    const unsigned grid_bin = (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((n + 255) / 256, (uint64_t)ctx->num_sms * 8));
    const uint32_t gl = ctx->tune.group_lanes;
    const int occ = ctx->persistent_blocks_per_sm[(packed ? 4 : 0) + group_index(gl)];
    const unsigned grid_main = (unsigned)std::max(1, ctx->num_sms * occ);
    cudaError_t e = enqueue_batched(ctx, R, S, d_r, d_s, n, d_verdict, d_scratch, packed, grid_bin, grid_main,
                                    std::max<unsigned>(1, max_ctas), alone, (cudaStream_t)stream, d_status);
    if (e != cudaSuccess) return cuda_fail(e, "enqueueing a serving request");
    return APRIL_OK;
}

int april_ctx_num_sms(const april_ctx *ctx) { return ctx->num_sms; }
int april_ctx_device(const april_ctx *ctx) { return ctx->device; }
uint32_t *april_ctx_status_word(april_ctx *ctx) { return ctx->d_status; }

extern "C" april_status april_filter_pairs(april_ctx *ctx, const april_dev_sets *R, const april_dev_sets *S,
                                           const uint32_t *d_r, const uint32_t *d_s, uint64_t n,
                                           uint8_t *d_verdict, int mode, void *d_scratch, size_t scratch_bytes,
                                           void *stream) {
    if (!ctx || !R || !S) return fail(APRIL_ERR_INVALID_ARG, "NULL argument");
    if (n == 0) return APRIL_OK;
    if (!d_r || !d_s || !d_verdict) return fail(APRIL_ERR_INVALID_ARG, "NULL pair or verdict array");
    const april_status chk = check_filter_args(R, S, n, mode);
    if (chk) return chk;
    cudaStream_t st = (cudaStream_t)stream;
    const DevSet dR = dev_set(R), dS = dev_set(S);
    const int sms = ctx->num_sms;
    switch (mode) {
        case APRIL_MODE_PLAIN: {
            uint64_t blocks = (n + 255) / 256;
            unsigned grid = (unsigned)std::min<uint64_t>(blocks, (uint64_t)sms * 8);
            k_plain<<<grid, 256, 0, st>>>(dR, dS, d_r, d_s, n, d_verdict, ctx->d_status);
            break;
        }
        case APRIL_MODE_WARP: {
            uint64_t blocks = (n + kBlock - 1) / kBlock;
            unsigned grid = (unsigned)std::min<uint64_t>(blocks, (uint64_t)sms * 16);
            k_warp<<<grid, kBlock, 0, st>>>(dR, dS, d_r, d_s, n, d_verdict, ctx->d_status, kWarpFirstWindow,
                                            join_order_of(ctx->tune.join_order));
            break;
        }
        case APRIL_MODE_BATCHED:
        case APRIL_MODE_BATCHED_PACKED: {
            size_t need = 0;
            april_filter_scratch_bytes(mode, n, &need);
            if (!d_scratch || scratch_bytes < need) return fail(APRIL_ERR_INVALID_ARG, "scratch missing or too small");
            if (((uintptr_t)d_scratch) & 255u) return fail(APRIL_ERR_INVALID_ARG, "scratch must be 256-byte aligned");
            return launch_batched(ctx, R, S, d_r, d_s, n, d_verdict, d_scratch, mode == APRIL_MODE_BATCHED_PACKED, st);
        }
        default: return fail(APRIL_ERR_INVALID_ARG, "unknown mode");
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "kernel launch");
    return APRIL_OK;
}

// Decision plans (see K7).  Verdict v is encoded as -(v + 1).
static Plan make_plan(int predicate, uint32_t order_r, uint32_t order_s, uint32_t jo) {
    Plan P{};
    const int8_t TN = -1, TH = -2, INC = -3;
    if (predicate == APRIL_PREDICATE_WITHIN) {
        // Sec. 4.3.2: AA (no overlap: not within), then "every A(r) interval
        // lies in one F(s) interval" (yes: within; a violation: refine)
        P.nst = 2;
        P.xf[0] = 0; P.yf[0] = 0; P.pred[0] = kOverlap; P.on_true[0] = 1; P.on_false[0] = TN;
        P.xf[1] = 0; P.yf[1] = 1; P.pred[1] = kContain; P.on_true[1] = INC; P.on_false[1] = TH;
        return P;
    }
    // intersects in join order jo (step_outcome): 1 is Algorithm 2's AA AF FA
    // (for different granularity: AA, then the coarse side's F-list join)
    if (jo == 1) {
        P.xf[0] = 0; P.yf[0] = 0; P.pred[0] = kOverlap; P.on_true[0] = 1; P.on_false[0] = TN;
        if (order_r == order_s) {
            P.nst = 3;
            P.xf[1] = 0; P.yf[1] = 1; P.pred[1] = kOverlap; P.on_true[1] = TH; P.on_false[1] = 2;
            P.xf[2] = 1; P.yf[2] = 0; P.pred[2] = kOverlap; P.on_true[2] = TH; P.on_false[2] = INC;
        } else {
            P.nst = 2;
            const bool r_finer = order_r > order_s;
            P.sx = r_finer ? (uint8_t)(2 * (order_r - order_s)) : 0;
            P.sy = r_finer ? 0 : (uint8_t)(2 * (order_s - order_r));
            P.xf[1] = r_finer ? 0 : 1; P.yf[1] = r_finer ? 1 : 0; P.pred[1] = kOverlap;
            P.on_true[1] = TH; P.on_false[1] = INC;
        }
        return P;
    }
    if (order_r == order_s) {  // Algorithm 2's verdicts in the order AF, AA, FA
        P.nst = 3;
        P.xf[0] = 0; P.yf[0] = 1; P.pred[0] = kOverlap; P.on_true[0] = TH; P.on_false[0] = 1;
        P.xf[1] = 0; P.yf[1] = 0; P.pred[1] = kOverlap; P.on_true[1] = 2; P.on_false[1] = TN;
        P.xf[2] = 1; P.yf[2] = 0; P.pred[2] = kOverlap; P.on_true[2] = TH; P.on_false[2] = INC;
    } else if (order_r > order_s) {  // Sec. 5.3: coarsen r, use only the coarse side's F-list
        P.nst = 2;
        P.sx = (uint8_t)(2 * (order_r - order_s));
        P.xf[0] = 0; P.yf[0] = 1; P.pred[0] = kOverlap; P.on_true[0] = TH; P.on_false[0] = 1;
        P.xf[1] = 0; P.yf[1] = 0; P.pred[1] = kOverlap; P.on_true[1] = INC; P.on_false[1] = TN;
    } else {
        P.nst = 2;
        P.sy = (uint8_t)(2 * (order_s - order_r));
        P.xf[0] = 1; P.yf[0] = 0; P.pred[0] = kOverlap; P.on_true[0] = TH; P.on_false[0] = 1;
        P.xf[1] = 0; P.yf[1] = 0; P.pred[1] = kOverlap; P.on_true[1] = INC; P.on_false[1] = TN;
    }
    return P;
}

// A variant's plan in the lanes' form.
static LanePlan lane_plan_of(const Plan &P) {
    LanePlan L{};
    auto code = [](int8_t v) { return v < 0 ? 8u + (uint32_t)(-(v + 1)) : (uint32_t)v; };
    for (uint32_t k = 0; k < P.nst; ++k) {
        L.xf |= (uint32_t)P.xf[k] << k;
        L.yf |= (uint32_t)P.yf[k] << k;
        L.contain |= (P.pred[k] == kContain ? 1u : 0u) << k;
        L.next |= code(P.on_false[k]) << (8 * k) | code(P.on_true[k]) << (8 * k + 4);
    }
    L.v.sx = P.sx;
    L.v.sy = P.sy;
    return L;
}

extern "C" april_status april_filter_pairs_ex(april_ctx *ctx, const april_dev_sets *R, const april_dev_sets *S,
                                              const uint32_t *d_r, const uint32_t *d_s, uint64_t n,
                                              uint8_t *d_verdict, int predicate, void *d_scratch,
                                              size_t scratch_bytes, void *stream) {
    if (!ctx || !R || !S) return fail(APRIL_ERR_INVALID_ARG, "NULL argument");
    if (n == 0) return APRIL_OK;
    if (!d_r || !d_s || !d_verdict) return fail(APRIL_ERR_INVALID_ARG, "NULL pair or verdict array");
    if (predicate != APRIL_PREDICATE_INTERSECTS && predicate != APRIL_PREDICATE_WITHIN)
        return fail(APRIL_ERR_INVALID_ARG, "unknown predicate");
    if (R->parts || S->parts) return fail(APRIL_ERR_INVALID_ARG, "april_filter_pairs_ex takes sets on one global grid");
    if (check_layout(R) || check_layout(S)) return APRIL_ERR_INVALID_ARG;
    if (predicate == APRIL_PREDICATE_WITHIN && R->order != S->order)
        return fail(APRIL_ERR_INVALID_ARG, "the within filter needs both sets on the same grid");
    if (n > 0xFFFFFFFFull) return fail(APRIL_ERR_INVALID_ARG, "at most 2^32-1 pairs per call");
    size_t need = 0;
    april_filter_scratch_bytes(APRIL_MODE_BATCHED, n, &need);
    if (!d_scratch || scratch_bytes < need) return fail(APRIL_ERR_INVALID_ARG, "scratch missing or too small");
    if (((uintptr_t)d_scratch) & 255u) return fail(APRIL_ERR_INVALID_ARG, "scratch must be 256-byte aligned");
    cudaStream_t st = (cudaStream_t)stream;
    uint32_t *counters = (uint32_t *)d_scratch;
    uint32_t *big_list = (uint32_t *)((char *)d_scratch + kCounterBytes);
    const RawSets dR{dev_set(R)}, dS{dev_set(S)};
    const Plan P = make_plan(predicate, R->order, S->order, join_order_of(ctx->tune.join_order));
    const unsigned grid_bin = (unsigned)std::min<uint64_t>((n + 255) / 256, (uint64_t)ctx->num_sms * 8);
    cudaError_t e;
    const april_tune &t = ctx->tune;
    if (triage_applies(t)) {  // in lanes, as for the batched filter, and K7 for the pairs left
        const LanePlan L = lane_plan_of(P);
        bool left = false;
        e = launch_lanes<true>(ctx->num_sms, ctx->lane_blocks_per_sm[2], 0xffffffffu, dR, dS, L, d_r, d_s, n, d_verdict,
                               ctx->d_status, big_list, counters, true, st, &left);
        if (e == cudaSuccess && left) {
            k_rest_general<<<rest_grid(n, ctx->num_sms, 0xffffffffu, kRestGeneralCtas), 32 * kRestWarps, 0, st>>>(
                P, dR.s, dS.s, d_r, d_s, d_verdict, ctx->d_status, counters, Rest{big_list, rest_stages(n)});
            e = cudaGetLastError();
        }
    } else {
        e = cudaMemsetAsync(counters, 0, kCounterBytes, st);
        if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync");
        int bps = 1;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k_general, kBlock, 0);
        const unsigned grid_main = (unsigned)std::max(1, ctx->num_sms * std::max(bps, 1));
        k_bin<<<grid_bin, 256, 0, st>>>(dR, dS, d_r, d_s, n, d_verdict, ctx->d_status, t.cta_threshold, big_list,
                                        counters);
        k_general<<<grid_main, kBlock, 0, st>>>(P, dR.s, dS.s, d_r, d_s, n, d_verdict, ctx->d_status, t.cta_threshold,
                                                big_list, counters, t.cta_window);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return cuda_fail(e, "kernel launch");
    return APRIL_OK;
}

extern "C" april_status april_autotune(april_ctx *ctx, const april_dev_sets *R, const april_dev_sets *S,
                                       const uint32_t *d_r, const uint32_t *d_s, uint64_t n, uint8_t *d_verdict,
                                       void *d_scratch, size_t scratch_bytes, void *stream, april_tune *out) {
    if (!ctx || !R || !S || !out) return fail(APRIL_ERR_INVALID_ARG, "NULL argument");
    if (n == 0) {
        *out = ctx->tune;
        return APRIL_OK;
    }
    cudaStream_t st = (cudaStream_t)stream;
    const uint32_t thresholds[] = {2048, 4096, 8192, 16384, kNoLongPairs};
    const uint32_t groups[][2] = {{4, 8}, {4, 16}, {4, 32}, {8, 16}, {8, 32}, {8, 64}, {16, 32}, {16, 64}, {16, 128},
                                  {32, 64}};
    const april_tune saved = ctx->tune;
    april_tune best = saved;
    float best_ms = 1e30f;
    cudaEvent_t a = nullptr, b = nullptr;
    cudaError_t e = cudaEventCreate(&a);
    if (e == cudaSuccess) e = cudaEventCreate(&b);
    if (e != cudaSuccess) return cuda_fail(e, "cudaEventCreate");
    april_status rc = APRIL_OK;
    // times tuning t on the sample (best of three replays after the capture)
    auto time_tune = [&](const april_tune &t, float &best_here) -> april_status {
        ctx->tune = t;
        best_here = 1e30f;
        for (int rep = 0; rep < 4; ++rep) {
            cudaError_t e2 = cudaEventRecord(a, st);
            if (e2 != cudaSuccess) return cuda_fail(e2, "cudaEventRecord");
            april_status r2 = april_filter_pairs(ctx, R, S, d_r, d_s, n, d_verdict, APRIL_MODE_BATCHED, d_scratch,
                                                 scratch_bytes, stream);
            if (r2) return r2;
            e2 = cudaEventRecord(b, st);
            if (e2 == cudaSuccess) e2 = cudaEventSynchronize(b);
            float ms = 0.f;
            if (e2 == cudaSuccess) e2 = cudaEventElapsedTime(&ms, a, b);
            if (e2 != cudaSuccess) return cuda_fail(e2, "timing an autotune candidate");
            if (rep > 0) best_here = std::min(best_here, ms);  // rep 0 captures the graph
        }
        return APRIL_OK;
    };
    // the context's tuning first: a candidate replaces it only if it is more
    // than 2% faster, so that the pick does not flip between shapes whose
    // times differ by noise
    float saved_ms = 1e30f;
    rc = time_tune(saved, saved_ms);
    // long pairs joined by one warp (first window 64 or 128) or by the whole CTA
    const uint32_t long_windows[] = {64u, 128u, saved.cta_window >= kBlock ? saved.cta_window : kBlock};
    auto candidate = [&](const april_tune &t) {
        float best_here = 1e30f;
        rc = time_tune(t, best_here);
        if (rc == APRIL_OK && best_here < best_ms) {
            best_ms = best_here;
            best = t;
        }
    };
    for (uint32_t jo = 0; jo < 2; ++jo) {
        april_tune t = saved;
        t.join_order = jo;
        // the single lanes, which read no group shape: one candidate
        const april_tune d = default_tune();
        t.cta_threshold = kNoLongPairs;
        t.group_lanes = d.group_lanes;
        t.group_window = d.group_window;
        t.triage_off = 0;
        if (rc == APRIL_OK) candidate(t);
        for (uint32_t T : thresholds)
            for (const auto &gw : groups)
                for (const uint32_t lw : long_windows) {
                    if (T == kNoLongPairs && lw != long_windows[0]) continue;  // no long pairs: one scope is enough
                    t.cta_threshold = T;
                    t.group_lanes = gw[0];
                    t.group_window = gw[1];
                    t.cta_window = lw;
                    t.triage_off = T == kNoLongPairs ? 1 : saved.triage_off;  // without a threshold, else lanes again
                    if (rc == APRIL_OK) candidate(t);
                }
    }
    if (rc == APRIL_OK && saved_ms <= 1.02f * best_ms) {
        best = saved;
        best_ms = saved_ms;
    }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    if (rc) {
        ctx->tune = saved;
        return rc;
    }
    best.ms = best_ms;
    ctx->tune = best;
    *out = best;
    return APRIL_OK;
}

// april_filter_pairs_host in the batched modes pipelines the pairs in chunks
// of at least kPipeChunkMin pairs (at most kPipeMaxChunks): a chunk's pairs
// are copied in while the previous chunk is filtered, and its verdicts are
// copied out while the next one is.  Chunks alternate between two kernel
// streams, each with its own scratch, so that one chunk's tail overlaps the
// next chunk's start.  Each chunk costs a launch and a tail, which measured
// more than the copies it hides below 2^22 pairs (the end-to-end overhead is
// mostly fixed latency); 10M pairs in three chunks end 5% sooner than in one.
#ifndef APRIL_PIPE_CHUNK_LOG2
#define APRIL_PIPE_CHUNK_LOG2 22
#endif
constexpr uint64_t kPipeChunkMin = 1ull << APRIL_PIPE_CHUNK_LOG2;
constexpr uint32_t kPipeMaxChunks = 8;
static uint32_t pipe_chunks(uint64_t n) {
    return (uint32_t)std::min<uint64_t>(kPipeMaxChunks, std::max<uint64_t>(1, (n + kPipeChunkMin - 1) / kPipeChunkMin));
}
static uint64_t pipe_chunk_size(uint64_t n) {
    const uint32_t k = pipe_chunks(n);
    return ((n + k - 1) / k + 63) / 64 * 64;
}

// With the triage (K2), the pipeline is finer, and only pairs that the device
// cannot read in place come to it: they are copied in
// chunks that double from kTriageChunk0 pairs up to kTriageChunkMax (at most
// kPipeMaxChunks, the last one taking what is left), and each chunk is
// triaged on one of two kernel streams as soon as it has arrived, while the
// next one is copied.  The triage appends to one rest list over all n pairs
// (indices plus the chunk's offset), which one launch then joins, and the
// verdicts are copied out.  The copies hide behind the triage.
constexpr uint64_t kTriageChunk0 = 1ull << 18;
constexpr uint64_t kTriageChunkMax = 1ull << 21;

extern "C" april_status april_filter_host_work_bytes(int mode, uint64_t n, size_t *bytes) {
    if (!bytes) return fail(APRIL_ERR_INVALID_ARG, "bytes is NULL");
    size_t sb = 0;
    april_status st = april_filter_scratch_bytes(mode, n, &sb);
    if (st) return st;
    if (mode == APRIL_MODE_BATCHED || mode == APRIL_MODE_BATCHED_PACKED) {
        size_t sc = 0;  // per chunk, one region per kernel stream; the triage pipeline takes n's
        april_filter_scratch_bytes(mode, pipe_chunk_size(n), &sc);
        sb = std::max<size_t>(round256(sb), round256(sc) * (pipe_chunks(n) > 1 ? 2 : 1));
    }
    *bytes = (size_t)(round256(4 * n) * 2 + round256(n) + round256(sb));
    return APRIL_OK;
}

static april_status ensure_pipeline(april_ctx *ctx) {
    if (ctx->pipe[0]) return APRIL_OK;
    cudaError_t e = cudaSuccess;
    for (cudaStream_t &p : ctx->pipe)
        if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&p, cudaStreamNonBlocking);
    for (cudaEvent_t &v : ctx->pev)
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&v, cudaEventDisableTiming);
    if (e != cudaSuccess) {
        for (cudaStream_t &p : ctx->pipe)
            if (p) cudaStreamDestroy(p), p = nullptr;
        for (cudaEvent_t &v : ctx->pev)
            if (v) cudaEventDestroy(v), v = nullptr;
        return cuda_fail(e, "creating the host pipeline's streams");
    }
    return APRIL_OK;
}

// The triage of pairs [off, off + cnt) of a call over n pairs (partition
// routing first for partitioned sets), appending to the call's rest list.
template <class SetsT>
static void enqueue_triage_chunk(april_ctx *ctx, const SetsT &R, const SetsT &S, const april_dev_sets *Rd,
                                 const april_dev_sets *Sd, const uint32_t *d_r, const uint32_t *d_s, uint64_t n,
                                 uint64_t off, uint64_t cnt, uint32_t chunk, uint8_t *out, void *scratch,
                                 cudaStream_t st) {
    uint32_t *counters = (uint32_t *)scratch;
    uint32_t *big_list = (uint32_t *)((char *)scratch + kCounterBytes);
    const unsigned grid_bin = (unsigned)std::min<uint64_t>((cnt + 255) / 256, (uint64_t)ctx->num_sms * 8);
    d_r += off;
    d_s += off;
    if (Rd->parts) {
        uint32_t *er = (uint32_t *)((char *)scratch + kCounterBytes + round256(4 * n)) + off;
        uint32_t *es = (uint32_t *)((char *)scratch + kCounterBytes + 2 * round256(4 * n)) + off;
        uint32_t lg = 0;
        while ((1u << lg) < Rd->parts) ++lg;
        k_route<<<grid_bin, 256, 0, st>>>(part_view(Rd), part_view(Sd), lg, d_r, d_s, cnt, er, es);
        d_r = er;
        d_s = es;
    }
    launch_triage(ctx->num_sms, ctx->lane_blocks_per_sm[SetsT::kPacked ? 1 : 0], tuned_ctas(ctx), R, S,
                  lane_plan(join_order_of(ctx->tune.join_order)), d_r, d_s, cnt, out + off, ctx->d_status, big_list,
                  counters, C_LANE_HEAD + chunk, (uint32_t)off, rest_stages(n), !SetsT::kPacked, st);
}

static cudaError_t host_triage_pipeline(april_ctx *ctx, const april_dev_sets *R, const april_dev_sets *S,
                                        const uint32_t *h_r, const uint32_t *h_s, uint64_t n, uint8_t *h_verdict,
                                        uint32_t *d_r, uint32_t *d_s, uint8_t *d_v, void *d_scr, bool packed) {
    cudaStream_t s_in = ctx->pipe[0], k1 = ctx->pipe[1], k2 = ctx->pipe[2];
    cudaError_t e = cudaMemsetAsync(d_scr, 0, kCounterBytes, k1);
    if (e == cudaSuccess) e = cudaEventRecord(ctx->pev[3], k1);  // the counters are reset
    if (e == cudaSuccess) e = cudaStreamWaitEvent(k2, ctx->pev[3], 0);
    uint64_t off = 0;
    for (uint32_t c = 0; off < n && e == cudaSuccess; ++c) {
        const uint64_t take = c + 1 == kPipeMaxChunks
                                  ? n - off
                                  : std::min<uint64_t>(std::min<uint64_t>(kTriageChunk0 << c, kTriageChunkMax), n - off);
        cudaStream_t ks = c & 1u ? k2 : k1;
        e = cudaMemcpyAsync(d_r + off, h_r + off, 4 * take, cudaMemcpyHostToDevice, s_in);
        if (e == cudaSuccess) e = cudaMemcpyAsync(d_s + off, h_s + off, 4 * take, cudaMemcpyHostToDevice, s_in);
        if (e == cudaSuccess) e = cudaEventRecord(ctx->pev[2 + 2 * c], s_in);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(ks, ctx->pev[2 + 2 * c], 0);
        if (e == cudaSuccess) {
            if (packed)
                enqueue_triage_chunk(ctx, packed_set(R), packed_set(S), R, S, d_r, d_s, n, off, take, c, d_v, d_scr,
                                     ks);
            else
                enqueue_triage_chunk(ctx, RawSets{dev_set(R)}, RawSets{dev_set(S)}, R, S, d_r, d_s, n, off, take, c,
                                     d_v, d_scr, ks);
            e = cudaGetLastError();
        }
        off += take;
    }
    // the rest list follows once both kernel streams' triages are done
    if (e == cudaSuccess) e = cudaEventRecord(ctx->pev[5], k2);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(k1, ctx->pev[5], 0);
    if (e == cudaSuccess) {
        const uint32_t *er = (const uint32_t *)((char *)d_scr + kCounterBytes + round256(4 * n));
        const uint32_t *es = (const uint32_t *)((char *)d_scr + kCounterBytes + 2 * round256(4 * n));
        e = enqueue_rest(ctx, R, S, R->parts ? er : d_r, R->parts ? es : d_s, n, d_v, d_scr, packed, tuned_ctas(ctx),
                         !packed, k1, ctx->d_status, (const uint32_t *)((char *)d_scr + kCounterBytes));
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(h_verdict, d_v, n, cudaMemcpyDeviceToHost, k1);
    return e;
}

// The device's address of the n words at host address h, where they lie in one
// page-locked allocation or registration (nullptr: elsewhere, or not aligned).
// The first pass reads each pair once, 32 of them by one load per array, so it
// can as well read them over the link: 2M pairs take 407 us that way, and 520
// copied in and filtered in overlapping chunks, whose launches and tails cost
// more than the copies (1,000 pairs: 50 us, copied in first 60).
static const uint32_t *pinned_words(const uint32_t *h, uint64_t n) {
    using Attribute = CUresult (*)(void *, CUpointer_attribute, CUdeviceptr);
    static const Attribute attribute = [] {
        void *f = nullptr;
        cudaDriverEntryPointQueryResult found;
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuPointerGetAttribute", &f, 12000, cudaEnableDefault, &found);
        return e == cudaSuccess && found == cudaDriverEntryPointSuccess ? (Attribute)f : nullptr;
    }();
    cudaPointerAttributes a{};
    if (((uintptr_t)h & 3u) || cudaPointerGetAttributes(&a, h) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    if (a.type != cudaMemoryTypeHost || !a.devicePointer || !attribute) return nullptr;
    const CUdeviceptr p = (CUdeviceptr)(uintptr_t)h;
    CUdeviceptr start = 0;
    size_t size = 0;
    if (attribute(&start, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, p) != CUDA_SUCCESS ||
        attribute(&size, CU_POINTER_ATTRIBUTE_RANGE_SIZE, p) != CUDA_SUCCESS || p < start || p + 4 * n > start + size)
        return nullptr;
    return (const uint32_t *)a.devicePointer;
}

extern "C" april_status april_filter_pairs_host(april_ctx *ctx, const april_dev_sets *R, const april_dev_sets *S,
                                                const uint32_t *h_r, const uint32_t *h_s, uint64_t n,
                                                uint8_t *h_verdict, int mode, void *d_work, size_t work_bytes,
                                                void *stream) {
    if (!ctx || !R || !S) return fail(APRIL_ERR_INVALID_ARG, "NULL argument");
    if (n == 0) return APRIL_OK;
    if (!h_r || !h_s || !h_verdict || !d_work) return fail(APRIL_ERR_INVALID_ARG, "NULL host or work buffer");
    if (((uintptr_t)d_work) & 255u) return fail(APRIL_ERR_INVALID_ARG, "work buffer must be 256-byte aligned");
    size_t need = 0;
    april_status st = april_filter_host_work_bytes(mode, n, &need);
    if (st) return st;
    if (work_bytes < need) return fail(APRIL_ERR_INVALID_ARG, "work buffer too small");
    char *w = (char *)d_work;
    uint32_t *d_r = (uint32_t *)w;
    uint32_t *d_s = (uint32_t *)(w + round256(4 * n));
    uint8_t *d_v = (uint8_t *)(w + 2 * round256(4 * n));
    char *d_scr = w + 2 * round256(4 * n) + round256(n);
    cudaStream_t cs = (cudaStream_t)stream;
    cudaError_t e;
    if (mode != APRIL_MODE_BATCHED && mode != APRIL_MODE_BATCHED_PACKED) {
        // the one-pair-per-thread and per-warp modes: copy in, filter, copy out
        e = cudaMemcpyAsync(d_r, h_r, 4 * n, cudaMemcpyHostToDevice, cs);
        if (e == cudaSuccess) e = cudaMemcpyAsync(d_s, h_s, 4 * n, cudaMemcpyHostToDevice, cs);
        if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpyAsync(pairs)");
        st = april_filter_pairs(ctx, R, S, d_r, d_s, n, d_v, mode, nullptr, 0, stream);
        if (st) return st;
        e = cudaMemcpyAsync(h_verdict, d_v, n, cudaMemcpyDeviceToHost, cs);
        if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpyAsync(verdicts)");
        return april_sync_status(ctx, stream);
    }
    st = check_filter_args(R, S, n, mode);
    if (st) return st;
    const bool packed = mode == APRIL_MODE_BATCHED_PACKED, triaged = triage_applies(ctx->tune, R, S, packed);
    const uint32_t *p_r = triaged ? pinned_words(h_r, n) : nullptr, *p_s = p_r ? pinned_words(h_s, n) : nullptr;
    const unsigned max_ctas = tuned_ctas(ctx);
    if (p_s || (triaged && few_pairs(n, lane_warps(ctx->num_sms, ctx->lane_blocks_per_sm[packed ? 1 : 0], max_ctas)))) {
        // in one piece: page-locked pairs are read where they are, a few are copied in
        if (!p_s) {
            e = cudaMemcpyAsync(d_r, h_r, 4 * n, cudaMemcpyHostToDevice, cs);
            if (e == cudaSuccess) e = cudaMemcpyAsync(d_s, h_s, 4 * n, cudaMemcpyHostToDevice, cs);
            if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpyAsync(pairs)");
            p_r = d_r;
            p_s = d_s;
        }
        const unsigned grid_bin = (unsigned)std::min<uint64_t>((n + 255) / 256, (uint64_t)ctx->num_sms * 8);
        e = enqueue_batched(ctx, R, S, p_r, p_s, n, d_v, d_scr, packed, grid_bin, 1u, max_ctas, !packed, cs);
        if (e == cudaSuccess) e = cudaMemcpyAsync(h_verdict, d_v, n, cudaMemcpyDeviceToHost, cs);
        if (e != cudaSuccess) return cuda_fail(e, "april_filter_pairs_host");
        return april_sync_status(ctx, stream);
    }
    st = ensure_pipeline(ctx);
    if (st) return st;
    const uint32_t K = pipe_chunks(n);
    const uint64_t cs_n = pipe_chunk_size(n);
    size_t sb = 0;
    april_filter_scratch_bytes(mode, cs_n, &sb);
    sb = round256(sb);
    const uint32_t gl = ctx->tune.group_lanes;
    const int occ = ctx->persistent_blocks_per_sm[(packed ? 4 : 0) + group_index(gl)];
    const int bps = ctx->tune.blocks_per_sm ? (int)std::min<uint32_t>(ctx->tune.blocks_per_sm, (uint32_t)occ) : occ;
    const unsigned grid_main = (unsigned)std::max(1, ctx->num_sms * bps);
    cudaStream_t s_in = ctx->pipe[0], s_out = ctx->pipe[3];
    cudaEvent_t ev_start = ctx->pev[0], ev_end = ctx->pev[1];
    // the pipeline follows the work already queued on the caller's stream
    e = cudaEventRecord(ev_start, cs);
    for (cudaStream_t p : ctx->pipe)
        if (e == cudaSuccess) e = cudaStreamWaitEvent(p, ev_start, 0);
    if (triaged && e == cudaSuccess)
        e = host_triage_pipeline(ctx, R, S, h_r, h_s, n, h_verdict, d_r, d_s, d_v, d_scr, packed);
    for (uint32_t c = 0; c < K && e == cudaSuccess && !triaged; ++c) {
        const uint64_t off = c * cs_n;
        if (off >= n) break;
        const uint64_t cnt = std::min<uint64_t>(cs_n, n - off);
        cudaStream_t ks = ctx->pipe[1 + (c & 1u)];
        cudaEvent_t ev_in = ctx->pev[2 + 2 * c], ev_k = ctx->pev[3 + 2 * c];
        e = cudaMemcpyAsync(d_r + off, h_r + off, 4 * cnt, cudaMemcpyHostToDevice, s_in);
        if (e == cudaSuccess) e = cudaMemcpyAsync(d_s + off, h_s + off, 4 * cnt, cudaMemcpyHostToDevice, s_in);
        if (e == cudaSuccess) e = cudaEventRecord(ev_in, s_in);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(ks, ev_in, 0);
        if (e == cudaSuccess) {
            const unsigned grid_bin = (unsigned)std::min<uint64_t>((cnt + 255) / 256, (uint64_t)ctx->num_sms * 8);
            e = enqueue_batched(ctx, R, S, d_r + off, d_s + off, cnt, d_v + off, d_scr + (K > 1 ? (c & 1u) * sb : 0),
                                packed, grid_bin, grid_main, max_ctas, !packed, ks);
        }
        if (e == cudaSuccess) e = cudaEventRecord(ev_k, ks);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s_out, ev_k, 0);
        if (e == cudaSuccess) e = cudaMemcpyAsync(h_verdict + off, d_v + off, cnt, cudaMemcpyDeviceToHost, s_out);
    }
    // the caller's stream waits for every stream of the pipeline
    for (uint32_t q = 0; q < 4 && e == cudaSuccess; ++q) {
        e = cudaEventRecord(ev_end, ctx->pipe[q]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(cs, ev_end, 0);
    }
    if (e != cudaSuccess) return cuda_fail(e, "april_filter_pairs_host pipeline");
    return april_sync_status(ctx, stream);
}

extern "C" april_status april_sync_status(april_ctx *ctx, void *stream) {
    if (!ctx) return fail(APRIL_ERR_INVALID_ARG, "ctx is NULL");
    cudaStream_t st = (cudaStream_t)stream;
    uint32_t h = 0;
    cudaError_t e = cudaMemcpyAsync(&h, ctx->d_status, 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "april_sync_status");
    if (h) {
        e = cudaMemsetAsync(ctx->d_status, 0, 4, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return cuda_fail(e, "april_sync_status(clear)");
    }
    if (h & ST_TIMEOUT) return fail(APRIL_ERR_DEVICE_TIMEOUT, "a bounded device wait ran out");
    if (h & ST_BAD_ID) return fail(APRIL_ERR_OUT_OF_RANGE_ID, "a pair named an out-of-range object id");
    return APRIL_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free entry point.
//
// For callers that cannot allocate device memory on the call path -- for
// example code running where cudaMalloc is forbidden or would synchronize
// the device (inside a real-time serving loop, or a plugin whose host owns
// every allocation) -- the batched filter can run with its scratch in this
// file-scope device array instead of caller memory.  The array is part of
// the loaded module, so every GPU that loads libapril holds it (16 MiB +
// 512 bytes) until the process exits.  Layout: the batched pipeline's
// 256-byte counter block (cleared by every call), a 256-byte status block
// (word 0: the ST_* bits of every call since the last status query), then
// the list of long pairs, one uint32 per pair.
constexpr uint64_t kNoAllocMaxPairs = 4ull << 20;
constexpr uint32_t kNoAllocStatusWord = kCounterBytes / 4;
constexpr uint32_t kNoAllocListWord = 2 * kCounterBytes / 4;
static __device__ __align__(256) uint32_t g_noalloc_scratch[kNoAllocListWord + kNoAllocMaxPairs];

namespace {

struct NoAllocDevice {
    bool ready = false;
    int num_sms = 0;
    int lane_blocks_per_sm = 1;
};
constexpr int kNoAllocMaxDevices = 64;
constexpr uint32_t kNoAllocGroup = 4;  // the default tuning's lane groups
std::mutex g_noalloc_mu;
NoAllocDevice g_noalloc_dev[kNoAllocMaxDevices];

}  // namespace

// Device address of g_noalloc_scratch on the current device.  Host code
// cannot use the array's name as an address (it names a host-side stand-in),
// so the address is looked up on every call (no allocation; after the first
// call on a device the module is loaded and the lookup is cheap).
static april_status noalloc_scratch(uint32_t **ptr) {
    cudaError_t e = cudaGetSymbolAddress((void **)ptr, g_noalloc_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
    return APRIL_OK;
}

extern "C" april_status april_filter_pairs_noalloc(const april_dev_sets *R, const april_dev_sets *S,
                                                   const uint32_t *d_r, const uint32_t *d_s, uint64_t n,
                                                   uint8_t *d_verdict, void *stream) {
    if (!R || !S) return fail(APRIL_ERR_INVALID_ARG, "NULL argument");
    if (n == 0) return APRIL_OK;
    if (!d_r || !d_s || !d_verdict) return fail(APRIL_ERR_INVALID_ARG, "NULL pair or verdict array");
    if (R->order != S->order) return fail(APRIL_ERR_INVALID_ARG, "R and S are on different grids");
    if (R->parts || S->parts) return fail(APRIL_ERR_INVALID_ARG, "april_filter_pairs_noalloc takes unpartitioned sets");
    if (check_layout(R) || check_layout(S)) return APRIL_ERR_INVALID_ARG;
    if (n > kNoAllocMaxPairs)
        return fail(APRIL_ERR_INVALID_ARG, "april_filter_pairs_noalloc: n exceeds APRIL_NOALLOC_MAX_PAIRS (4194304); "
                                           "split the pairs or use april_filter_pairs with caller scratch");
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
    if (dev < 0 || dev >= kNoAllocMaxDevices) return fail(APRIL_ERR_INVALID_ARG, "device index out of range");
    uint32_t *scratch = nullptr;
    april_status rc = noalloc_scratch(&scratch);
    if (rc) return rc;
    NoAllocDevice nd;
    {
        // first call on this device: the launch shape (the current device is
        // the one being set up)
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        NoAllocDevice &slot = g_noalloc_dev[dev];
        if (!slot.ready) {
            int sms = 0, lane_bps = 0;
            e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (e == cudaSuccess)
                e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&lane_bps, k_triage<RawSets, false>, kBlock, 0);
            if (e != cudaSuccess) return cuda_fail(e, "april_filter_pairs_noalloc set-up");
            slot.num_sms = sms;
            slot.lane_blocks_per_sm = lane_bps < 1 ? 1 : lane_bps;
            slot.ready = true;
        }
        nd = slot;
    }
    cudaStream_t st = (cudaStream_t)stream;
    uint32_t *counters = scratch;
    uint32_t *status = scratch + kNoAllocStatusWord;
    uint32_t *big_list = scratch + kNoAllocListWord;
    // the array keeps the previous call's contents: launch_lanes resets the
    // counters that it has read (the status block keeps its bits until
    // april_noalloc_sync_status reads them)
    const RawSets dR{dev_set(R)}, dS{dev_set(S)};
    const april_tune t = default_tune();
    const uint32_t jo = join_order_of(t.join_order);
    bool left = false;
    e = launch_lanes(nd.num_sms, nd.lane_blocks_per_sm, 0xffffffffu, dR, dS, lane_plan(jo), d_r, d_s, n, d_verdict, status,
                     big_list, counters, true, st, &left);
    if (e == cudaSuccess && left) {
        const unsigned grid = rest_grid(n, nd.num_sms, 0xffffffffu, kRestCtas);
        k_persistent_rest<kNoAllocGroup, RawSets><<<grid, 32 * kRestWarps, 0, st>>>(
            dR, dS, d_r, d_s, d_verdict, status, counters, t.group_window, jo, 0u, nullptr, 0u,
            Rest{big_list, rest_stages(n)});
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) return cuda_fail(e, "april_filter_pairs_noalloc launch");
    return APRIL_OK;
}

extern "C" april_status april_noalloc_sync_status(void *stream) {
    uint32_t *scratch = nullptr;
    april_status rc = noalloc_scratch(&scratch);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    uint32_t h = 0;  // pageable: the copy has completed when the call returns
    cudaError_t e = cudaMemcpyAsync(&h, scratch + kNoAllocStatusWord, 4, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "april_noalloc_sync_status");
    if (h) {
        e = cudaMemsetAsync(scratch + kNoAllocStatusWord, 0, 4, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return cuda_fail(e, "april_noalloc_sync_status(clear)");
    }
    if (h & ST_TIMEOUT) return fail(APRIL_ERR_DEVICE_TIMEOUT, "a bounded device wait ran out");
    if (h & ST_BAD_ID) return fail(APRIL_ERR_OUT_OF_RANGE_ID, "a pair named an out-of-range object id");
    return APRIL_OK;
}

// ---------------------------------------------------------------------------
// Diagnostic: the iteration limit of the kernels' bounded waits.
extern "C" april_status april_debug_set_wait_limit(uint32_t spins) {
    cudaError_t e = cudaMemcpyToSymbol(c_wait_limit, &spins, sizeof(spins));
    if (e == cudaSuccess) e = (cudaError_t)april_build_wait_limit(spins);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpyToSymbol(c_wait_limit)");
    return APRIL_OK;
}
