// spread.cu -- the Monte-Carlo estimate of the expected spread E(S, G[V \ B]) (Def. 3; the
// paper evaluates the spread of every blocker set it reports by simulating the cascade on
// sampled graphs): the sum over theta sampled graphs of the number of vertices reachable from the
// seeds, seeds included, on the same Philox stream as Alg. 2 (sample j of call `round` under `key`).
// The comparison algorithms of Sec. 5 (BaselineGreedy, Exact) score many blocker sets this way on
// common samples, so the work is a list of (set, sample) items and the single estimate is the
// list of one empty set.
//
// Two launches per slice of the items:
//   * k_spread_warp: a warp per item. Only reachability counts, so there are no parents, levels or
//     local ids: a frontier queue and a hash of the visited vertices, 4 KB per warp in shared
//     memory, and no barriers. It is bound by instruction issue (Philox, hashing), like the warp
//     tier of Alg. 2.
//   * k_spread_block: the block-per-sample BFS of sample_cta.cuh for the cascades that outgrow the
//     queue; each resumes from the vertices the warp had found.
// Before, every item ran in the block kernel. Measured with both: 10^5 samples of a 50-vertex
// blocker set on R-MAT 2^17 / 2^20 2.86 -> 2.27 ms; BaselineGreedy (n = 2,000, b = 2, r = 2,000:
// 8*10^6 items of about 35 vertices) 82.2 -> 27.7 ms.
#include <algorithm>
#include <cstddef>

#include "internal.h"

#include "sample_cta.cuh"

namespace imin {

namespace {

using namespace cta;

constexpr uint32_t kWarps = 8;         // warps per block of the warp kernel
// Non-seed vertices a warp can hold; the hash has twice as many slots, which leaves room for the
// 32 insertions in flight and for a set of up to 64 blocked vertices. Larger cascades lose nothing but
// the chunk in which the queue ran full, so one size serves every graph.
constexpr uint32_t kQueue = 256;
constexpr uint32_t kSlots = 512;
constexpr uint32_t kSlotShift = 23;    // 32 - log2(kSlots)
constexpr uint32_t kHeader = 8;        // words before the queue in a hand-off
constexpr uint32_t kHandoffWords = kHeader + kQueue;

// Items [first, last) of a call: item i is set i / theta, sample i % theta.
struct SpreadWork {
    const int32_t* sets;                // k vertices per set, blocked on top of P.excl
    uint32_t k;
    unsigned long long first, last;
    uint32_t grab;                      // items a warp takes at a time
    unsigned long long* sums;           // per set
    uint32_t* handoff;                  // kHandoffWords per entry: set, sample, chunk start, queue
                                        // length (kQueue), examined and live edges (64 bits each), queue
};

struct __align__(16) WarpSpread {
    uint32_t hash[kSlots];
    uint32_t queue[kQueue];
    WarpStage stage;
};

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long x)
{
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) x += __shfl_down_sync(kFull, x, o);
    return __shfl_sync(kFull, x, 0);
}

// Find-or-insert of v in the warp's visited hash: true if v is new.
__device__ __forceinline__ bool insert_new(uint32_t* hash, uint32_t v)
{
    uint32_t slot = (v * 0x9E3779B1u) >> kSlotShift;
    for (uint32_t probe = 0; probe < kSlots; ++probe) {
        const uint32_t k = *reinterpret_cast<volatile uint32_t*>(hash + slot);
        if (k == v) return false;
        if (k == kEmpty) {
            const uint32_t prev = atomicCAS(hash + slot, kEmpty, v);
            if (prev == kEmpty) return true;
            if (prev == v) return false;
        }
        slot = (slot + 1) & (kSlots - 1);
    }
    return false;  // full: cannot happen, the queue overflows first
}

// One item of the warp kernel: |R| without the seeds, or kEmpty when the queue is too small; then
// *at is the queue index of the chunk it stopped in, the queue is full, and examined and live are the
// counts before that chunk (per lane). The hash is empty on entry and on return.
template <int M>
__device__ __forceinline__ uint32_t spread_sample(const SampleParams& P, WarpSpread& w, const int32_t* set, uint32_t k,
                                                  uint32_t j, uint32_t lane, uint32_t* at, uint32_t& examined,
                                                  uint32_t& live)
{
    // a set's vertices count as visited from the start, so nothing discovers them
    for (uint32_t i = lane; i < k; i += 32) insert_new(w.hash, static_cast<uint32_t>(set[i]));
    __syncwarp();
    const uint32_t ns = P.ns;
    uint32_t head = 0, end_q = ns;  // the seeds come first, read from P.seeds
    bool over = false;
    while (head < end_q) {
        const uint32_t next = min(head + 32, end_q);  // what this chunk finds comes after it
        const uint32_t idx = head + lane;
        int32_t beg = 0, end = 0;
        if (idx < next) {
            const uint32_t u = idx < ns ? static_cast<uint32_t>(__ldg(P.seeds + idx)) : w.queue[idx - ns];
            beg = __ldg(P.g.row_ptr + u);
            end = __ldg(P.g.row_ptr + u + 1);
        }
        const ChunkRows rows = publish_rows(&w.stage, beg, end, lane);
        uint32_t owners = 0, staged = 0, lv = 0;
        for (uint32_t t0 = 0; t0 < rows.total && !over; t0 += 32) {
            const uint32_t r = window_owner(rows, t0, owners);
            uint32_t m = 0;
            int32_t e0 = 0;
            if (t0 + lane < rows.total) {
                const uint32_t q = w.stage.qoff[r] + t0 + lane;
                e0 = static_cast<int32_t>(q << 2);
                m = group_live<M>(P.g, q, __ldg(P.g.thr4 + q), w.stage.beg[r], w.stage.end[r], j, P.round, P.key_lo,
                                  P.key_hi);
            }
            staged = stage_live(&w.stage, staged, m & 1u, m & 2u, m & 4u, m & 8u, e0, r, lane);
            const bool last = t0 + 32 >= rows.total;
            while (staged >= 32 || (last && staged > 0)) {
                const uint32_t take = staged < 32 ? staged : 32;
                staged -= take;
                bool fresh = false;
                uint32_t v = 0;
                if (lane < take) {
                    v = static_cast<uint32_t>(__ldg(P.g.col + w.stage.edge[staged + lane]));
                    if (!excluded(P.excl, v)) {
                        ++lv;
                        fresh = insert_new(w.hash, v);
                    }
                }
                const uint32_t won = __ballot_sync(kFull, fresh);
                const uint32_t p = end_q - ns + __popc(won & lanemask_lt());
                if (fresh && p < kQueue) w.queue[p] = v;
                end_q += __popc(won);
                if (end_q - ns > kQueue) {
                    over = true;
                    break;
                }
            }
            __syncwarp();
        }
        if (over) break;
        examined += static_cast<uint32_t>(end - beg);
        live += lv;
        head = next;
    }
    for (uint32_t i = lane; i < kSlots / 4; i += 32)
        reinterpret_cast<uint4*>(w.hash)[i] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
    __syncwarp();
    *at = head;
    return over ? kEmpty : end_q - ns;
}

template <int M>
__global__ void __launch_bounds__(kWarps * 32, 5) k_spread_warp(SampleParams P, SpreadWork W)
{
    __shared__ WarpSpread space[kWarps];
    const uint32_t lane = threadIdx.x & 31;
    WarpSpread& w = space[threadIdx.x >> 5];
    for (uint32_t i = lane; i < kSlots; i += 32) w.hash[i] = kEmpty;
    __syncwarp();
    const uint32_t items = static_cast<uint32_t>(W.last - W.first);
    unsigned long long reached = 0, examined = 0, live = 0, done = 0;
    for (;;) {
        uint32_t i0 = 0;
        if (lane == 0) i0 = atomicAdd(&P.ctl->cursor[0], W.grab);
        i0 = __shfl_sync(kFull, i0, 0);
        if (i0 >= items) break;
        const uint32_t i1 = min(i0 + W.grab, items);
        uint32_t set = static_cast<uint32_t>((W.first + i0) / P.theta);
        uint32_t j = static_cast<uint32_t>((W.first + i0) % P.theta);
        unsigned long long sum = 0;
        for (uint32_t i = i0; i < i1; ++i) {
            uint32_t ex = 0, lv = 0, at = 0;
            const uint32_t found = spread_sample<M>(P, w, W.sets + static_cast<uint64_t>(set) * W.k, W.k, j, lane, &at,
                                                    ex, lv);
            if (found != kEmpty) {
                sum += P.ns + found;
                reached += P.ns + found;
                examined += ex;
                live += lv;
                ++done;
            } else {
                const unsigned long long exs = warp_sum(ex), lvs = warp_sum(lv);
                uint32_t pos = 0;
                if (lane == 0) pos = atomicAdd(&P.ctl->count[kTierCta], 1u);
                pos = __shfl_sync(kFull, pos, 0);
                uint32_t* h = W.handoff + static_cast<uint64_t>(pos) * kHandoffWords;
                if (lane == 0) {
                    h[0] = set;
                    h[1] = j;
                    h[2] = at;
                    h[3] = kQueue;
                    *reinterpret_cast<unsigned long long*>(h + 4) = exs;
                    *reinterpret_cast<unsigned long long*>(h + 6) = lvs;
                }
                for (uint32_t t = lane; t < kQueue; t += 32) h[kHeader + t] = w.queue[t];
                __syncwarp();
            }
            if (++j == P.theta || i + 1 == i1) {
                if (lane == 0 && sum > 0) atomicAdd(W.sums + set, sum);
                sum = 0;
                if (j == P.theta) {
                    j = 0;
                    ++set;
                }
            }
        }
    }
    if (P.stats != nullptr) {
        examined = warp_sum(examined);
        live = warp_sum(live);
        if (lane == 0 && done > 0) {
            atomicAdd(P.stats + kStSamples, done);
            atomicAdd(P.stats + kStReached, reached);
            atomicAdd(P.stats + kStExamined, examined);
            atomicAdd(P.stats + kStLive, live);
        }
    }
}

// The items the warp kernel handed over: the block resumes each at the frontier chunk the warp
// stopped in, with the seeds and the queue as the vertices found so far.
template <bool kSmemBitmap, int M>
__global__ void __launch_bounds__(cta_threads<kSmemBitmap>(), 1024 / cta_threads<kSmemBitmap>())
k_spread_block(SampleParams P, CtaCfg C, SpreadWork W)
{
    constexpr uint32_t kCtaThreads = cta_threads<kSmemBitmap>();
    extern __shared__ __align__(16) uint32_t dsm[];
    __shared__ CtaShared<kCtaThreads> sh;
    const uint32_t tid = threadIdx.x;
    const uint32_t count = *reinterpret_cast<const volatile uint32_t*>(&P.ctl->count[kTierCta]);
    if (blockIdx.x >= count) return;  // the resident blocks hold at least as many items as blocks
    uint8_t* base = C.scratch + static_cast<uint64_t>(blockIdx.x) * C.slot_bytes;
    Slot S;
    S.gid = reinterpret_cast<int32_t*>(base + C.off_gid);
    S.par = reinterpret_cast<uint32_t*>(base + C.off_par);
    S.idom = reinterpret_cast<uint32_t*>(base + C.off_idom);
    S.rows = reinterpret_cast<int2*>(base + C.off_rows);
    S.edges = reinterpret_cast<uint2*>(base + C.off_edges);
    uint32_t* bm = kSmemBitmap ? dsm : reinterpret_cast<uint32_t*>(base + C.off_bm);
    if constexpr (kSmemBitmap) {
        for (uint32_t i = tid; i < C.bm_words; i += kCtaThreads) bm[i] = 0;
    }
    SampleCounters sc;
    unsigned long long examined = 0, live = 0;
    for (;;) {
        __syncthreads();
        if (tid == 0) sh.item = atomicAdd(&P.ctl->cursor[kTierCta], 1u);
        __syncthreads();
        if (sh.item >= count) break;
        const uint32_t* h = W.handoff + static_cast<uint64_t>(sh.item) * kHandoffWords;
        const uint32_t set = h[0], at = h[2], found = P.ns + h[3];
        // slot ids start at 1, as in Alg. 2's slots
        for (uint32_t i = tid; i < found; i += kCtaThreads) {
            const uint32_t v = i < P.ns ? static_cast<uint32_t>(P.seeds[i]) : h[kHeader + i - P.ns];
            S.gid[1 + i] = static_cast<int32_t>(v);
            if (i >= at) S.rows[1 + i] = make_int2(__ldg(P.g.row_ptr + v), __ldg(P.g.row_ptr + v + 1));
            if (i >= P.ns) atomicOr(bm + (v >> 5), 1u << (v & 31));
        }
        if (tid == 0) {
            sh.lvl[0] = 1;
            sh.nR = 1 + found;
            sh.nE = 0;
            sh.flag = 0;
            examined += *reinterpret_cast<const unsigned long long*>(h + 4);
            live += *reinterpret_cast<const unsigned long long*>(h + 6);
        }
        __syncthreads();
        const uint32_t from[3] = {1 + at, 1 + found, 1};
        const unsigned long long before = sc.reached;
        const int rc = run_sample_cta<kSmemBitmap, true, M>(
            P, C, bm, dsm, sh, S, h[1], tid, sc, examined, live,
            ExtraBlocked{W.sets + static_cast<uint64_t>(set) * W.k, W.k}, from);
        if (tid == 0) {
            // only a cascade beyond the slot capacity can fail
            if (rc != kSampleDone) atomicOr(&P.ctl->error, rc == kSampleOverflow ? kErrCapacity : kErrInternal);
            else atomicAdd(W.sums + set, sc.reached - before);
        }
    }

    if (P.stats != nullptr) {
        const uint32_t lane = tid & 31;
        unsigned long long ex = examined, lv = live;
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) {
            ex += __shfl_down_sync(kFull, ex, o);
            lv += __shfl_down_sync(kFull, lv, o);
        }
        unsigned long long* st = P.stats + kTierCta * kStPerTier;
        if (lane == 0) {
            if (ex) atomicAdd(st + kStExamined, ex);
            if (lv) atomicAdd(st + kStLive, lv);
        }
        if (tid == 0 && sc.done > 0) {
            atomicAdd(st + kStSamples, sc.done);
            atomicAdd(st + kStReached, sc.reached);
        }
    }
}

// In place of k_spread_block where no hand-off fits a slot: a slot of a large graph holds at most 2^18
// ids, and a cascade that has outgrown it will not fit later.
__global__ void k_spread_refuse(RoundCtl* ctl)
{
    if (ctl->count[kTierCta] > 0) atomicOr(&ctl->error, kErrCapacity);
}

template <int M>
cudaError_t launch_slice(const SampleParams& P, const CtaCfg& cfg, uint32_t warp_blocks, uint32_t blocks,
                         uint64_t smem, const SpreadWork& W, cudaStream_t s)
{
    k_spread_warp<M><<<warp_blocks, kWarps * 32, 0, s>>>(P, W);
    if (1 + P.ns + kQueue > cfg.rcap && cfg.rcap <= static_cast<uint32_t>(P.g.n)) k_spread_refuse<<<1, 1, 0, s>>>(P.ctl);
    else if (cfg.global_bitmap) k_spread_block<false, M><<<blocks, cta_threads<false>(), smem, s>>>(P, cfg, W);
    else k_spread_block<true, M><<<blocks, cta_threads<true>(), smem, s>>>(P, cfg, W);
    return cudaGetLastError();
}

}  // namespace

// One hand-off per item at most: 277 MB for a whole kSpreadSlice.
uint64_t spread_handoff_words(unsigned long long items) { return items * kHandoffWords; }

cudaError_t prepare_spread(const CtaCfg& c)
{
    const DeviceInfo dev = device_info();
    const cudaError_t e = c.global_bitmap ? allow_max_dynamic_smem(k_spread_block<false, kModelIC>, dev)
                                          : allow_max_dynamic_smem(k_spread_block<true, kModelIC>, dev);
    if (e != cudaSuccess) return e;
    return c.global_bitmap ? allow_max_dynamic_smem(k_spread_block<false, kModelLT>, dev)
                           : allow_max_dynamic_smem(k_spread_block<true, kModelLT>, dev);
}

cudaError_t launch_spread_slice(const SampleParams& P, const CtaCfg& c, uint32_t blocks, uint64_t smem,
                                uint8_t* scratch, const int32_t* sets, uint32_t k, unsigned long long first,
                                unsigned long long last, uint32_t* handoff, unsigned long long* sums,
                                cudaStream_t s)
{
    const DeviceInfo dev = device_info();
    CtaCfg cfg = c;
    cfg.scratch = scratch;
    // the slice's work cursors and hand-off count (the error bits stay)
    const cudaError_t e = cudaMemsetAsync(P.ctl, 0, offsetof(RoundCtl, error), s);
    if (e != cudaSuccess) return e;
    SpreadWork W{};
    W.sets = sets;
    W.k = k;
    W.first = first;
    W.last = last;
    const uint32_t n = static_cast<uint32_t>(W.last - W.first);
    const uint32_t warp_blocks = std::min((n + kWarps - 1) / kWarps, 5u * dev.sms);
    // at least 8 grabs per warp, so that no warp is left with the last long run
    W.grab = std::max(1u, std::min(16u, n / (8u * kWarps * warp_blocks)));
    W.sums = sums;
    W.handoff = handoff;
    return P.g.lo4 != nullptr ? launch_slice<kModelLT>(P, cfg, warp_blocks, blocks, smem, W, s)
                              : launch_slice<kModelIC>(P, cfg, warp_blocks, blocks, smem, W, s);
}

}  // namespace imin
