// noalloc.cu -- imin_estimate_decrease_noalloc: one Alg. 2 call that allocates no memory.
//
// Who needs it: callers that must not allocate device memory when they call in -- code whose
// device memory is owned by another allocator with a fixed budget (a framework's caching
// allocator, a serving process that sizes everything at start-up and must not grow later), and
// latency-critical paths that cannot afford cudaMalloc/cudaFree, which may synchronize the whole
// device. The call itself is synchronous: it reads a validation flag back from the device before
// its kernel runs and the kernel's status after it, so it returns only when the counters are
// final, and it cannot be recorded into a CUDA graph by stream capture.
//
// What it does: exactly what imin_estimate_decrease computes, with the block-per-sample tier
// (sample_cta.cu) and, for many samples, the warp tier at a fixed cutoff (sample.cu) in front of it.
// But every byte of working memory it needs besides the caller's inputs and output comes from one
// file-scope device array of kNoAllocBytes (64 MiB). Every GPU that loads the library holds that
// array until the process exits. Its limits follow from its size:
// graphs with at most kNoAllocMaxVertices vertices and at most kNoAllocMaxTheta samples per call;
// bigger requests are rejected with IMIN_ERR_INVALID. A sampled cascade that would need the
// whole-graph fallback tier (more non-tree live edges or BFS levels than the block tier holds)
// makes the call fail with IMIN_ERR_CAPACITY instead of running that tier; out_delta then holds
// partial counters and must not be used.
//
// The array is shared by every call on a device and keeps the last call's contents; each call
// clears the parts that must start at zero. Calls that overlap on the GPU (different streams or
// threads without ordering between them) race on it.
//
// Set-up: the first call on each device resolves the array's device address with
// cudaGetSymbolAddress (in host code the array's name is only a host-side stand-in, never a
// device address). The block tier's launch plan (slot layout, grid, shared memory) is computed
// once per device and graph size (n, m) and kept in a fixed table, so later calls of the same
// size make no attribute or occupancy queries; the plan's test hooks (IMIN_CTA_EDGE_CAP) are read
// only when a plan is made.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <mutex>

#include "imin.h"
#include "internal.h"

namespace imin {

namespace {

constexpr int32_t kNoAllocMaxVertices = 1 << 16;
constexpr uint32_t kNoAllocMaxTheta = 1u << 17;
constexpr uint64_t kNoAllocBytes = 64ull << 20;
constexpr int kMaxDevices = 64;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

std::mutex g_setup_mu;
void* g_scratch_ptr[kMaxDevices] = {};

// Launch plans of the block tier, per device and graph size, in a fixed table (no heap use).
struct PlanEntry {
    int device;
    int32_t n, m;
    CtaCfg cfg;
    uint32_t blocks;
    uint64_t smem;
};
// Slot capacities of the first block-tier launch (vertices, non-tree edges): the smallest that hold
// all but the rare cascades, so that a slot for every resident block (8 per SM) fits the array.
constexpr uint32_t kSmallVertices = 2048;
constexpr uint32_t kSmallEdges = 1024;
constexpr int kPlanSlots = 16;
PlanEntry g_plans[kPlanSlots];
int g_plan_count = 0, g_plan_next = 0;

// The block tier's plan for (device, n, m), made on first use.
bool cta_plan(const imin_graph* g, CtaCfg* cfg, uint32_t* blocks, uint64_t* smem)
{
    std::lock_guard<std::mutex> lk(g_setup_mu);
    for (int i = 0; i < g_plan_count; ++i) {
        const PlanEntry& e = g_plans[i];
        if (e.device == g->device && e.n == g->n && e.m == g->m) {
            *cfg = e.cfg;
            *blocks = e.blocks;
            *smem = e.smem;
            return true;
        }
    }
    uint64_t slot_total = 0;
    if (!plan_cta_tier(g->dev, g->n, g->m, cfg, blocks, smem, &slot_total)) return false;
    allow_tier0_smem(g->dev);
    PlanEntry& e = g_plans[g_plan_next];
    e = PlanEntry{g->device, g->n, g->m, *cfg, *blocks, *smem};
    g_plan_next = (g_plan_next + 1) % kPlanSlots;
    if (g_plan_count < kPlanSlots) ++g_plan_count;
    return true;
}

// Device address of the static array on `device` (resolved once per device).
int scratch_address(int device, uint8_t** out)
{
    if (device < 0 || device >= kMaxDevices) return fail_msg(IMIN_ERR_CUDA, "device index out of range");
    std::lock_guard<std::mutex> lk(g_setup_mu);
    if (g_scratch_ptr[device] == nullptr) {
        void* p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) {
            cudaGetLastError();
            char msg[160];
            std::snprintf(msg, sizeof(msg), "cudaGetSymbolAddress of the static scratch failed: %s",
                          cudaGetErrorString(e));
            return fail_msg(IMIN_ERR_CUDA, msg);
        }
        g_scratch_ptr[device] = p;
    }
    *out = static_cast<uint8_t*>(g_scratch_ptr[device]);
    return IMIN_OK;
}

// Marks every id in the seed/blocked bitmask; flags ids out of range (bit 0) and ids that were
// already marked -- duplicates, or a blocked vertex that is a seed (bit 1).
__global__ void k_mark_ids(const int32_t* ids, int32_t count, int32_t n, uint32_t* excl, uint32_t* bad)
{
    for (int32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        const int32_t v = ids[i];
        if (v < 0 || v >= n) {
            atomicOr(bad, 1u);
            continue;
        }
        const uint32_t bit = 1u << (v & 31);
        if (atomicOr(excl + (v >> 5), bit) & bit) atomicOr(bad, 2u);
    }
}

uint64_t up256(uint64_t x) { return (x + 255) & ~uint64_t(255); }

// 1: device (or managed) memory of `device`; 0: host memory; -1: device memory of another GPU.
int device_pointer(const void* p, int device)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if (a.type != cudaMemoryTypeDevice && a.type != cudaMemoryTypeManaged) return 0;
    return a.device == device ? 1 : -1;
}

int cuda_fail(cudaError_t e, const char* what)
{
    cudaGetLastError();
    char msg[200];
    std::snprintf(msg, sizeof(msg), "%s: %s", what, cudaGetErrorString(e));
    return fail_msg(IMIN_ERR_CUDA, msg);
}

#define NA_CUDA(call)                                 \
    do {                                              \
        const cudaError_t e_ = (call);                \
        if (e_ != cudaSuccess) return cuda_fail(e_, #call); \
    } while (0)

}  // namespace

}  // namespace imin

using namespace imin;

extern "C" int imin_estimate_decrease_noalloc(const imin_graph* g, const int32_t* seeds,
                                              int32_t n_seeds, const int32_t* blocked,
                                              int32_t n_blocked, uint32_t theta, uint64_t key,
                                              uint32_t round, uint64_t* out_delta, void* stream)
{
    fail_msg(IMIN_OK, "");
    if (g == nullptr) return fail_msg(IMIN_ERR_INVALID, "graph handle is NULL");
    if (out_delta == nullptr) return fail_msg(IMIN_ERR_INVALID, "out_delta is NULL");
    if (seeds == nullptr) return fail_msg(IMIN_ERR_INVALID, "seeds is NULL");
    if (n_seeds < 1 || n_seeds > g->n) return fail_msg(IMIN_ERR_INVALID, "n_seeds must be in [1, n]");
    if (n_blocked < 0 || (n_blocked > 0 && blocked == nullptr))
        return fail_msg(IMIN_ERR_INVALID, "n_blocked must be >= 0 and blocked non-NULL when > 0");
    if (n_seeds + static_cast<int64_t>(n_blocked) > g->n)
        return fail_msg(IMIN_ERR_INVALID, "more seeds and blocked vertices than vertices");
    if (theta < 1) return fail_msg(IMIN_ERR_INVALID, "theta must be >= 1");
    if (g->n > kNoAllocMaxVertices) {
        char msg[160];
        std::snprintf(msg, sizeof(msg),
                      "imin_estimate_decrease_noalloc: n = %d exceeds its static limit of %d vertices",
                      g->n, kNoAllocMaxVertices);
        return fail_msg(IMIN_ERR_INVALID, msg);
    }
    if (theta > kNoAllocMaxTheta) {
        char msg[160];
        std::snprintf(msg, sizeof(msg),
                      "imin_estimate_decrease_noalloc: theta = %u exceeds its static limit of %u",
                      theta, kNoAllocMaxTheta);
        return fail_msg(IMIN_ERR_INVALID, msg);
    }
    const cudaStream_t s = static_cast<cudaStream_t>(stream);
    NA_CUDA(cudaSetDevice(g->device));
    uint8_t* base = nullptr;
    int rc = scratch_address(g->device, &base);
    if (rc) return rc;

    // layout of the static array for this call
    const uint32_t words = static_cast<uint32_t>((g->n + 31) / 32);
    const int where_out = device_pointer(out_delta, g->device);
    if (where_out < 0)
        return fail_msg(IMIN_ERR_INVALID, "out_delta is device memory of another GPU than the graph's");
    const bool dev_out = where_out > 0;
    uint64_t o = 0;
    const uint64_t off_ctl = o;     o = up256(o + sizeof(RoundCtl));
    const uint64_t off_bad = o;     o = up256(o + sizeof(uint32_t));
    const uint64_t off_excl = o;    o = up256(o + 4ull * words);
    const uint64_t off_seeds = o;   o = up256(o + 4ull * n_seeds);
    const uint64_t off_blocked = o; o = up256(o + 4ull * n_blocked);
    const uint64_t off_delta = o;   o = up256(o + (dev_out ? 0ull : 8ull * g->n));
    const uint64_t off_lists = o;   o = up256(o + 4ull * kTiers * theta);
    const uint64_t off_slots = o;

    CtaCfg cfg{};
    uint32_t blocks = 0;
    uint64_t smem = 0;
    if (!cta_plan(g, &cfg, &blocks, &smem))
        return fail_msg(IMIN_ERR_INTERNAL, "the block-per-sample kernel cannot be configured");
    if (off_slots + cfg.slot_bytes > kNoAllocBytes)
        return fail_msg(IMIN_ERR_INVALID, "imin_estimate_decrease_noalloc: request exceeds the static scratch");
    const uint64_t room = kNoAllocBytes - off_slots;
    // Whole-graph slots are so large that few fit (56 at n = 50,000, where 1,216 blocks could be
    // resident). So a call has up to three launches: the warp tier, which needs no slots; the block
    // tier on slots of kSmallVertices, one per resident block; and the block tier on whole-graph
    // slots for the samples that outgrow those. The launches follow one another on the stream and
    // share the array. n = 50,021, m = 400,009, theta = 10^4, |S| = 50: 6.26 -> 2.40 ms. The second
    // launch must read the first's overflow count either way, so it is always enqueued.
    CtaCfg small = cfg;
    small.rcap = std::min(cfg.rcap, std::max(kSmallVertices, 2u * (1u + static_cast<uint32_t>(n_seeds))));
    small.ecap = std::min(cfg.ecap, kSmallEdges);
    cta_slot_layout(&small);
    const uint32_t small_blocks = static_cast<uint32_t>(std::min<uint64_t>(blocks, room / small.slot_bytes));
    const uint32_t whole_blocks = static_cast<uint32_t>(std::min<uint64_t>(blocks, room / cfg.slot_bytes));
    // Few samples are done sooner by the last launch alone: the launches' latencies add up, and a
    // cascade that outgrows the warp and a small slot runs three times. Both routes were timed on six
    // kinds of graph (Chung-Lu and R-MAT; weighted cascade, trivalency, p = 0.15) of 256 to 65,536
    // vertices, theta = 250 to 32,000. With b whole-graph slots the times cross between 2 and 10 b for
    // b > 375, between 1 and 13 b (mostly 500 to 2,000 samples) down to b = 146, and near 3 to 20 b
    // below. ms with one launch / three, theta = 2,000; 8,000: n = 2,048 (b = 389), R-MAT, 216 reached
    // 0.25 / 0.20; 0.72 / 0.37. n = 4,096 (b = 314), R-MAT trivalency, 466 reached 0.52 / 0.30;
    // 1.78 / 0.78. n = 16,384 (b = 146), p = 0.15, 420 reached 0.82 / 0.35; 2.79 / 0.90, but R-MAT
    // weighted cascade, 63 reached, 0.26 / 0.43; 0.65 / 0.49. n = 65,536 (b = 46), R-MAT, 207 reached
    // 1.09 / 0.68; 3.68 / 1.47. Where most cascades outgrow the small slots the three launches lose at
    // any theta: R-MAT trivalency at 16,384 (1,749 reached) 12 %, at 65,536 2 %; likewise where every
    // block has a whole-graph slot and most cascades outgrow the warp (500 vertices, 177 reached) 18 %.
    const uint32_t few = whole_blocks >= 375 ? 4 * whole_blocks : std::min(20 * whole_blocks, 2000u);
    const bool whole_only = theta <= few;
    TierPlan warp{};
    if (!whole_only) {
        plan_tier0(g->dev, static_cast<uint32_t>(n_seeds), kDefaultCutoff, &warp);
        warp.few = few_per_warp(warp, theta);
    }

    RoundCtl* ctl = reinterpret_cast<RoundCtl*>(base + off_ctl);
    uint32_t* bad = reinterpret_cast<uint32_t*>(base + off_bad);
    uint32_t* excl = reinterpret_cast<uint32_t*>(base + off_excl);
    int32_t* dseeds = reinterpret_cast<int32_t*>(base + off_seeds);
    int32_t* dblocked = reinterpret_cast<int32_t*>(base + off_blocked);
    unsigned long long* delta =
        dev_out ? reinterpret_cast<unsigned long long*>(out_delta)
                : reinterpret_cast<unsigned long long*>(base + off_delta);

    // zero what must start at zero; bring the ids into the array
    NA_CUDA(cudaMemsetAsync(base, 0, off_seeds, s));  // control block, flag, bitmask
    NA_CUDA(cudaMemsetAsync(delta, 0, 8ull * g->n, s));
    NA_CUDA(cudaMemcpyAsync(dseeds, seeds, 4ull * n_seeds, cudaMemcpyDefault, s));
    if (n_blocked > 0)
        NA_CUDA(cudaMemcpyAsync(dblocked, blocked, 4ull * n_blocked, cudaMemcpyDefault, s));
    k_mark_ids<<<(n_seeds + 255) / 256, 256, 0, s>>>(dseeds, n_seeds, g->n, excl, bad);
    if (n_blocked > 0) k_mark_ids<<<(n_blocked + 255) / 256, 256, 0, s>>>(dblocked, n_blocked, g->n, excl, bad);
    NA_CUDA(cudaGetLastError());
    count_launches(n_blocked > 0 ? 2 : 1);
    uint32_t hbad = 0;
    NA_CUDA(cudaMemcpyAsync(&hbad, bad, sizeof(hbad), cudaMemcpyDeviceToHost, s));
    NA_CUDA(cudaStreamSynchronize(s));
    if (hbad & 1u) return fail_msg(IMIN_ERR_INVALID, "seeds/blocked: vertex id out of range");
    if (hbad & 2u) return fail_msg(IMIN_ERR_INVALID, "seeds/blocked: duplicate vertex or blocked seed");

    SampleParams P{};
    P.g = dev_graph(g);
    P.seeds = dseeds;
    P.ns = static_cast<uint32_t>(n_seeds);
    P.excl = excl;
    P.key_lo = static_cast<uint32_t>(key);
    P.key_hi = static_cast<uint32_t>(key >> 32);
    P.round = round;
    P.theta = theta;
    P.delta = delta;
    P.ctl = ctl;
    P.lists = reinterpret_cast<uint32_t*>(base + off_lists);
    P.done = nullptr;
    P.stats = nullptr;
    if (!whole_only) {
        bool warp_ran = false;
        NA_CUDA(launch_sample_tier(0, P, warp, nullptr, s, &warp_ran));
        small.from_list = warp_ran ? 1u : 0u;
        NA_CUDA(launch_cta_tier(P, small, small_blocks, smem, base + off_slots, s));
        count_launches(warp_ran ? 2 : 1);
        cfg.from_list = 1;
        cfg.in_tier = kTierWhole;
    }
    cfg.out_tier = 1;  // the warp tier 1 does not run here: its list takes what nothing here holds
    NA_CUDA(launch_cta_tier(P, cfg, whole_blocks, smem, base + off_slots, s));
    count_launches(1);

    RoundCtl hctl;
    NA_CUDA(cudaMemcpyAsync(&hctl, ctl, sizeof(hctl), cudaMemcpyDeviceToHost, s));
    if (!dev_out)
        NA_CUDA(cudaMemcpyAsync(out_delta, delta, 8ull * g->n, cudaMemcpyDeviceToHost, s));
    NA_CUDA(cudaStreamSynchronize(s));
    if (hctl.error & kErrInternal) return fail_msg(IMIN_ERR_INTERNAL, "dominator iteration did not converge");
    if (hctl.count[1] > 0)
        return fail_msg(IMIN_ERR_CAPACITY,
                        "imin_estimate_decrease_noalloc: a sampled cascade needs the whole-graph "
                        "tier, which this entry point does not run");
    return IMIN_OK;
}
