// Host side of the C ABI declared in omni_mla.h: argument checks, the split-KV plan,
// workspace carving and kernel launches.  Nothing here allocates device memory.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <mutex>

#include "combine.cuh"
#include "common.cuh"
#include "host_gather.cuh"
#include "simt_decode.cuh"
#include "tc_decode.cuh"
#include "tc2_decode.cuh"
#include "tc2q8_decode.cuh"
#include "topk_select.cuh"

namespace omni {
namespace {

constexpr int kMaxSplits = 32;

cudaEvent_t g_profile_before = nullptr, g_profile_after = nullptr;

struct DeviceInfo {
    int sm_count = 0;
    int cc_major = 0;
    int index = -1;
    bool ok = false;
};

// Per-device facts, looked up once per device and process.
const DeviceInfo &device_info()
{
    static DeviceInfo info[64];
    static std::mutex mu;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        static DeviceInfo none;
        return none;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (!info[dev].ok) {
        int sms = 0, major = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) == cudaSuccess) {
            info[dev].sm_count = sms;
            info[dev].cc_major = major;
            info[dev].index = dev;
            info[dev].ok = true;
        }
    }
    return info[dev];
}

bool desc_ok(const omni_mla_desc_t *d)
{
    return d && d->batch >= 1 && d->num_heads >= 1 && d->num_heads <= 128 && d->d_qk == kDqk &&
           d->d_v == kDv && d->page_size == kPage && d->num_pages >= 1 &&
           d->num_pages <= (int64_t)0x7fffffff / kPage && d->max_pages_per_req >= 1 &&
           d->max_sel >= 1 && d->num_splits >= 0 && d->num_splits <= kMaxSplits;
}

// Pages of a compressed layer's rolling cache: the sink pages are kept for good, the ring holds
// the recent window (which can straddle one more page than it fills).
int64_t rolling_sink_pages(int32_t n_sink) { return ((int64_t)n_sink + kPage - 1) / kPage; }
int64_t rolling_ring_pages(int32_t n_recent) { return ((int64_t)n_recent + kPage - 1) / kPage + 1; }

bool aligned(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; }

// Which tensor-core kernel serves a problem: the paired-CTA one (a cluster of two CTAs per work unit)
// unless there are few heads and little to read.  Up to 64 heads leave half of a pair's rows empty, but an M = 128 pair
// runs the tensor pipe at full rate where the single CTA's M = 64 runs it at half rate, with 2 tiles of
// buffers to the pair's 4.  What the single-CTA kernel has is the shorter start and twice as many work units, which
// shows up to 32 heads while two tiles per unit spread over all SMs in one wave (one request of 13 tiles of 16 heads 9.3
// against 9.7 us on pairs, 4 x 33 11.2 against 12.0, 8 x 33 12.8 against 14.8).
// From 40 tiles for one request and 80 for each of two on, pairs are faster all the same: a split (32 at most) is two and more tiles then, at half
// the pair's rate.  One request of 48 tiles 11.1 us against 10.8 on pairs, of 96 13.3 against 12.3, of 192 18.9 against 14.3; two requests of 64
// tiles 11.8 against 13.2, of 96 13.4 against 12.7; four of 64 13.2 against 13.5.  (Three and more reach the limit of one wave before.)
constexpr int kSingleCtaHeads = 32, kSingleCtaUnits = 148, kSingleCtaTiles = 40;     // (units: the SMs of the device this library is for)
bool use_pair_kernel(const omni_mla_desc_t *d)
{
    if (d->flags & OMNI_FLAG_SIMT) return false;
    const int tiles = (d->max_sel + kTile - 1) / kTile;
    return d->num_heads > kSingleCtaHeads || (long)d->batch * ((tiles + 1) / 2) > kSingleCtaUnits || tiles > (long)kSingleCtaTiles * d->batch;
}

// The 8-bit entry point takes more than 64 heads, as the header says: fewer would leave half of a pair's rows and more empty.
bool q8_shape_ok(const omni_mla_desc_t *d) { return !(d->flags & OMNI_FLAG_SIMT) && d->num_heads > kTcHeads; }

// Work units one split of one request occupies in the kernel that will run.
int units_per_request(const omni_mla_desc_t *d)
{
    if (d->flags & OMNI_FLAG_SIMT)
        return (d->num_heads + kSimtWarps * kSimtHeadsPerWarp - 1) / (kSimtWarps * kSimtHeadsPerWarp);
    return 1;
}

// Two splits of a request can be merged inside a cluster of two CTA pairs as long as all those
// clusters are resident at once.
bool merge_in_cluster(const omni_mla_desc_t *d, int splits, int resident_merge_clusters = -1)
{
    if (!(splits == 2 && use_pair_kernel(d) && !(d->flags & (OMNI_FLAG_FUSED_MERGE | OMNI_FLAG_NO_CLUSTER_MERGE))))
        return false;
    if (resident_merge_clusters < 0) resident_merge_clusters = tc2_max_merge_clusters();
    return d->batch <= resident_merge_clusters;
}

// How the requests are split: the first `whole` of them (in the order they are taken) not at all, the others in `splits`.
struct SplitPlan {
    int splits, whole;
};

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

size_t part_out_bytes(const omni_mla_desc_t *d, const SplitPlan &plan)
{
    return align_up((size_t)(d->batch - plan.whole) * plan.splits * d->num_heads * kDv * sizeof(float), 256);
}

size_t part_lse_bytes(const omni_mla_desc_t *d, const SplitPlan &plan)
{
    return align_up((size_t)(d->batch - plan.whole) * plan.splits * d->num_heads * sizeof(float), 256);
}

// Arrival counters of the in-kernel merge: one per (request, CTA of a pair); where only the last requests are cut,
// which ones these are.
size_t counter_bytes(const omni_mla_desc_t *d)
{
    return align_up((size_t)d->batch * 2 * sizeof(int32_t), 256);
}

size_t workspace_need(const omni_mla_desc_t *d, const SplitPlan &plan)
{
    return part_out_bytes(d, plan) + part_lse_bytes(d, plan) + counter_bytes(d);
}

// The number of split-KV partitions per request: minimises waves * (units per split + fixed part) + merge, where the work
// runs in waves over the SMs and the unit of cost is the time of 64 tokens (0.65 to 0.9 us, by how many pairs read):
//  * a unit of the single-CTA kernel takes twice as long, and the merge of its few heads costs 5.5;
//  * on pairs, up to 8 units stay whole (one launch without any merge);
//  * two splits merged inside a cluster of two CTA pairs cost about 3.5;
//  * partial results in global memory and the merge kernel cost about 8 (its launch, latencies), and from 24
//    partial results on a sixteenth more for each of them (up to 256 KiB written and read back);
//    5.5 more per wave when there are several, since the partials then compete with the next wave's loads.
// Fitted to 460 measured (heads, batch, units, splits), whole pages and scattered tokens, which the host cannot tell
// apart.  Against a flat 8 for the merge kernel and 5 for the cluster merge: 4 requests of 16 units 17.6 -> 13.3 us, 16 of
// them 17.6 -> 13.8, 24 x 33 26.6 -> 22.3, 6 x 12 16.4 -> 11.4.
// most_bytes: where the workspace is given, no plan that needs a larger one (a plan without splits needs none).
SplitPlan split_plan(const omni_mla_desc_t *d, int sm_count, int resident_merge_clusters = -1, size_t most_bytes = SIZE_MAX)
{
    if (d->num_splits >= 1) return {d->num_splits, 0};
    if (sm_count <= 0) sm_count = 148;
    constexpr long kUnit = 16;                           // costs are in sixteenths of a unit
    constexpr int kWholeUnits = 8, kTailUnits = 64;
    const bool pair = use_pair_kernel(d), single = !pair && !(d->flags & OMNI_FLAG_SIMT);
    const int granule = pair ? kC2Tile : kTile;
    const int granules = (d->max_sel + granule - 1) / granule;
    const long units = (long)d->batch * units_per_request(d);
    if (pair) sm_count /= 2;                             // a work unit occupies two SMs
    const int most = pair && granules <= kWholeUnits ? 1 : kMaxSplits;
    long best_cost = -1;
    int best = 1;
    for (int s = 1; s <= most && s <= granules; ++s) {
        if (s > 1 && workspace_need(d, {s, 0}) > most_bytes) break;
        const long waves = (units * s + sm_count - 1) / sm_count;
        const long per = (granules + s - 1) / s;
        long cost;
        if (single)
            cost = waves * (2 * per + 6 + (s > 1 && waves > 1 ? 4 : 0)) * kUnit + (s > 1 ? 88 : 0);
        else
            cost = waves * (per + 2) * kUnit;
        if (!single && s > 1) {
            if (merge_in_cluster(d, s, resident_merge_clusters))
                cost += 56;
            else
                cost += 124 + std::max(0l, units * s - 24) + (waves > 1 ? 88 * waves : 0);
        }
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = s;
        }
    }
    // One wave of whole requests and a few more: whole, these would keep at most a third of the pairs busy for as
    // long again, so they are cut into as many pieces as there are pairs.  Requests of one size, and of sizes up to 1 : 1.5,
    // gain 1.08 to 1.46 times (76 x 64 units 118 -> 94 us, 80 x 128 253 -> 179, 98 x 96 192 -> 173).  The host does
    // not see the sizes.  Where they differ so much that the few run beside the longest ones the kernel takes them whole after
    // all (c2_rank_requests) and the merge kernel finds nothing to do; spread over 1 : 3 to 1 : 8 that costs up to
    // 9 % with 88 or 98 requests (98 x 64 89 -> 98 us, 98 x 128 170 -> 176) and still gains with 76 or 80 long ones
    // (80 x 128 163 -> 152).  Below 64 units the loss is the larger part.
    const int tail = d->batch - sm_count;
    if (pair && tail > 0 && 3 * tail <= sm_count && granules >= kTailUnits && !(d->flags & OMNI_FLAG_FUSED_MERGE)) {
        const int pieces = std::min(kMaxSplits, sm_count / tail), per = std::max(2, (granules + pieces - 1) / pieces);
        const int s = (granules + per - 1) / per;
        const long cost = (granules + 2 + per + 2) * kUnit + 212 + std::max(0, tail * s - 24);
        if (s > 1 && d->batch <= 256 && cost < best_cost && workspace_need(d, {s, sm_count}) <= most_bytes) return {s, sm_count};
    }
    return {best, 0};
}

// Splits of every request, as the queries report them (1 if only the last few are cut).
int choose_splits(const omni_mla_desc_t *d, int sm_count, int resident_merge_clusters = -1)
{
    const SplitPlan plan = split_plan(d, sm_count, resident_merge_clusters);
    return plan.whole > 0 ? 1 : plan.splits;
}

// On request the paired-CTA kernel merges the splits itself (the last CTA to finish a request's
// head half does it); by default a second, programmatically dependent kernel spreads the merge
// over all SMs, which is faster when every split of a batch finishes at about the same time.
bool merge_in_kernel(const omni_mla_desc_t *d)
{
    return use_pair_kernel(d) && (d->flags & OMNI_FLAG_FUSED_MERGE);
}

// The form of the paired-CTA kernel that serves a problem (see tc2_kernel_for): two splits merged inside a cluster, several work units per
// pair, or one.  Several where there are more units than pairs and they are taken by size (not more than 256 requests), short, and
// neither cut at the end only nor merged by the last CTA of a request; the units are dealt out as pairs become free.  What is saved is
// part of the start and the end of every unit but a pair's first; the longer a unit, the more its main loop weighs, which takes longer in this form.
// One unit per pair -> several, us, by the longest unit: 100 alike 16 46.8 -> 44.0, 24 63.5 -> 62.9, 32 79.1 -> 80.5, 40 95.5 -> 96.8, 48 113 -> 115; 148 alike 16
// 58.7 -> 55.5, 24 79.4 -> 80.4, 32 102 -> 100, 40 126 -> 125, 48 143 -> 148, 64 182 -> 189; 200 from 4 units up to 32 89.4 -> 83.0, to 40 103 -> 99, to 48
// 118 -> 116, to 64 146 -> 146.
constexpr int kMultiUnits = 32;
int pair_form(const omni_mla_desc_t *d, int splits, int whole, bool cluster_merge, bool fused_merge, int pairs)
{
    if (cluster_merge) return 1;
    const int longest = ((d->max_sel + kC2Tile - 1) / kC2Tile + splits - 1) / splits;
    return whole == 0 && !fused_merge && d->batch <= 256 && (long)d->batch * splits > pairs && longest <= kMultiUnits ? 2 : 0;
}

// Launch whose blocks may become resident while the kernel in front of it in the stream still runs
// (programmatic dependent launch); the kernel itself waits (griddepcontrol.wait) before it touches
// global memory, so only the launch gap between the two kernels goes away.
template <class... KernelArgs, class... CallArgs>
omni_status_t launch_overlapped(void (*kernel)(KernelArgs...), unsigned blocks, unsigned threads, cudaStream_t stream, CallArgs... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, KernelArgs(args)...) == cudaSuccess ? OMNI_OK : OMNI_ERR_CUDA;
}

// Merges `sets` sets of partial results; the s-th is that of request[s] (null: of request s) among `batch`.
omni_status_t launch_combine(int sets, int batch, int heads, int max_splits, const float *part_out,
                             const float *part_lse, const int32_t *num_splits, const int32_t *request, void *out,
                             float *lse, cudaStream_t stream)
{
    // Keep the shared-memory / L1 split the decode kernel needs: alternating between two splits
    // makes every launch wait for the SMs to be reconfigured.
    static const bool carveout_set = [] {
        cudaFuncSetAttribute(combine_kernel<1>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        cudaFuncSetAttribute(combine_kernel<4>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        return true;
    }();
    (void)carveout_set;
    // Four thread groups per block while all blocks fit the SMs at once (three of 512 threads per SM)
    // and there are more splits than one thread keeps in flight.
    const int blocks = sets * heads;
    const bool wide = max_splits > kCombineAhead && blocks <= 3 * device_info().sm_count;
    return launch_overlapped(wide ? combine_kernel<4> : combine_kernel<1>, (unsigned)blocks, wide ? 512 : 128, stream, part_out,
                             part_lse, num_splits, request, batch, max_splits, heads, static_cast<__nv_bfloat16 *>(out), lse);
}

omni_status_t launch_resolve(const omni_mla_desc_t *d, const int32_t *page_table,
                             const int32_t *sel_idx, const int32_t *sel_len, int64_t *rows,
                             int32_t *status, cudaStream_t stream)
{
    dim3 grid((unsigned)min(64, (d->max_sel + 255) / 256), (unsigned)d->batch);
    resolve_rows_kernel<<<grid, 256, 0, stream>>>(page_table, sel_idx, sel_len,
                                                  d->max_pages_per_req, d->max_sel, d->num_pages,
                                                  rows, status);
    return cudaPeekAtLastError() == cudaSuccess ? OMNI_OK : OMNI_ERR_CUDA;
}

// Self-test of the bounded wait every kernel here relies on: one warp waits, with the given
// limit, on a barrier that nobody ever arrives on.  No copy and no tensor memory is involved;
// the warp reports what the product kernels report when a wait runs out and returns.
__global__ void __launch_bounds__(32) bounded_wait_selftest_kernel(long long limit_cycles, int32_t *status,
                                                                   long long *waited_cycles)
{
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    const long long t0 = clock64();
    bool ok = mbar_wait(&bar, 0, limit_cycles);
    ok = __all_sync(0xffffffffu, ok);
    const long long t1 = clock64();
    if (threadIdx.x == 0) {
        if (!ok) flag_status(status, OMNI_DEV_TIMEOUT | OMNI_DEV_ROLE_SOFTMAX);
        if (waited_cycles) *waited_cycles = t1 - t0;
    }
}

}  // namespace
}  // namespace omni

using namespace omni;

extern "C" {

int omni_version(void) { return 1000; }

void omni_sparse_mla_set_profile_events(void *before, void *after)
{
    g_profile_before = static_cast<cudaEvent_t>(before);
    g_profile_after = static_cast<cudaEvent_t>(after);
}

const char *omni_status_string(omni_status_t status)
{
    switch (status) {
        case OMNI_OK: return "ok";
        case OMNI_ERR_NULL: return "null pointer";
        case OMNI_ERR_SHAPE: return "unsupported or inconsistent shape";
        case OMNI_ERR_ALIGN: return "misaligned pointer";
        case OMNI_ERR_WORKSPACE: return "workspace too small";
        case OMNI_ERR_INDEX: return "index out of range";
        case OMNI_ERR_TIMEOUT: return "device wait timed out";
        case OMNI_ERR_CUDA: return "CUDA call failed";
        case OMNI_ERR_ARCH: return "device is not compute capability 10.x";
    }
    return "unknown status";
}

int32_t omni_sparse_mla_num_splits(const omni_mla_desc_t *desc)
{
    if (!desc_ok(desc)) return 0;
    return choose_splits(desc, device_info().sm_count);
}

int32_t omni_sparse_mla_num_launches(const omni_mla_desc_t *desc)
{
    if (!desc_ok(desc)) return 0;
    const SplitPlan plan = split_plan(desc, device_info().sm_count);
    const int s = plan.splits;
    int n = 1 + ((desc->flags & OMNI_FLAG_VALIDATE) ? 1 : 0);
    if (plan.whole > 0) return n + 1;
    if (s > 1 && !merge_in_cluster(desc, s) && !(use_pair_kernel(desc) && (desc->flags & OMNI_FLAG_FUSED_MERGE))) ++n;
    return n;
}

int32_t omni_sparse_mla_plan_query(const omni_mla_desc_t *desc, int32_t sm_count, int32_t resident_merge_clusters,
                                   int32_t *num_launches)
{
    if (!desc_ok(desc) || sm_count < 1 || resident_merge_clusters < 0) return 0;
    const SplitPlan plan = split_plan(desc, sm_count, resident_merge_clusters);
    const int s = plan.whole > 0 ? 1 : plan.splits;
    if (num_launches) {
        int n = 1 + ((desc->flags & OMNI_FLAG_VALIDATE) ? 1 : 0);
        if (plan.whole > 0) ++n;
        if (s > 1 && !merge_in_cluster(desc, s, resident_merge_clusters) &&
            !(use_pair_kernel(desc) && (desc->flags & OMNI_FLAG_FUSED_MERGE)))
            ++n;
        *num_launches = n;
    }
    return s;
}

// Part of the tests of the dispatch: the form of the paired-CTA kernel that a call with a workspace takes, or -1 where another kernel serves it.
int32_t omni_internal_pair_form(const omni_mla_desc_t *desc, int32_t sm_count, int32_t resident_merge_clusters)
{
    if (!desc_ok(desc) || sm_count < 1 || resident_merge_clusters < 0 || !use_pair_kernel(desc)) return -1;
    const SplitPlan plan = split_plan(desc, sm_count, resident_merge_clusters);
    return pair_form(desc, plan.splits, plan.whole, plan.whole == 0 && merge_in_cluster(desc, plan.splits, resident_merge_clusters),
                     plan.splits > 1 && merge_in_kernel(desc), sm_count / 2);
}

size_t omni_sparse_mla_workspace_bytes(const omni_mla_desc_t *desc)
{
    if (!desc_ok(desc)) return 0;
    return workspace_need(desc, split_plan(desc, device_info().sm_count));
}

// Everything about a decode call that depends only on the descriptor, q and the pool: which
// kernel, the split plan, workspace carving, tensor maps.  The ordinary entry points build
// one per call (maps come from the cache); omni_sparse_mla_plan_init stores one in caller
// memory so that omni_sparse_mla_decode_planned only fills in pointers and launches.
constexpr uint32_t kPlanMagic = 0x4c504d4fu;
struct LaunchPlan {
    uint32_t magic;
    int32_t kernel;            // 0 plain-FMA, 1 single-CTA tensor-core, 2 paired-CTA tensor-core, 3 the same over the 8-bit cache
    int32_t splits, whole;     // the first `whole` requests are not split
    int32_t cluster_merge, longest_first, fused_merge, pairs;   // pairs: that the device holds
    int32_t device;
    size_t need, part_out, part_lse, counters;
    omni_mla_desc_t desc;
    const void *q, *kv;
    const float *kv_scale;     // 8-bit cache only
    alignas(64) CUtensorMap maps[5];
};
static_assert(sizeof(LaunchPlan) <= sizeof(omni_mla_plan_t), "plan does not fit its public container");
static_assert(alignof(LaunchPlan) <= 64, "plan alignment");

// most_bytes: see split_plan
static omni_status_t build_plan(const omni_mla_desc_t *desc, const void *q, const void *kv_cache, bool cached_maps,
                                LaunchPlan *plan, const float *kv_scale = nullptr, bool q8 = false, size_t most_bytes = SIZE_MAX)
{
    if (!desc || !q || !kv_cache || (q8 && !kv_scale)) return OMNI_ERR_NULL;
    if (!desc_ok(desc)) return OMNI_ERR_SHAPE;
    if (q8 && !q8_shape_ok(desc)) return OMNI_ERR_SHAPE;
    if (!aligned(q, 16) || !aligned(kv_cache, 128) || !aligned(kv_scale, 4)) return OMNI_ERR_ALIGN;
    const DeviceInfo &dev = device_info();
    if (!dev.ok) return OMNI_ERR_CUDA;
    if (dev.cc_major != 10) return OMNI_ERR_ARCH;
    plan->desc = *desc;
    plan->q = q;
    plan->kv = kv_cache;
    plan->kv_scale = kv_scale;
    plan->device = dev.index;
    plan->kernel = q8 ? 3 : (desc->flags & OMNI_FLAG_SIMT) ? 0 : use_pair_kernel(desc) ? 2 : 1;
    const SplitPlan cut = split_plan(desc, dev.sm_count, -1, most_bytes);
    const int splits = cut.splits;
    plan->splits = splits;
    plan->whole = cut.whole;
    plan->part_out = part_out_bytes(desc, cut);
    plan->part_lse = part_lse_bytes(desc, cut);
    plan->counters = counter_bytes(desc);
    plan->need = workspace_need(desc, cut);
    // Two splits of a request can be merged inside a cluster of two CTA pairs, without partial
    // results in global memory, as long as all those clusters are resident at once.
    plan->cluster_merge = (cut.whole == 0 && merge_in_cluster(desc, splits)) ? 1 : 0;
    plan->fused_merge = (splits > 1 && merge_in_kernel(desc)) ? 1 : 0;
    // several waves of work units: start the longest requests first (the kernel ranks them itself)
    plan->longest_first = (plan->kernel >= 2 && !plan->cluster_merge && desc->batch <= 256 &&
                           (long)desc->batch * splits > dev.sm_count / 2)
                              ? 1
                              : 0;
    plan->pairs = dev.sm_count / 2;
    DecodeParams shape = {};
    shape.q = static_cast<const __nv_bfloat16 *>(q);
    shape.kv = static_cast<const __nv_bfloat16 *>(kv_cache);
    shape.num_pages = desc->num_pages;
    shape.batch = desc->batch;
    shape.heads = desc->num_heads;
    if (plan->kernel == 3) {
        if (!tc2q8_prepare_device() || !tc2q8_make_maps(shape, plan->maps, cached_maps)) return OMNI_ERR_CUDA;
    } else if (plan->kernel == 2) {
        if (!tc2_prepare_device() || !tc2_make_maps(shape, plan->maps, cached_maps)) return OMNI_ERR_CUDA;
    } else if (plan->kernel == 1) {
        if (!tc_prepare_device() || !tc_make_maps(shape, plan->maps, cached_maps)) return OMNI_ERR_CUDA;
    }
    plan->magic = kPlanMagic;
    return OMNI_OK;
}

// Checks of the per-step arguments that need no device.
static omni_status_t check_step_args(const omni_mla_desc_t *desc, const int32_t *page_table, const int32_t *sel_idx,
                                     const int32_t *sel_len, const int32_t *ctx_len, int32_t n_sink, int32_t n_recent,
                                     bool rolling, const void *out, const float *lse)
{
    const bool ranges = sel_idx == nullptr;
    if (!page_table || !out || !lse) return OMNI_ERR_NULL;
    if (ranges ? !ctx_len : !sel_len) return OMNI_ERR_NULL;
    if (ranges) {
        // max_sel bounds the selection size the split plan is made for
        if (n_sink < 0 || n_recent < 0) return OMNI_ERR_SHAPE;
        const int64_t longest = (int64_t)desc->max_pages_per_req * kPage;
        // a rolling cache holds contexts of any length, so only N_sink + N_recent bounds the selection
        const int64_t bound = (rolling || (int64_t)n_sink + n_recent < longest) ? (int64_t)n_sink + n_recent : longest;
        if ((int64_t)desc->max_sel < bound) return OMNI_ERR_SHAPE;
        if (rolling && (int64_t)desc->max_pages_per_req < rolling_sink_pages(n_sink) + rolling_ring_pages(n_recent))
            return OMNI_ERR_SHAPE;
    }
    if (!aligned(out, 16) || !aligned(lse, 4) || !aligned(page_table, 4) || !aligned(sel_idx, 4) || !aligned(sel_len, 4) ||
        !aligned(ctx_len, 4))
        return OMNI_ERR_ALIGN;
    return OMNI_OK;
}

// The per-call half: pointer checks, workspace carving, launches.  The selection is an index
// list (sel_idx, sel_len) or, with sel_idx == nullptr, Eq. 2's ranges (ctx_len, n_sink, n_recent).
static omni_status_t run_plan(const LaunchPlan &plan, const int32_t *page_table, const int32_t *sel_idx,
                              const int32_t *sel_len, const int32_t *ctx_len, int32_t n_sink, int32_t n_recent,
                              bool rolling, void *out, float *lse, void *workspace, size_t workspace_bytes,
                              int32_t *device_status, void *stream_)
{
    const omni_mla_desc_t *desc = &plan.desc;
    const bool ranges = sel_idx == nullptr;
    omni_status_t args = check_step_args(desc, page_table, sel_idx, sel_len, ctx_len, n_sink, n_recent, rolling, out, lse);
    if (args != OMNI_OK) return args;
    // Without a workspace nothing is cut, unless the caller asked for the cut: which requests the plan cuts is the library's
    // own affair, and a caller who brings none must not depend on it.
    const bool whole = !workspace && desc->num_splits == 0;
    const int splits = whole ? 1 : plan.splits;
    const bool cluster_merge = !whole && plan.cluster_merge, fused_merge = !whole && plan.fused_merge;
    if (splits > 1) {
        if (!workspace) return OMNI_ERR_NULL;
        if (!aligned(workspace, 256)) return OMNI_ERR_ALIGN;
        if (workspace_bytes < plan.need) return OMNI_ERR_WORKSPACE;
    }
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);

    if ((desc->flags & OMNI_FLAG_VALIDATE) && !ranges) {
        omni_status_t st = launch_resolve(desc, page_table, sel_idx, sel_len, nullptr, device_status, stream);
        if (st != OMNI_OK) return st;
    }

    DecodeParams p;
    p.q = static_cast<const __nv_bfloat16 *>(plan.q);
    p.kv = static_cast<const __nv_bfloat16 *>(plan.kv);
    p.kv_scale = plan.kv_scale;
    p.page_table = page_table;
    p.sel_idx = sel_idx;
    p.sel_len = sel_len;
    p.ctx_len = ctx_len;
    p.n_sink = n_sink;
    p.n_recent = n_recent;
    p.sink_pages = rolling ? (int32_t)rolling_sink_pages(n_sink) : 0;
    p.ring_pages = rolling ? (int32_t)rolling_ring_pages(n_recent) : 0;
    p.out = static_cast<__nv_bfloat16 *>(out);
    p.lse = lse;
    p.part_out = static_cast<float *>(workspace);
    p.part_lse = splits > 1 ? reinterpret_cast<float *>(static_cast<char *>(workspace) + plan.part_out) : nullptr;
    p.status = device_status;
    p.counters = nullptr;
    p.whole = whole ? 0 : plan.whole;
    p.tail_request = p.whole > 0 ? reinterpret_cast<int32_t *>(static_cast<char *>(workspace) + plan.part_out + plan.part_lse) : nullptr;
    p.cluster_merge = cluster_merge ? 1 : 0;
    const int form = pair_form(desc, splits, p.whole, cluster_merge, fused_merge, plan.pairs);
    p.longest_first = plan.longest_first || (plan.kernel == 2 && form == 2);
    if (fused_merge) {
        p.counters = reinterpret_cast<int32_t *>(static_cast<char *>(workspace) + plan.part_out + plan.part_lse);
        if (cudaMemsetAsync(p.counters, 0, plan.counters, stream) != cudaSuccess) return OMNI_ERR_CUDA;
    }
    p.num_pages = desc->num_pages;
    p.batch = desc->batch;
    p.heads = desc->num_heads;
    p.max_pages = desc->max_pages_per_req;
    p.max_sel = desc->max_sel;
    p.splits = splits;
    p.scale_log2 = desc->softmax_scale * kLog2e;

    const bool profile = g_profile_before && g_profile_after;
    if (profile) cudaEventRecord(g_profile_before, stream);
    omni_status_t st = OMNI_OK;
    if (plan.kernel == 0) {
        const int grid = desc->batch * splits * units_per_request(desc);
        simt_decode_kernel<<<grid, kSimtWarps * 32, 0, stream>>>(p);
        if (cudaPeekAtLastError() != cudaSuccess) st = OMNI_ERR_CUDA;
    } else {
        st = plan.kernel == 3   ? tc2q8_launch(plan.maps, p, stream)
             : plan.kernel == 2 ? tc2_launch(plan.maps, p, form, stream)
                                : tc_launch(plan.maps, p, stream);
    }
    if (st != OMNI_OK) return st;
    if (profile) cudaEventRecord(g_profile_after, stream);
    if (splits > 1 && p.counters == nullptr && !p.cluster_merge)
        return launch_combine(desc->batch - p.whole, desc->batch, desc->num_heads, splits, p.part_out, p.part_lse, nullptr, p.tail_request,
                              out, lse, stream);
    return OMNI_OK;
}

static omni_status_t decode_impl(const omni_mla_desc_t *desc, const void *q, const void *kv_cache,
                                 const int32_t *page_table, const int32_t *sel_idx,
                                 const int32_t *sel_len, const int32_t *ctx_len, int32_t n_sink,
                                 int32_t n_recent, bool rolling, void *out, float *lse, void *workspace,
                                 size_t workspace_bytes, int32_t *device_status, void *stream, size_t most_bytes = SIZE_MAX)
{
    // everything the host can check is checked before the device is asked anything
    if (!desc || !q || !kv_cache || !page_table || !out || !lse) return OMNI_ERR_NULL;
    if (sel_idx == nullptr ? !ctx_len : !sel_len) return OMNI_ERR_NULL;
    if (!desc_ok(desc)) return OMNI_ERR_SHAPE;
    omni_status_t st = check_step_args(desc, page_table, sel_idx, sel_len, ctx_len, n_sink, n_recent, rolling, out, lse);
    if (st == OMNI_OK && (!aligned(q, 16) || !aligned(kv_cache, 128))) st = OMNI_ERR_ALIGN;
    if (st != OMNI_OK) return st;
    LaunchPlan plan;
    st = build_plan(desc, q, kv_cache, true, &plan, nullptr, false, most_bytes);
    if (st != OMNI_OK) return st;
    return run_plan(plan, page_table, sel_idx, sel_len, ctx_len, n_sink, n_recent, rolling, out, lse, workspace,
                    workspace_bytes, device_status, stream);
}

omni_status_t omni_sparse_mla_decode_q8(const omni_mla_desc_t *desc, const void *q, const void *kv_q8,
                                        const float *kv_scale, const int32_t *page_table, const int32_t *sel_idx,
                                        const int32_t *sel_len, void *out, float *lse, void *workspace,
                                        size_t workspace_bytes, int32_t *device_status, void *stream)
{
    if (!desc || !q || !kv_q8 || !kv_scale || !page_table || !sel_idx || !sel_len || !out || !lse) return OMNI_ERR_NULL;
    if (!desc_ok(desc) || !q8_shape_ok(desc)) return OMNI_ERR_SHAPE;
    omni_status_t st = check_step_args(desc, page_table, sel_idx, sel_len, nullptr, 0, 0, false, out, lse);
    if (st == OMNI_OK && (!aligned(q, 16) || !aligned(kv_q8, 128) || !aligned(kv_scale, 4))) st = OMNI_ERR_ALIGN;
    if (st != OMNI_OK) return st;
    LaunchPlan plan;
    st = build_plan(desc, q, kv_q8, true, &plan, kv_scale, true);
    if (st != OMNI_OK) return st;
    return run_plan(plan, page_table, sel_idx, sel_len, nullptr, 0, 0, false, out, lse, workspace, workspace_bytes,
                    device_status, stream);
}

omni_status_t omni_kv_quantize_q8(const void *kv_rows, int64_t num_rows, void *kv_q8, float *kv_scale, void *stream)
{
    if (!kv_rows || !kv_q8 || !kv_scale) return OMNI_ERR_NULL;
    if (num_rows < 1 || num_rows > (int64_t)0x7fffffff * 8) return OMNI_ERR_SHAPE;
    if (!aligned(kv_rows, 16) || !aligned(kv_q8, 128) || !aligned(kv_scale, 4)) return OMNI_ERR_ALIGN;
    constexpr int kRowsPerBlock = kQ8QuantWarps * kQ8RowsPerWarp;
    return launch_overlapped(quantize_q8_kernel, (unsigned)((num_rows + kRowsPerBlock - 1) / kRowsPerBlock), kQ8QuantWarps * 32,
                             static_cast<cudaStream_t>(stream), static_cast<const __nv_bfloat16 *>(kv_rows), num_rows,
                             static_cast<uint8_t *>(kv_q8), kv_scale);
}

omni_status_t omni_sparse_mla_plan_init(const omni_mla_desc_t *desc, const void *q, const void *kv_cache,
                                        omni_mla_plan_t *plan)
{
    if (!plan) return OMNI_ERR_NULL;
    if (!aligned(plan, 64)) return OMNI_ERR_ALIGN;
    LaunchPlan *lp = reinterpret_cast<LaunchPlan *>(plan);
    lp->magic = 0;
    return build_plan(desc, q, kv_cache, false, lp);
}

omni_status_t omni_sparse_mla_decode_planned(const omni_mla_plan_t *plan, const int32_t *page_table,
                                             const int32_t *sel_idx, const int32_t *sel_len, void *out,
                                             float *lse, void *workspace, size_t workspace_bytes,
                                             int32_t *device_status, void *stream)
{
    if (!plan || !sel_idx) return OMNI_ERR_NULL;
    if (!aligned(plan, 64)) return OMNI_ERR_ALIGN;
    const LaunchPlan *lp = reinterpret_cast<const LaunchPlan *>(plan);
    if (lp->magic != kPlanMagic) return OMNI_ERR_SHAPE;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != lp->device) return OMNI_ERR_CUDA;
    return run_plan(*lp, page_table, sel_idx, sel_len, nullptr, 0, 0, false, out, lse, workspace, workspace_bytes,
                    device_status, stream);
}

omni_status_t omni_sparse_mla_decode(const omni_mla_desc_t *desc, const void *q,
                                     const void *kv_cache, const int32_t *page_table,
                                     const int32_t *sel_idx, const int32_t *sel_len, void *out,
                                     float *lse, void *workspace, size_t workspace_bytes,
                                     int32_t *device_status, void *stream)
{
    if (!sel_idx) return OMNI_ERR_NULL;
    return decode_impl(desc, q, kv_cache, page_table, sel_idx, sel_len, nullptr, 0, 0, false, out, lse, workspace,
                       workspace_bytes, device_status, stream);
}

omni_status_t omni_sparse_mla_decode_sink_recent(const omni_mla_desc_t *desc, const void *q,
                                                 const void *kv_cache, const int32_t *page_table,
                                                 const int32_t *ctx_len, int32_t n_sink,
                                                 int32_t n_recent, void *out, float *lse,
                                                 void *workspace, size_t workspace_bytes,
                                                 int32_t *device_status, void *stream)
{
    return decode_impl(desc, q, kv_cache, page_table, nullptr, nullptr, ctx_len, n_sink, n_recent, false, out, lse,
                       workspace, workspace_bytes, device_status, stream);
}

omni_status_t omni_sparse_mla_decode_rolling(const omni_mla_desc_t *desc, const void *q,
                                             const void *kv_cache, const int32_t *page_table,
                                             const int32_t *ctx_len, int32_t n_sink, int32_t n_recent,
                                             void *out, float *lse, void *workspace,
                                             size_t workspace_bytes, int32_t *device_status, void *stream)
{
    return decode_impl(desc, q, kv_cache, page_table, nullptr, nullptr, ctx_len, n_sink, n_recent, true, out, lse,
                       workspace, workspace_bytes, device_status, stream);
}

// Part of omni_sparse_mla_decode_static (static_scratch.cu): the plan is the best one that the library's own scratch holds.
// Only a cut that the caller asked for can be too large.
omni_status_t omni_internal_decode_fitting(const omni_mla_desc_t *desc, const void *q, const void *kv_cache, const int32_t *page_table,
                                           const int32_t *sel_idx, const int32_t *sel_len, void *out, float *lse, void *scratch,
                                           size_t scratch_bytes, int32_t *device_status, void *stream)
{
    if (!sel_idx) return OMNI_ERR_NULL;
    return decode_impl(desc, q, kv_cache, page_table, sel_idx, sel_len, nullptr, 0, 0, false, out, lse, scratch, scratch_bytes,
                       device_status, stream, scratch_bytes);
}

omni_status_t omni_topk_select(const float *scores, const int32_t *ctx_len, int32_t batch, int32_t stride,
                               int32_t k, int32_t *sel_idx, int32_t *sel_len, void *stream)
{
    if (!scores || !ctx_len || !sel_idx || !sel_len) return OMNI_ERR_NULL;
    if (batch < 1 || stride < 1 || stride > kTopkMaxContext || k < 1 || k > stride) return OMNI_ERR_SHAPE;
    if (!aligned(scores, 4) || !aligned(ctx_len, 4) || !aligned(sel_idx, 4) || !aligned(sel_len, 4)) return OMNI_ERR_ALIGN;
    const DeviceInfo &dev = device_info();
    if (!dev.ok) return OMNI_ERR_CUDA;
    if (dev.cc_major != 10) return OMNI_ERR_ARCH;
    return launch_topk_select(scores, ctx_len, batch, stride, k, sel_idx, sel_len, static_cast<cudaStream_t>(stream));
}

int32_t omni_rolling_pages_per_request(int32_t n_sink, int32_t n_recent)
{
    if (n_sink < 0 || n_recent < 0) return 0;
    const int64_t pages = rolling_sink_pages(n_sink) + rolling_ring_pages(n_recent);
    return pages > 0x7fffffff ? 0 : (int32_t)pages;
}

omni_status_t omni_kv_append_rolling(const omni_mla_desc_t *desc, void *kv_cache,
                                     const int32_t *page_table, const int32_t *ctx_len,
                                     const void *new_rows, int32_t n_sink, int32_t n_recent,
                                     int32_t *device_status, void *stream)
{
    if (!desc || !kv_cache || !page_table || !ctx_len || !new_rows) return OMNI_ERR_NULL;
    if (!desc_ok(desc) || n_sink < 0 || n_recent < 0) return OMNI_ERR_SHAPE;
    if ((int64_t)desc->max_pages_per_req < rolling_sink_pages(n_sink) + rolling_ring_pages(n_recent)) return OMNI_ERR_SHAPE;
    if (!aligned(kv_cache, 128) || !aligned(new_rows, 16) || !aligned(page_table, 4) || !aligned(ctx_len, 4))
        return OMNI_ERR_ALIGN;
    return launch_overlapped(append_rolling_kernel, (unsigned)desc->batch, 72, static_cast<cudaStream_t>(stream),
                             static_cast<__nv_bfloat16 *>(kv_cache), page_table, ctx_len, static_cast<const __nv_bfloat16 *>(new_rows),
                             desc->max_pages_per_req, desc->num_pages, (int)rolling_sink_pages(n_sink),
                             (int)rolling_ring_pages(n_recent), device_status);
}

omni_status_t omni_sparse_mla_combine(const omni_mla_desc_t *desc, int32_t max_splits,
                                      const float *part_out, const float *part_lse,
                                      const int32_t *num_splits, void *out, float *lse,
                                      void *stream)
{
    if (!desc || !part_out || !part_lse || !out || !lse) return OMNI_ERR_NULL;
    if (desc->batch < 1 || desc->num_heads < 1 || desc->d_v != kDv || max_splits < 1)
        return OMNI_ERR_SHAPE;
    if (!aligned(part_out, 16) || !aligned(out, 8) || !aligned(part_lse, 4) || !aligned(lse, 4))
        return OMNI_ERR_ALIGN;
    return launch_combine(desc->batch, desc->batch, desc->num_heads, max_splits, part_out, part_lse, num_splits, nullptr,
                          out, lse, static_cast<cudaStream_t>(stream));
}

omni_status_t omni_selftest_bounded_wait(int64_t limit_cycles, int32_t *device_status, int64_t *waited_cycles,
                                         void *stream)
{
    if (!device_status) return OMNI_ERR_NULL;
    if (limit_cycles < 1 || limit_cycles > ((int64_t)1 << 31)) return OMNI_ERR_SHAPE;
    if (!aligned(device_status, 4) || !aligned(waited_cycles, 8)) return OMNI_ERR_ALIGN;
    bounded_wait_selftest_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(
        (long long)limit_cycles, device_status, reinterpret_cast<long long *>(waited_cycles));
    return cudaPeekAtLastError() == cudaSuccess ? OMNI_OK : OMNI_ERR_CUDA;
}

omni_status_t omni_sparse_mla_validate(const omni_mla_desc_t *desc, const int32_t *page_table,
                                       const int32_t *sel_idx, const int32_t *sel_len,
                                       int32_t *device_status, void *stream)
{
    if (!desc || !page_table || !sel_idx || !sel_len || !device_status) return OMNI_ERR_NULL;
    if (!desc_ok(desc)) return OMNI_ERR_SHAPE;
    return launch_resolve(desc, page_table, sel_idx, sel_len, nullptr, device_status,
                          static_cast<cudaStream_t>(stream));
}

omni_status_t omni_sparse_mla_resolve_rows(const omni_mla_desc_t *desc,
                                           const int32_t *page_table, const int32_t *sel_idx,
                                           const int32_t *sel_len, int64_t *rows, void *stream)
{
    if (!desc || !page_table || !sel_idx || !sel_len || !rows) return OMNI_ERR_NULL;
    if (!desc_ok(desc)) return OMNI_ERR_SHAPE;
    return launch_resolve(desc, page_table, sel_idx, sel_len, rows, nullptr,
                          static_cast<cudaStream_t>(stream));
}


// The host-buffer entry point moves q and the index arrays in and out and lse back over PCIe, which carries
// both directions at once.  With pinned buffers, which is what they are for, one kernel reads the index arrays (see
// host_gather.cuh).  A small batch runs as one part: that kernel reads q too, and the decode
// kernels store out and lse straight into the host buffers (a copy out would start only after their last
// store, and costs 4-7 us of its own): one request of 16 heads 49 -> 20 us, four of 128 77 -> 47.
// A large batch runs as up to four parts: on one stream of the library's the copy engine brings q,
// part after part, on another it takes the results of a part back, and the kernels run on the
// caller's stream, which both fork from and join back into.  The copy engines do it there because
// reads and writes of the SMs over PCIe hold each other up (5 MB each way: 201 us together, 125 with
// the copy engine reading); only the last part, which has PCIe to itself, stores its results in
// place.  32 requests: 203 -> 178 us, of which 125 are the transfers if both directions overlapped
// throughout.
// Other host memory goes through copies, a large batch in two halves.
static size_t host_copy_bytes(const omni_mla_desc_t *desc)
{
    const size_t B = desc->batch, H = desc->num_heads;
    return align_up(B * H * kDqk * 2, 256) + align_up(B * desc->max_pages_per_req * 4, 256) +
           align_up(B * desc->max_sel * 4, 256) + align_up(B * 4, 256) +
           align_up(B * H * kDv * 2, 256) + align_up(B * H * 4, 256);
}

static bool host_pipelined(const omni_mla_desc_t *desc)
{
    const size_t B = desc->batch, H = desc->num_heads;
    return desc->batch >= 4 && B * H * (kDqk + kDv) * 2 >= (size_t)(2u << 20);
}

static omni_mla_desc_t host_half_desc(const omni_mla_desc_t *desc, int half)
{
    omni_mla_desc_t d = *desc;
    const int first = (desc->batch + 1) / 2;       // even halves measured better than 5/8 : 3/8
    d.batch = half == 0 ? first : desc->batch - first;
    return d;
}

static size_t host_half_workspace(const omni_mla_desc_t *desc, int half)
{
    const omni_mla_desc_t d = host_half_desc(desc, half);
    return align_up(workspace_need(&d, split_plan(&d, device_info().sm_count)), 256);
}

// Side streams of the host-buffer entry point: a few per device, chosen by the caller's stream, so
// that calls in flight on different streams do not queue their second halves behind one another.
constexpr int kHostSideStreams = 4;
static cudaStream_t host_side_stream(cudaStream_t caller, int which = 0)
{
    static std::mutex lock;
    static cudaStream_t all[2][64][kHostSideStreams] = {};
    cudaStream_t(*streams)[kHostSideStreams] = all[which];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    const uintptr_t h = reinterpret_cast<uintptr_t>(caller);
    const int slot = (int)(((h >> 4) ^ (h >> 12) ^ (h >> 20)) % kHostSideStreams);
    std::lock_guard<std::mutex> guard(lock);
    if (!streams[dev][slot] && cudaStreamCreateWithFlags(&streams[dev][slot], cudaStreamNonBlocking) != cudaSuccess)
        streams[dev][slot] = nullptr;
    return streams[dev][slot];
}

// Parts of a large batch in pinned buffers.  The last part is the smallest: its kernel and its results are what
// nothing overlaps.  Where the kernels take longer than the transfers, parts only cost efficiency:
// two halves keep the first transfer in and the last one out short.  Returns how many, their sizes in `size`.
constexpr int kHostParts = 4;
static int host_parts(const omni_mla_desc_t *desc, int *size)
{
    const int B = desc->batch;
    size[0] = B;
    // one part up to 3.5 MB of q and out (12 requests of 128 heads: 105 us either way, 20: 152 against 142)
    if (!host_pipelined(desc) || (size_t)B * desc->num_heads * (kDqk + kDv) * 2 <= (size_t)(3584u << 10)) return 1;
    const double tiles = (desc->max_sel + kTile - 1) / kTile;
    const double kernel_us = 0.9 * B * tiles / 74, copy_us = (double)B * desc->num_heads * (kDqk * 2) / 50e3;
    if (B < 8 || kernel_us > copy_us) {
        size[0] = (B + 1) / 2;
        size[1] = B - size[0];
        return 2;
    }
    size[3] = B / 8;
    size[2] = B / 4;
    size[1] = (B - size[3] - size[2]) / 2;
    size[0] = B - size[3] - size[2] - size[1];
    return 4;
}

static size_t host_part_workspace(const omni_mla_desc_t *desc)
{
    int size[kHostParts];
    const int n = host_parts(desc, size);
    size_t need = 0;
    for (int i = 0; i < n; ++i) {
        omni_mla_desc_t d = *desc;
        d.batch = size[i];
        const size_t w = workspace_need(&d, split_plan(&d, device_info().sm_count));
        need = w > need ? w : need;
    }
    return align_up(need, 256);
}

size_t omni_sparse_mla_host_staging_bytes(const omni_mla_desc_t *desc)
{
    if (!desc_ok(desc)) return 0;
    size_t n = host_copy_bytes(desc);
    if (host_pipelined(desc)) {
        const size_t halves = host_half_workspace(desc, 0) + host_half_workspace(desc, 1), parts = host_part_workspace(desc);
        n += halves > parts ? halves : parts;
    }
    return n;
}

// Whether kernels can use a host buffer in place: pinned from its first to its last byte, at the same address
// on the device, 16-byte aligned.
static bool mapped_host(const void *p, size_t bytes)
{
    if (!aligned(p, 16)) return false;
    const void *ends[2] = {p, static_cast<const char *>(p) + bytes - 1};
    for (const void *e : ends) {
        cudaPointerAttributes at = {};
        if (cudaPointerGetAttributes(&at, e) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        if (at.type != cudaMemoryTypeHost || at.devicePointer != e) return false;
    }
    return true;
}

// Events that order a call's streams: one set per host thread and device.  A recorded event may be recorded
// again while an earlier wait on it is still pending, so a set serves every call of its thread.
struct HostEvents {
    cudaEvent_t ev[64][2 * kHostParts + 1] = {};
    ~HostEvents()
    {
        for (auto &device : ev)
            for (cudaEvent_t e : device)
                if (e) cudaEventDestroy(e);
    }
    cudaEvent_t *of(int dev)
    {
        if (dev < 0 || dev >= 64) return nullptr;
        for (cudaEvent_t &e : ev[dev])
            if (!e && cudaEventCreateWithFlags(&e, cudaEventDisableTiming) != cudaSuccess) return nullptr;
        return ev[dev];
    }
};

omni_status_t omni_sparse_mla_decode_host(const omni_mla_desc_t *desc, const void *q_host,
                                          const void *kv_cache,
                                          const int32_t *page_table_host,
                                          const int32_t *sel_idx_host,
                                          const int32_t *sel_len_host, void *out_host,
                                          float *lse_host, void *staging, size_t staging_bytes,
                                          void *workspace, size_t workspace_bytes,
                                          int32_t *device_status, void *stream_)
{
    if (!desc || !q_host || !kv_cache || !page_table_host || !sel_idx_host || !sel_len_host ||
        !out_host || !lse_host || !staging)
        return OMNI_ERR_NULL;
    if (!desc_ok(desc)) return OMNI_ERR_SHAPE;
    if (!aligned(staging, 256)) return OMNI_ERR_ALIGN;
    if (staging_bytes < omni_sparse_mla_host_staging_bytes(desc)) return OMNI_ERR_WORKSPACE;
    cudaStream_t stream = static_cast<cudaStream_t>(stream_);
    const size_t B = desc->batch, H = desc->num_heads;
    const size_t rq = H * kDqk * 2, rpt = (size_t)desc->max_pages_per_req * 4, rsi = (size_t)desc->max_sel * 4,
                 rsl = 4, rout = H * kDv * 2, rlse = H * 4;                      // bytes per request
    char *base = static_cast<char *>(staging);
    char *dq = base;
    char *dpt = dq + align_up(B * rq, 256);
    char *dsi = dpt + align_up(B * rpt, 256);
    char *dsl = dsi + align_up(B * rsi, 256);
    char *dout = dsl + align_up(B * rsl, 256);
    char *dlse = dout + align_up(B * rout, 256);
    char *half_ws = dlse + align_up(B * rlse, 256);

    auto h2d = [](void *dst, const void *src, size_t n, cudaStream_t s) {
        return cudaMemcpyAsync(dst, src, n, cudaMemcpyHostToDevice, s) == cudaSuccess;
    };
    // the three index arrays of all requests (small: one copy each)
    auto copy_indices = [&](cudaStream_t s) {
        return h2d(dpt, page_table_host, B * rpt, s) && h2d(dsi, sel_idx_host, B * rsi, s) && h2d(dsl, sel_len_host, B * rsl, s);
    };
    auto copy_q = [&](size_t b0, size_t n, cudaStream_t s) {
        return h2d(dq + b0 * rq, static_cast<const char *>(q_host) + b0 * rq, n * rq, s);
    };
    // requests [b0, b0 + d.batch) on stream s: decode and copies out
    auto decode_and_copy_out = [&](const omni_mla_desc_t &d, size_t b0, void *ws, size_t ws_bytes, cudaStream_t s) -> omni_status_t {
        const size_t n = d.batch;
        omni_status_t st = omni_sparse_mla_decode(
            &d, dq + b0 * rq, kv_cache, reinterpret_cast<int32_t *>(dpt + b0 * rpt), reinterpret_cast<int32_t *>(dsi + b0 * rsi),
            reinterpret_cast<int32_t *>(dsl + b0 * rsl), dout + b0 * rout, reinterpret_cast<float *>(dlse + b0 * rlse), ws,
            ws_bytes, device_status, s);
        if (st != OMNI_OK) return st;
        if (cudaMemcpyAsync(static_cast<char *>(out_host) + b0 * rout, dout + b0 * rout, n * rout, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaMemcpyAsync(reinterpret_cast<char *>(lse_host) + b0 * rlse, dlse + b0 * rlse, n * rlse, cudaMemcpyDeviceToHost, s) != cudaSuccess)
            return OMNI_ERR_CUDA;
        return OMNI_OK;
    };

    cudaStream_t side = host_pipelined(desc) ? host_side_stream(stream) : nullptr;
    if (mapped_host(q_host, B * rq) && mapped_host(page_table_host, B * rpt) && mapped_host(sel_idx_host, B * rsi) &&
        mapped_host(sel_len_host, B * rsl) && mapped_host(out_host, B * rout) && mapped_host(lse_host, B * rlse)) {
        int size[kHostParts];
        int parts = host_parts(desc, size), dev = -1;
        static thread_local HostEvents pool;
        cudaStream_t back = parts > 1 ? host_side_stream(stream, 1) : nullptr;
        cudaEvent_t *ev = side && back && cudaGetDevice(&dev) == cudaSuccess ? pool.of(dev) : nullptr;
        auto gather = [&](const GatherParts &g) {
            size_t vectors = 0;
            for (const GatherPart &a : g.part) vectors += a.bytes / 16;
            const unsigned blocks = (unsigned)std::min<size_t>(16, vectors / (kGatherThreads * kGatherAhead) + 1);
            return launch_overlapped(host_gather_kernel, blocks, kGatherThreads, stream, g);
        };
        if (!ev) {
            const omni_status_t st =
                gather({{{page_table_host, dpt, B * rpt}, {sel_idx_host, dsi, B * rsi}, {sel_len_host, dsl, B * rsl}, {q_host, dq, B * rq}}});
            if (st != OMNI_OK) return st;
            // a batch that other host memory would run in halves has its scratch in `staging` whatever its parts are
            const bool own = parts == 1 && host_pipelined(desc);
            return omni_sparse_mla_decode(desc, dq, kv_cache, reinterpret_cast<int32_t *>(dpt), reinterpret_cast<int32_t *>(dsi),
                                          reinterpret_cast<int32_t *>(dsl), out_host, lse_host, own ? half_ws : workspace,
                                          own ? host_part_workspace(desc) : workspace_bytes, device_status, stream);
        }
        // side:   q of part 0 | q of part 1 | ...
        // caller: indices     | kernels 0   | kernels 1     | ... | join
        // back:                             | out of part 0 | ...
        cudaEvent_t *in_done = ev, *part_done = ev + kHostParts, start = ev[2 * kHostParts];
        if (cudaEventRecord(start, stream) != cudaSuccess || cudaStreamWaitEvent(side, start, 0) != cudaSuccess) return OMNI_ERR_CUDA;
        // indices of more than a megabyte or so come with the parts that use them
        const bool indices_at_once = B * (rpt + rsi + rsl) <= (size_t)(1u << 20);
        bool ok = true;
        size_t b0 = 0;
        for (int i = 0; i < parts; b0 += size[i], ++i) {
            if (!indices_at_once) {
                const size_t n = size[i];
                ok = ok && h2d(dpt + b0 * rpt, reinterpret_cast<const char *>(page_table_host) + b0 * rpt, n * rpt, side) &&
                     h2d(dsi + b0 * rsi, reinterpret_cast<const char *>(sel_idx_host) + b0 * rsi, n * rsi, side) &&
                     h2d(dsl + b0 * rsl, reinterpret_cast<const char *>(sel_len_host) + b0 * rsl, n * rsl, side);
            }
            ok = ok && copy_q(b0, size[i], side);
            ok = cudaEventRecord(in_done[i], side) == cudaSuccess && ok;
        }
        omni_status_t st = ok ? OMNI_OK : OMNI_ERR_CUDA;
        if (st == OMNI_OK && indices_at_once)
            st = gather({{{page_table_host, dpt, B * rpt}, {sel_idx_host, dsi, B * rsi}, {sel_len_host, dsl, B * rsl}, {nullptr, nullptr, 0}}});
        const size_t part_ws = host_part_workspace(desc);
        b0 = 0;
        for (int i = 0; i < parts; b0 += size[i], ++i) {
            // (after an error the waits still join the streams)
            if (cudaStreamWaitEvent(stream, in_done[i], 0) != cudaSuccess) st = OMNI_ERR_CUDA;
            if (st != OMNI_OK) continue;
            omni_mla_desc_t d = *desc;
            d.batch = size[i];
            const bool last = i == parts - 1;
            char *to = static_cast<char *>(out_host) + b0 * rout;
            st = omni_sparse_mla_decode(&d, dq + b0 * rq, kv_cache, reinterpret_cast<int32_t *>(dpt + b0 * rpt),
                                        reinterpret_cast<int32_t *>(dsi + b0 * rsi), reinterpret_cast<int32_t *>(dsl + b0 * rsl),
                                        last ? to : dout + b0 * rout,
                                        reinterpret_cast<float *>((last ? reinterpret_cast<char *>(lse_host) : dlse) + b0 * rlse), half_ws,
                                        part_ws, device_status, stream);
            if (st == OMNI_OK && !last &&
                (cudaEventRecord(part_done[i], stream) != cudaSuccess || cudaStreamWaitEvent(back, part_done[i], 0) != cudaSuccess ||
                 cudaMemcpyAsync(to, dout + b0 * rout, size[i] * rout, cudaMemcpyDeviceToHost, back) != cudaSuccess ||
                 // (lse of all parts but the last in one copy)
                 (i == parts - 2 && cudaMemcpyAsync(lse_host, dlse, (b0 + size[i]) * rlse, cudaMemcpyDeviceToHost, back) != cudaSuccess)))
                st = OMNI_ERR_CUDA;
        }
        if (cudaEventRecord(start, back) != cudaSuccess || cudaStreamWaitEvent(stream, start, 0) != cudaSuccess)
            st = st != OMNI_OK ? st : OMNI_ERR_CUDA;
        return st;
    }
    if (!side) {
        if (!copy_q(0, B, stream) || !copy_indices(stream)) return OMNI_ERR_CUDA;
        return decode_and_copy_out(*desc, 0, workspace, workspace_bytes, stream);
    }
    const omni_mla_desc_t first = host_half_desc(desc, 0), second = host_half_desc(desc, 1);
    const size_t ws0 = host_half_workspace(desc, 0), ws1 = host_half_workspace(desc, 1);
    cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};     // first q in | indices in | second half done
    for (int e = 0; e < 3; ++e)
        if (cudaEventCreateWithFlags(&ev[e], cudaEventDisableTiming) != cudaSuccess) {
            for (int f = 0; f < e; ++f) cudaEventDestroy(ev[f]);
            return OMNI_ERR_CUDA;
        }
    // caller's stream: q of the first half | indices | kernel | copies out           | join
    // side stream:                         | q of the second half     | kernel | copies out
    bool ok = copy_q(0, (size_t)first.batch, stream) && cudaEventRecord(ev[0], stream) == cudaSuccess &&
              cudaStreamWaitEvent(side, ev[0], 0) == cudaSuccess;
    const bool forked = ok;
    ok = ok && copy_q((size_t)first.batch, (size_t)second.batch, side);
    ok = ok && copy_indices(stream) && cudaEventRecord(ev[1], stream) == cudaSuccess &&
         cudaStreamWaitEvent(side, ev[1], 0) == cudaSuccess;
    omni_status_t st = ok ? OMNI_OK : OMNI_ERR_CUDA;
    if (st == OMNI_OK) st = decode_and_copy_out(first, 0, half_ws, ws0, stream);
    if (st == OMNI_OK) st = decode_and_copy_out(second, (size_t)first.batch, half_ws + ws0, ws1, side);
    if (forked && (cudaEventRecord(ev[2], side) != cudaSuccess || cudaStreamWaitEvent(stream, ev[2], 0) != cudaSuccess))
        st = st != OMNI_OK ? st : OMNI_ERR_CUDA;
    for (int e = 0; e < 3; ++e) cudaEventDestroy(ev[e]);  // released by the runtime once the work that uses them is done
    return st;
}

}  // extern "C"
