// Split-KV merge and the small index kernels (validation, row export).
#pragma once

#include "common.cuh"

namespace omni {

// One block per (request, head): lse = ln sum_s exp(lse_s); out = sum_s exp(lse_s - lse) * out_s.
// 128 * kGroups threads: thread t owns value columns 4 (t % 128) .. + 3 of the splits t / 128,
// t / 128 + kGroups, ...; the partial sums of a column meet in shared memory.  The kernel is a chain of
// latencies, not of bytes (the partials sit in L2): every log-sum-exp at once (a lane per split in every
// warp) and with them a thread's first kCombineAhead partial rows, then the others, as many in flight.  With one thread
// per column walking the splits one after the other, 32 splits of one request took 11 us; with the rows behind the
// log-sum-exps about 3.  Steps with and without the rows in front of the weights: one request of 16 heads in
// 13 splits 10.26 -> 9.70 us, of 128 heads in 32 splits 15.73 -> 15.55, 4 x 64 units of 64 heads 17.09 -> 15.91.
// Four groups pay where a launch has few blocks and many splits; with more blocks than the
// SMs hold at once the larger blocks only make more waves (64 requests of 64 heads, two splits: 80 us
// per step with four groups, 66 with one), see launch_combine.
constexpr int kCombineAhead = 4;
template <int kGroups>
__global__ void __launch_bounds__(128 * kGroups) combine_kernel(const float *__restrict__ part_out,
                                                                const float *__restrict__ part_lse,
                                                                const int32_t *__restrict__ num_splits,
                                                                const int32_t *__restrict__ request,
                                                                int batch, int max_splits, int heads,
                                                                __nv_bfloat16 *__restrict__ out,
                                                                float *__restrict__ lse)
{
    __shared__ float4 sums[kGroups > 1 ? kGroups - 1 : 1][128];
    const int b = blockIdx.x / heads, h = blockIdx.x % heads;
    const int lane = threadIdx.x & 31, col = threadIdx.x & 127, group = threadIdx.x >> 7;
    const float4 *rows = reinterpret_cast<const float4 *>(part_out + ((size_t)b * max_splits * heads + h) * kDv) + col;
    const size_t row_pitch = (size_t)heads * (kDv / 4);
    const float *pl = part_lse + (size_t)b * max_splits * heads + h;
    // no-op unless launched as a programmatic dependent: then wait for the producing kernel;
    // the kernel that follows may be scheduled early in turn (it waits before it reads)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // Which of the `batch` requests the b-th set of partial results belongs to; negative: there are none after all.
    // (Nor does a decode kernel that gave up before it wrote the number leave one: the word is then whatever the
    // workspace held.)
    const int owner = request ? __ldg(request + b) : b;
    if ((unsigned)owner >= (unsigned)batch) return;
    int ns = num_splits ? __ldg(num_splits + b) : max_splits;
    ns = max(0, min(ns, max_splits));
    // The first rows of this thread are on their way while the weights are worked out (what an empty split's holds is dropped below).
    float4 ahead[kCombineAhead];
#pragma unroll
    for (int k = 0; k < kCombineAhead; ++k) {
        const int i = group + k * kGroups;
        ahead[k] = i < min(ns, 32) ? __ldg(rows + (size_t)i * row_pitch) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    // total over all splits, 32 at a time: every warp does it for itself
    float mx = -INFINITY, z = 0.f, first = -INFINITY;      // z: sum of exp(lse - mx)
    bool nan = false;                                      // one of them is: it never is the maximum, but it is in the sum
    for (int s0 = 0; s0 < ns; s0 += 32) {
        const float v = s0 + lane < ns ? __ldg(pl + (size_t)(s0 + lane) * heads) : -INFINITY;
        if (s0 == 0) first = v;
        float m = v;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, d));
        m = fmaxf(m, mx);
        if (m == -INFINITY) {                                  // (beside a number the sum itself becomes NaN)
            nan |= __any_sync(0xffffffffu, v != v) != 0;
            continue;
        }
        float e = exp2f((v - m) * kLog2e);
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) e += __shfl_xor_sync(0xffffffffu, e, d);
        z = (mx == -INFINITY ? 0.f : z * exp2f((mx - m) * kLog2e)) + e;
        mx = m;
    }
    const float total = nan ? NAN : mx > -INFINITY ? mx + logf(z) : -INFINITY;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = 0; s0 < ns; s0 += 32) {
        const float v = s0 == 0 ? first : (s0 + lane < ns ? __ldg(pl + (size_t)(s0 + lane) * heads) : -INFINITY);
        // Of split s0 + lane.  The row of an empty split does not count: it may hold anything.  A weight that is merely too small
        // for fp32 does multiply its row, whose infinities and NaNs count.
        const uint32_t some = __ballot_sync(0xffffffffu, v != -INFINITY);
        const float weight = v != -INFINITY ? exp2f((v - total) * kLog2e) : 0.f;
        const int here = min(32, ns - s0);
        for (int i0 = group; i0 < here; i0 += kGroups * kCombineAhead) {
            float4 x[kCombineAhead];
            float w[kCombineAhead];
#pragma unroll
            for (int k = 0; k < kCombineAhead; ++k) {
                const int i = i0 + k * kGroups;
                w[k] = __shfl_sync(0xffffffffu, weight, i & 31);
                // (a row that does not count is zero, whatever weight stands beside it: a finite one, or the sum is NaN anyway)
                x[k] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (i < here && ((some >> i) & 1u)) x[k] = s0 == 0 && i0 == group ? ahead[k] : __ldg(rows + (size_t)(s0 + i) * row_pitch);
            }
#pragma unroll
            for (int k = 0; k < kCombineAhead; ++k) {
                acc.x = fmaf(w[k], x[k].x, acc.x);
                acc.y = fmaf(w[k], x[k].y, acc.y);
                acc.z = fmaf(w[k], x[k].z, acc.z);
                acc.w = fmaf(w[k], x[k].w, acc.w);
            }
        }
    }
    if (kGroups > 1) {
        if (group > 0) sums[group - 1][col] = acc;
        __syncthreads();
        if (group > 0) return;
#pragma unroll
        for (int g = 0; g < kGroups - 1; ++g) {
            const float4 x = sums[g][col];
            acc.x += x.x;
            acc.y += x.y;
            acc.z += x.z;
            acc.w += x.w;
        }
    }
    __nv_bfloat162 lo = __floats2bfloat162_rn(acc.x, acc.y), hi = __floats2bfloat162_rn(acc.z, acc.w);
    uint2 packed;
    packed.x = *reinterpret_cast<uint32_t *>(&lo);
    packed.y = *reinterpret_cast<uint32_t *>(&hi);
    const size_t to = (size_t)owner * heads + h;
    reinterpret_cast<uint2 *>(out + to * kDv)[col] = packed;
    if (threadIdx.x == 0) lse[to] = total;
}

// rows[b][j] = physical row of the j-th selected token (-1 outside sel_len or on a contract
// violation); with rows == nullptr it only checks and flags.
__global__ void __launch_bounds__(256) resolve_rows_kernel(const int32_t *__restrict__ page_table,
                                                           const int32_t *__restrict__ sel_idx,
                                                           const int32_t *__restrict__ sel_len,
                                                           int max_pages, int max_sel,
                                                           int64_t num_pages, int64_t *rows,
                                                           int32_t *status)
{
    const int b = blockIdx.y;
    int n = __ldg(sel_len + b);
    bool bad = false;
    if (n < 0 || n > max_sel) {
        bad = true;
        n = 0;
    }
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < max_sel; j += gridDim.x * blockDim.x) {
        int64_t r = -1;
        if (j < n) {
            r = resolve_row(page_table + (size_t)b * max_pages, __ldg(sel_idx + (size_t)b * max_sel + j),
                            max_pages, num_pages);
            bad |= (r < 0);
        }
        if (rows) rows[(size_t)b * max_sel + j] = r;
    }
    if (bad) flag_status(status, OMNI_DEV_BAD_INDEX);
}

// Appends one latent row per request to the rolling cache of a compressed layer: the row of the
// token at absolute position ctx_len[b] goes to rolling_position(ctx_len[b]) of the request's
// page table.  72 threads per request, 16 bytes each.
__global__ void __launch_bounds__(72) append_rolling_kernel(__nv_bfloat16 *__restrict__ kv,
                                                            const int32_t *__restrict__ page_table,
                                                            const int32_t *__restrict__ ctx_len,
                                                            const __nv_bfloat16 *__restrict__ new_rows,
                                                            int max_pages, int64_t num_pages, int sink_pages,
                                                            int ring_pages, int32_t *status)
{
    // launched as a programmatic dependent between two decode steps: the launch gaps on either side would
    // cost more than the copy (the step it precedes waits for this one before it reads)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int b = blockIdx.x;
    const int32_t t = __ldg(ctx_len + b);
    int64_t row = -1;
    if (t >= 0) {
        const int32_t pos = rolling_position(t, sink_pages, ring_pages);
        row = resolve_row(page_table + (size_t)b * max_pages, pos, max_pages, num_pages);
    }
    if (row < 0) {
        if (threadIdx.x == 0) flag_status(status, OMNI_DEV_BAD_INDEX);
        return;
    }
    const uint4 *src = reinterpret_cast<const uint4 *>(new_rows + (size_t)b * kDqk);
    uint4 *dst = reinterpret_cast<uint4 *>(kv + (size_t)row * kDqk);
    dst[threadIdx.x] = __ldg(src + threadIdx.x);
}

}  // namespace omni
