// Paired-CTA decode kernel over the 8-bit latent cache (sm_100a).
//
// Cache row of a token: 512 FP8 E4M3 codes (the latent columns), then the 64 rope columns as
// bf16 (128 bytes): 640 bytes, five 128-byte panels.  One fp32 scale per row in a separate array:
// latent value = code * scale.  The result is attention over those de-quantised rows.
//
// The kernel keeps the structure of tc2_decode_kernel (a CTA pair = all heads of one (request,
// split), cta_group::2 MMAs with M = 128, K role / V role loads, eight softmax warps) and changes
// what the 8-bit rows change:
//
//  * Scores.  The latent part runs on the 8-bit tensor-core kind (kind::f8f6f4, K = 32 per
//    instruction): S8 = Q8 K8^T.  q arrives as bf16; at the start of a work unit the softmax warps
//    rewrite its 512 latent columns as TWO E4M3 terms per value, hi = E4M3(q / a) and
//    lo = E4M3(q / a - hi), with a a power of two per head row, so that hi + lo carries the eight
//    significant bits of the bf16 value; both terms accumulate into the same S8.  The rope part
//    is an ordinary bf16 MMA (K = 64) into a second accumulator Sr, because S8 still has to be
//    multiplied by a[row] * scale[token]:  x = (a * scale_t * S8 + Sr) * softmax_scale.
//  * Weighted sum.  V = code * scale_t, so the token's scale is folded into its weight: the
//    softmax runs on y = x + log2(scale_t), P' = exp2(y - m) = p * scale_t is what multiplies the
//    codes, and the row sum uses p = P' / scale_t.  Because the reference m follows max y, P' stays
//    below 448 whatever the data, which is what lets it be written as E4M3: again as two
//    terms hi + lo, side by side in one 128-byte row of the P buffer, [hi tokens 0..63 | lo tokens
//    0..63], so that O += [P_hi | P_lo] [V8 ; V8] is four K = 32 steps per accumulator.
//  * Shared memory.  The K rows of a tile are 40 KiB a CTA and the V columns of a unit 16 KiB (72 and 32
//    for bf16 rows), so the same budget holds two whole tiles of K and three units of V.  The bf16 copy
//    of q (latent panels) sits in the V stages and P buffers while it is converted.
//  * Tensor memory holds two score buffers (of two accumulators each) instead of three.
//
// What bounds it: the tensor core takes as long as for bf16 rows (two terms of half the width), and the
// softmax warps go through about 16 instructions a token in one long chain per tile.  On tiles
// of 64 tokens that chain took 2100 clocks a tile and nothing overlapped it; on tiles of 128 a thread
// has twice the independent work for the same chain: 32 requests x 33 units 33.6 -> 28.3 us, 128 x 64
// 181 -> 148.
//
// Work split, merge paths, index handling, time-outs: as in tc2_decode_kernel.
#pragma once

#include <cuda_fp16.h>

#include "tc2_decode.cuh"

namespace omni {

constexpr int kQ8RowBytes = 640;
constexpr int kQ8Panels = 5;                              // four panels of 128 codes, one of 64 bf16 rope columns
constexpr int kQ8KStages = 2, kQ8VStages = 3;
constexpr int kQ8KBytes = kQ8Panels * kPanelBytes;        // K role: 64 tokens x 640 B
constexpr int kQ8VBytes = 2 * kPanelBytes;                // V role: 64 tokens x 256 codes
constexpr int kQ8SmemQHi = 0;                             // 4 panels x [64 heads x 128 codes]
constexpr int kQ8SmemQLo = 4 * kPanelBytes;
constexpr int kQ8SmemQRope = 8 * kPanelBytes;             // [64 heads x 64 bf16]
constexpr int kQ8SmemK = kTileBytes;
constexpr int kQ8SmemV = kQ8SmemK + kQ8KStages * kQ8KBytes;
constexpr int kQ8SmemP = kQ8SmemV + kQ8VStages * kQ8VBytes;     // 2 units x [64 heads x (64 hi + 64 lo codes)]
constexpr int kQ8SmemAux = kQ8SmemP + 2 * kPanelBytes;
constexpr int kQ8SmemQTemp = kQ8SmemV;                    // 8 bf16 panels of q during set-up: V stages + P buffers
// Masks and scales travel from the K producer to the softmax warps through rings.  Those of tile t + 2 are
// written once the score MMAs of tile t have retired; these were issued only after every softmax warp
// had read the scores of tile t - 2 (two score buffers), i.e. after tile t - 3 was finished: five
// tiles can be live.
constexpr int kQ8Ring = 5;
constexpr uint32_t kQ8ColS8 = 256, kQ8ColSr = 384;        // two buffers of 64 columns each
// The weights P' = exp2(y - m) are written as E4M3, whose range is [2^-9, 448].  The reference m is
// therefore kept below the running maximum of y: it is set kQ8Headroom under the tile maximum
// whenever that maximum has risen more than kQ8RescaleWindow above it, so the largest weight
// lies in (2^-.., 2^8.75 = 431] and a token is only lost to underflow when its weight is more
// than 2^18 times smaller than the largest one seen.
constexpr float kQ8Headroom = 8.f, kQ8RescaleWindow = 8.75f;

struct Q8Aux {
    float q_scale[64];                    // a[row]
    float tok_scale[kQ8Ring][128];        // scale of each token of a tile
    float tok_log2[kQ8Ring][128];         // its base-2 logarithm
    float tok_rcp[kQ8Ring][128];          // its reciprocal
};
static_assert(kQ8SmemQRope + kPanelBytes == kTileBytes, "q area");
static_assert(kQ8SmemAux + (int)sizeof(Q8Aux) <= kC2SmemCtl, "auxiliary arrays must end below the control block");
static_assert(kQ8SmemQTemp + 8 * kPanelBytes <= kQ8SmemAux, "the temporary copy of q must not reach the auxiliary arrays");

struct Q8Control {
    uint64_t q_full;                     // this CTA's bf16 q has landed (local)
    uint64_t q_ready;                    // leader: both CTAs have rewritten q as E4M3 terms
    uint64_t q_conv;                     // local: the temporary copy of q is dead
    uint64_t k_full[kQ8KStages];
    uint64_t k_empty[kQ8KStages];
    uint64_t v_full[kQ8VStages];
    uint64_t v_empty[kQ8VStages];
    uint64_t s_full[2];
    uint64_t s_empty[2];
    uint64_t p_full;                     // both P units of a tile are written (and O rescaled)
    uint64_t pv_done[2];                 // P V of a unit retired: its P unit may be rewritten, O may be rescaled
    uint64_t x_bar;
    uint64_t exit_bar;
    uint64_t recv_bar[4];
    uint64_t ready_bar;
    uint64_t taken_bar;
    uint64_t valid_mask[kQ8Ring][2];     // [tile][unit]
    float xchg[2][4][64];
    uint32_t tmem_base;
    uint32_t abort;
    uint32_t merge_flag;
    uint32_t xfail;
    int32_t k_progress;
};
static_assert(sizeof(Q8Control) <= kC2SmemCtlBytes, "control block too large");

// Instruction descriptor of kind::f8f6f4 with E4M3 inputs and fp32 accumulation (same fields as
// instr_desc; the two format fields are 0 for E4M3).
__host__ __device__ constexpr uint32_t instr_desc_e4m3(int m, int n, int b_mn_major)
{
    return (1u << 4) | ((uint32_t)b_mn_major << 16) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

template <bool kAccumulate>
__device__ __forceinline__ void tc_mma8_pair_elect(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo,
                                                   uint32_t b_hi, uint32_t idesc)
{
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], da, db, %5, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "n"(kAccumulate ? 1 : 0)
        : "memory");
}

__device__ __forceinline__ void tc_mma8_pair_elect(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                                   uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], da, db, %5, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Two floats -> two E4M3 codes (round to nearest even, saturating), `lo` in the low byte.
__device__ __forceinline__ uint32_t e4m3x2(float lo, float hi)
{
    uint16_t r;
    asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
    return r;
}
// Two E4M3 codes -> their exact values.
__device__ __forceinline__ float2 e4m3x2_values(uint32_t codes)
{
    uint32_t h2;
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)codes));
    return __half22float2(*reinterpret_cast<const __half2 *>(&h2));
}
// Sixteen values as two-term E4M3: hi codes and lo codes (value ~ hi + lo), 16 bytes each.
__device__ __forceinline__ void split_e4m3(const float (&v)[16], uint4 &hi, uint4 &lo)
{
    uint32_t h[4], l[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t h0 = e4m3x2(v[4 * k], v[4 * k + 1]), h1 = e4m3x2(v[4 * k + 2], v[4 * k + 3]);
        const float2 b0 = e4m3x2_values(h0), b1 = e4m3x2_values(h1);
        const f32x2 minus = pack2(-1.f, -1.f);            // (v - b is exact, whatever the form)
        const float2 r0 = unpack2(fma2(pack2(b0.x, b0.y), minus, pack2(v[4 * k], v[4 * k + 1])));
        const float2 r1 = unpack2(fma2(pack2(b1.x, b1.y), minus, pack2(v[4 * k + 2], v[4 * k + 3])));
        const uint32_t l0 = e4m3x2(r0.x, r0.y), l1 = e4m3x2(r1.x, r1.y);
        h[k] = h0 | (h1 << 16);
        l[k] = l0 | (l1 << 16);
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// Row gathers of the 8-bit layout (see gather_rows): 64 rows of 640 bytes, kCount panels.
template <int kCount>
__device__ __noinline__ void gather_rows_q8(uint32_t dst, const char *cols, int row_lo, int row_hi, int lane)
{
    const int ch = lane & 7;
#pragma unroll
    for (int g = 0; g < 16; ++g) {
        const int r = 4 * g + (lane >> 3);
        const int src_row = __shfl_sync(0xffffffffu, g < 8 ? row_lo : row_hi, r & 31);
        const char *src = cols + (size_t)src_row * kQ8RowBytes + ch * 16;
        const uint32_t d = dst + r * 128 + ((ch ^ (r & 7)) << 4);
#pragma unroll
        for (int c = 0; c < kCount; ++c) cp_async16(d + c * kPanelBytes, src + c * 128);
    }
    cp_async_commit();
}

__device__ __forceinline__ void prefetch_row_q8(const char *kv, int row)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(kv + (size_t)row * kQ8RowBytes), "n"(kQ8RowBytes) : "memory");
}

// Two instances, as for the bf16 kernel: with and without the in-cluster merge of two splits, each
// carrying only its own merge and epilogue code.  The 8-bit entry point takes an index list only.
template <bool kClusterMerge>
__device__ __forceinline__ void tc2q8_decode_body(const CUtensorMap &q_nope_map, const CUtensorMap &q_rope_map,
                                                  const CUtensorMap &kv_k_map, const CUtensorMap &kv_v_map,
                                                  const CUtensorMap &kv_page_map, const DecodeParams &p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = smem_raw;
    if (smem_u32(smem_raw) & 1023u) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (threadIdx.x == 0) flag_status(p.status, OMNI_DEV_TIMEOUT);
        return;
    }
    Q8Control *ctl = reinterpret_cast<Q8Control *>(smem + kC2SmemCtl);
    Q8Aux *aux = reinterpret_cast<Q8Aux *>(smem + kQ8SmemAux);
    const uint32_t smem_base = smem_u32(smem);
    const uint32_t crank = cluster_rank();
    const uint32_t rank = crank & 1u, leader = crank & ~1u, peer = crank ^ 1u;
    const uint16_t pair_mask = (uint16_t)(3u << leader);

    const int pair = blockIdx.x >> 1;
    C2Unit unit = kClusterMerge ? C2Unit{(int)(blockIdx.x >> 2), (int)(crank >> 1), 2, 0} : c2_unit(p, pair);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // warp-uniform
    const int rows = c2_rows(p.heads);
    const int h0 = (int)rank * rows;                          // (dealt out evenly, as in tc2_decode_kernel)
    const int head_rows = min(rows, p.heads - h0);

    // ---- set-up (no global memory access before the dependent-launch wait) -------------------
    if (threadIdx.x == 0) {
        mbar_init(&ctl->q_full, 1);
        mbar_init(&ctl->q_ready, 16);
        mbar_init(&ctl->q_conv, 8);
        for (int i = 0; i < kQ8KStages; ++i) {
            mbar_init(&ctl->k_full[i], 1);
            mbar_init(&ctl->k_empty[i], 1);
        }
        for (int i = 0; i < kQ8VStages; ++i) {
            mbar_init(&ctl->v_full[i], 1);
            mbar_init(&ctl->v_empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&ctl->s_full[i], 1);
            mbar_init(&ctl->s_empty[i], 16);
            mbar_init(&ctl->pv_done[i], 1);
        }
        mbar_init(&ctl->p_full, 16);
        mbar_init(&ctl->x_bar, 256);
        mbar_init(&ctl->exit_bar, 2);
        for (int i = 0; i < 4; ++i) mbar_init(&ctl->recv_bar[i], 1);
        mbar_init(&ctl->ready_bar, 1);
        mbar_init(&ctl->taken_bar, 8);
        ctl->abort = 0;
        ctl->xfail = 0;
        ctl->k_progress = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_after_init();
    tc_fence_after();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (!kClusterMerge) {
        bool cut = true;
        int request = unit.b;
        if (p.longest_first) {
            uint8_t *order = smem + 4096;                 // (behind the sizes; shared memory nobody uses yet)
            cut = c2_rank_requests(p, reinterpret_cast<int *>(smem), order);
            request = order[unit.b];
            c2_release_scratch();
        }
        c2_name_request(p, unit, request, cut, rank == 0 && threadIdx.x == 0);
    }
    const int b = unit.b, s = unit.s;
    const Selection selection = load_selection(p, b);
    __builtin_assume(selection.list != nullptr);
    const int n = !kClusterMerge && unit.splits == 0 ? 0 : selection.n;
    const bool bad_len = selection.bad;
    int begin, end;
    split_range(n, max(unit.splits, 1), s, begin, end, kC2Tile);
    const int units = (end - begin + kC2Tile - 1) / kC2Tile, tiles = (units + 1) / 2;

    const bool active = units > 0;
    if (!active && bad_len && threadIdx.x == 0 && crank == 0) flag_status(p.status, OMNI_DEV_BAD_INDEX);
    if (!kClusterMerge && !active) c2_store_empty(p, unit, h0, head_rows, warp, kC2Threads / 32, lane);

    const uint32_t tmem = ctl->tmem_base;
    volatile uint32_t *abort_flag = &ctl->abort;
    const int32_t *pt = p.page_table + (size_t)b * p.max_pages;
    const char *kv_bytes = reinterpret_cast<const char *>(p.kv);

    // Index pipeline of the producers: as in tc2_decode_kernel (lane l serves tokens l and l+32 of a unit).
    struct TileIdx {
        int t0, t1;
        int pg0, pg1;
    };
    const uint32_t t_limit = (uint32_t)min((int64_t)p.max_pages * kPage, (int64_t)1 << 31);
    const uint32_t page_limit = (uint32_t)p.num_pages;
    auto stage_tokens = [&](int unit, TileIdx &x) {
        const int j0 = begin + unit * kC2Tile + lane, j1 = j0 + 32;
        x.t0 = j0 < end ? selection_at(selection, j0) : -1;
        x.t1 = j1 < end ? selection_at(selection, j1) : -1;
    };
    auto stage_pages = [&](TileIdx &x) {
        x.pg0 = (uint32_t)x.t0 < t_limit ? ldg_index(pt + (x.t0 >> 6), selection.keep) : -1;
        x.pg1 = (uint32_t)x.t1 < t_limit ? ldg_index(pt + (x.t1 >> 6), selection.keep) : -1;
    };
    auto stage_rows = [&](int unit, const TileIdx &x, int &row_lo, int &row_hi, uint64_t &mask, bool &contig,
                          bool &any_bad) {
        const bool ok0 = (uint32_t)x.pg0 < page_limit, ok1 = (uint32_t)x.pg1 < page_limit;
        row_lo = x.pg0 * kPage + (x.t0 & (kPage - 1));
        row_hi = x.pg1 * kPage + (x.t1 & (kPage - 1));
        const int base = __shfl_sync(0xffffffffu, row_lo, 0);
        contig = __all_sync(0xffffffffu, ok0 && ok1 && row_lo == base + lane && row_hi == base + 32 + lane);
        mask = ~0ull;
        if (contig) return;
        const int j0 = begin + unit * kC2Tile + lane, j1 = j0 + 32;
        any_bad |= (j0 < end && !ok0) || (j1 < end && !ok1);
        const uint32_t m0 = __ballot_sync(0xffffffffu, ok0), m1 = __ballot_sync(0xffffffffu, ok1);
        mask = (uint64_t)m0 | ((uint64_t)m1 << 32);
        int stand_in = 0;
        if (m0)
            stand_in = __shfl_sync(0xffffffffu, row_lo, __ffs(m0) - 1);
        else if (m1)
            stand_in = __shfl_sync(0xffffffffu, row_hi, __ffs(m1) - 1);
        row_lo = ok0 ? row_lo : stand_in;
        row_hi = ok1 ? row_hi : stand_in;
    };

    float cm_lse = -INFINITY, cm_inv = 0.f;
    bool softmax_ok = true;

    if (!active) {
        // an empty split inside a merging cluster: no pipeline, but it takes part in the exchange
    } else if (warp == 0) {
        // =========================== K-role producer =====================================
        if (lane == 0) {
            // q, bf16: the eight latent panels go to a temporary place, the rope panel to its own
            mbar_expect_tx(&ctl->q_full, kTileBytes);
            tma_box3d(smem_base + kQ8SmemQTemp, &q_nope_map, &ctl->q_full, b * p.heads + h0, 0);
            tma_box3d(smem_base + kQ8SmemQRope, &q_rope_map, &ctl->q_full, b * p.heads + h0, 8);
        }
        // This CTA's K rows are unit 2 t + rank of every tile t.
        bool any_bad = bad_len;
        TileIdx x1[2], x2[2];
        int row_lo = 0, row_hi = 0;          // of this CTA's unit of the tile about to be loaded
        bool contig = false;
        uint64_t mask[2];
        float sc[2][2];                      // scales of the rows of that tile: [unit][token half]
        auto resolve_tile = [&](int tile, const TileIdx (&x)[2]) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                int lo, hi;
                bool whole;
                stage_rows(2 * tile + h, x[h], lo, hi, mask[h], whole, any_bad);
                // a unit without tokens has no row whose scale could be read
                sc[h][0] = mask[h] ? __ldg(p.kv_scale + lo) : 1.f;
                sc[h][1] = mask[h] ? __ldg(p.kv_scale + hi) : 1.f;
                if (h == (int)rank) {
                    row_lo = lo;
                    row_hi = hi;
                    contig = whole;
                }
            }
        };
        {
            TileIdx x0[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                stage_tokens(h, x0[h]);
                stage_tokens(2 + h, x1[h]);
                stage_tokens(4 + h, x2[h]);
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                stage_pages(x0[h]);
                stage_pages(x1[h]);
            }
            resolve_tile(0, x0);
        }
        bool ok = true;
        int pending = -1;
        const uint32_t k_full_leader = map_to_rank(smem_u32(&ctl->k_full[0]), leader);
        for (int i = 0; ok && i < tiles; ++i) {
            const int st = i & 1;
            if (i >= 2) {
                if (pending >= 0 && !__all_sync(0xffffffffu, mbar_test(&ctl->k_empty[st], ((i >> 1) - 1) & 1))) {
                    retire_gathered_stage(k_full_leader + 8 * pending, kQ8KBytes, 0, lane);
                    pending = -1;
                }
                ok = mbar_wait(&ctl->k_empty[st], ((i >> 1) - 1) & 1);
            }
            ok = __all_sync(0xffffffffu, ok) && (*abort_flag == 0);
            if (!ok) break;
            {
                // what the softmax warps need to know about tile i, published before its copy is
                // requested: which tokens count, and every token's scale, its logarithm and reciprocal
                const int ring = i % kQ8Ring;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float s1 = sc[k >> 1][k & 1];
                    aux->tok_scale[ring][32 * k + lane] = s1;
                    aux->tok_log2[ring][32 * k + lane] = log2f(s1);
                    aux->tok_rcp[ring][32 * k + lane] = 1.f / s1;
                }
                if (lane < 2) ctl->valid_mask[ring][lane] = lane ? mask[1] : mask[0];
                __threadfence_block();
                __syncwarp();
            }
            if (lane == 0 && rank == 0) mbar_expect_tx(&ctl->k_full[st], 2 * kQ8KBytes);
            // The last tile has a single unit when their number is odd: CTA 1 then leaves its rows as they are and
            // credits the bytes all the same, so that the scores wait for what it has just written and for
            // its own wait above (as in tc2_decode_kernel).
            bool gathered = false;
            if (2 * i + (int)rank >= units) {
                if (lane == 0) credit_bytes(k_full_leader + 8 * st, kQ8KBytes);
            } else {
                const uint32_t dst = smem_base + kQ8SmemK + st * kQ8KBytes;
                if (contig) {
                    if (lane == 0) tma_box3d_pair(dst, &kv_k_map, k_full_leader + 8 * st, row_lo, 0);
                } else {
                    gathered = true;
                    gather_rows_q8<kQ8Panels>(dst, kv_bytes, row_lo, row_hi, lane);
                }
            }
            if (lane == 0) *const_cast<volatile int32_t *>(&ctl->k_progress) = 2 * i + 2;
            if (pending >= 0) {
                retire_gathered_stage(k_full_leader + 8 * pending, kQ8KBytes, gathered ? 1 : 0, lane);
                pending = -1;
            }
            if (gathered) pending = st;
            if (i + 1 < tiles) resolve_tile(i + 1, x1);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                x1[h] = x2[h];
                stage_pages(x1[h]);
                stage_tokens(2 * i + 6 + h, x2[h]);
            }
        }
        if (pending >= 0) retire_gathered_stage(k_full_leader + 8 * pending, kQ8KBytes, 0, lane);
        if (lane == 0) *const_cast<volatile int32_t *>(&ctl->k_progress) = 0x7fffffff;
        if (!ok && lane == 0) {
            flag_status(p.status, OMNI_DEV_TIMEOUT | OMNI_DEV_ROLE_PRODUCER_K);
            *abort_flag = 1;
        }
        if (__any_sync(0xffffffffu, any_bad) && lane == 0 && rank == 0) flag_status(p.status, OMNI_DEV_BAD_INDEX);
    } else if (warp == 6) {
        // =========================== V-role producer =====================================
        // This CTA's V columns are [256*rank, 256*rank+256): code panels 2*rank and 2*rank+1.
        bool any_bad = false;
        TileIdx x1, x2;
        int row_lo, row_hi;
        uint64_t mask_unused;
        bool contig;
        {
            TileIdx x0;
            stage_tokens(0, x0);
            stage_tokens(1, x1);
            stage_tokens(2, x2);
            stage_pages(x0);
            stage_pages(x1);
            stage_rows(0, x0, row_lo, row_hi, mask_unused, contig, any_bad);
        }
        // the V stages hold the temporary copy of q until the softmax warps have converted it
        bool ok = mbar_wait(&ctl->q_conv, 0);
        ok = __all_sync(0xffffffffu, ok);
        int pending = -1;
        for (int i = 0; ok && i < units; ++i) {
            const int st = i % kQ8VStages;
            if (i >= kQ8VStages) {
                if (pending >= 0 && !__all_sync(0xffffffffu, mbar_test(&ctl->v_empty[st], ((i / kQ8VStages) - 1) & 1))) {
                    retire_gathered_stage(map_to_rank(smem_u32(&ctl->v_full[pending]), leader), kQ8VBytes, 0, lane);
                    pending = -1;
                }
                ok = mbar_wait(&ctl->v_empty[st], ((i / kQ8VStages) - 1) & 1);
            }
            ok = __all_sync(0xffffffffu, ok) && (*abort_flag == 0);
            if (!ok) break;
            const uint32_t bar = map_to_rank(smem_u32(&ctl->v_full[st]), leader);
            if (lane == 0 && rank == 0) mbar_expect_tx(&ctl->v_full[st], 2 * kQ8VBytes);
            __syncwarp();
            const uint32_t dst = smem_base + kQ8SmemV + st * kQ8VBytes;
            bool gathered = false;
            if (contig) {
                if (lane == 0) tma_box3d_pair(dst, &kv_v_map, bar, row_lo, 2 * (int)rank);
            } else {
                gathered = true;
                gather_rows_q8<2>(dst, kv_bytes + (int)rank * 256, row_lo, row_hi, lane);
            }
            if (pending >= 0) {
                retire_gathered_stage(map_to_rank(smem_u32(&ctl->v_full[pending]), leader), kQ8VBytes, gathered ? 1 : 0, lane);
                pending = -1;
            }
            if (gathered) pending = st;
            if (i + 1 < units) stage_rows(i + 1, x1, row_lo, row_hi, mask_unused, contig, any_bad);
            x1 = x2;
            stage_pages(x1);
            stage_tokens(i + 3, x2);
        }
        if (pending >= 0) retire_gathered_stage(map_to_rank(smem_u32(&ctl->v_full[pending]), leader), kQ8VBytes, 0, lane);
        if (!ok && lane == 0) {
            flag_status(p.status, OMNI_DEV_TIMEOUT | OMNI_DEV_ROLE_PRODUCER_V);
            *abort_flag = 1;
        }
    } else if (warp == 7) {
        // =========================== L2 prefetcher (as in tc2_decode_kernel) =============
        for (int t0 = (int)rank; t0 < units; t0 += 64) {
            const int t = t0 + 2 * lane;
            const int j0 = begin + t * kC2Tile;
            int row = -1;
            if (t < units && j0 + kC2Tile <= end) {
                const int first = selection_at(selection, j0), last = selection_at(selection, j0 + kC2Tile - 1);
                if (first >= 0 && first % kPage == 0 && last == first + kC2Tile - 1 && first / kPage < p.max_pages) {
                    const int pg = ldg_index(pt + first / kPage, selection.keep);
                    if (pg >= 0 && (int64_t)pg < p.num_pages) row = pg * kPage;
                }
            }
            __syncwarp();
            bool ok = true;
            TileIdx x = {-1, -1, -1, -1};    // of a unit that is not a whole page
            for (int k = 0; ok && k < 32 && t0 + 2 * k < units; ++k) {
                const int i = t0 + 2 * k;
                const bool page = __shfl_sync(0xffffffffu, row, k) >= 0;
                if (!page) {
                    stage_tokens(i, x);
                    stage_pages(x);
                }
                const volatile int32_t *progress = &ctl->k_progress;
                for (int naps = 0; *progress < i - (int)rank - (page ? 0 : kScatterAhead) && *abort_flag == 0; ++naps) {
                    if (naps > (1 << 22)) {
                        ok = false;
                        break;
                    }
                    __nanosleep(200);
                }
                ok = ok && (*abort_flag == 0);
                ok = __all_sync(0xffffffffu, ok);
                if (ok && page && lane == k)
                    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(&kv_page_map),
                                 "r"(0), "r"(row), "r"(0)
                                 : "memory");
                if (ok && !page && *progress <= i) {
                    if ((uint32_t)x.pg0 < page_limit) prefetch_row_q8(kv_bytes, x.pg0 * kPage + (x.t0 & (kPage - 1)));
                    if ((uint32_t)x.pg1 < page_limit) prefetch_row_q8(kv_bytes, x.pg1 * kPage + (x.t1 & (kPage - 1)));
                }
                __syncwarp();
            }
            if (!ok) break;
        }
    } else if (warp == 1) {
        // =========================== MMA issuer (CTA 0 only) =============================
        if (rank == 0) {
            constexpr uint32_t idesc_qk8 = instr_desc_e4m3(128, 2 * kC2Tile, 0);
            constexpr uint32_t idesc_qkr = instr_desc(128, 2 * kC2Tile, 0);
            constexpr uint32_t idesc_pv8 = instr_desc_e4m3(128, 256, 1);
            const uint64_t q_desc = smem_desc(smem_base + kQ8SmemQHi, 16, 1024);
            const uint64_t k_desc = smem_desc(smem_base + kQ8SmemK, 16, 1024);
            const uint64_t p_desc = smem_desc(smem_base + kQ8SmemP, 16, 1024);
            const uint64_t v_desc = smem_desc(smem_base + kQ8SmemV, kPanelBytes, 1024);
            const uint32_t q_lo = (uint32_t)q_desc, k_lo = (uint32_t)k_desc, p_lo = (uint32_t)p_desc, v_lo = (uint32_t)v_desc;
            const uint32_t kmaj_hi = (uint32_t)(q_desc >> 32), v_hi = (uint32_t)(v_desc >> 32);
            const int tiles_u = __shfl_sync(0xffffffffu, tiles, 0), units_u = __shfl_sync(0xffffffffu, units, 0);
            const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem, 0);
            // S8(t) = [Q_hi | Q_lo] [K8 ; K8]^T: two terms x 16 steps of 32 codes; Sr(t) = Q_rope K_rope^T: 4 steps of 16 bf16
            auto issue_qk = [&](int kst, int sbuf) {
                const uint32_t d8 = tmem_u + kQ8ColS8 + 64 * sbuf, dr = tmem_u + kQ8ColSr + 64 * sbuf;
                const uint32_t kb = k_lo + ((kst * kQ8KBytes) >> 4);
                tc_mma8_pair_elect<false>(d8, q_lo, kmaj_hi, kb, kmaj_hi, idesc_qk8);
#pragma unroll
                for (int kk = 1; kk < 32; ++kk) {
                    const int term = kk >> 4, c = kk & 15;
                    tc_mma8_pair_elect<true>(d8, q_lo + ((term * kQ8SmemQLo + (c >> 2) * kPanelBytes + (c & 3) * 32) >> 4), kmaj_hi,
                                             kb + (((c >> 2) * kPanelBytes + (c & 3) * 32) >> 4), kmaj_hi, idesc_qk8);
                }
                tc_mma_pair_elect<false>(dr, q_lo + (kQ8SmemQRope >> 4), kmaj_hi, kb + ((4 * kPanelBytes) >> 4), kmaj_hi, idesc_qkr);
#pragma unroll
                for (int kk = 1; kk < 4; ++kk)
                    tc_mma_pair_elect<true>(dr, q_lo + ((kQ8SmemQRope + kk * 32) >> 4), kmaj_hi,
                                            kb + ((4 * kPanelBytes + kk * 32) >> 4), kmaj_hi, idesc_qkr);
                tc_commit_pair_elect(&ctl->k_empty[kst], pair_mask);
                tc_commit_pair_elect(&ctl->s_full[sbuf], pair_mask);
            };
            // O += [P_hi | P_lo] [V8 ; V8]: four steps of 32 codes of a P row (hi tokens 0..31, 32..63,
            // then lo), each against the matching 32 tokens of the stage, two N = 256 accumulators
            auto issue_pv = [&](int vst, int pbuf, bool first) {
                const uint32_t a = p_lo + ((pbuf * kPanelBytes) >> 4);
                const uint32_t bd = v_lo + ((vst * kQ8VBytes) >> 4);
                tc_mma8_pair_elect(tmem_u + kColO, a, kmaj_hi, bd, v_hi, idesc_pv8, first ? 0u : 1u);
                tc_mma8_pair_elect(tmem_u + kColO + 128, a, kmaj_hi, bd + (kPanelBytes >> 4), v_hi, idesc_pv8, first ? 0u : 1u);
#pragma unroll
                for (int k = 1; k < 4; ++k) {
                    const uint32_t ak = a + ((k * 32) >> 4), bk = bd + (((k & 1) * 4096) >> 4);
                    tc_mma8_pair_elect<true>(tmem_u + kColO, ak, kmaj_hi, bk, v_hi, idesc_pv8);
                    tc_mma8_pair_elect<true>(tmem_u + kColO + 128, ak, kmaj_hi, bk + (kPanelBytes >> 4), v_hi, idesc_pv8);
                }
                tc_commit_pair_elect(&ctl->v_empty[vst], pair_mask);
                tc_commit_pair_elect(&ctl->pv_done[pbuf], pair_mask);
            };
            // as in tc2_decode_kernel: whatever is ready goes next, scores first
            bool ok = mbar_wait(&ctl->q_ready, 0);
            ok = __all_sync(0xffffffffu, ok);
            if (ok) tc_fence_after();
            int t = 0, u = 0, vst = 0, vph = 0;
            long long start = 0;
            uint32_t idle = 0;
            while (ok && u < units_u) {
                const int sbuf = t & 1;
                const bool qk = t < tiles_u && mbar_test(&ctl->k_full[sbuf], (t >> 1) & 1) && mbar_test(&ctl->s_empty[sbuf], ((t >> 1) & 1) ^ 1);
                if (__all_sync(0xffffffffu, qk)) {
                    tc_fence_after();
                    issue_qk(sbuf, sbuf);
                    ++t;
                    idle = 0;
                    continue;
                }
                const bool pv = mbar_test(&ctl->p_full, (u >> 1) & 1) && mbar_test(&ctl->v_full[vst], vph);
                if (__all_sync(0xffffffffu, pv)) {
                    tc_fence_after();
                    issue_pv(vst, u & 1, u == 0);
                    ++u;
                    if (++vst == kQ8VStages) {
                        vst = 0;
                        vph ^= 1;
                    }
                    idle = 0;
                    continue;
                }
                if ((++idle & 63u) == 0u) {
                    const long long now = __shfl_sync(0xffffffffu, clock64(), 0);
                    if (idle == 64u)
                        start = now;
                    else
                        ok = now - start <= kWaitCycles;
                    ok = ok && __shfl_sync(0xffffffffu, *abort_flag, 0) == 0u;
                }
            }
            if (!ok && lane == 0) {
                flag_status(p.status, OMNI_DEV_TIMEOUT | OMNI_DEV_ROLE_MMA);
                *abort_flag = 1;
            }
        }
        __syncwarp();
    } else {
        // =========================== softmax + epilogue =================================
        const int quarter = warp & 3;
        const int sub = warp >= 8 ? 1 : 0;
        const int row = (quarter & 1) * 32 + lane;
        const int half = quarter >> 1;
        const int part = half * 2 + sub;
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        const uint32_t s_empty_leader = map_to_rank(smem_u32(&ctl->s_empty[0]), leader);
        const uint32_t p_full_leader = map_to_rank(smem_u32(&ctl->p_full), leader);
        bool ok = true;
        float a_row = 1.f;
        {
            // ---- rewrite q's latent columns as two E4M3 terms per value -------------------
            // This thread: head row `row`, latent columns [128 * part, 128 * part + 128), i.e. bf16
            // panels 2*part and 2*part+1 of the temporary copy and code panel `part` of each term.
            ok = mbar_wait(&ctl->q_full, 0);
            ok = __all_sync(0xffffffffu, ok);
            float amax = 0.f;
            const uint8_t *src = smem + kQ8SmemQTemp + (size_t)(2 * part) * kPanelBytes + row * 128;
            if (ok) {
#pragma unroll
                for (int c = 0; c < 16; ++c) {
                    const uint4 w = *reinterpret_cast<const uint4 *>(src + (c >> 3) * kPanelBytes + (((c & 7) ^ (row & 7)) << 4));
                    const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        amax = fmaxf(amax, fabsf(__uint_as_float(ws[k] << 16)));
                        amax = fmaxf(amax, fabsf(__uint_as_float(ws[k] & 0xffff0000u)));
                    }
                }
                ctl->xchg[0][part][row] = amax;
            }
            asm volatile("bar.sync 2, 256;" ::: "memory");        // the eight softmax warps
            if (ok) {
                amax = fmaxf(fmaxf(ctl->xchg[0][0][row], ctl->xchg[0][1][row]), fmaxf(ctl->xchg[0][2][row], ctl->xchg[0][3][row]));
                // a power of two with |q| / a < 448: the division is exact
                int e = 0;
                if (amax > 0.f) (void)frexpf(amax * (1.f / 448.f), &e);
                a_row = amax > 0.f ? ldexpf(1.f, e) : 1.f;
                const float inv_a = 1.f / a_row;
                uint8_t *hi_row = smem + kQ8SmemQHi + (size_t)part * kPanelBytes + row * 128;
                uint8_t *lo_row = smem + kQ8SmemQLo + (size_t)part * kPanelBytes + row * 128;
#pragma unroll
                for (int c = 0; c < 8; ++c) {                    // 16 columns = one 16-byte chunk of codes
                    float v[16];
#pragma unroll
                    for (int hc = 0; hc < 2; ++hc) {
                        const int cc = 2 * c + hc;               // bf16 chunk (8 columns) within the thread's 128
                        const uint4 w = *reinterpret_cast<const uint4 *>(src + (cc >> 3) * kPanelBytes + (((cc & 7) ^ (row & 7)) << 4));
                        const uint32_t ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            v[8 * hc + 2 * k] = __uint_as_float(ws[k] << 16) * inv_a;
                            v[8 * hc + 2 * k + 1] = __uint_as_float(ws[k] & 0xffff0000u) * inv_a;
                        }
                    }
                    uint4 hi, lo;
                    split_e4m3(v, hi, lo);
                    *reinterpret_cast<uint4 *>(hi_row + ((c ^ (row & 7)) << 4)) = hi;
                    *reinterpret_cast<uint4 *>(lo_row + ((c ^ (row & 7)) << 4)) = lo;
                }
                if (part == 0) aux->q_scale[row] = a_row;
            }
            fence_async_smem();                                   // the tensor core reads what the threads wrote
            asm volatile("bar.sync 2, 256;" ::: "memory");        // every read of the temporary copy is done
            if (lane == 0) {
                mbar_arrive(&ctl->q_conv);
                mbar_arrive_cluster(map_to_rank(smem_u32(&ctl->q_ready), leader));
            }
            a_row = aux->q_scale[row];
        }
        float m_ref = -INFINITY, l = 0.f;
        // this thread: head row `row`, tokens [64 half + 32 sub, + 32) of every tile, i.e. quarter `part`
        const float ac = a_row * p.scale_log2;
        for (int i = 0; ok && i < tiles; ++i) {
            const int sbuf = i & 1, ring = i % kQ8Ring;
            ok = mbar_wait(&ctl->s_full[sbuf], (i >> 1) & 1);
            if (!__all_sync(0xffffffffu, ok)) {
                ok = false;
                break;
            }
            tc_fence_after();
            uint32_t s8[32], sr[32];
            tc_ld32(tmem + lane_base + kQ8ColS8 + 64 * sbuf + 32 * sub, s8);
            tc_ld32(tmem + lane_base + kQ8ColSr + 64 * sbuf + 32 * sub, sr);
            tc_wait_ld();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(s_empty_leader + 8 * sbuf);
            const uint32_t valid = (uint32_t)(ctl->valid_mask[ring][half] >> (32 * sub));
            const float4 *ts = reinterpret_cast<const float4 *>(&aux->tok_scale[ring][32 * part]);
            const float4 *tl = reinterpret_cast<const float4 *>(&aux->tok_log2[ring][32 * part]);
            float y[32];
            const f32x2 ac2 = pack2(ac, ac), scale2 = pack2(p.scale_log2, p.scale_log2);
#pragma unroll
            for (int g = 0; g < 8; ++g) {
                const float4 sc = ts[g], lg = tl[g];
#pragma unroll
                for (int k = 0; k < 4; k += 2) {
                    const int j = 4 * g + k;
                    const f32x2 rope = fma2(pack2(__uint_as_float(sr[j]), __uint_as_float(sr[j + 1])), scale2, k ? pack2(lg.z, lg.w) : pack2(lg.x, lg.y));
                    const float2 v = unpack2(fma2(pack2(__uint_as_float(s8[j]), __uint_as_float(s8[j + 1])),
                                                  mul2(ac2, k ? pack2(sc.z, sc.w) : pack2(sc.x, sc.y)), rope));
                    y[j] = v.x;
                    y[j + 1] = v.y;
                }
            }
            if (valid != 0xffffffffu) {
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    if (!((valid >> j) & 1u)) y[j] = -INFINITY;
            }
            float mt = fmaxf(max32([&](int j) { return y[j]; }), -INFINITY);
            ctl->xchg[i & 1][part][row] = mt;
            mbar_arrive(&ctl->x_bar);
            ok = mbar_wait(&ctl->x_bar, i & 1);
            if (!__all_sync(0xffffffffu, ok)) {
                ok = false;
                break;
            }
            mt = fmaxf(fmaxf(ctl->xchg[i & 1][0][row], ctl->xchg[i & 1][1][row]),
                       fmaxf(ctl->xchg[i & 1][2][row], ctl->xchg[i & 1][3][row]));
            float factor = 1.f;
            bool moved = false;
            if (mt > m_ref + kQ8RescaleWindow || (m_ref == -INFINITY && mt > -INFINITY)) {
                // the new reference sits kQ8Headroom below the tile maximum (see the constants)
                factor = exp2f(m_ref - (mt - kQ8Headroom));
                m_ref = mt - kQ8Headroom;
                moved = true;
            }
            const float mr = (m_ref == -INFINITY) ? 0.f : m_ref;
            const float4 *tr = reinterpret_cast<const float4 *>(&aux->tok_rcp[ring][32 * part]);
            const f32x2 mr2 = pack2(-mr, -mr);
            f32x2 sums = pack2(0.f, 0.f);
            uint4 p_hi[2], p_lo[2];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                float pw[16];
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const float4 rc = tr[4 * c + g];
#pragma unroll
                    for (int k = 0; k < 4; k += 2) {
                        const int j = 4 * g + k;
                        const float2 d = unpack2(add2(pack2(y[16 * c + j], y[16 * c + j + 1]), mr2));
                        pw[j] = fast_exp2(d.x);                      // p * scale_t, below 448; 0 for a masked token
                        pw[j + 1] = fast_exp2(d.y);
                        sums = fma2(pack2(pw[j], pw[j + 1]), k ? pack2(rc.z, rc.w) : pack2(rc.x, rc.y), sums);   // p (a masked token repeats a selected row's scale)
                    }
                }
                split_e4m3(pw, p_hi[c], p_lo[c]);
            }
            const float2 sum = unpack2(sums);
            l = l * factor + (sum.x + sum.y);
            // P and O are free once P V of the tile before retired
            if (i >= 1) {
                ok = mbar_wait(&ctl->pv_done[1], (i - 1) & 1);
                if (!__all_sync(0xffffffffu, ok)) {
                    ok = false;
                    break;
                }
                if (__any_sync(0xffffffffu, moved)) {
                    tc_fence_after();
#pragma unroll 1
                    for (int c = 0; c < 128; c += 32) {
                        uint32_t ov[32];
                        tc_ld32(tmem + lane_base + kColO + 128 * sub + c, ov);
                        tc_wait_ld();
#pragma unroll
                        for (int j = 0; j < 32; ++j) ov[j] = __float_as_uint(__uint_as_float(ov[j]) * factor);
                        tc_st32(tmem + lane_base + kColO + 128 * sub + c, ov);
                    }
                    tc_wait_st();
                }
            }
            // a P row of unit 2 i + half: hi codes of its 64 tokens in chunks 0-3, lo codes in chunks 4-7
            uint8_t *p_row = smem + kQ8SmemP + half * kPanelBytes + row * 128;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                *reinterpret_cast<uint4 *>(p_row + (((2 * sub + c) ^ (row & 7)) << 4)) = p_hi[c];
                *reinterpret_cast<uint4 *>(p_row + (((4 + 2 * sub + c) ^ (row & 7)) << 4)) = p_lo[c];
            }
            fence_async_smem();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(p_full_leader);
        }
        if (ok) {
            ok = mbar_wait(&ctl->pv_done[(units - 1) & 1], ((units - 1) >> 1) & 1);
            ok = __all_sync(0xffffffffu, ok);
        }
        if (ok) {
            ctl->xchg[tiles & 1][part][row] = l;
            mbar_arrive(&ctl->x_bar);
            ok = mbar_wait(&ctl->x_bar, tiles & 1);
            ok = __all_sync(0xffffffffu, ok);
        }
        if (kClusterMerge && ok) {
            if (warp == 2 && lane == 0) mbar_arrive_cluster(map_to_rank(smem_u32(&ctl->ready_bar), crank ^ 2u));
            const float lt = (ctl->xchg[tiles & 1][0][row] + ctl->xchg[tiles & 1][1][row]) +
                             (ctl->xchg[tiles & 1][2][row] + ctl->xchg[tiles & 1][3][row]);
            cm_inv = lt > 0.f ? 1.f / lt : 0.f;
            cm_lse = row_lse(lt, m_ref, true);
        } else if (!kClusterMerge && ok) {
            tc_fence_after();
            const float lt = (ctl->xchg[tiles & 1][0][row] + ctl->xchg[tiles & 1][1][row]) +
                             (ctl->xchg[tiles & 1][2][row] + ctl->xchg[tiles & 1][3][row]);
            c2_store_result<128>(p, smem, tmem, warp, lane, unit, h0, head_rows, lt, m_ref);
            if (unit.splits != 1 && p.counters != nullptr) __threadfence();
        }
        if (!ok && lane == 0) {
            flag_status(p.status, OMNI_DEV_TIMEOUT | OMNI_DEV_ROLE_SOFTMAX);
            *abort_flag = 1;
        }
        softmax_ok = ok;
    }

    // ---- tear-down (as in tc2_decode_kernel) ---------------------------------------------------
    if (*abort_flag) nap_after_abort();
    if (kClusterMerge) cluster_merge_exchange(p, ctl, smem, tmem, b, s, crank, h0, rows, head_rows, active, softmax_ok, cm_lse, cm_inv);
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        if (kClusterMerge) {
            mbar_wait(&ctl->taken_bar, 0, kLeaveCycles);
            if (*const_cast<volatile uint32_t *>(&ctl->xfail)) nap_after_abort();
        }
        if (lane == 0) {
            mbar_arrive(&ctl->exit_bar);
            mbar_arrive_cluster(map_to_rank(smem_u32(&ctl->exit_bar), peer));
        }
        mbar_wait(&ctl->exit_bar, 0, kLeaveCycles);
        __syncwarp();
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
    if (!kClusterMerge && p.splits > 1 && p.counters != nullptr)
        merge_if_last(p, b, (int)rank, 2, h0, head_rows, reinterpret_cast<float *>(smem), &ctl->merge_flag);
}

__global__ void __launch_bounds__(kC2Threads, 1)
tc2q8_decode_kernel(const __grid_constant__ CUtensorMap q_nope_map, const __grid_constant__ CUtensorMap q_rope_map,
                    const __grid_constant__ CUtensorMap kv_k_map, const __grid_constant__ CUtensorMap kv_v_map,
                    const __grid_constant__ CUtensorMap kv_page_map, DecodeParams p)
{
    tc2q8_decode_body<false>(q_nope_map, q_rope_map, kv_k_map, kv_v_map, kv_page_map, p);
}

__global__ void __launch_bounds__(kC2Threads, 1)
tc2q8_decode_cm_kernel(const __grid_constant__ CUtensorMap q_nope_map, const __grid_constant__ CUtensorMap q_rope_map,
                       const __grid_constant__ CUtensorMap kv_k_map, const __grid_constant__ CUtensorMap kv_v_map,
                       const __grid_constant__ CUtensorMap kv_page_map, DecodeParams p)
{
    tc2q8_decode_body<true>(q_nope_map, q_rope_map, kv_k_map, kv_v_map, kv_page_map, p);
}

// Quantiser of the 8-bit cache: kQ8RowsPerWarp rows per warp.  scale = max(amax, 2^-60) / 448 with amax
// the largest magnitude of the row's 512 latent columns, code = E4M3(value / scale) with the
// division in fp32 and round-to-nearest-even, saturating conversion; the 64 rope columns are copied.
//
// Every value is read once and every code written once, so memory bounds the kernel as long as the
// arithmetic stays under it.  A correctly rounded division per value does not (sixteen per lane
// and row, each an order of magnitude more instructions than a multiplication).  All divisions of a
// row share their divisor, so the quotient comes from its correctly rounded reciprocal and one
// remainder step (Markstein, "Computation of elementary functions on the IBM RISC System/6000
// processor", 1990).  Over every pair of a bf16 value and a bf16 row maximum the codes were checked to be
// those of the division.  57344 rows: 26.7 us with divisions, 17.4 us now (5.9 TB/s, 90 % of a copy).  The remainder is rounded down, so that an exact one is -0 and a
// quotient of -0 keeps its sign.  A row whose maximum is infinite takes the division.
constexpr int kQ8RowsPerWarp = 2;
constexpr int kQ8QuantWarps = 8;
__device__ __forceinline__ float q8_quotient(float x, float scale, float rcp)
{
    const float q = x * rcp;
    return fmaf(__fmaf_rd(-q, scale, x), rcp, q);
}
__global__ void __launch_bounds__(kQ8QuantWarps * 32) quantize_q8_kernel(const __nv_bfloat16 *__restrict__ rows, int64_t num_rows,
                                                                         uint8_t *__restrict__ out, float *__restrict__ scale)
{
    // launched with programmatic stream serialization: nothing is read or written before the kernel
    // in front has finished, and the one behind may get ready meanwhile
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int64_t r0 = ((int64_t)blockIdx.x * kQ8QuantWarps + (threadIdx.x >> 5)) * kQ8RowsPerWarp;
    const int lane = threadIdx.x & 31;
    // lane l: columns [8l, 8l + 8) and [256 + 8l, 256 + 8l + 8), lanes 0-7 the rope columns too; all
    // loads of the warp's rows go out before the first is used
    uint4 w[kQ8RowsPerWarp][2], rope[kQ8RowsPerWarp];
#pragma unroll
    for (int j = 0; j < kQ8RowsPerWarp; ++j) {
        if (r0 + j < num_rows) {
            const uint4 *src = reinterpret_cast<const uint4 *>(rows + (r0 + j) * kDqk);
            w[j][0] = __ldg(src + lane);
            w[j][1] = __ldg(src + 32 + lane);
            if (lane < 8) rope[j] = __ldg(src + 64 + lane);
        }
    }
#pragma unroll
    for (int j = 0; j < kQ8RowsPerWarp; ++j) {
        const int64_t r = r0 + j;
        if (r >= num_rows) return;
        const uint32_t ws[8] = {w[j][0].x, w[j][0].y, w[j][0].z, w[j][0].w, w[j][1].x, w[j][1].y, w[j][1].z, w[j][1].w};
        // the maximum on bf16 pairs: exact, and a NaN never wins (it starts from zero)
        __nv_bfloat162 top = __float2bfloat162_rn(0.f);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t mag = ws[k] & 0x7fff7fffu;
            top = __hmax2(top, *reinterpret_cast<const __nv_bfloat162 *>(&mag));
        }
        const uint32_t bits = *reinterpret_cast<const uint32_t *>(&top);
        // magnitudes order like their bit patterns
        const uint32_t amax_bits = __reduce_max_sync(0xffffffffu, max(bits << 16, bits & 0xffff0000u));
        const float sc = __fdiv_rn(fmaxf(__uint_as_float(amax_bits), 0x1p-60f), 448.f);
        uint32_t c[4];
        if (amax_bits < 0x7f800000u) {
            const float rcp = __frcp_rn(sc);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t u0 = ws[2 * k], u1 = ws[2 * k + 1];
                c[k] = e4m3x2(q8_quotient(__uint_as_float(u0 << 16), sc, rcp), q8_quotient(__uint_as_float(u0 & 0xffff0000u), sc, rcp)) |
                       (e4m3x2(q8_quotient(__uint_as_float(u1 << 16), sc, rcp), q8_quotient(__uint_as_float(u1 & 0xffff0000u), sc, rcp)) << 16);
            }
        } else {
#pragma unroll 1
            for (int k = 0; k < 4; ++k) {
                const uint32_t u0 = k == 0 ? ws[0] : k == 1 ? ws[2] : k == 2 ? ws[4] : ws[6];
                const uint32_t u1 = k == 0 ? ws[1] : k == 1 ? ws[3] : k == 2 ? ws[5] : ws[7];
                const uint32_t v = e4m3x2(__fdiv_rn(__uint_as_float(u0 << 16), sc), __fdiv_rn(__uint_as_float(u0 & 0xffff0000u), sc)) |
                                   (e4m3x2(__fdiv_rn(__uint_as_float(u1 << 16), sc), __fdiv_rn(__uint_as_float(u1 & 0xffff0000u), sc)) << 16);
                (k == 0 ? c[0] : k == 1 ? c[1] : k == 2 ? c[2] : c[3]) = v;
            }
        }
        uint8_t *dst = out + r * kQ8RowBytes;
        *reinterpret_cast<uint2 *>(dst + 8 * lane) = make_uint2(c[0], c[1]);
        *reinterpret_cast<uint2 *>(dst + 256 + 8 * lane) = make_uint2(c[2], c[3]);
        if (lane < 8) *reinterpret_cast<uint4 *>(dst + 512 + 16 * lane) = rope[j];
        if (lane == 0) scale[r] = sc;
    }
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------
// The 8-bit pool seen as [rows, 5 panels of 128 bytes]: boxes {128 bytes, box_rows, n panels}.
inline bool encode_q8_panel_map(CUtensorMap *map, const void *base, uint64_t rows, uint32_t box_rows, uint32_t box_panels)
{
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t dims[3] = {128, (cuuint64_t)rows, (cuuint64_t)kQ8Panels};
    const cuuint64_t strides[2] = {(cuuint64_t)kQ8RowBytes, 128};
    const cuuint32_t box[3] = {128, box_rows, box_panels};
    const cuuint32_t estr[3] = {1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<void *>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

inline bool tc2q8_prepare_device()
{
    static bool attr_set[64] = {};
    static std::mutex mu;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    std::lock_guard<std::mutex> lock(mu);
    if (!attr_set[dev]) {
        if (cudaFuncSetAttribute(tc2q8_decode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kC2SmemBytes) !=
                cudaSuccess ||
            cudaFuncSetAttribute(tc2q8_decode_cm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kC2SmemBytes) !=
                cudaSuccess)
            return false;
        attr_set[dev] = true;
    }
    return true;
}

// maps[0] = q latent panels, maps[1] = q rope panel, maps[2] = K role, maps[3] = V role, maps[4] = whole pages
inline bool tc2q8_make_maps(const DecodeParams &p, CUtensorMap *maps, bool cached)
{
    const uint64_t rows = (uint64_t)p.num_pages * kPage, qrows = (uint64_t)p.batch * p.heads;
    if (cached)
        return cached_map(&maps[0], p.q, qrows, kTcHeads, 8, 1, encode_panel_map) &&
               cached_map(&maps[1], p.q, qrows, kTcHeads, 1, 1, encode_panel_map) &&
               cached_map(&maps[2], p.kv, rows, kTile, kQ8Panels, 2, encode_q8_panel_map) &&
               cached_map(&maps[3], p.kv, rows, kTile, 2, 2, encode_q8_panel_map) &&
               cached_map(&maps[4], p.kv, rows, kTile, kQ8Panels, 2, encode_q8_panel_map);
    return encode_panel_map(&maps[0], p.q, qrows, kTcHeads, 8) && encode_panel_map(&maps[1], p.q, qrows, kTcHeads, 1) &&
           encode_q8_panel_map(&maps[2], p.kv, rows, kTile, kQ8Panels) && encode_q8_panel_map(&maps[3], p.kv, rows, kTile, 2) &&
           encode_q8_panel_map(&maps[4], p.kv, rows, kTile, kQ8Panels);
}

inline omni_status_t tc2q8_launch(const CUtensorMap *maps, const DecodeParams &p, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((p.whole + (p.batch - p.whole) * p.splits) * 2));
    cfg.blockDim = dim3(kC2Threads);
    cfg.dynamicSmemBytes = kC2SmemBytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = p.cluster_merge ? 4 : 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, p.cluster_merge ? tc2q8_decode_cm_kernel : tc2q8_decode_kernel, maps[0], maps[1], maps[2],
                              maps[3], maps[4], p) == cudaSuccess
               ? OMNI_OK
               : OMNI_ERR_CUDA;
}

}  // namespace omni
