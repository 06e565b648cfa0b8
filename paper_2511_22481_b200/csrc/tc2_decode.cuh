// Paired-CTA tensor-core decode kernel for sm_100a (every problem but the smallest with few heads).
//
// A cluster of two CTAs owns all heads of one (request, split), each CTA half of them, up to 64
// rows.  The pair issues cta_group::2 MMAs with M = 128 (64 rows per CTA), which run
// the tensor pipe of each SM at full rate where a lone M = 64 MMA runs it at half rate, and it
// halves the operand bytes each SM must hold.  Per tile of 128 tokens, two units of 64:
//   S = Q K^T   M=128, N=128 tokens, K=576: every CTA supplies its 64 Q rows and the K rows of
//               ITS unit of the tile ("K role": 64 tokens x 576 columns, 72 KiB)
//   O += P V    per unit: M=128, N=256 per instruction (two of them), K=64 tokens: every CTA
//               supplies its 64 P rows and, for all 64 tokens, ITS 256 value columns ("V role":
//               64 tokens x 256 columns, 32 KiB; CTA r holds columns [256r, 256r+256))
// The two roles overlap only in a quarter of the tile, at different addresses in the two CTAs,
// so each role is loaded on its own (1.9x the tile's bytes cross L2 -> shared memory, which L2
// sustains; each byte leaves HBM once because the pair runs together).
//
// What bounds it: a score MMA over N = 64 tokens is bound by its operand reads from shared memory (24
// clocks for 16 clocks of math), over N = 128 by the math (32 clocks), so a tile of 128 tokens costs
// the tensor core 2176 clocks where two of 64 cost 2750; and it reads 23 % fewer operand bytes,
// which is power, and long runs are held back by the power limit.  From there on it is the refill of the
// operands: there is room for one tile of K rows and one of V columns, about one HBM latency of
// work, so each is refilled piece by piece as it is used up: K in three groups of three column panels,
// V in its two units.  Where 64 pairs read 17 units each (32 requests x 33 units), HBM delivers at its rate
// throughout the main loop, and what is left is the start and the end of a launch.  Against tiles
// of 64 tokens with two whole stages, both measured in one call: 32 requests x 33 units 25.6 ->
// 24.5 us, 64 x 33 43.2 -> 40.7, 128 x 64 156 -> 147, one request of 128 units 16.4 -> 15.7.
//
// The loads of a piece are requested as soon as its last reader retires, S is triple buffered, and
// Q K^T runs up to two tiles ahead of P V.  Every piece is ONE 3-D TMA box {64 columns, 64 rows,
// panels}: requesting one costs a warp 50 to 90 clocks.  Units that are not 64 consecutive pool rows
// are gathered row by row with cp.async (see below).
//
// All MMAs are issued by warp 1 of CTA 0 in "whatever is ready" order: the whole warp runs the
// loop with warp-uniform control flow and one elected lane issues each instruction (a lone
// diverged thread cannot feed the tensor pipe: it needs ~110 clocks per MMA, the elected form
// issues one every 25-64 clocks).  Completion is broadcast to both CTAs with multicast commits.
//
// Warps per CTA: 0 K-role producer, 1 MMA issuer (CTA 0 only) + tensor-memory owner, 2-5 and 8-11
// softmax / epilogue (a thread serves one head row and 32 of a tile's 128 tokens), 6 V-role
// producer, 7 L2 prefetcher: the rows of each unit are pulled into L2 ahead of their K-role load, so
// that the shared-memory refills start from a line already on its way.
//
// Tensor memory per CTA (a 64-row slice of an M=128 pair accumulator keeps columns [0, N/2) in
// lanes 0-63 and columns [N/2, N) in lanes 64-127):
//   columns   0..255  O: two N=256 accumulators; lane L, column x  <->  head row L%64,
//                        value column 256*(L/64) + x
//   columns 256..319  S buffer 0: lane L, column x <-> head row L%64, token 64*(L/64) + x
//   columns 320..383, 384..447  S buffers 1, 2
//
// Splits of a request are merged in one of three ways chosen by the host: inside a cluster of
// two pairs (two splits, see cluster_merge_exchange), by a separate merge kernel over fp32
// partial results, or by the last CTA to finish a request's head half (a counter per (request,
// head half) in the workspace).
#pragma once

#include <type_traits>

#include "merge.cuh"
#include "tc_decode.cuh"

namespace omni {

constexpr int kC2Tile = 64;                              // tokens per unit: the granule of splits, index handling and P V
constexpr int kC2Threads = 384;
// Tiles the L2 prefetch of scattered rows runs ahead of that of whole pages.  A page is prefetched when the K
// loads of the tile in front of its own have been requested: a prefetch that competes with the loads of
// an earlier tile delays them (requested one tile earlier 25.8 us per step of 32 requests x 33 units, just
// before those loads 25.5, just after them 24.5).
constexpr int kScatterAhead = 1;
// Long work units prefetch whole pages for their first tiles only.  In a short launch the prefetch hides a memory latency per tile; in a
// long one HBM has the requests of many pairs at once anyway, and a prefetch is a third pass through L2 and the copy
// engine on launches that are held back by power: 32 x 1024 units 703 -> 680 us, 74 x 128 200 -> 186, 128 requests of 8 to
// 128 units 185.5 -> 182.  Cut there as well, 32 x 33 units (17 a pair) would go from 27.2 to 27.9.  Scattered rows are prefetched
// throughout: a gathered group waits a latency of its own, however long the unit (without: 37 x 96 units of scattered tokens 99 ->
// 103 us, 74 x 96 181 -> 184, 32 x 128 183 -> 195, 4 x 256 on a pair each 349 -> 381).
// Where few pairs run, HBM is not busy and the prefetch pays up to longer units (never cut -> always, one unit to a pair): 16 and 32 pairs of
// 48 units 41.7 -> 42.6 and 44.9 -> 46.2, 32 of 64 58.5 -> 59.4, of 96 86.3 -> 85.8; 40 pairs of 48 53.9 -> 53.8, 56 of them 63.4 -> 61.3, 74 of 64
// 98.3 -> 95.9, 8 of 96 79.7 -> 76.7.  The instances that merge in a cluster prefetch throughout: cut as well, 32 requests of 192 units go from
// 128 to 121 us and 32 x 128 from 86.5 to 84.3, but the code of the test alone makes 32 x 33 27.04 -> 27.41.
constexpr int kPrefetchAllUnits = 48, kPrefetchManyPairs = 40, kPrefetchLongUnits = 96, kPrefetchFirstUnits = 8;
constexpr int kC2GroupPanels = 3;                        // K role: refilled in three groups of three panels
constexpr int kC2Groups = kPanels / kC2GroupPanels;
constexpr int kC2GroupBytes = kC2GroupPanels * kPanelBytes;   // [64 tokens x 128 B] x 3
constexpr int kC2VBytes = 4 * kPanelBytes;               // V role: 4 panels x [64 tokens x 128 B]
constexpr int kC2SmemQ = 0;                              // 9 panels x [64 heads x 128 B]
constexpr int kC2SmemK = kC2SmemQ + kTileBytes;          // 9 panels x [64 tokens x 128 B]
constexpr int kC2SmemV = kC2SmemK + kTileBytes;          // 2 stages
constexpr int kC2SmemP = kC2SmemV + 2 * kC2VBytes;       // 2 units x [64 heads x 128 B]
constexpr int kC2SmemCtl = kC2SmemP + 2 * kPanelBytes;
constexpr int kC2SmemCtlBytes = 3072;
constexpr int kC2SmemBytes = kC2SmemCtl + kC2SmemCtlBytes;   // no alignment slack: the base is checked at run time
constexpr uint32_t kC2ColS = 256;
// Validity masks travel from the K producer to the softmax warps through a small ring, in units.  The
// producer resolves up to tile t + 2 once the score MMAs of tile t have retired.  Those were issued only
// after every softmax warp had read the scores of tile t - 3 (three score buffers), i.e. after tile
// t - 4 was finished: six tiles can be live, and the ring holds eight.
constexpr int kMaskRing = 16;

// Limit of the waits for the other CTAs at the end of a launch.  After a wait that ran out (in a cluster merge after up
// to five in a row) a CTA still arrives at the others' barriers; had they left by then, which waits of the same
// length make certain, the time-out would end as an access to shared memory that is gone: a failed launch.
constexpr long long kLeaveCycles = 8 * kWaitCycles;

// A wait ran out: gives copies that are still in flight time to land before anyone exits.
__device__ __forceinline__ void nap_after_abort()
{
    for (int i = 0; i < 200; ++i) __nanosleep(1000);
}

// Head rows per CTA of a pair.
__host__ __device__ __forceinline__ int c2_rows(int heads) { return (heads + 1) >> 1; }

// What a pair works on: split s of `splits` of request b (splits = 0: nothing), whose partial results are those
// of request `slot`.
struct C2Unit {
    int b, s, splits, slot;
};

// A further unit of a pair, as it is dealt out: request and split (negative: there is none), the length the caller gave and the entries
// [begin, end) of the selection.
struct alignas(16) C2Work {
    int request_split, length, begin, end;
};
// A pair takes at most this many work units one after the other.
constexpr int kC2Rounds = 16;

struct C2Control {
    uint64_t k_full[kC2Groups];          // per tile; those of the first tile wait for q's panels too
    uint64_t k_empty[kC2Groups];
    uint64_t v_full[2];
    uint64_t s_full[3];
    uint64_t s_empty[3];
    uint64_t p_full;                     // both P units of a tile are written (and O rescaled)
    uint64_t pv_done[2];                 // P V of a unit retired: frees its V stage and its P unit
    uint64_t x_bar;                      // all softmax threads: exchange of the final row sums
    uint64_t exit_bar;                   // both CTAs of the pair are done with tensor memory
    uint64_t valid_mask[kMaskRing];      // per unit: validity of its 64 tokens
    float xchg[2][4][64];                // row maxima: [tile parity][quarter of the tile's tokens][head row]; at the end the parity no longer in use carries the partial row sums
    uint32_t tmem_base;
    uint32_t abort;
    uint32_t merge_flag;
    uint32_t xfail;                      // cluster merge: some wait of this CTA ran out (decided CTA-wide)
    int32_t k_progress;                  // tiles whose K loads have been requested (L2 prefetch pacing)
    uint64_t recv_bar[4];                // cluster merge: the partner's chunks have arrived
    uint64_t ready_bar;                  // cluster merge: the partner's main loop is over
    uint64_t taken_bar;                  // cluster merge: the partner's softmax warps have received this CTA's block
    uint64_t xg_bar;                     // row-maximum exchange of a tile
    // several units per pair: the next cluster that has not begun (grant, asked for by CTA 0) and the unit it is, written to both CTAs
    uint64_t grant_bar;
    uint64_t work_full[kC2Rounds];
    alignas(16) uint4 grant;
    C2Work work[kC2Rounds];
};
static_assert(sizeof(C2Control) <= kC2SmemCtlBytes, "control block too large");
static_assert(kC2SmemBytes <= 232448, "shared memory budget");

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// Address of the same shared-memory location in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr)
{
    // default (CTA-scope release) semantics: a cluster-scope release costs ~0.6 us per arrive here,
    // and what must be ordered before it is already ordered by the tcgen05 / async-proxy fences
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

// Rendezvous of the cluster after the barriers were initialised.  The initialising thread has
// issued the barrier-init fence, so the arrive needs no release of its own (a release-ordered
// arrive cost half a microsecond of every launch); nothing else that the other CTAs read was
// written before it.
__device__ __forceinline__ void cluster_sync_after_init()
{
    __syncwarp();                        // the aligned forms want whole warps
    asm volatile("barrier.cluster.arrive.relaxed.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// 3-D box {64 columns, box rows, n column panels} loaded by one CTA of a pair: lands panel-major,
// i.e. as n consecutive [rows x 128 B] swizzled panels.  The transaction bytes are credited to
// `bar_cluster_addr`, which may be a barrier of the other CTA of the pair.
__device__ __forceinline__ void tma_box3d_pair(uint32_t dst, const CUtensorMap *map, uint32_t bar_cluster_addr,
                                               int row, int panel)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(0), "r"(row), "r"(panel), "r"(bar_cluster_addr)
        : "memory");
}

// The same of q: box {64 columns, 64 rows, 3 panels} of one CTA's heads of one request (see encode_q_map).
__device__ __forceinline__ void tma_box5d_pair(uint32_t dst, const CUtensorMap *map, uint32_t bar_cluster_addr, int row, int panel,
                                               int side, int request)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
        ::"r"(dst), "l"(map), "r"(0), "r"(row), "r"(panel), "r"(side), "r"(request), "r"(bar_cluster_addr)
        : "memory");
}

// Row gathers without the copy engine.  A 4-row TMA gather moves 512 bytes per instruction and
// the engine takes ~60 clocks for each, which bounds token-level selections; a warp-wide 16-byte
// cp.async moves the same 512 bytes (four rows x 128 B, eight lanes per row) through the load/store
// path at several times that rate.  The lanes place their chunks in the 128-byte-swizzled operand
// layout themselves, and the warp credits the bytes to the stage's barrier with an explicit
// complete_tx once its copies have landed, exactly as a TMA copy would have.
__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory");
}
// One thread: credits bytes to a barrier of the pair, behind what this thread has written or seen written.
__device__ __forceinline__ void credit_bytes(uint32_t bar_cluster_addr, uint32_t bytes)
{
    asm volatile("fence.acq_rel.cta;" ::: "memory");
    asm volatile("mbarrier.complete_tx.relaxed.cluster.shared::cluster.b64 [%0], %1;" ::"r"(bar_cluster_addr), "r"(bytes)
                 : "memory");
}
// All lanes: wait for this lane's copies of the stage (all but the `newer` most recent groups of them, at
// most two), make them visible to the tensor core's proxy, then lane 0 credits `bytes` to the barrier.
__device__ __noinline__ void retire_gathered_stage(uint32_t bar_cluster_addr, uint32_t bytes, int newer, int lane)
{
    if (newer >= 2)
        cp_async_wait<2>();
    else if (newer == 1)
        cp_async_wait<1>();
    else
        cp_async_wait<0>();
    fence_async_smem();
    __syncwarp();
    // The rows are in this CTA's shared memory (wait_group returned in every lane, the proxy
    // fence and the warp barrier order them before this point) and it is this CTA's own
    // tensor core that will read them, so a CTA-scope fence is what orders them before the
    // credit.  A cluster-scope fence here would also wait for the next tile's copies and the
    // index loads this lane has in flight: measured at ~0.9 us per tile.
    if (lane == 0) credit_bytes(bar_cluster_addr, bytes);
}

// Gathers 64 rows x kCount panels, `cols` pointing at the first panel of row 0: eight lanes per row, four rows
// per instruction, chunk c of row r lands at chunk c ^ (r % 8) of its 128-byte line.  Kept out of
// line so that the producers' loops stay as small as they are for selections that never need it.
template <int kCount>
__device__ __noinline__ void gather_rows(uint32_t dst, const char *cols, int row_lo, int row_hi, int lane)
{
    const int ch = lane & 7;
#pragma unroll
    for (int g = 0; g < 16; ++g) {
        const int r = 4 * g + (lane >> 3);
        const int src_row = __shfl_sync(0xffffffffu, g < 8 ? row_lo : row_hi, r & 31);
        const char *src = cols + (size_t)src_row * (kDqk * 2) + ch * 16;
        const uint32_t d = dst + r * 128 + ((ch ^ (r & 7)) << 4);
#pragma unroll
        for (int c = 0; c < kCount; ++c) cp_async16(d + c * kPanelBytes, src + c * 128);
    }
    cp_async_commit();
}

// One cache row into L2.
__device__ __forceinline__ void prefetch_row(const __nv_bfloat16 *kv, int row)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(kv + (size_t)row * kDqk), "n"(kDqk * 2) : "memory");
}

// Pair MMA executed by a whole converged warp: one elected lane issues the instruction.  The
// descriptors arrive as 32-bit halves so that stepping through a tile is a 32-bit add.
template <bool kAccumulate>
__device__ __forceinline__ void tc_mma_pair_elect(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo,
                                                  uint32_t b_hi, uint32_t idesc)
{
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %5, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "n"(kAccumulate ? 1 : 0)
        : "memory");
}

// The same with the accumulate flag as a run-time value.
__device__ __forceinline__ void tc_mma_pair_elect(uint32_t d_tmem, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                                  uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %2};\n\t"
        "mov.b64 db, {%3, %4};\n\t"
        "setp.ne.b32 p, %6, 0;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.mma.cta_group::2.kind::f16 [%0], da, db, %5, p;\n\t}"
        ::"r"(d_tmem), "r"(a_lo), "r"(a_hi), "r"(b_lo), "r"(b_hi), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Arrive on the barrier at this shared-memory offset in BOTH CTAs once all MMAs issued so far by
// the elected lane have retired.
__device__ __forceinline__ void tc_commit_pair_elect(uint64_t *bar, uint16_t both)
{
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "elect.sync _|q, 0xffffffff;\n\t"
        "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n\t}"
        ::"r"(smem_u32(bar)), "h"(both)
        : "memory");
}

// Asks for the next cluster of this grid that has not begun, which then never will: 16 bytes that say which one it is, or that there was none
// to be had, arrive at `response`.  One thread.
__device__ __forceinline__ void try_cancel_cluster(uint4 *response, uint64_t *bar)
{
    asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];" ::"r"(smem_u32(response)),
                 "r"(smem_u32(bar))
                 : "memory");
}
// The first CTA of the cluster that such an answer names, or -1.
__device__ __forceinline__ int cancelled_cluster(const uint4 *response)
{
    int first;
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b128 answer;\n\t"
        "ld.shared.b128 answer, [%1];\n\t"
        "mov.b32 %0, -1;\n\t"
        "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, answer;\n\t"
        "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %0, answer;\n\t}"
        : "=&r"(first)
        : "r"(smem_u32(response))
        : "memory");
    return first;
}
// 16 bytes to a CTA of the cluster, credited to a barrier there.
__device__ __forceinline__ void st_async16(uint32_t dst_cluster_addr, uint32_t bar_cluster_addr, const int4 &v)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(dst_cluster_addr), "r"(v.x),
                 "r"(v.y), "r"(v.z), "r"(v.w), "r"(bar_cluster_addr)
                 : "memory");
}

// Split-KV merge inside a cluster of two pairs, i.e. the two splits of one request (cluster
// merge).  CTA `crank` and its partner `crank ^ 2` serve the same 64 heads in the two splits.
// Instead of writing fp32 partial results to global memory for a second kernel to read back,
// the two exchange what the other needs through distributed shared memory.  Of every head row
// split 0 finishes value columns [0,128) and [256,384), split 1 the other two quarters: these are
// the columns of softmax warps 2-5 and 8-11 in tensor memory, so in either CTA one warp per
// scheduler is a "sender" (its columns are finished by the partner) and one a "keeper":
//   1. the senders normalise their half by the row sums and write it to a block of shared memory, behind
//      the log-sum-exp of the split for every head row, which four bulk shared-memory-to-shared-memory
//      copies take to the partner, each as soon as its quarter of the block is written;
//   2. every softmax warp finishes 64 columns of its tensor-memory lane quarter as the quarters of the
//      partner's block come in (each has a barrier of its own): it weighs its own half (still in tensor
//      memory) and the received one by exp(lse_split - lse_total), adds them and stores bf16 rows
//      as whole 128-byte lines through warp-private staging tiles.
// What bounds it: the block takes about 4000 clocks through the network between SMs (17 bytes a clock), so
// everything else overlaps it; with one barrier for the whole block, and the cluster's last
// rendezvous behind the stores, the exchange took 7800 clocks after the later main loop, now 5800 (28.2 ->
// 27.6 us per step of 32 requests x 33 units).  Its barriers are mbarriers: an aligned cluster barrier in
// one branch of the kernel makes the compiler give up warp uniformity everywhere, 11 KB more code and
// a main loop 1.6 times slower.
// The copy lands in shared memory that held the partner's operand tiles, so it is not sent
// before the partner has said that its main loop is over (`ready_bar`, a remote arrive that the
// partner fires as soon as its last P V has retired, while this CTA is still staging).
// Called by every thread of the CTA after the main loop.  rows: head rows per CTA; only these are sent.
template <class Control>
__device__ __forceinline__ void cluster_merge_exchange(const DecodeParams &p, Control *ctl, uint8_t *smem,
                                                       uint32_t tmem, int b, int s, uint32_t crank, int h0,
                                                       int rows, int head_rows, bool active, bool main_ok, float cm_lse, float cm_inv)
{
    // The block travels as four chunks, so that the copy of one overlaps the staging of the next and the mixing
    // of the one before: chunk q holds, for every head row, the q-th 32 columns of both 128-column runs
    // that are sent.  The log-sum-exps go with the first.
    constexpr uint32_t kChunkPitch = 2 * 128 + 16;       // row-per-lane 16-byte accesses do not conflict
    constexpr uint32_t kChunkBytes = 64 * kChunkPitch;   // 17,408
    constexpr uint32_t kLseBytes = 256;
    constexpr uint32_t kBlockBytes = kLseBytes + 4 * kChunkBytes;      // 69,888
    constexpr uint32_t kStagePitch = 144, kStageBytes = 32 * kStagePitch;
    static_assert(2 * kBlockBytes + 8 * kStageBytes <= 221184, "exchange tiles must end below the control block and the 8-bit kernel's auxiliary arrays");
    uint8_t *send = smem, *stages = smem + kBlockBytes, *recv = smem + kBlockBytes + 8 * kStageBytes;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const bool is_softmax = (warp >= 2 && warp <= 5) || warp >= 8;
    if (!is_softmax) return;
    const int quarter = warp & 3, sub = warp >= 8 ? 1 : 0;
    const int row = (quarter & 1) * 32 + lane, half = quarter >> 1;
    const uint32_t partner = crank ^ 2u;
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    volatile uint32_t *xfail = &ctl->xfail;
    if (!main_ok && lane == 0) *xfail = 1u;
    // The partner may overwrite this CTA's operand tiles once it has been told that the main loop
    // here is over.  Warp 2 says so at the end of a main loop that went well; after one that did
    // not (or that never ran: an empty split) the same thread says so here, so that the arrive is
    // fired exactly once per launch whatever happened.
    if (warp == 2 && lane == 0 && (!active || !main_ok)) mbar_arrive_cluster(map_to_rank(smem_u32(&ctl->ready_bar), partner));

    // No warp leaves this function early and no barrier below depends on how a wait ended: the
    // four sending warps always meet at their named barrier, every wait is bounded, and a wait
    // that ran out only marks the launch as failed (its results are then unspecified).
    tc_fence_after();
    if (sub != s) {
        // ---- sender: this thread's 128 value columns are finished by the other split ----------
        if (half == 0) reinterpret_cast<float *>(send)[row] = cm_lse;
        // (sending warp) chunks go out as soon as they are staged and the partner's operand tiles are dead; a
        // split that finishes first has staged all of them by the time it hears that
        int sent = 0;
        auto send_chunks = [&](int upto) {
#pragma unroll 1
            for (; sent <= upto; ++sent) {
                const uint32_t from = sent == 0 ? 0u : kLseBytes + sent * kChunkBytes, bytes = rows * kChunkPitch + (sent == 0 ? kLseBytes : 0u);
                const uint32_t dst = map_to_rank(smem_u32(recv + from), partner);
                const uint32_t bar = map_to_rank(smem_u32(&ctl->recv_bar[sent]), partner);
                if (lane == 0)
                    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                                 ::"r"(dst), "r"(smem_u32(send + from)), "r"(bytes), "r"(bar)
                                 : "memory");
            }
        };
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
            uint32_t ov[32];
            __syncwarp();
            if (active) {
                tc_ld32(tmem + lane_base + kColO + 128 * sub + q * 32, ov);
                tc_wait_ld();
            }
            uint4 *o = reinterpret_cast<uint4 *>(send + kLseBytes + q * kChunkBytes + (size_t)row * kChunkPitch + half * 128);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                // an empty or fully masked split contributes exact zeros
                o[j] = (active && cm_inv != 0.f)
                           ? make_uint4(__float_as_uint(__uint_as_float(ov[4 * j]) * cm_inv),
                                        __float_as_uint(__uint_as_float(ov[4 * j + 1]) * cm_inv),
                                        __float_as_uint(__uint_as_float(ov[4 * j + 2]) * cm_inv),
                                        __float_as_uint(__uint_as_float(ov[4 * j + 3]) * cm_inv))
                           : make_uint4(0u, 0u, 0u, 0u);
            }
            fence_async_smem();                           // the bulk copy reads what the threads wrote
            asm volatile("bar.sync 2, 128;" ::: "memory"); // the four sending warps
            if (quarter == 0 && __all_sync(0xffffffffu, mbar_test(&ctl->ready_bar, 0))) send_chunks(q);
        }
        if (quarter == 0 && sent < 4) {
            bool ready = mbar_wait(&ctl->ready_bar, 0);
            ready = __all_sync(0xffffffffu, ready);
            if (ready) send_chunks(3);
            if (!ready && lane == 0) {
                *xfail = 1u;
                flag_status(p.status, OMNI_DEV_TIMEOUT | OMNI_DEV_ROLE_SOFTMAX);
            }
        }
    } else if (quarter == 0 && lane == 0) {
        for (int q = 0; q < 4; ++q) mbar_expect_tx(&ctl->recv_bar[q], rows * kChunkPitch + (q == 0 ? kLseBytes : 0u));
    }

    // ---- finish: the columns kept here (those of the warps with sub == s) never left tensor
    // memory.  All eight warps take part: a warp can read any column of its tensor-memory lane
    // quarter, so the keeping warp of a quarter finishes the first 64 of its 128 columns (chunks 0 and 1)
    // and the sending warp of the same quarter, its block gone, the other 64 (chunks 2 and 3).  A thread
    // mixes its accumulator row with the received one and the warp writes the bf16 rows out as
    // whole 128-byte lines through its private staging tile.
    auto received = [&](int q) {
        bool got = mbar_wait(&ctl->recv_bar[q], 0);
        got = __all_sync(0xffffffffu, got);
        if (!got && lane == 0) {
            *xfail = 1u;
            flag_status(p.status, OMNI_DEV_TIMEOUT | OMNI_DEV_ROLE_SOFTMAX);
        }
    };
    received(0);
    // weights of the two splits for this head row, final log-sum-exp
    const float other = reinterpret_cast<const float *>(recv)[row];
    const float mx = fmaxf(cm_lse, other);
    float total = -INFINITY, w_own = 0.f, w_other = 0.f;
    if (mx > -INFINITY) {
        total = mx + logf(exp2f((cm_lse - mx) * kLog2e) + exp2f((other - mx) * kLog2e));
        if (cm_lse > -INFINITY) w_own = exp2f((cm_lse - total) * kLog2e);
        if (other > -INFINITY) w_other = exp2f((other - total) * kLog2e);
    }
    if (cm_lse != cm_lse || other != other) total = w_other = NAN;        // a split whose sum is NaN, see row_lse
    if (s == 0 && sub == 0 && half == 0 && row < head_rows) p.lse[(size_t)b * p.heads + h0 + row] = total;
    // An accumulator row that carries no weight counts as zeros (that of an empty split was never written, that of a
    // fully masked one may hold anything); the partner sends exact zeros then.  The read itself is the whole warp's or
    // nobody's: rows of one warp differ in whether they carry weight (where one split's sum is below 2^-126 of the
    // other's, or a NaN or an infinity meets some of the heads), and a diverged tcgen05.ld does not return.
    const bool use_own = active && cm_inv != 0.f && w_own != 0.f;
    const float f_own = use_own ? w_own * cm_inv : 0.f, f_other = w_other;
    const int col = 128 * s + (sub == s ? 0 : 64);                        // first of this thread's 64 columns within its half
    uint8_t *buf = stages + (size_t)(sub * 4 + quarter) * kStageBytes;
    const int row0 = (quarter & 1) * 32;                                  // first head row of this warp
    uint8_t *gq = reinterpret_cast<uint8_t *>(p.out + ((size_t)b * p.heads + h0 + row0) * kDv + half * 256 + col);
    const int rows_here = max(0, min(32, head_rows - row0));
    const int first_chunk = sub == s ? 0 : 2;
    const uint8_t *theirs = recv + kLseBytes + first_chunk * kChunkBytes + (size_t)row * kChunkPitch + half * 128;
    uint4 *mine = reinterpret_cast<uint4 *>(buf + lane * kStagePitch);
    tc_fence_after();
#pragma unroll 1
    for (int c2 = 0; c2 < 2; ++c2) {
        received(first_chunk + c2);
        uint32_t ov[32];
        __syncwarp();
        if (active) {
            tc_ld32(tmem + lane_base + kColO + col + c2 * 32, ov);
            tc_wait_ld();
        }
#pragma unroll
        for (int j = 0; j < 32; ++j) ov[j] = use_own ? ov[j] : 0u;
        const uint4 *r4 = reinterpret_cast<const uint4 *>(theirs + c2 * kChunkBytes);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const uint4 ra = r4[2 * j], rb = r4[2 * j + 1];
            auto mix = [&](uint32_t own, uint32_t got) { return fmaf(f_own, __uint_as_float(own), f_other * __uint_as_float(got)); };
            uint4 w;
            w.x = pack_bf16(mix(ov[8 * j], ra.x), mix(ov[8 * j + 1], ra.y));
            w.y = pack_bf16(mix(ov[8 * j + 2], ra.z), mix(ov[8 * j + 3], ra.w));
            w.z = pack_bf16(mix(ov[8 * j + 4], rb.x), mix(ov[8 * j + 5], rb.y));
            w.w = pack_bf16(mix(ov[8 * j + 6], rb.z), mix(ov[8 * j + 7], rb.w));
            mine[c2 * 4 + j] = w;
        }
    }
    // this warp has seen its chunks land: once all eight have said so, the partner may leave
    __syncwarp();
    if (lane == 0) mbar_arrive_cluster(map_to_rank(smem_u32(&ctl->taken_bar), partner));
    __syncwarp();
    uint4 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k)
        v[k] = *reinterpret_cast<const uint4 *>(buf + (4 * k + (lane >> 3)) * kStagePitch + (lane & 7) * 16);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const int r = 4 * k + (lane >> 3);
        if (r < rows_here) *reinterpret_cast<uint4 *>(gq + (size_t)r * (kDv * 2) + (lane & 7) * 16) = v[k];
    }
}

// The unit of the pair-th pair.  Only the requests behind the first p.whole are split (whole = 0: all of
// them); b is their place in the order they are taken in, until c2_name_request.
__device__ __forceinline__ C2Unit c2_unit(const DecodeParams &p, int pair)
{
    C2Unit w;
    const int behind = pair - p.whole, tail = p.batch - p.whole;
    w.slot = -1;
    if (p.whole == 0) {
        w.splits = p.splits;
        w.s = pair % p.splits;
        w.b = pair / p.splits;
    } else if (behind < 0) {
        w.splits = 1;
        w.s = 0;
        w.b = pair;
    } else {
        w.splits = p.splits;
        w.s = behind / tail;             // first pieces first: they are all there is when nothing is cut
        w.slot = behind % tail;
        w.b = p.whole + w.slot;
    }
    return w;
}

// Names the request.  cut: see c2_rank_requests; without it the first piece of a request is all of it.
// One thread of the pair (`first`) tells the merge kernel which request, or that there is nothing to do.
__device__ __forceinline__ void c2_name_request(const DecodeParams &p, C2Unit &w, int b, bool cut, bool first)
{
    w.b = b;
    if (p.whole == 0) {
        w.slot = b;
    } else if (w.slot >= 0) {
        if (w.s == 0 && first) p.tail_request[w.slot] = cut ? b : -1;
        if (!cut) w.splits = w.s == 0 ? 1 : 0;
    }
}

// An empty split (no tokens): zeros and -inf in place of a result.  Called by warps `warp` of `warps`.
__device__ __forceinline__ void c2_store_empty(const DecodeParams &p, const C2Unit &w, int h0, int head_rows, int warp, int warps, int lane)
{
    if (w.splits == 0) return;
    for (int r = warp; r < head_rows; r += warps) {
        const int h = h0 + r;
        if (w.splits == 1) {
            uint4 *o = reinterpret_cast<uint4 *>(p.out + ((size_t)w.b * p.heads + h) * kDv);
            for (int i = lane; i < kDv * 2 / 16; i += 32) o[i] = make_uint4(0, 0, 0, 0);
            if (lane == 0) p.lse[(size_t)w.b * p.heads + h] = -INFINITY;
        } else {
            const size_t u = ((size_t)w.slot * p.splits + w.s) * p.heads + h;
            float4 *o = reinterpret_cast<float4 *>(p.part_out + u * kDv);
            for (int i = lane; i < kDv / 4; i += 32) o[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (lane == 0) p.part_lse[u] = -INFINITY;
        }
    }
    if (w.splits > 1 && p.counters != nullptr) __threadfence();
}

// Where there are more work units than pairs, the requests are taken longest first (ties by index).  Every CTA ranks
// the (at most 256) selection sizes itself: request j has rank #{i : n_i > n_j, or n_i = n_j and i < j}.
// lens: shared memory nobody uses yet (batch + 3 ints); order: the same, the request of every rank.  Called by all threads; the caller hands
// the memory to the producers' copies with c2_release_scratch once it has read `order`.  Returns, where only the
// requests behind the first wave are split (p.whole > 0), whether that pays.  Whole, the longest of them would
// start when the shortest of the first wave ends; only if it then ends after the longest of all, by more than
// a merge costs (12 units), do pieces help.
constexpr int kCutGain = 12 * kC2Tile;
__device__ __forceinline__ bool c2_rank_requests(const DecodeParams &p, int *lens, uint8_t *order)
{
    int *mark = lens + p.batch;                               // sizes of three ranks
    for (int j = threadIdx.x; j < p.batch; j += kC2Threads) lens[j] = load_selection(p, j).n;
    __syncthreads();
    for (int j = threadIdx.x; j < p.batch; j += kC2Threads) {
        const int nj = lens[j];
        int before = 0;
        for (int i = 0; i < p.batch; ++i) before += (lens[i] > nj) || (lens[i] == nj && i < j);
        order[before] = (uint8_t)j;
        if (before == 0) mark[0] = nj;
        if (before == p.whole - 1) mark[1] = nj;
        if (before == p.whole) mark[2] = nj;
    }
    __syncthreads();
    return p.whole == 0 || (int64_t)mark[1] + mark[2] > (int64_t)mark[0] + kCutGain;
}

// Shared memory that threads have written and read goes to the asynchronous copies: their writes must not pass the threads' accesses.
__device__ __forceinline__ void c2_release_scratch()
{
    fence_async_smem();
    __syncthreads();
}

// Epilogue of a work unit whose result leaves through global memory (final bf16 rows, or fp32
// partial rows of a split).  Each of the eight softmax warps owns 32 rows x 128 value columns
// of the accumulator: warp quarter q = warp % 4 serves head rows 32 * (q % 2) + lane and value
// columns 256 * (q / 2) + 128 * sub + [0, 128), sub = 1 for warps 8-11.  It moves them out in
// rounds of kRow bytes per row: tensor memory -> registers (scaled by 1 / lt) -> a warp-private
// staging tile of 32 x kRow bytes in shared memory (chunk c of row r at c ^ a hash of r, so neither the
// row-per-lane writes nor the reads conflict) -> global memory, 512 bytes per instruction.
// lt: the row's sum of weights; m_ref: its reference maximum (log2 units).
template <int kRow>
__device__ __forceinline__ void c2_store_result(const DecodeParams &p, uint8_t *stages, uint32_t tmem, int warp, int lane,
                                                const C2Unit &w, int h0, int head_rows, float lt, float m_ref)
{
    const int quarter = warp & 3;
    const int sub = warp >= 8 ? 1 : 0;
    const int row = (quarter & 1) * 32 + lane;
    const int part = (quarter >> 1) * 2 + sub;
    const uint32_t from = tmem + ((uint32_t)(quarter * 32) << 16) + kColO + 128 * sub;
    const float inv = lt > 0.f ? 1.f / lt : 0.f;
    const int h = h0 + row;
    const bool final_out = w.splits == 1;
    const size_t first = final_out ? (size_t)w.b * p.heads : ((size_t)w.slot * p.splits + w.s) * p.heads;
    const size_t u = first + h;
    constexpr int kChunks = kRow / 16, kRowsAtOnce = 32 / kChunks;       // rows of a store instruction
    const int widx = sub * 4 + ((warp - 2) & 3);                         // 0..7
    uint8_t *stage = stages + (size_t)widx * 32 * kRow;
    auto chunk_at = [&](int r, int c) { return stage + r * kRow + ((c ^ ((kChunks == 8 ? r : r >> 1) & (kChunks - 1))) << 4); };
    const uint32_t row_bytes = final_out ? kDv * 2 : kDv * 4;
    const int row0 = (quarter & 1) * 32;                                  // first head row of this warp
    // global address of (row0, this warp's first value column)
    const size_t u0 = first + h0 + row0;
    uint8_t *gbase = (final_out ? reinterpret_cast<uint8_t *>(p.out + u0 * kDv)
                                : reinterpret_cast<uint8_t *>(p.part_out + u0 * kDv)) + part * (row_bytes / 4);
    const int rows_here = max(0, min(32, head_rows - row0));              // rows of this warp that exist
    const int rounds = rows_here > 0 ? (int)(row_bytes / 4) / kRow : 0;
    constexpr int kCols16 = kRow / 2, kCols32 = kRow / 4;                 // columns of a round, bf16 and fp32
#pragma unroll 1
    for (int q = 0; q < rounds; ++q) {
        __syncwarp();
        if (final_out) {
#pragma unroll
            for (int c2 = 0; c2 < kCols16 / 32; ++c2) {
                uint32_t ov[32];
                tc_ld32(from + q * kCols16 + c2 * 32, ov);
                tc_wait_ld();
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint4 w;
                    w.x = pack_bf16(__uint_as_float(ov[8 * j]) * inv, __uint_as_float(ov[8 * j + 1]) * inv);
                    w.y = pack_bf16(__uint_as_float(ov[8 * j + 2]) * inv, __uint_as_float(ov[8 * j + 3]) * inv);
                    w.z = pack_bf16(__uint_as_float(ov[8 * j + 4]) * inv, __uint_as_float(ov[8 * j + 5]) * inv);
                    w.w = pack_bf16(__uint_as_float(ov[8 * j + 6]) * inv, __uint_as_float(ov[8 * j + 7]) * inv);
                    *reinterpret_cast<uint4 *>(chunk_at(lane, c2 * 4 + j)) = w;
                }
            }
        } else {
#pragma unroll
            for (int c2 = 0; c2 < kCols32 / 16; ++c2) {
                uint32_t ov[16];
                tc_ld16(from + q * kCols32 + c2 * 16, ov);
                tc_wait_ld();
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    *reinterpret_cast<uint4 *>(chunk_at(lane, c2 * 4 + j)) =
                        make_uint4(__float_as_uint(__uint_as_float(ov[4 * j]) * inv), __float_as_uint(__uint_as_float(ov[4 * j + 1]) * inv),
                                   __float_as_uint(__uint_as_float(ov[4 * j + 2]) * inv), __float_as_uint(__uint_as_float(ov[4 * j + 3]) * inv));
            }
        }
        __syncwarp();
        uint8_t *gq = gbase + q * kRow;
        uint4 v[kChunks];
#pragma unroll
        for (int k = 0; k < kChunks; ++k)
            v[k] = *reinterpret_cast<const uint4 *>(chunk_at(kRowsAtOnce * k + lane / kChunks, lane % kChunks));
#pragma unroll
        for (int k = 0; k < kChunks; ++k) {
            const int r = kRowsAtOnce * k + lane / kChunks;
            if (r < rows_here) *reinterpret_cast<uint4 *>(gq + (size_t)r * row_bytes + (lane % kChunks) * 16) = v[k];
        }
    }
    if (row < head_rows && part == 0) {
        const float lse = row_lse(lt, m_ref, !final_out);
        if (final_out)
            p.lse[u] = lse;
        else
            p.part_lse[u] = lse;
    }
}

// Zeroes 128 columns of the warp's tensor-memory lanes.  (The lanes come here from stores that not all of them took part in.)
__device__ __forceinline__ void c2_clear(uint32_t at)
{
    const uint32_t zero[32] = {};
    __syncwarp();
#pragma unroll
    for (int c = 0; c < 128; c += 32) tc_st32(at + c, zero);
    tc_wait_st();
}

// The kernel body in six instances.  kClusterMerge: the two splits of a request merged inside a cluster of two pairs;
// kMulti: several work units per pair, one after the other; neither: every other form (one unit per pair: no split, merge
// kernel, fused merge).  kRanges = false: the selection is the caller's index list; true: Eq. 2's two ranges (with or
// without a rolling cache).  Each instance carries only its own merge, epilogue and index code.
//
// Several units per pair (kMulti).  As many clusters as units are launched, and a pair that is nearly through with its unit takes
// the place of the next one that has not begun (cluster launch control), so that the units go out longest first to whichever pair
// becomes free, as they do where the hardware starts a cluster for each.  Dealt out in a fixed pattern instead, a pair with long units waits for nobody
// and is waited for.  One unit per pair / fixed pattern / this, us: 10 requests of 32 units and 246 of 4 60.1 / 55.6 / 45.3, 30 of 18 and 98 of 4
// 36.2 / 34.6 / 29.9, 256 sizes spread evenly in the logarithm over 1 to 32 72.9 / 64.1 / 60.7, 128 of them 37.4 / 40.2 / 38.5, 40 of 32 and 100 of 2
// 42.6 / 46.3 / 43.6, 128 of 18 57.9 / 56.7 / 56.1.  (The two that one unit per pair would do faster have few long
// units; this form has a longer start and end, and where few pairs run its main loop takes up to 2 % longer.)
// Every role goes through the units on its own; the barriers' phases, the score buffers and the
// mask ring go on by a running tile number.  So the loads and the first scores of a unit overlap the end of the one
// before: q and K follow as its last scores retire, V as its last P V does, and what remains between two units is
// the epilogue of one and the first softmax of the next.  An odd last tile's second unit is a gap that the barriers count.
// Launched only with the requests ranked, none cut at the end only (p.whole = 0) and no merge by the last CTA (p.counters null).
// (`unit` is set where the kernel begins although some instances set it anew: with that line further down the compiler makes
// 10 % more code of every instance and the merging ones run 1.4 times slower.)
template <bool kClusterMerge, bool kRanges, bool kMulti>
__device__ __forceinline__ void tc2_decode_body(const CUtensorMap &q_map, const CUtensorMap &kv_k_map,
                                                const CUtensorMap &kv_v_map, const CUtensorMap &kv_tile_map,
                                                const DecodeParams &p)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = smem_raw;
    if (smem_u32(smem_raw) & 1023u) {
        // the swizzled operand layouts need a 1024-byte aligned base; never seen otherwise, but say so
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (threadIdx.x == 0) flag_status(p.status, OMNI_DEV_TIMEOUT);
        return;
    }
    C2Control *ctl = reinterpret_cast<C2Control *>(smem + kC2SmemCtl);
    const uint32_t smem_base = smem_u32(smem);
    // A cluster is one pair, or (cluster merge) the two pairs that serve the two splits of a
    // request.  `rank` is the CTA's place within its pair; the pair's barriers live in `leader`.
    const uint32_t crank = cluster_rank();
    const uint32_t rank = crank & 1u, leader = crank & ~1u, peer = crank ^ 1u;
    const uint16_t pair_mask = (uint16_t)(3u << leader);

    const int pair = blockIdx.x >> 1;
    C2Unit unit = kClusterMerge ? C2Unit{(int)(blockIdx.x >> 2), (int)(crank >> 1), 2, 0} : c2_unit(p, pair);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // warp-uniform
    // The heads are dealt out evenly, so that neither CTA has more rows than it must to exchange and store.  The rows of q behind
    // them are zeros, see encode_q_map.
    const int rows = c2_rows(p.heads);
    const int h0 = (int)rank * rows;
    const int head_rows = min(rows, p.heads - h0);

    // ---- set-up: barriers and tensor memory (nothing here touches global memory, so with a
    // programmatic dependent launch it overlaps the tail of the kernel before this one) --------
    if (threadIdx.x == 0) {
        // arrivals per tile on the pair's score / weight barriers: one per softmax warp, in either CTA
        constexpr uint32_t kTileWarps = 16;
        for (int i = 0; i < kC2Groups; ++i) {
            mbar_init(&ctl->k_full[i], 1);
            mbar_init(&ctl->k_empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&ctl->v_full[i], 1);
            mbar_init(&ctl->pv_done[i], 1);
        }
        for (int i = 0; i < 3; ++i) {
            mbar_init(&ctl->s_full[i], 1);
            mbar_init(&ctl->s_empty[i], kTileWarps);
        }
        mbar_init(&ctl->p_full, kTileWarps);
        mbar_init(&ctl->xg_bar, 256);
        mbar_init(&ctl->x_bar, 256);
        mbar_init(&ctl->exit_bar, 2);
        if (kMulti) {
            mbar_init(&ctl->grant_bar, 1);
            for (int i = 1; i < kC2Rounds; ++i) {
                mbar_init(&ctl->work_full[i], 1);
                mbar_expect_tx(&ctl->work_full[i], sizeof(C2Work));
            }
        }
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
    // Programmatic dependent launch, both ways.  This grid may have been scheduled while the
    // kernel before it in the stream was still finishing: nothing in global memory is touched
    // until that kernel has completed and its writes are visible.  And the kernel after this one
    // may be scheduled as soon as resources allow; it waits in the same way before it reads.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    uint2 order_here = {0, 0};           // kMulti: the requests of ranks 8 lane, ... + 7, a byte each
    if (!kClusterMerge) {
        bool cut = true;
        int request = unit.b;
        if (p.longest_first) {
            uint8_t *order = smem + 4096;                     // (behind the sizes; shared memory nobody uses yet)
            cut = c2_rank_requests(p, reinterpret_cast<int *>(smem), order);
            request = order[unit.b];
            if (kMulti) order_here = reinterpret_cast<const uint2 *>(order)[lane];
            c2_release_scratch();
        }
        c2_name_request(p, unit, request, cut, rank == 0 && threadIdx.x == 0);
    }
    volatile uint32_t *abort_flag = &ctl->abort;
    // The work unit that a warp has in hand; take() moves on to the next.  Its tiles are numbered on from those of the one before,
    // [tile0, tile_end), and so are its 64-token units, two a tile, [2 tile0, unit_end); `begin` is the entry where unit 0 would begin.
    Selection selection;
    bool bad_len;
    int begin, end, units, tile0 = 0, tile_end = 0, unit_end;
    const int32_t *pt;
    auto take = [&](int round) {
        if (round == 0) {
            selection = load_selection(p, unit.b);
            split_range(!kClusterMerge && unit.splits == 0 ? 0 : selection.n, max(unit.splits, 1), unit.s, begin, end, kC2Tile);
        } else {
            if (!kMulti || round >= kC2Rounds) return false;
            if (!__all_sync(0xffffffffu, mbar_wait(&ctl->work_full[round], 0))) {
                if (lane == 0) {
                    flag_status(p.status, OMNI_DEV_TIMEOUT);
                    *abort_flag = 1;
                }
                return false;
            }
            const int4 w = *reinterpret_cast<const int4 *>(&ctl->work[round]);
            if (w.x < 0) return false;
            unit.b = unit.slot = w.x & 0xff;
            unit.s = w.x >> 8;
            begin = w.z;
            end = w.w;
            selection = make_selection(p, unit.b, w.y);
        }
        __builtin_assume(kRanges ? selection.list == nullptr : selection.list != nullptr);
        bad_len = selection.bad;
        units = (end - begin + kC2Tile - 1) / kC2Tile;
        if (kMulti) {
            tile0 = tile_end;
            begin -= 2 * tile0 * kC2Tile;
        }
        tile_end = tile0 + (units + 1) / 2;
        unit_end = 2 * tile0 + units;
        pt = p.page_table + (size_t)unit.b * p.max_pages;
        return true;
    };
    take(0);
    const bool active = kMulti || units > 0;
    if (!active && bad_len && threadIdx.x == 0 && crank == 0) flag_status(p.status, OMNI_DEV_BAD_INDEX);
    // an empty split (the same decision in both CTAs of the pair): zeros and -inf, no pipeline
    if (!kClusterMerge && !active) c2_store_empty(p, unit, h0, head_rows, warp, kC2Threads / 32, lane);

    const uint32_t tmem = ctl->tmem_base;

    // Index pipeline of the producers.  Lane l serves tokens l and l+32 of a unit.  The three
    // dependent steps (token position -> page id -> pool row) run in different loop iterations, so no
    // load is consumed in the iteration that issued it.  A lone warp takes 5-8 clocks an
    // instruction and a producer has about 1100 clocks a unit, so the common unit (64 consecutive pool
    // rows) is recognised with one vote and everything else is left to a slower path.
    struct TileIdx {
        int t0, t1;        // token positions (stage 1)
        int pg0, pg1;      // physical page ids, -1 if the position breaks the contract (stage 2)
    };
    // positions from here on (as unsigned numbers: negative ones too) break the contract
    const uint32_t t_limit = (uint32_t)min((int64_t)p.max_pages * kPage, (int64_t)1 << 31);
    const uint32_t page_limit = (uint32_t)p.num_pages;
    auto stage_tokens = [&](int unit, TileIdx &x) {
        const int first = begin + unit * kC2Tile;
        if (kRanges && first >= selection.vstart && first + kC2Tile <= end) {
            // a unit inside the recent range: 64 consecutive positions of one page, rolled once for all
            int t = selection.rs + (first - selection.vstart);
            if ((t & (kPage - 1)) == 0) {
                if (selection.ring_pages > 0) t = rolling_position(t, selection.sink_pages, selection.ring_pages);
                x.t0 = t + lane;
                x.t1 = t + lane + 32;
                return;
            }
        }
        const int j0 = first + lane, j1 = j0 + 32;
        x.t0 = j0 < end ? selection_at(selection, j0) : -1;
        x.t1 = j1 < end ? selection_at(selection, j1) : -1;
    };
    auto stage_pages = [&](TileIdx &x) {
        x.pg0 = (uint32_t)x.t0 < t_limit ? ldg_index(pt + (x.t0 >> 6), selection.keep) : -1;
        x.pg1 = (uint32_t)x.t1 < t_limit ? ldg_index(pt + (x.t1 >> 6), selection.keep) : -1;
    };
    static_assert(kPage == 64, "positions are split by shifts");
    // row_lo / row_hi: pool rows of tokens lane and lane+32 (a masked token repeats the row of the
    // unit's first valid token: real cache contents, multiplied by a weight of exactly zero);
    // contig: all 64 tokens valid and in consecutive rows.  box: first of 64 consecutive rows that hold every valid
    // token at its place, or -1.  Under ranges that includes the part of a page at either end of the recent
    // window: the K role may take such a box although it brings rows along that are not selected, since
    // their scores are masked whatever they hold (the V role may not: a weight of zero does not mask a
    // NaN).  128 requests with 1024 recent tokens on a rolling cache: 55.9 -> 54.0 us per step.
    auto stage_rows = [&](int unit, const TileIdx &x, int &row_lo, int &row_hi, uint64_t &mask, bool &contig, int &box,
                          bool &any_bad) {
        const bool ok0 = (uint32_t)x.pg0 < page_limit, ok1 = (uint32_t)x.pg1 < page_limit;
        row_lo = x.pg0 * kPage + (x.t0 & (kPage - 1));
        row_hi = x.pg1 * kPage + (x.t1 & (kPage - 1));
        const int base = __shfl_sync(0xffffffffu, row_lo, 0);
        contig = __all_sync(0xffffffffu, ok0 && ok1 && row_lo == base + lane && row_hi == base + 32 + lane);
        mask = ~0ull;
        box = contig ? base : -1;
        if (contig) return;
        const int j0 = begin + unit * kC2Tile + lane, j1 = j0 + 32;
        any_bad |= (j0 < end && !ok0 && !is_padding(selection, x.t0)) || (j1 < end && !ok1 && !is_padding(selection, x.t1));
        const uint32_t m0 = __ballot_sync(0xffffffffu, ok0), m1 = __ballot_sync(0xffffffffu, ok1);
        mask = (uint64_t)m0 | ((uint64_t)m1 << 32);
        int stand_in = 0;
        if (m0)
            stand_in = __shfl_sync(0xffffffffu, row_lo, __ffs(m0) - 1);
        else if (m1)
            stand_in = __shfl_sync(0xffffffffu, row_hi, __ffs(m1) - 1);
        if (kRanges) {
            const int first = stand_in - (m0 ? __ffs(m0) - 1 : 31 + __ffs(m1));
            const bool in_place = (!ok0 || row_lo == first + lane) && (!ok1 || row_hi == first + 32 + lane);
            if (__all_sync(0xffffffffu, in_place) && mask != 0ull && first >= 0 && (first & (kPage - 1)) == 0) box = first;
        }
        row_lo = ok0 ? row_lo : stand_in;
        row_hi = ok1 ? row_hi : stand_in;
    };

    // what the cluster merge needs from the softmax warps after the main loop
    float cm_lse = -INFINITY, cm_inv = 0.f;
    bool softmax_ok = true;              // false in a softmax warp whose main loop ran into a bounded wait

    if (!active) {
        // an empty split inside a merging cluster: no pipeline, but it takes part in the exchange
    } else if (warp == 0) {
        // =========================== K-role producer =====================================
        // This CTA's K rows are unit 2 t + rank of every tile t, refilled in three groups of three panels as the
        // score MMAs of the tile before retire.
        const uint32_t k_full_leader = map_to_rank(smem_u32(&ctl->k_full[0]), leader);
        // the columns of q that group g is scored against
        auto load_q = [&](int g) {
            const bool odd = p.heads & 1;
            tma_box5d_pair(smem_base + kC2SmemQ + g * kC2GroupBytes, &q_map, k_full_leader + 8 * g, odd ? h0 : 0,
                           g * kC2GroupPanels, odd ? 0 : (int)rank, unit.b);
        };
        bool any_bad = false, ok = true;
        int round = 0;
        do {
            any_bad |= bad_len;
            if (kMulti && units == 0) continue;
            if (tile0 == 0 && lane == 0) {
#pragma unroll
                for (int g = 0; g < kC2Groups; ++g) load_q(g);
            }
            // index pipeline, a tile (two units) at a time: page ids are one tile, positions two tiles ahead
            TileIdx x1[2], x2[2];
            int row_lo = 0, row_hi = 0, box = -1;    // of this CTA's unit of the tile about to be loaded
            bool boxed = false;
            // Resolves the rows of a tile and publishes the masks of its units (store + fence), BEFORE the next
            // index loads go out: a fence waits for the loads its thread has in flight, so a fence placed
            // after them put their whole latency in front of every refill.
            auto resolve_tile = [&](int tile, const TileIdx (&x)[2]) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    int lo, hi, first;
                    uint64_t mask;
                    bool whole;
                    stage_rows(2 * tile + h, x[h], lo, hi, mask, whole, first, any_bad);
                    if (lane == 0) ctl->valid_mask[(2 * tile + h) % kMaskRing] = mask;
                    if (h == (int)rank) {
                        row_lo = lo;
                        row_hi = hi;
                        // (the flag straight from a vote: the compiler has to see that it is the same in all lanes, or
                        // the steady state is 5 % slower)
                        box = kRanges ? first : lo;
                        boxed = kRanges ? __all_sync(0xffffffffu, first >= 0) != 0 : whole;
                    }
                }
                if (lane == 0) __threadfence_block();
            };
            {
                // the position loads of the first three tiles go out together, then the page-id loads that
                // depend on them: two cache misses in a row before the first copy, not four
                TileIdx x0[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    stage_tokens(2 * tile0 + h, x0[h]);
                    stage_tokens(2 * tile0 + 2 + h, x1[h]);
                    stage_tokens(2 * tile0 + 4 + h, x2[h]);
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    stage_pages(x0[h]);
                    stage_pages(x1[h]);
                }
                resolve_tile(tile0, x0);
            }
            // gathered groups whose bytes are not credited yet, first in first out: a single scattered group takes
            // about a memory latency, so all three are requested before the first is waited for
            int waiting = 0, oldest = 0;
            auto credit_oldest = [&]() {
                retire_gathered_stage(k_full_leader + 8 * oldest, kC2GroupBytes, --waiting, lane);
                oldest = oldest == kC2Groups - 1 ? 0 : oldest + 1;
            };
            const char *kv_bytes = reinterpret_cast<const char *>(p.kv);
            for (int tile = tile0; ok && tile < tile_end; ++tile) {
                // The last tile has a single unit when their number is odd: CTA 1 then leaves its half of the K
                // rows as it is (the scores of those tokens are masked) and credits the bytes all the same.  Every
                // tile's scores thus wait for this warp of either CTA: for the masks it has written by then, and
                // because k_empty must not get two phases ahead of a wait below, whose parity would then match again and
                // the wait run out.
                const bool mine = 2 * tile + (int)rank < unit_end;
                const uint32_t bytes = (tile == tile0 ? 4 : 2) * kC2GroupBytes;
#pragma unroll 1
                for (int g = 0; g < kC2Groups; ++g) {
                    if (tile > 0) {
                        // nothing to do until the group is free: credit what has landed meanwhile
                        while (waiting > 0 && !__all_sync(0xffffffffu, mbar_test(&ctl->k_empty[g], (tile - 1) & 1))) credit_oldest();
                        ok = __all_sync(0xffffffffu, mbar_wait(&ctl->k_empty[g], (tile - 1) & 1));
                        if (!ok) break;
                    }
                    if (lane == 0 && rank == 0) mbar_expect_tx(&ctl->k_full[g], bytes);
                    if (kMulti && tile == tile0 && tile0 > 0 && lane == 0) load_q(g);  // (the scores that read the q before have retired)
                    if (!mine) {
                        if (lane == 0) credit_bytes(k_full_leader + 8 * g, kC2GroupBytes);
                        continue;
                    }
                    const uint32_t dst = smem_base + kC2SmemK + g * kC2GroupBytes;
                    if (boxed) {
                        if (lane == 0) tma_box3d_pair(dst, &kv_k_map, k_full_leader + 8 * g, box, g * kC2GroupPanels);
                    } else {
                        gather_rows<kC2GroupPanels>(dst, kv_bytes + g * (kC2GroupPanels * 128), row_lo, row_hi, lane);
                        if (waiting++ == 0) oldest = g;
                    }
                }
                if (lane == 0) *const_cast<volatile int32_t *>(&ctl->k_progress) = tile + 1;
                // (before the index work: that fits into the time the score MMAs then take)
                while (waiting > 0) credit_oldest();
                ok = ok && (*abort_flag == 0);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                // advance the index pipeline: rows of the next tile, page ids of the one after, positions of the third
                if (tile + 1 < tile_end) resolve_tile(tile + 1, x1);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    x1[h] = x2[h];
                    stage_pages(x1[h]);
                    stage_tokens(2 * tile + 6 + h, x2[h]);
                }
            }
        } while (ok && take(++round));
        if (lane == 0) *const_cast<volatile int32_t *>(&ctl->k_progress) = 0x7fffffff;
        if (!ok && lane == 0) {
            flag_status(p.status, OMNI_DEV_TIMEOUT | OMNI_DEV_ROLE_PRODUCER_K);
            *abort_flag = 1;
        }
        if (__any_sync(0xffffffffu, any_bad) && lane == 0 && rank == 0) flag_status(p.status, OMNI_DEV_BAD_INDEX);
    } else if (warp == 6) {
        // =========================== V-role producer =====================================
        // This CTA's V columns are [256*rank, 256*rank+256) = panels [4*rank, 4*rank+4) of all 64 tokens.
        bool any_bad = false, ok = true;
        int round = 0;
        int pending = -1;                    // stage of a gathered unit whose bytes are not credited yet
        const char *kv_bytes = reinterpret_cast<const char *>(p.kv);
        do {
            TileIdx x1, x2;
            int row_lo, row_hi, box_unused;
            uint64_t mask_unused;
            bool contig;
            {
                // the position loads of the first three units go out together, then the two page-id
                // loads that depend on them: two cache misses in a row before the first copy, not four
                TileIdx x0;
                const int first = 2 * tile0;
                stage_tokens(first, x0);
                stage_tokens(first + 1, x1);
                stage_tokens(first + 2, x2);
                stage_pages(x0);
                stage_pages(x1);
                stage_rows(first, x0, row_lo, row_hi, mask_unused, contig, box_unused, any_bad);
            }
            for (int i = 2 * tile0; ok && i < (kMulti ? 2 * tile_end : unit_end); ++i) {
                const int st = i & 1;
                if (i >= 2) {
                    if (pending >= 0 && !__all_sync(0xffffffffu, mbar_test(&ctl->pv_done[st], ((i >> 1) - 1) & 1))) {
                        retire_gathered_stage(map_to_rank(smem_u32(&ctl->v_full[pending]), leader), kC2VBytes, 0, lane);
                        pending = -1;
                    }
                    ok = mbar_wait(&ctl->pv_done[st], ((i >> 1) - 1) & 1);
                }
                ok = __all_sync(0xffffffffu, ok) && (*abort_flag == 0);
                if (!ok) break;
                if (kMulti && i >= unit_end) {
                    // an odd last tile has no second unit: only the phases of its barriers go on
                    if (pending >= 0) retire_gathered_stage(map_to_rank(smem_u32(&ctl->v_full[pending]), leader), kC2VBytes, 0, lane);
                    pending = -1;
                    if (lane == 0 && rank == 0) mbar_arrive(&ctl->v_full[st]);
                    break;
                }
                const uint32_t bar = map_to_rank(smem_u32(&ctl->v_full[st]), leader);
                if (lane == 0 && rank == 0) mbar_expect_tx(&ctl->v_full[st], 2 * kC2VBytes);
                __syncwarp();
                const uint32_t dst = smem_base + kC2SmemV + st * kC2VBytes;
                bool gathered = false;
                if (contig) {
                    if (lane == 0) tma_box3d_pair(dst, &kv_v_map, bar, row_lo, 4 * (int)rank);
                } else {
                    // scattered rows: the four panels of this CTA's value columns, 64 tokens
                    gathered = true;
                    gather_rows<4>(dst, kv_bytes + (int)rank * 512, row_lo, row_hi, lane);
                }
                if (pending >= 0) {
                    retire_gathered_stage(map_to_rank(smem_u32(&ctl->v_full[pending]), leader), kC2VBytes, gathered ? 1 : 0, lane);
                    pending = -1;
                }
                if (gathered) {
                    pending = st;
                    // the next stage is still in use: credit this one before the index work
                    if (i >= 1 && !__all_sync(0xffffffffu, mbar_test(&ctl->pv_done[st ^ 1], (((i + 1) >> 1) - 1) & 1))) {
                        retire_gathered_stage(map_to_rank(smem_u32(&ctl->v_full[pending]), leader), kC2VBytes, 0, lane);
                        pending = -1;
                    }
                }
                if (i + 1 < unit_end) stage_rows(i + 1, x1, row_lo, row_hi, mask_unused, contig, box_unused, any_bad);
                x1 = x2;
                stage_pages(x1);
                stage_tokens(i + 3, x2);
            }
        } while (ok && take(++round));
        if (pending >= 0) retire_gathered_stage(map_to_rank(smem_u32(&ctl->v_full[pending]), leader), kC2VBytes, 0, lane);
        if (!ok && lane == 0) {
            flag_status(p.status, OMNI_DEV_TIMEOUT | OMNI_DEV_ROLE_PRODUCER_V);
            *abort_flag = 1;
        }
    } else if (warp == 7) {
        // =========================== L2 prefetcher =======================================
        // A hint only.  CTA r pulls the units that are ITS K rows into L2 ahead of their loads: a whole page in
        // order (first position page-aligned, last position 63 further) by one tensor prefetch, anything
        // else row by row.  Lane l looks at the ends of unit r + 2 l, ... of a batch of 32 in parallel.
        bool ok = true;
        int round = 0;
        // Several units per pair: CTA 0 asks for the next one and hands it to both CTAs, some 3 us before the pair is free; the answer takes
        // 0.3 us.  Where the unit in hand ends in a whole page it asks once the K loads of the last tile have been requested (the earlier, the less
        // is known of who is free first: a tile earlier 256 x 8 units take 60.9 us, not 58.2), behind scattered rows at once, two
        // tiles earlier, since the next unit's are late without a prefetch (100 x 11 after a selection 57.1 -> 55.7).
        auto deal = [&](int round) {
            if (lane == 0) {
                mbar_expect_tx(&ctl->grant_bar, sizeof(ctl->grant));
                try_cancel_cluster(&ctl->grant, &ctl->grant_bar);
            }
            if (!__all_sync(0xffffffffu, mbar_wait(&ctl->grant_bar, (round - 1) & 1))) {
                if (lane == 0) {
                    flag_status(p.status, OMNI_DEV_TIMEOUT);
                    *abort_flag = 1;
                }
                return;
            }
            const int first = __shfl_sync(0xffffffffu, cancelled_cluster(&ctl->grant), 0);
            fence_async_smem();                               // (the next answer is written by the asynchronous proxy)
            int4 w = {-1, 0, 0, 0};
            if (first >= 0) {
                const C2Unit next = c2_unit(p, first >> 1);
                const uint32_t word = __shfl_sync(0xffffffffu, (next.b & 4) ? order_here.y : order_here.x, next.b >> 3);
                const int b = (int)(word >> (8 * (next.b & 3))) & 0xff;
                w.x = b | (next.s << 8);
                w.y = load_length(p, b);
                split_range(make_selection(p, b, w.y).n, p.splits, next.s, w.z, w.w, kC2Tile);
            }
            if (lane < 2) st_async16(map_to_rank(smem_u32(&ctl->work[round]), lane), map_to_rank(smem_u32(&ctl->work_full[round]), lane), w);
        };
        do {
            const int all_upto = (int)(gridDim.x >> 1) < kPrefetchManyPairs ? kPrefetchLongUnits : kPrefetchAllUnits;
            bool paged = false;                               // the last of these units is a whole page
            const int pages_upto = kClusterMerge || units < all_upto ? unit_end : kPrefetchFirstUnits;
            for (int t0 = 2 * tile0 + (int)rank; ok && t0 < unit_end; t0 += 64) {
                const int t = t0 + 2 * lane;
                const int j0 = begin + t * kC2Tile;
                int row = -1;
                if (t < unit_end && j0 + kC2Tile <= end) {
                    const int first = selection_at(selection, j0), last = selection_at(selection, j0 + kC2Tile - 1);
                    if (first >= 0 && first % kPage == 0 && last == first + kC2Tile - 1 && first / kPage < p.max_pages) {
                        const int pg = ldg_index(pt + first / kPage, selection.keep);
                        if (pg >= 0 && (int64_t)pg < p.num_pages) row = pg * kPage;
                    }
                }
                __syncwarp();
                TileIdx x = {-1, -1, -1, -1};    // of a unit that is not a whole page
                for (int k = 0; ok && k < 32 && t0 + 2 * k < unit_end; ++k) {
                    const int i = t0 + 2 * k, tile = i >> 1;
                    const bool page = __shfl_sync(0xffffffffu, row, k) >= 0;
                    if (kMulti) paged = page;
                    if (page && i >= pages_upto) continue;
                    if (!page) {
                        stage_tokens(i, x);
                        stage_pages(x);
                    }
                    // a page is prefetched once the K loads of the tile before have been requested (a monotonic
                    // counter, polled with a bounded number of naps)
                    const volatile int32_t *progress = &ctl->k_progress;
                    for (int naps = 0; *progress < tile - (page ? 0 : kScatterAhead) && *abort_flag == 0; ++naps) {
                        if (naps > (1 << 22)) {
                            ok = false;
                            break;
                        }
                        __nanosleep(200);
                    }
                    ok = ok && (*abort_flag == 0);
                    ok = __all_sync(0xffffffffu, ok);
                    if (ok && page && lane == k)
                        asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(&kv_tile_map),
                                     "r"(0), "r"(row), "r"(0)
                                     : "memory");
                    if (ok && !page && *progress <= tile) {      // (not once the unit's own loads are out)
                        if ((uint32_t)x.pg0 < page_limit) prefetch_row(p.kv, x.pg0 * kPage + (x.t0 & (kPage - 1)));
                        if ((uint32_t)x.pg1 < page_limit) prefetch_row(p.kv, x.pg1 * kPage + (x.t1 & (kPage - 1)));
                    }
                    __syncwarp();
                }
            }
            if (kMulti && rank == 0 && ok && round + 1 < kC2Rounds) {
                const volatile int32_t *progress = &ctl->k_progress;
                for (int naps = 0; paged && *progress < tile_end && *abort_flag == 0 && naps < (1 << 22); ++naps) __nanosleep(100);
                __syncwarp();
                deal(round + 1);
            }
        } while (ok && take(++round));
    } else if (warp == 1) {
        // =========================== MMA issuer (CTA 0 only) =============================
        if (rank == 0) {
            constexpr uint32_t idesc_qk = instr_desc(128, 2 * kC2Tile, 0);
            constexpr uint32_t idesc_pv = instr_desc(128, 256, 1);
            const uint64_t q_desc = smem_desc(smem_base + kC2SmemQ, 16, 1024);
            const uint64_t k_desc = smem_desc(smem_base + kC2SmemK, 16, 1024);
            const uint64_t p_desc = smem_desc(smem_base + kC2SmemP, 16, 1024);
            const uint64_t v_desc = smem_desc(smem_base + kC2SmemV, kPanelBytes, 1024);
            const uint32_t q_lo = (uint32_t)q_desc, k_lo = (uint32_t)k_desc, p_lo = (uint32_t)p_desc, v_lo = (uint32_t)v_desc;
            const uint32_t kmaj_hi = (uint32_t)(q_desc >> 32), v_hi = (uint32_t)(v_desc >> 32);
            // Values that steer the loop are broadcast from lane 0 so that the compiler can see
            // they are warp-uniform and keep the descriptor arithmetic on the uniform datapath;
            // with thread-dependent control flow every MMA costs ~70 clocks to issue instead of ~25.
            const int tiles_u = __shfl_sync(0xffffffffu, tile_end, 0), units_u = __shfl_sync(0xffffffffu, units, 0);
            const uint32_t tmem_u = __shfl_sync(0xffffffffu, tmem, 0);
            // One copy of each issue routine: group, stage and buffer enter as warp-uniform run-time values
            // (every operand of an MMA is then a uniform base plus a compile-time offset), which
            // keeps the issuing warp's code a few kilobytes instead of several tens (an issue loop
            // unrolled over the buffer parities ran config-2-sized launches 5 % slower, token-level
            // ones 8 %: a launch starts with cold instruction caches and this loop is its critical path).
            auto issue_qk = [&](int g, int sbuf) {
                const uint32_t d = tmem_u + kC2ColS + 64 * sbuf, at = (uint32_t)((g * kC2GroupBytes) >> 4);
                tc_mma_pair_elect(d, q_lo + at, kmaj_hi, k_lo + at, kmaj_hi, idesc_qk, g != 0 ? 1u : 0u);
#pragma unroll
                for (int kk = 1; kk < 4 * kC2GroupPanels; ++kk) {
                    const uint32_t off = at + (((kk >> 2) * kPanelBytes + (kk & 3) * 32) >> 4);
                    tc_mma_pair_elect<true>(d, q_lo + off, kmaj_hi, k_lo + off, kmaj_hi, idesc_qk);
                }
                tc_commit_pair_elect(&ctl->k_empty[g], pair_mask);
                if (g == kC2Groups - 1) tc_commit_pair_elect(&ctl->s_full[sbuf], pair_mask);
            };
            auto issue_pv = [&](int par, bool first) {
                const uint32_t a = p_lo + ((par * kPanelBytes) >> 4);
                const uint32_t bd = v_lo + ((par * kC2VBytes) >> 4);
                tc_mma_pair_elect(tmem_u + kColO, a, kmaj_hi, bd, v_hi, idesc_pv, first ? 0u : 1u);
                tc_mma_pair_elect(tmem_u + kColO + 128, a, kmaj_hi, bd + ((2 * kPanelBytes) >> 4), v_hi, idesc_pv, first ? 0u : 1u);
#pragma unroll
                for (int k = 1; k < 4; ++k) {
                    const uint32_t ak = a + ((k * 32) >> 4), bk = bd + ((k * 2048) >> 4);
                    tc_mma_pair_elect<true>(tmem_u + kColO, ak, kmaj_hi, bk, v_hi, idesc_pv);
                    tc_mma_pair_elect<true>(tmem_u + kColO + 128, ak, kmaj_hi, bk + ((2 * kPanelBytes) >> 4), v_hi, idesc_pv);
                }
            };
            // Whatever is ready goes next, scores first (P V first was 1 to 5 % slower): group g of tile t once its
            // K panels have landed and (first group) the score buffer t % 3 is free; P V of unit u once the
            // weights of its tile are written and its V rows have landed.
            // u counts steps of P V, two a tile.  Several units per pair: scores run ahead of P V across the units, and every step but the
            // first adds to O, which the softmax warps clear between two units.
            bool ok = true;
            int t = 0, g = 0, u = 0, sbuf = 0, sph = 1;     // sph: parity of the wait on s_empty (the first use passes at once)
            int round = 0, stop = units_u;                  // stop: the step behind the unit that P V is at, a gap if that is odd
            long long start = 0;
            uint32_t idle = 0;
            do {
                while (ok && u < stop) {
                    const bool qk = (kMulti || t < tiles_u) && mbar_test(&ctl->k_full[g], t & 1) && (g > 0 || mbar_test(&ctl->s_empty[sbuf], sph));
                    if (__all_sync(0xffffffffu, qk)) {
                        tc_fence_after();
                        issue_qk(g, sbuf);
                        if (++g == kC2Groups) {
                            g = 0;
                            ++t;
                            if (++sbuf == 3) {
                                sbuf = 0;
                                sph ^= 1;
                            }
                        }
                        idle = 0;
                        continue;
                    }
                    const bool pv = mbar_test(&ctl->p_full, (u >> 1) & 1) && mbar_test(&ctl->v_full[u & 1], (u >> 1) & 1);
                    if (__all_sync(0xffffffffu, pv)) {
                        tc_fence_after();
                        issue_pv(u & 1, u == 0);
                        tc_commit_pair_elect(&ctl->pv_done[u & 1], pair_mask);
                        ++u;
                        idle = 0;
                        continue;
                    }
                    // bounded: the clock is read now and then while nothing is ready
                    if ((++idle & 63u) == 0u) {
                        const long long now = __shfl_sync(0xffffffffu, clock64(), 0);
                        if (idle == 64u)
                            start = now;
                        else
                            ok = now - start <= kWaitCycles;
                        ok = ok && __shfl_sync(0xffffffffu, *abort_flag, 0) == 0u;
                    }
                }
                if (!kMulti || !ok) break;
                if (u & 1) {
                    // the gap: its barriers' phases only
                    ok = __all_sync(0xffffffffu, mbar_wait(&ctl->v_full[1], (u >> 1) & 1));
                    if (!ok) break;
                    tc_commit_pair_elect(&ctl->pv_done[1], pair_mask);
                    ++u;
                }
                if (!take(++round)) break;
                stop = u + __shfl_sync(0xffffffffu, units, 0);
            } while (true);
            if (!ok && lane == 0) {
                flag_status(p.status, OMNI_DEV_TIMEOUT | OMNI_DEV_ROLE_MMA);
                *abort_flag = 1;
            }
        }
        __syncwarp();
    } else {
        // =========================== softmax + epilogue =================================
        // Eight warps (2-5 and 8-11): two per tensor-memory lane quarter (sub = 0 for warps 2-5, 1 for warps
        // 8-11).  A thread serves head row L % 64 (L = its
        // tensor-memory lane); in the epilogue it owns value columns 256 * (L / 64) + 128 * sub +
        // [0, 128) of that row.
        const int quarter = warp & 3;
        const int sub = warp >= 8 ? 1 : 0;
        const int row = (quarter & 1) * 32 + lane;          // head row within this CTA
        const int half = quarter >> 1;                      // token half of S / column half of O
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        const uint32_t s_empty_leader = map_to_rank(smem_u32(&ctl->s_empty[0]), leader);   // [1], [2] follow at +8, +16
        const uint32_t p_full_leader = map_to_rank(smem_u32(&ctl->p_full), leader);
        bool ok = true;
        int round = 0, sbuf = 0, sph = 0;        // sph: parity of the wait on s_full
        // Every tile is worked on by all eight warps: a thread serves head row `row` and 32 of the 128 tokens,
        // [64 half + 32 sub, + 32), and the four threads of a row meet over its maximum through shared
        // memory.  (Two groups of four warps that take the tiles in turn, 64 tokens a thread, overlap one
        // tile's exchange with the other's exponentials, but the weights of a tile are then ready about 450
        // clocks later, which every launch pays at its first and at its last tile: one request of 128
        // units 16.8 us that way, 16.2 this way.)
        const int tq = half * 2 + sub;                     // quarter of the tile's tokens
        do {
            if (kMulti && units == 0) {
                // an empty split (the same decision in both CTAs of the pair): zeros and -inf, no pipeline
                c2_store_empty(p, unit, h0, head_rows, warp < 8 ? warp - 2 : warp - 4, 8, lane);
                continue;
            }
            float m_ref = -INFINITY, l = 0.f;
            for (int i = tile0; i < tile_end; ++i) {
                ok = mbar_wait(&ctl->s_full[sbuf], sph);
                if (!__all_sync(0xffffffffu, ok)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                uint32_t sv[32];
                tc_ld32(tmem + lane_base + kC2ColS + 64 * sbuf + 32 * sub, sv);
                tc_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(s_empty_leader + 8 * sbuf);
                if (++sbuf == 3) {
                    sbuf = 0;
                    sph ^= 1;
                }
                const uint32_t valid = (uint32_t)(ctl->valid_mask[(2 * i + half) % kMaskRing] >> (32 * sub));
                // x * xs is the scaled score of a token.  Under a positive scale x is the raw score: the
                // maximum is taken on them and the scale rides on the fused multiply-add in front of the
                // exponential, one instruction less per token.
                float xs = p.scale_log2;
                if (!(p.scale_log2 > 0.f)) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) sv[j] = __float_as_uint(__uint_as_float(sv[j]) * p.scale_log2);
                    xs = 1.f;
                }
                if (valid != 0xffffffffu) {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (!((valid >> j) & 1u)) sv[j] = __float_as_uint(-INFINITY);
                }
                float mt = fmaxf(max32([&](int j) { return __uint_as_float(sv[j]); }), -INFINITY) * xs;
                float *xg = &ctl->xchg[i & 1][0][row];
                // (the row sums of the unit before went through the same slots: everybody has read them)
                if (kMulti && i == tile0 && tile0 > 0) ok = mbar_wait(&ctl->x_bar, 1);
                xg[tq * 64] = mt;
                mbar_arrive(&ctl->xg_bar);
                ok = mbar_wait(&ctl->xg_bar, i & 1) && ok;
                if (!__all_sync(0xffffffffu, ok)) {
                    ok = false;
                    break;
                }
                mt = fmaxf(fmaxf(xg[0], xg[64]), fmaxf(xg[128], xg[192]));
                // move the reference only when the tile maximum leaves the window above it
                float factor = 1.f;
                bool moved = false;
                if (mt > m_ref + kRescaleThreshold || (m_ref == -INFINITY && mt > -INFINITY)) {
                    factor = m_ref == -INFINITY ? 0.f : exp2f(m_ref - mt);
                    m_ref = mt;
                    moved = true;
                }
                const float mr = (m_ref == -INFINITY) ? 0.f : m_ref;
                const f32x2 xs2 = pack2(xs, xs), mr2 = pack2(-mr, -mr);
                f32x2 sums = pack2(0.f, 0.f);
                uint32_t pk[16];
#pragma unroll
                for (int j = 0; j < 32; j += 2) {
                    const float2 y = unpack2(fma2(pack2(__uint_as_float(sv[j]), __uint_as_float(sv[j + 1])), xs2, mr2));
                    const float e0 = fast_exp2(y.x), e1 = fast_exp2(y.y);
                    sums = add2(sums, pack2(e0, e1));
                    pk[j >> 1] = pack_bf16(e0, e1);
                }
                const float2 sum = unpack2(sums);
                l = l * factor + (sum.x + sum.y);
                // P and O are free once P V of the tile before (its second unit: only the last tile can have a
                // single one) retired
                if (i > tile0) {
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
                // half a P row of unit 2 i + half: 32 tokens x bf16 = four 16-byte chunks, chunk c stored at c ^ (row % 8)
                uint8_t *p_row = smem + kC2SmemP + half * kPanelBytes + row * 128;
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    *reinterpret_cast<uint4 *>(p_row + (((sub * 4 + c) ^ (row & 7)) << 4)) =
                        make_uint4(pk[4 * c], pk[4 * c + 1], pk[4 * c + 2], pk[4 * c + 3]);
                fence_async_smem();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(p_full_leader);
            }
            // The row sums are final as soon as the last tile's weights are written, before its P V has
            // run: their exchange and what follows from them overlap that last P V.
            // Their slots: the parity that the last tile did not use.  Every thread has passed the exchange barrier of
            // that tile, which it reached only after reading the slots of the tile before.
            float lt = 0.f;
            if (ok) {
                float *sums = &ctl->xchg[tile_end & 1][0][row];
                sums[tq * 64] = l;
                mbar_arrive(&ctl->x_bar);
                ok = mbar_wait(&ctl->x_bar, 0);
                ok = __all_sync(0xffffffffu, ok);
                lt = (sums[0] + sums[64]) + (sums[128] + sums[192]);
                if (kMulti) mbar_arrive(&ctl->x_bar);
            }
            if (ok) {
                cm_inv = lt > 0.f ? 1.f / lt : 0.f;
                cm_lse = row_lse(lt, m_ref, true);
                // now the last P V
                const int last = kMulti ? 2 * tile_end - 1 : units - 1;
                ok = mbar_wait(&ctl->pv_done[last & 1], (last >> 1) & 1);
                ok = __all_sync(0xffffffffu, ok);
            }
            if (kClusterMerge && ok) {
                // every MMA of the pair has retired and every copy has landed: the partner in the other
                // split may overwrite this CTA's operand tiles from now on.  The result stays in tensor
                // memory: the exchange after the main loop normalises it and hands half of it to the CTA
                // that serves the same heads in the other split.
                if (warp == 2 && lane == 0) mbar_arrive_cluster(map_to_rank(smem_u32(&ctl->ready_bar), crank ^ 2u));
            } else if (!kClusterMerge && ok) {
                tc_fence_after();
                // With more units to come only the P buffer is free to stage in: the next tile's weights are written once all eight warps
                // are through.
                if (kMulti) {
                    c2_store_result<64>(p, smem + kC2SmemP, tmem, warp, lane, unit, h0, head_rows, lt, m_ref);
                    c2_clear(tmem + lane_base + kColO + 128 * sub);
                } else {
                    c2_store_result<128>(p, smem, tmem, warp, lane, unit, h0, head_rows, lt, m_ref);
                }
                tc_fence_before();
                // with the in-kernel merge the partial results must be visible before this CTA is counted
                if (!kMulti && unit.splits != 1 && p.counters != nullptr) __threadfence();
            }
        } while (ok && take(++round));
        if (!ok && lane == 0) {
            flag_status(p.status, OMNI_DEV_TIMEOUT | OMNI_DEV_ROLE_SOFTMAX);
            *abort_flag = 1;
        }
        softmax_ok = ok;
    }

    // ---- tear-down: nobody leaves while the other CTA may still touch this one's memory --
    if (*abort_flag) nap_after_abort();
    if (kClusterMerge) cluster_merge_exchange(p, ctl, smem, tmem, unit.b, unit.s, crank, h0, rows, head_rows, active, softmax_ok, cm_lse, cm_inv);
    tc_fence_before();
    __syncthreads();
    // Tensor memory was allocated for the pair, so it is released only when both CTAs are done
    // with it.  The rendezvous is an mbarrier in each CTA that both CTAs arrive on (the hardware
    // cluster barrier took 6-9 us at this point); warp 1 stays until the peer's arrival has
    // landed, which also keeps this CTA's shared memory alive for it.
    if (warp == 1) {
        // the bulk copies sent to the partner read this CTA's shared memory: it has to stay until they are in
        // (a cluster barrier here would wait for the partner's last stores too)
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
    // ---- split merge by whichever CTA finishes a (request, head half) last ---------------
    if (!kClusterMerge && !kMulti && p.splits > 1 && p.counters != nullptr)
        merge_if_last(p, unit.b, (int)rank, 2, h0, head_rows, reinterpret_cast<float *>(smem), &ctl->merge_flag);
}

#define OMNI_C2_KERNEL(name, cluster_merge, ranges, multi)                                                                  \
    __global__ void __launch_bounds__(kC2Threads, 1)                                                                   \
    name(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap kv_k_map,                      \
         const __grid_constant__ CUtensorMap kv_v_map, const __grid_constant__ CUtensorMap kv_tile_map, DecodeParams p) \
    {                                                                                                                  \
        tc2_decode_body<cluster_merge, ranges, multi>(q_map, kv_k_map, kv_v_map, kv_tile_map, p);                             \
    }
OMNI_C2_KERNEL(tc2_decode_kernel, false, false, false)
OMNI_C2_KERNEL(tc2_decode_cm_kernel, true, false, false)
OMNI_C2_KERNEL(tc2_decode_multi_kernel, false, false, true)
OMNI_C2_KERNEL(tc2_decode_rng_kernel, false, true, false)
OMNI_C2_KERNEL(tc2_decode_cm_rng_kernel, true, true, false)
OMNI_C2_KERNEL(tc2_decode_multi_rng_kernel, false, true, true)
#undef OMNI_C2_KERNEL

using C2KernelFn = void (*)(CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, DecodeParams);
// form: 0 one work unit per pair, 1 two splits merged inside a cluster, 2 several work units per pair
inline C2KernelFn tc2_kernel_for(int form, bool ranges)
{
    static const C2KernelFn table[3][2] = {{tc2_decode_kernel, tc2_decode_rng_kernel},
                                           {tc2_decode_cm_kernel, tc2_decode_cm_rng_kernel},
                                           {tc2_decode_multi_kernel, tc2_decode_multi_rng_kernel}};
    return table[form][ranges ? 1 : 0];
}

// Clusters of two pairs (cluster merge) that can be resident at once on the current device, or 0.
inline int tc2_max_merge_clusters()
{
    static int cached[64];
    static bool known[64] = {};
    static std::mutex mu;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> lock(mu);
    if (!known[dev]) {
        int n = 0;
        if (cudaFuncSetAttribute(tc2_decode_cm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kC2SmemBytes) == cudaSuccess) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(4 * 64);
            cfg.blockDim = dim3(kC2Threads);
            cfg.dynamicSmemBytes = kC2SmemBytes;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = 4;
            attr[0].val.clusterDim.y = 1;
            attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            if (cudaOccupancyMaxActiveClusters(&n, tc2_decode_cm_kernel, &cfg) != cudaSuccess) {
                cudaGetLastError();
                n = 0;
            }
        }
        cached[dev] = n;
        known[dev] = true;
    }
    return cached[dev];
}

inline bool tc2_prepare_device()
{
    static bool attr_set[64] = {};
    static std::mutex mu;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    std::lock_guard<std::mutex> lock(mu);
    if (!attr_set[dev]) {
        for (int k = 0; k < 6; ++k)
            if (cudaFuncSetAttribute(tc2_kernel_for(k >> 1, (k & 1) != 0), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     kC2SmemBytes) != cudaSuccess)
                return false;
        attr_set[dev] = true;
    }
    return true;
}

// q [requests * heads, 576] as the pair kernel loads it: {64 columns, head rows, 9 panels, CTA of the pair, request}.  A CTA's rows
// end where its half of the heads does, so that a box of 64 rows brings zeros for the others: rows that hold other
// heads' values would be multiplied for nothing, and long launches are held back by power (64 requests x 33 units of
// 64 heads 46.1 us with zeros, 48.7 with the neighbours' rows).  An odd number of heads does not halve: there the rows
// are all heads of the request, and the first CTA's box brings some that are the second's.
inline bool encode_q_map(CUtensorMap *map, const void *base, uint64_t qrows, uint32_t heads, uint32_t panels)
{
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const bool odd = heads & 1;
    const cuuint64_t row = (cuuint64_t)kDqk * 2, rows = odd ? heads : heads / 2;
    const cuuint64_t dims[5] = {64, rows, (cuuint64_t)kPanels, odd ? 1u : 2u, qrows / heads};
    const cuuint64_t strides[4] = {row, 128, rows * row, heads * row};
    const cuuint32_t box[5] = {64, kTcHeads, panels, 1, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void *>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// maps[0] = q, maps[1] = K role boxes, maps[2] = V role boxes, maps[3] = whole pages
inline bool tc2_make_maps(const DecodeParams &p, CUtensorMap *maps, bool cached)
{
    const uint64_t rows = (uint64_t)p.num_pages * kPage, qrows = (uint64_t)p.batch * p.heads;
    if (cached)
        return cached_map(&maps[0], p.q, qrows, p.heads, kC2GroupPanels, 2, encode_q_map) &&
               make_panel_map(&maps[1], p.kv, rows, kTile, kC2GroupPanels) && make_panel_map(&maps[2], p.kv, rows, kTile, 4) &&
               make_panel_map(&maps[3], p.kv, rows, kTile, kPanels);
    return encode_q_map(&maps[0], p.q, qrows, p.heads, kC2GroupPanels) && encode_panel_map(&maps[1], p.kv, rows, kTile, kC2GroupPanels) &&
           encode_panel_map(&maps[2], p.kv, rows, kTile, 4) && encode_panel_map(&maps[3], p.kv, rows, kTile, kPanels);
}

// form: see tc2_kernel_for
inline omni_status_t tc2_launch(const CUtensorMap *maps, const DecodeParams &p, int form, cudaStream_t stream)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((p.whole + (p.batch - p.whole) * p.splits) * 2));
    cfg.blockDim = dim3(kC2Threads);
    cfg.dynamicSmemBytes = kC2SmemBytes;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = p.cluster_merge ? 4 : 2;      // cluster merge: both splits of a request in one cluster
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    // the launch may overlap the tail of the previous kernel in the stream (the kernel waits
    // before its first global access), which hides the launch latency between decode steps
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, tc2_kernel_for(form, p.sel_idx == nullptr), maps[0], maps[1],
                                               maps[2], maps[3], p);
    return err == cudaSuccess ? OMNI_OK : OMNI_ERR_CUDA;
}

}  // namespace omni
