// Backward packed variable-length attention for sm_100a: the main kernel for sequences of more than one tile and
// head dimensions above 64, on CTA pairs.
//
// A cluster of two CTAs (one pair of SMs, cta_group::2) works on (sequence, head, 256 keys): CTA r of the pair
// holds keys 128 r .. 128 r + 127 of the block, and both walk over every Q tile that sees the block.  As in the
// one-CTA kernel everything is transposed (keys on tensor-memory lanes, queries on columns):
//
//     S'^T  = K Q^T - 1 (lse/scale)^T      M = 256 keys                      P^T  = exp2(S'^T scale log2e) -> tensor memory
//     dP'^T = V dO^T - 1 D^T               M = 256                           dS^T = P^T o dP'^T            -> tensor memory
//     dV += P^T dO    dK += dS^T Q         M = 256, A from tensor memory          and, for dQ, shared memory
//     dQ_tile = dS K                       M = 128 queries, contraction over all 256 keys
//
// What this form is for: the fp32 dQ tile leaves an SM at 25.6 bytes per clock (measured, the SM's outbound
// port), 64 KB per 128 keys in the one-CTA kernel, as long as all five products take, and the next tiles' loads
// queue behind it.  Here the pair adds the dQ of 256 keys in tensor memory and each CTA sends half of the tile's
// rows: 32 KB per CTA and Q tile.  In exchange half of dS^T (16 KB) crosses to the partner through distributed
// shared memory, because CTA r multiplies the dS of queries 64 r .. 64 r + 63 with all 256 keys.  Each MMA reads
// its own half of B from each SM and A of dV and dK from tensor memory, so the shared-memory port carries
// 192 KB of operands per tile instead of 288.
//
// One continuous pipeline over all tiles of all items of the pair.  The leader's MMA warp issues, per tile k,
//
//     dV(k) | S(k+1) | dK(k) | dP(k+1) | dQ(k)
//
// so that the compute warps rarely wait: S(k+1) runs while they form dS(k), dP(k+1) while they form P(k+1).  Above head
// dimension 96 dQ lives in the middle columns of S^T, which are free once S(k+1) has been read into registers (P^T is packed
// into the outer ones); up to 96 it has columns of its own, so that S(k+1) does not wait for dQ(k-1) to be drained.  Every
// operand tile is used by exactly one product (Q and dO are loaded twice, as rows for S and dP and as columns for dK and dV,
// since a CTA supplies half of B's columns), which leaves each single-buffered load most of a period.  Between items nothing
// drains: the first S of an item follows the last dV of the previous one, and the drain warps write dV and dK of an item while
// the next one is under way.
//
// The issuing warp paces the pipe (an MMA issue blocks while the pipe is busy, so what it does between two products
// is idle time of the tensor cores; a barrier poll takes 100-250 cycles under load).  So there is one commit per
// product, which also releases the operands' buffers, and the barriers a product waits on are polled by different
// lanes at the same time.
//
// Measured (16 heads of 128, fwd + bwd in turn under the power cap; the one-CTA kernel in brackets): two sequences of
// 16384 tokens 9.1 ms = 1200 TFLOP/s (10.5 ms = 1046); the video batch's step 69.8 ms (75.2), the 2-D model's spatial axis
// 8.31 (8.83), at head_dim 72 7.90 (8.16), causal text 4.99 (5.08).  Without the reductions the first is 8.7 ms.  A Q tile
// of the first takes 2.54 us and pair at the 1460 MHz that the power cap leaves, 3720 cycles, and 2.24 us, 4180 cycles,
// when the kernel runs with pauses at 1870-1965 MHz (the loads, the exchange and the reductions do not get faster with the
// clock).  The products need 3300 cycles per tile (dQ 1024 of them: M = 128 on a pair runs at half the rate of M = 256),
// barrier latency the rest; an item's first tile takes 3200 more, most of it waiting for the drain warps to have read the
// previous dK and dQ.
//
// Sequences of one block (at most 256 tokens) write dQ directly; longer ones add it to the fp32 accumulator that
// the pre kernel zeroes and the post kernel converts (layout as in the one-CTA kernel).
//
// Roles (512 threads per CTA): warps 0-7 compute (two groups, 64 of the 128 query columns each, one key per
// thread), warp 8 MMA issue in the leader and, in the partner, the relay that tells the leader when its share
// of dS has arrived; warp 9 TMA producer; warp 11 of the leader pulls work items; warps 12-15 drain dQ.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "attn_kernels.h"
#include "launch.h"
#include "sched.cuh"
#include "sm100_ptx.cuh"

namespace dcp {
namespace {

constexpr int kPairThreads = 512;
constexpr int kRing = 4;                                 // work items in flight between the scheduler and the slowest role
constexpr int kBoxBytes = kTile * 128;                   // 128 rows of 64 columns
constexpr uint32_t kHalfTileBytes = kTile * 128;         // what one CTA loads of a Q or dO tile per use
// shared-memory map (offsets from a 1024-byte aligned base)
constexpr int kOffK = 0;                                 // this CTA's 128 keys, all columns (A of S^T)
constexpr int kOffV = 32768;                             // likewise V
constexpr int kOffKx = 65536;                            // all 256 keys, this CTA's half of the columns (B of dQ)
constexpr int kOffDs = 98304;                            // dS^T of all 256 keys, this CTA's 64 queries (A of dQ)
constexpr int kOffSend = 131072;                         // dS^T of this CTA's keys, the partner's 64 queries
constexpr int kOffQr = 147456;                           // Q: this CTA's 64 rows (B of S^T)
constexpr int kOffQc = 163840;                           // Q: all 128 rows, half of the columns (B of dK)
constexpr int kOffDor = 180224;                          // dO: likewise for dP^T
constexpr int kOffDoc = 196608;                          // ... and dV
constexpr int kOffOnes = 212992;                         // ones, zeros, ones (2 KB each): A of the rank-1 products
constexpr int kStatBytes = 2048;                         // per-query terms of this CTA's 64 queries
constexpr int kOffStat = kOffOnes + 6144;
constexpr int kOffCtl = kOffStat + 2 * kStatBytes;
constexpr int kOffStage = kOffCtl + 512;                  // 2 KB per drain warp, for dV and dK on their way out
constexpr int kSmemBytes = kOffStage + 8192;
static_assert(kSmemBytes <= 232448, "exceeds the 227 KB a CTA may use");
// tensor-memory columns.  P^T (dS^T) overwrites S^T (dP^T) packed: group 0's 64 columns go to the first 32, group
// 1's to the last 32, which leaves 64 adjacent ones in the middle of S^T for dQ.
// Up to head dimension 96 the three results take 96 columns (a pair's products come in steps of 32) and dQ, 48 then, has room
// of its own.  Main kernel, 65536 tokens x 16 heads of 72, us with 128 columns and dQ in S^T: sequences of 200 tokens 477 ->
// 445, 256: 398 -> 373, 1200: 1456 -> 1440, causal 512: 591 -> 559, causal 1200: 1011 -> 955; of 96: 300 814 -> 780.
template <int KS>
struct PairCols {
    static constexpr int kW = KS <= 6 ? 96 : 128;
    static constexpr bool kOwnDq = kW == 96;
    static constexpr uint32_t kS = 0, kDp = 128, kDv = 256, kDk = 256 + kW, kDq = kOwnDq ? 256 + 2 * kW : kS + 32;
};

// The reductions of a dQ tile go out half a tile later: sent at once they delay the exchange of the next dS^T, which the next dQ
// waits for (2 % of a tile's time on long sequences; 500 ns had no effect).  With columns of its own a dQ may leave later still,
// which pays on long sequences: 65536 tokens x 16 heads of 72 and 96, without a mask, kRedDelayLongNs instead of kRedDelayNs at 384
// tokens + 2 and + 6 %, 600 + 2 and + 4, 1000 + 1 and + 1, 2048 - 2 and - 1, 3000 - 3 and - 2, 8192 - 3 and - 3; causal 600 + 1
// and + 3, 2048 + 1 and + 1, 8192 - 2 and - 2.  An item that writes its dQ directly sends none and does not wait: its dK is out
// sooner (16 heads of 128: sequences of 200 tokens 597 -> 578 us, 256 494 -> 478, causal 598 -> 576; of 72 to 96 0 to - 2 %).
constexpr unsigned kRedDelayNs = 900, kRedDelayLongNs = 1344;
constexpr int kLongRed = 2048;

struct PairControl {
    uint64_t work_full[kRing], work_empty[kRing];
    uint64_t ld_s, ld_p, ld_k, ld_v;                     // operands of S (and per-query terms), dP, dK and dQ, dV have landed
    uint64_t s_done, dp_done, dk_done, dq_done, dv_done; // products completed, in both CTAs
    uint64_t s_read, p_full, ds_tmem, ds_smem, ds_recv, dq_free, dv_free, dk_free;
    uint32_t tmem_base;
    uint32_t abort_flag;
    alignas(16) int32_t work[kRing][8];                  // WorkItem and padding
};
static_assert(sizeof(PairControl) <= 512, "control block must fit its slot");
static_assert(sizeof(WorkItem) == 20, "work ring slots are written as five words");

__device__ __forceinline__ void red_add_v4(float* addr, float a, float b, float c, float d) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// dV or dK of a drain warp's 32 keys, all columns: tensor memory -> bf16 in registers (the accumulator is free again),
// then 32 columns at a time through 2 KB of staging (rows of 64 bytes, 16-byte chunks swizzled) to global memory, eight
// rows per instruction.
template <int W>
__device__ __forceinline__ void store_block(__nv_bfloat16* out, const BwdParams& p, uint8_t* stage, uint32_t src_tmem, uint32_t free_bar,
                                            float mul, int head, int tok_row0, int rows_left) {
    const int lane = threadIdx.x & 31;
    uint32_t pk[W / 2];
#pragma unroll
    for (int c = 0; c < W / 32; ++c) {
        uint32_t acc[32];
        tmem_ld_x32(src_tmem + c * 32, acc);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 16; ++e) pk[c * 16 + e] = pack_bf16x2(__uint_as_float(acc[2 * e]) * mul, __uint_as_float(acc[2 * e + 1]) * mul);
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive_at(free_bar);
    const int sub = lane >> 2, chunk = lane & 3;
    __nv_bfloat16* dst = out + ((size_t)tok_row0 + sub) * p.row_stride + head * p.head_dim + chunk * 8;
#pragma unroll
    for (int c = 0; c < W / 32; ++c) {
        if (c * 32 >= p.head_dim) break;
#pragma unroll
        for (int v4 = 0; v4 < 4; ++v4)
            *reinterpret_cast<uint4*>(stage + lane * 64 + ((v4 ^ ((lane >> 1) & 3)) << 4)) =
                make_uint4(pk[c * 16 + v4 * 4], pk[c * 16 + v4 * 4 + 1], pk[c * 16 + v4 * 4 + 2], pk[c * 16 + v4 * 4 + 3]);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int row = i * 8 + sub;
            const uint4 val = *reinterpret_cast<const uint4*>(stage + row * 64 + ((chunk ^ ((row >> 1) & 3)) << 4));
            if (row < rows_left && c * 32 + chunk * 8 < p.head_dim)
                *reinterpret_cast<uint4*>(dst + c * 32 + (size_t)(i * 8) * p.row_stride) = val;
        }
        __syncwarp();                                    // the staging rows have been read
    }
}

// KS = ceil(head_dim / 16), the steps S and dP sum over (5 to 8; a template parameter, because a step count that the issuing
// warp reads at run time costs it 650 of 4500 cycles per tile, more than the skipped steps save).  dV, dK and dQ have 96 or
// 128 columns (PairCols).  S(k+1) overwrites the P^T that dV(k) reads, and dP(k+1) the dS^T that dK(k) reads.  With 128 columns
// these products have one shape (256 x 128), and the pipe has always run them in the order of their issue.  Of 256 x 96 and 256 x
// 128 nothing says so (the PTX ISA does of one accumulator and shape), so there the one waits until the other has completed.
// S(k+1) is ready long before it is read, so that this costs little (backward, 65536 tokens x 16 heads of 72, us without and with
// the waits: 256 tokens 476 and 474, causal 300 907 and 919, 1200 1689 and 1704, causal 1217 and 1228, 16384 16039 and 16120,
// causal 8601 and 8634; of 88 and 96 - 3 to + 1 %).
template <bool CAUSAL, int KS>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
attn_bwd_pair_kernel(const __grid_constant__ PairMaps maps, const __grid_constant__ BwdParams p) {
    using Cols = PairCols<KS>;
    extern __shared__ __align__(1024) uint8_t smem[];
    PairControl& sh = *reinterpret_cast<PairControl*>(smem + kOffCtl);

    const int tid = threadIdx.x;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int lane = tid & 31;
    const uint32_t rank = cluster_ctarank();
    const bool lead = rank == 0;
    const WaitGuard guard{&sh.abort_flag, &p.sched.hdr->status};
    // shared::cluster address of a barrier in the leader
    auto at_leader = [&](const uint64_t* bar) { return map_to_rank(smem_u32(bar), 0); };

    if (tid == 0) {
        for (int i = 0; i < kRing; ++i) {
            mbar_init(&sh.work_full[i], 1);
            mbar_init(&sh.work_empty[i], 28);            // both CTAs: 8 compute + 4 drain warps, warp 8 and the producer
        }
        for (uint64_t* b : {&sh.ld_s, &sh.ld_p, &sh.ld_k, &sh.ld_v, &sh.s_done, &sh.dp_done, &sh.dk_done, &sh.dq_done, &sh.dv_done,
                            &sh.ds_recv})
            mbar_init(b, 1);
        for (uint64_t* b : {&sh.s_read, &sh.p_full, &sh.ds_tmem}) mbar_init(b, 16);      // the compute warps of both CTAs
        mbar_init(&sh.ds_smem, 9);                       // the four warps of each CTA that keep their dS^T, and the relay
        for (uint64_t* b : {&sh.dq_free, &sh.dv_free, &sh.dk_free}) mbar_init(b, 8);      // the drain warps of both CTAs
        sh.abort_flag = 0;
        fence_mbar_init();
        mbar_expect_tx(&sh.ds_recv, kBoxBytes);          // armed one tile ahead by whoever waits on it
        if ((smem_u32(smem) & 1023u) != 0) sh.abort_flag = 1;      // the swizzled layouts need an aligned base; refuse to run otherwise
    }
    {   // A operands of the rank-1 products, [128 keys x 16] in 8x8 core matrices, the two column halves 2 KB apart:
        // ones in columns 0-2 and nothing else (adds the lse term) starts at the first block, ones in columns 8-10 at the second
        uint32_t* ones = reinterpret_cast<uint32_t*>(smem + kOffOnes);
        for (int i = tid; i < 6144 / 4; i += kPairThreads) {
            const int blk = i / 512, in_row = i % 4;
            ones[i] = blk == 1 ? 0u : in_row == 0 ? 0x3f803f80u : in_row == 1 ? 0x00003f80u : 0u;   // 1,1 | 1,0 | 0..
        }
        fence_async_smem();
    }
    __syncthreads();
    cluster_sync();                                      // both CTAs run and their barriers are initialised
    if (warp == 0) {
        tmem_alloc_pair(&sh.tmem_base, 512);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();                                      // the products write both CTAs' tensor memory
    tc_fence_after();
    const uint32_t tmem = sh.tmem_base;
    grid_trigger();
    grid_wait();
    if (tid == 0 && sh.abort_flag) atomicMax(&p.sched.hdr->status, (uint32_t)kStatusBadSmemAlign);
    if (tid == 0) span_begin(p.sched, 1);

    // Q tiles that see key block `blk`: [first_q, n_q)
    auto first_q_of = [](const WorkItem& w) { return CAUSAL ? 2 * w.blk : 0; };
    auto n_q_of = [](const WorkItem& w) { return (w.len + kTile - 1) / kTile; };
    // next item of the ring, for one warp; false at the end of the list
    auto take_item = [&](uint32_t n, WorkItem& w) -> bool {
        const uint32_t slot = n % kRing;
        const bool got = mbar_wait_cluster(&sh.work_full[slot], (n / kRing) & 1u, guard);
        if (!__all_sync(0xffffffffu, got)) return false;
        w.tok0 = sh.work[slot][0];
        w.len = sh.work[slot][1];
        w.head = sh.work[slot][2];
        w.blk = sh.work[slot][3];
        w.tile0 = sh.work[slot][4];
        __syncwarp();
        if (lane == 0) mbar_arrive_at(at_leader(&sh.work_empty[slot]));
        return w.len >= 0;
    };

    if (warp >= 8 && warp < 12) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 104;");
    if (warp == 11) {
        // ------------------------------------------------- scheduler (leader): items of the list to both CTAs
        if (lead) {
            const uint32_t n_items = p.sched.hdr->n_long_items;
            SeqCursor cur;
            for (uint32_t n = 0;; ++n) {
                const uint32_t slot = n % kRing;
                if (n >= kRing) mbar_wait_cluster(&sh.work_empty[slot], (n / kRing - 1) & 1u, guard);
                uint32_t item = 0;
                if (lane == 0) item = claim_item(p.sched.hdr, n, blockIdx.x / 2, gridDim.x / 2, sh.abort_flag);
                item = __shfl_sync(0xffffffffu, item, 0);
                WorkItem w{0, -1, 0, 0, 0};
                if (item < n_items) w = decode_item(p.sched, p.cu_seqlens, item, 2 * kTile, p.n_heads, gridDim.x / 2, CAUSAL, false, cur);
                if (lane < 2) {                     // a lane for each CTA
                    const uint32_t dst = map_to_rank(smem_u32(&sh.work[slot][0]), (uint32_t)lane);
                    st_cluster_v4(dst, (uint32_t)w.tok0, (uint32_t)w.len, (uint32_t)w.head, (uint32_t)w.blk);
                    st_cluster_v4(dst + 16, (uint32_t)w.tile0, 0u, 0u, 0u);
                    mbar_arrive_release_at(map_to_rank(smem_u32(&sh.work_full[slot]), (uint32_t)lane));
                }
                __syncwarp();
                if (w.len < 0) break;
            }
        }
    } else if (warp == 9) {
        // ------------------------------------------------- TMA producer
        // Loads are issued in the order in which the buffers come free: those of dK one tile later than those of S.
        const int x_half = (int)rank * (Cols::kW / 2);               // columns of B this CTA supplies to dV, dK, dQ
        if (lane == 0) {
            tma_prefetch_desc(&maps.q);
            tma_prefetch_desc(&maps.q_rows);
            tma_prefetch_desc(&maps.k);
            tma_prefetch_desc(&maps.v);
            tma_prefetch_desc(&maps.d_o);
            tma_prefetch_desc(&maps.do_rows);
            tma_prefetch_desc(&maps.stats);
        }
        const uint32_t bar_s = at_leader(&sh.ld_s), bar_p = at_leader(&sh.ld_p), bar_k = at_leader(&sh.ld_k), bar_v = at_leader(&sh.ld_v);
        uint32_t n_work = 0, k = 0;
        WorkItem w, prev{0, 0, 0, 0, 0};
        int prev_row = 0;                                // token of tile k - 1's first query
        bool prev_first = false;
        auto load_late = [&](uint32_t c) {               // operands of dK(c) and, new with an item, dQ
            if (c >= 1) mbar_wait(&sh.dk_done, (c - 1) & 1u, guard);
            if (lead) mbar_expect_tx(&sh.ld_k, 2 * (kHalfTileBytes + (prev_first ? 2 * kBoxBytes : 0)));
            tma_load_3d_pair(smem + kOffQc, &maps.q, bar_k, x_half, prev.head, prev_row);
            if (prev_first) {
                if (c >= 1) mbar_wait(&sh.dq_done, (c - 1) & 1u, guard);
                const int key_tok0 = prev.tok0 + prev.blk * 2 * kTile;
                tma_load_3d_pair(smem + kOffKx, &maps.k, bar_k, x_half, prev.head, key_tok0);
                tma_load_3d_pair(smem + kOffKx + kBoxBytes, &maps.k, bar_k, x_half, prev.head, key_tok0 + kTile);
            }
        };
        while (take_item(n_work, w)) {
            const int first_q = first_q_of(w), n_q = n_q_of(w);
            const int key_tok = w.tok0 + w.blk * 2 * kTile + (int)rank * kTile;
            if (lane == 0) {
                for (int i = first_q; i < n_q; ++i, ++k) {
                    const bool first = i == first_q;
                    const int row = w.tok0 + i * kTile;
                    // S(k-1) having completed also frees the per-query terms of tile k-2: dP(k-2) was issued before it
                    if (k >= 1) mbar_wait(&sh.s_done, (k - 1) & 1u, guard);
                    if (lead) mbar_expect_tx(&sh.ld_s, 2 * (kHalfTileBytes + kStatBytes + (first ? 2 * kBoxBytes : 0)));
                    if (first) {
                        tma_load_3d_pair(smem + kOffK, &maps.k, bar_s, 0, w.head, key_tok);
                        tma_load_3d_pair(smem + kOffK + kBoxBytes, &maps.k, bar_s, 64, w.head, key_tok);
                    }
                    tma_load_3d_pair(smem + kOffQr, &maps.q_rows, bar_s, 0, w.head, row + (int)rank * 64);
                    tma_load_3d_pair(smem + kOffQr + 8192, &maps.q_rows, bar_s, 64, w.head, row + (int)rank * 64);
                    tma_load_4d_pair(smem + kOffStat + (k & 1u) * kStatBytes, &maps.stats, bar_s, 0, 0, (int)rank,
                                     2 * ((w.tile0 + i) * p.n_heads + w.head));
                    if (k >= 1) load_late(k - 1);
                    if (k >= 1) mbar_wait(&sh.dp_done, (k - 1) & 1u, guard);
                    if (lead) mbar_expect_tx(&sh.ld_p, 2 * (kHalfTileBytes + (first ? 2 * kBoxBytes : 0)));
                    if (first) {
                        tma_load_3d_pair(smem + kOffV, &maps.v, bar_p, 0, w.head, key_tok);
                        tma_load_3d_pair(smem + kOffV + kBoxBytes, &maps.v, bar_p, 64, w.head, key_tok);
                    }
                    tma_load_3d_pair(smem + kOffDor, &maps.do_rows, bar_p, 0, w.head, row + (int)rank * 64);
                    tma_load_3d_pair(smem + kOffDor + 8192, &maps.do_rows, bar_p, 64, w.head, row + (int)rank * 64);
                    if (k >= 1) mbar_wait(&sh.dv_done, (k - 1) & 1u, guard);
                    if (lead) mbar_expect_tx(&sh.ld_v, 2 * kHalfTileBytes);
                    tma_load_3d_pair(smem + kOffDoc, &maps.d_o, bar_v, x_half, w.head, row);
                    prev = w;
                    prev_row = row;
                    prev_first = first;
                }
            }
            __syncwarp();
            ++n_work;
        }
        if (lane == 0 && k >= 1) load_late(k - 1);
    } else if (warp == 8 && !lead) {
        // ------------------------------------------------- relay: the leader's dQ product reads this CTA's dS^T as well
        uint32_t n_work = 0, k = 0;
        WorkItem w;
        while (take_item(n_work, w)) {
            ++n_work;
            if (lane == 0) {
                for (int i = first_q_of(w); i < n_q_of(w); ++i, ++k) {
                    mbar_wait(&sh.ds_recv, k & 1u, guard);
                    mbar_expect_tx(&sh.ds_recv, kBoxBytes);
                    mbar_arrive_at(at_leader(&sh.ds_smem));
                }
            }
            __syncwarp();
        }
    } else if (warp == 8) {
        // ------------------------------------------------- MMA issue (all lanes in lock step, one elected lane issues)
        const bool leader = elect_one();
        constexpr uint32_t idesc_abt = make_idesc_bf16(256, 128, false, false);  // S^T, dP^T: both operands K-contiguous
        constexpr uint32_t idesc_acc = make_idesc_bf16(256, Cols::kW, false, true);   // dV, dK: A in tensor memory, B N-contiguous
        constexpr uint32_t idesc_dq = make_idesc_bf16(128, Cols::kW, true, true);     // dQ: A M-contiguous, B N-contiguous
        const uint64_t k_km = make_sdesc_sw128(smem_u32(smem + kOffK), 16, 1024);
        const uint64_t v_km = make_sdesc_sw128(smem_u32(smem + kOffV), 16, 1024);
        const uint64_t qr_km = make_sdesc_sw128(smem_u32(smem + kOffQr), 16, 1024);
        const uint64_t dor_km = make_sdesc_sw128(smem_u32(smem + kOffDor), 16, 1024);
        const uint64_t qc_mn = make_sdesc_sw128(smem_u32(smem + kOffQc), kBoxBytes, 1024);
        const uint64_t doc_mn = make_sdesc_sw128(smem_u32(smem + kOffDoc), kBoxBytes, 1024);
        const uint64_t ds_mn = make_sdesc_sw128(smem_u32(smem + kOffDs), kBoxBytes, 1024);
        const uint64_t kx_mn = make_sdesc_sw128(smem_u32(smem + kOffKx), kBoxBytes, 1024);
        const uint64_t ones_s = make_sdesc_nosw(smem_u32(smem + kOffOnes), 2048, 128);
        const uint64_t ones_d = make_sdesc_nosw(smem_u32(smem + kOffOnes + 2048), 2048, 128);
        const uint64_t stat0 = make_sdesc_nosw(smem_u32(smem + kOffStat), 1024, 128);
        // D[256 x 128] = A B^T over head_dim: A in two boxes of 128 rows, B in two boxes of 64 rows; then the per-query terms
        auto issue_abt = [&](uint32_t d_tmem, uint64_t a, uint64_t b, uint64_t ones, uint64_t stat) {
#pragma unroll
            for (int ks = 0; ks < KS; ++ks)
                if (leader)
                    tc_mma_ss_pair(d_tmem, a + (uint64_t)(((ks / 4) * kBoxBytes + (ks % 4) * 32) >> 4),
                                   b + (uint64_t)(((ks / 4) * 8192 + (ks % 4) * 32) >> 4), idesc_abt, ks > 0);
            if (leader) tc_mma_ss_pair(d_tmem, ones, stat, idesc_abt, true);
        };
        // D[256 x 96 or 128] (+)= A B over the 128 queries; A = packed bf16 in tensor memory (columns 0-31 and 96-127 of `a_tmem`)
        auto issue_acc = [&](uint32_t d_tmem, uint32_t a_tmem, uint64_t b, bool accumulate) {
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
                if (leader)
                    tc_mma_ts_pair(d_tmem, a_tmem + (ks < 4 ? ks * 8 : 96 + (ks - 4) * 8), b + (uint64_t)((ks * 2048) >> 4), idesc_acc,
                                   accumulate || ks > 0);
        };
        auto commit = [&](uint64_t* bar) { if (leader) tc_commit_pair(bar); };
        // Up to three barriers, each polled by a lane of its own (the others poll the first).  The loop is left by a vote:
        // lanes that leave a wait one by one would run what follows diverged, and MMA operands live in registers that the
        // whole warp shares.
        auto wait = [&](int n, uint64_t* b0, uint32_t p0, uint64_t* b1, uint32_t p1, uint64_t* b2, uint32_t p2) {
            uint64_t* b = n > 1 && lane == 1 ? b1 : n > 2 && lane == 2 ? b2 : b0;
            const uint32_t par = n > 1 && lane == 1 ? p1 : n > 2 && lane == 2 ? p2 : p0;
            mbar_wait_all(b, par & 1u, guard);
            tc_fence_after();
        };
        auto wait1 = [&](uint64_t* b, uint32_t par) { wait(1, b, par, b, par, b, par); };

        uint32_t n_work = 0, k = 0;                      // items taken; current tile
        WorkItem w{0, 0, 0, 0, 0};
        bool cur = take_item(n_work, w);
        if (cur) {
            uint32_t item = 0;                           // of the current tile
            int left = n_q_of(w) - first_q_of(w);        // tiles of its item from the current one on
            bool first = true;
            ++n_work;
            wait1(&sh.ld_s, 0);
            issue_abt(tmem + Cols::kS, k_km, qr_km, ones_s, stat0);
            commit(&sh.s_done);
            wait1(&sh.ld_p, 0);
            issue_abt(tmem + Cols::kDp, v_km, dor_km, ones_d, stat0);
            commit(&sh.dp_done);
            while (cur) {
                // the tile after this one
                bool next = true, next_first = false;
                if (--left == 0) {
                    next = take_item(n_work, w);
                    next_first = true;
                    if (next) {
                        left = n_q_of(w) - first_q_of(w);
                        ++n_work;
                    }
                }
                const uint64_t stat = stat0 + ((k + 1) & 1u) * (kStatBytes >> 4);
                wait(first && item >= 1 ? 3 : 2, &sh.p_full, k, &sh.ld_v, k, &sh.dv_free, item - 1);
                issue_acc(tmem + Cols::kDv, tmem + Cols::kS, doc_mn, !first);
                commit(&sh.dv_done);
                if (next) {
                    // until its columns are free: of the P^T that dV(k) reads (a product of another shape), or of dQ(k-1)
                    if (Cols::kOwnDq) wait(2, &sh.ld_s, k + 1, &sh.dv_done, k, &sh.ld_s, k + 1);
                    else wait(k >= 1 ? 2 : 1, &sh.ld_s, k + 1, &sh.dq_free, k - 1, &sh.ld_s, k + 1);
                    issue_abt(tmem + Cols::kS, k_km, qr_km, ones_s, stat);
                    commit(&sh.s_done);
                }
                wait(first && item >= 1 ? 3 : 2, &sh.ds_tmem, k, &sh.ld_k, k, &sh.dk_free, item - 1);
                issue_acc(tmem + Cols::kDk, tmem + Cols::kDp, qc_mn, !first);
                commit(&sh.dk_done);
                if (next) {
                    wait(Cols::kOwnDq ? 2 : 1, &sh.ld_p, k + 1, &sh.dk_done, k, &sh.ld_p, k + 1);   // (dK(k) reads dS^T)
                    issue_abt(tmem + Cols::kDp, v_km, dor_km, ones_d, stat);
                    commit(&sh.dp_done);
                }
                // the columns of dQ: S(k+1) has been read, which was issued after the drain of dQ(k-1); for the last tile
                // that drain itself
                if (next && !Cols::kOwnDq) wait(3, &sh.ds_smem, k, &sh.ds_recv, k, &sh.s_read, k + 1);
                else wait(k >= 1 ? 3 : 2, &sh.ds_smem, k, &sh.ds_recv, k, &sh.dq_free, k - 1);
                if (leader) mbar_expect_tx(&sh.ds_recv, kBoxBytes);
#pragma unroll
                for (int ks = 0; ks < 16; ++ks)
                    if (leader)
                        tc_mma_ss_pair(tmem + Cols::kDq, ds_mn + (uint64_t)((ks * 2048) >> 4), kx_mn + (uint64_t)((ks * 2048) >> 4),
                                       idesc_dq, ks > 0);
                commit(&sh.dq_done);
                cur = next;
                first = next_first;
                if (next_first) item = n_work - 1;
                ++k;
            }
        }
    }
    } else if (warp < 8) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 136;");
        // ------------------------------------------------- compute: P^T and dS^T
        const int half = warp >> 2;                                  // which 64 query columns
        const int key_in_tile = (warp & 3) * 32 + lane;              // tensor-memory lane = key
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t st_tmem = tmem + lane_base + Cols::kS + half * 64;
        const uint32_t dp_tmem = tmem + lane_base + Cols::kDp + half * 64;
        const uint32_t pt_tmem = tmem + lane_base + Cols::kS + half * 96;       // packed: columns 0-31 or 96-127
        const uint32_t dst_tmem = tmem + lane_base + Cols::kDp + half * 96;
        // dS^T of the queries whose dQ this CTA computes stays here, the other half goes to the partner
        const bool keep = half == (int)rank;
        uint8_t* ds_box = smem + (keep ? kOffDs + (int)rank * kBoxBytes : kOffSend);
        const uint32_t send_dst = map_to_rank(smem_u32(smem + kOffDs + (int)rank * kBoxBytes + (warp & 3) * 4096), rank ^ 1u);
        const uint32_t send_bar = map_to_rank(smem_u32(&sh.ds_recv), rank ^ 1u);
        const uint32_t bar_s_read = at_leader(&sh.s_read), bar_p = at_leader(&sh.p_full), bar_ds_tmem = at_leader(&sh.ds_tmem),
                       bar_ds_smem = at_leader(&sh.ds_smem);
        const uint64_t sc2 = pack_f32x2(p.scale_log2, p.scale_log2);
        uint32_t n_work = 0, k = 0;
        WorkItem w;
        while (take_item(n_work, w)) {
            const int key0 = w.blk * 2 * kTile + (int)rank * kTile, key = key0 + key_in_tile;
            const bool key_valid = key < w.len, key_tail = key0 + kTile > w.len;
            const int n_q = n_q_of(w);
            for (int i = first_q_of(w); i < n_q; ++i, ++k) {
                const bool diag = CAUSAL && i * kTile < key0 + kTile;
                float pf[64];
                mbar_wait_warp(&sh.s_done, k & 1u, guard);
                tc_fence_after();
                {
                    uint32_t sr[64];
                    tmem_ld_x32(st_tmem, *reinterpret_cast<uint32_t(*)[32]>(&sr[0]));
                    tmem_ld_x32(st_tmem + 32, *reinterpret_cast<uint32_t(*)[32]>(&sr[32]));
                    tmem_wait_ld();
                    if constexpr (!Cols::kOwnDq) {                   // dQ may have the columns
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive_at(bar_s_read);
                    }
                    // the key is seen by the queries from `lo` of this thread's 64 on
                    const bool edge = key_tail || diag;
                    const int lo = !key_valid ? 64 : diag ? key - (i * kTile + half * 64) : -64;
                    auto form_p = [&](auto masked) {
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
#pragma unroll
                            for (int e = 0; e < 32; e += 2) {
                                float x0, x1;
                                unpack_f32x2(mul_f32x2(pack_f32x2(__uint_as_float(sr[c * 32 + e]), __uint_as_float(sr[c * 32 + e + 1])), sc2),
                                             x0, x1);
                                pf[c * 32 + e] = fast_exp2(x0);
                                pf[c * 32 + e + 1] = fast_exp2(x1);
                            }
                            if constexpr (decltype(masked)::value) {
#pragma unroll
                                for (int e = 0; e < 32; ++e) pf[c * 32 + e] = c * 32 + e >= lo ? pf[c * 32 + e] : 0.f;
                            }
                            uint32_t pk[16];
#pragma unroll
                            for (int e = 0; e < 16; ++e) pk[e] = pack_bf16x2(pf[c * 32 + 2 * e], pf[c * 32 + 2 * e + 1]);
                            tmem_st_x16(pt_tmem + c * 16, pk);
                        }
                    };
                    // One select per element, and where the masks stand decides how the loop is compiled.  Before, with a test of
                    // (key_valid, diag, key > query) on every element of a masked tile: causal 256-token sequences, 16 heads of 128,
                    // 527 -> 494 us for 65536 tokens, of 72 448 -> 398; causal 1200 1165 -> 1116 and 998 -> 956; the text batch 2.8 %,
                    // the 2-D model's spatial axis (no mask but at sequence ends) 1.7 %.  At 96 columns the form of 128, with its
                    // second copy of the loop body, costs batches without a mask 1 to 4 %; at 128 that of 96 costs them 1 to 2 %.
                    if constexpr (Cols::kOwnDq) {
                        if (edge) {
#pragma unroll
                            for (int e = 0; e < 64; ++e) sr[e] = e >= lo ? sr[e] : 0xff800000u;         // -inf
                        }
                        form_p(std::false_type{});
                    } else if (edge) {
                        form_p(std::true_type{});
                    } else {
                        form_p(std::false_type{});
                    }
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_at(bar_p);

                // dS^T = P^T o (dP^T - D)
                mbar_wait_warp(&sh.dp_done, k & 1u, guard);
                tc_fence_after();
                uint32_t ds[32];
                {
                    uint32_t dr[64];
                    tmem_ld_x32(dp_tmem, *reinterpret_cast<uint32_t(*)[32]>(&dr[0]));
                    tmem_ld_x32(dp_tmem + 32, *reinterpret_cast<uint32_t(*)[32]>(&dr[32]));
                    tmem_wait_ld();
#pragma unroll
                    for (int e = 0; e < 32; ++e) {
                        float x0, x1;
                        unpack_f32x2(mul_f32x2(pack_f32x2(pf[2 * e], pf[2 * e + 1]),
                                               pack_f32x2(__uint_as_float(dr[2 * e]), __uint_as_float(dr[2 * e + 1]))), x0, x1);
                        ds[e] = pack_bf16x2(x0, x1);
                    }
                }
                tmem_st_x32(dst_tmem, ds);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_at(bar_ds_tmem);
                // shared memory: dQ of the previous tile, which read it (in both CTAs), was issued before dV of this one
                if (k >= 1) mbar_wait_warp(&sh.dq_done, (k - 1) & 1u, guard);
#pragma unroll
                for (int c = 0; c < 8; ++c)
                    *reinterpret_cast<uint4*>(ds_box + sw128_offset(key_in_tile, c)) =
                        make_uint4(ds[c * 4], ds[c * 4 + 1], ds[c * 4 + 2], ds[c * 4 + 3]);
                fence_async_smem();
                __syncwarp();
                if (lane == 0) {
                    if (!keep) bulk_copy_to_partner(send_dst, ds_box + (warp & 3) * 4096, 4096, send_bar);
                    else mbar_arrive_at(bar_ds_smem);
                }
            }
            ++n_work;
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 136;");
        // ------------------------------------------------- drain: dQ (64 queries of the tile, half of the columns per warp
        // pair) and, after an item's last tile, its dV and dK: the stores wait for the way out of the SM, 5000 cycles per
        // item, which the compute warps cannot afford on short items and these can
        const int q_in_half = (warp & 1) * 32 + lane;
        const int col0 = ((warp >> 1) & 1) * (Cols::kW / 2);
        const int n_c4 = min(Cols::kW / 2, p.head_dim - col0) / 4;             // groups of four columns that hold data
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t dq_tmem = tmem + lane_base + Cols::kDq;
        uint8_t* stage = smem + kOffStage + (warp & 3) * 2048;
        const uint32_t bar_free = at_leader(&sh.dq_free);
        uint32_t n_work = 0, k = 0;
        WorkItem w;
        while (take_item(n_work, w)) {
            ++n_work;
            const int n_q = n_q_of(w);
            const int key0 = w.blk * 2 * kTile + (int)rank * kTile + (warp & 3) * 32;
            for (int i = first_q_of(w); i < n_q; ++i, ++k) {
                if (i == n_q - 1) {                      // dV is complete before the last dQ
                    mbar_wait_warp(&sh.dv_done, k & 1u, guard);
                    tc_fence_after();
                    store_block<Cols::kW>(p.dv, p, stage, tmem + lane_base + Cols::kDv, at_leader(&sh.dv_free), 1.0f, w.head, w.tok0 + key0, w.len - key0);
                }
                mbar_wait_warp(&sh.dq_done, k & 1u, guard);
                tc_fence_after();
                uint32_t acc[Cols::kW / 2];
                tmem_ld_x32(dq_tmem, *reinterpret_cast<uint32_t(*)[32]>(&acc[0]));
                if constexpr (Cols::kW == 128) tmem_ld_x32(dq_tmem + 32, *reinterpret_cast<uint32_t(*)[32]>(&acc[32]));
                else tmem_ld_x16(dq_tmem + 32, *reinterpret_cast<uint32_t(*)[16]>(&acc[32]));
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_at(bar_free);
                if (w.len > 2 * kTile) __nanosleep(Cols::kOwnDq && w.len > kLongRed ? kRedDelayLongNs : kRedDelayNs);
                const int row_in_tile = (int)rank * 64 + q_in_half, qrow = i * kTile + row_in_tile;
                const bool live = qrow < w.len;
                if (w.len <= 2 * kTile) {
                    // the sequence's only key block: this is the whole dQ
                    __nv_bfloat16* out = p.dq + ((size_t)w.tok0 + qrow) * p.row_stride + w.head * p.head_dim + col0;
#pragma unroll
                    for (int c = 0; c < Cols::kW / 16; ++c) {
                        uint4 val;
                        val.x = pack_bf16x2(__uint_as_float(acc[c * 8 + 0]) * p.scale, __uint_as_float(acc[c * 8 + 1]) * p.scale);
                        val.y = pack_bf16x2(__uint_as_float(acc[c * 8 + 2]) * p.scale, __uint_as_float(acc[c * 8 + 3]) * p.scale);
                        val.z = pack_bf16x2(__uint_as_float(acc[c * 8 + 4]) * p.scale, __uint_as_float(acc[c * 8 + 5]) * p.scale);
                        val.w = pack_bf16x2(__uint_as_float(acc[c * 8 + 6]) * p.scale, __uint_as_float(acc[c * 8 + 7]) * p.scale);
                        if (live && c * 2 < n_c4) *reinterpret_cast<uint4*>(out + c * 8) = val;
                    }
                } else {
                    float* dst = p.dq_acc + (((size_t)w.tile0 + i) * p.n_heads + w.head) * (size_t)(kTile * 128) + row_in_tile * 4 +
                                 (col0 / 4) * (kTile * 4);
#pragma unroll
                    for (int c = 0; c < Cols::kW / 8; ++c)
                        if (live && c < n_c4)
                            red_add_v4(dst + c * (kTile * 4), __uint_as_float(acc[c * 4]), __uint_as_float(acc[c * 4 + 1]),
                                       __uint_as_float(acc[c * 4 + 2]), __uint_as_float(acc[c * 4 + 3]));
                }
            }
            // dK was issued before the last dQ
            store_block<Cols::kW>(p.dk, p, stage, tmem + lane_base + Cols::kDk, at_leader(&sh.dk_free), p.scale, w.head, w.tok0 + key0, w.len - key0);
        }
    }

    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (tid == 0) span_end(p.sched, 1);
    // after an abandoned wait a copy to the partner may still be under way: give it time before the CTAs leave
    if (sh.abort_flag) for (int i = 0; i < 64; ++i) __nanosleep(1000);
    __syncwarp();
    cluster_sync();                                      // all work of the pair is done
    tc_fence_after();
    if (warp == 0) tmem_dealloc_pair(tmem, 512);
    __syncwarp();
    cluster_sync();                                      // neither CTA leaves while the other may still address it
}

template <int KS>
cudaError_t launch_one(const PairMaps& maps, const BwdParams& p, bool causal, int n_ctas, cudaStream_t stream) {
    auto launch = [&](auto kern) { return launch_dependent(kern, n_ctas & ~1, kPairThreads, kSmemBytes, stream, maps, p); };
    if (causal) {
        if (cudaError_t e = allow_smem<attn_bwd_pair_kernel<true, KS>>(kSmemBytes)) return e;
        return launch(attn_bwd_pair_kernel<true, KS>);
    }
    if (cudaError_t e = allow_smem<attn_bwd_pair_kernel<false, KS>>(kSmemBytes)) return e;
    return launch(attn_bwd_pair_kernel<false, KS>);
}

}  // namespace

cudaError_t launch_attn_bwd_pair(const PairMaps& maps, const BwdParams& p, int head_dim, bool causal, int n_ctas, cudaStream_t stream) {
    switch ((head_dim + 15) / 16) {
        case 5: return launch_one<5>(maps, p, causal, n_ctas, stream);
        case 6: return launch_one<6>(maps, p, causal, n_ctas, stream);
        case 7: return launch_one<7>(maps, p, causal, n_ctas, stream);
        default: return launch_one<8>(maps, p, causal, n_ctas, stream);
    }
}

}  // namespace dcp
