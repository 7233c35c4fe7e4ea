// Backward packed variable-length attention for sm_100a (main kernel).
//
// One persistent CTA per SM.  A work item is (sequence, head, 128 keys); the CTA keeps that K and V
// tile in shared memory and walks over every Q tile that sees it.  Everything is computed in the
// transposed orientation, keys on tensor-memory lanes and queries on columns, so that P^T can feed
// the dV product straight from tensor memory:
//
//     S'^T  = K Q^T - 1 (lse/scale)^T   (tcgen05, fp32 in tensor memory)
//     P^T   = exp2(S'^T * scale*log2e), masked                     -> bf16, overwrites S'^T
//     dP'^T = V dO^T - 1 D^T
//     dS^T  = P^T o dP'^T                                          -> bf16, shared memory
//     dV  += P^T dO          dK += dS^T Q          dQ_tile = dS K  (dQ aliases dP^T's columns)
//
// The per-query terms -lse/scale and -D are columns in this orientation; instead of every thread
// reading them (a shared-memory broadcast costs one wavefront per value, on the port that feeds the
// MMAs), they are added by one extra K=16 MMA per product: A = a constant tile of ones, B = a
// [128 queries x 16] bf16 tile holding each term split into three bf16 parts (24 bits, exact sum in
// the fp32 accumulator), prepared per (tile, head) by the pre kernel and fetched by bulk copy.
//
// dQ tiles are added into an fp32 accumulator in global memory with vector atomics because every
// key block of a sequence contributes to the same query rows.  The accumulator is a workspace, so
// its layout is chosen for the atomics: per (tile, head) a block [16][128 rows][4 floats], which
// makes the 32 rows a warp holds contiguous (full 32-byte sectors, four 128-byte lines per
// instruction instead of 32 scattered ones); a small kernel converts it to [T, H, d] bf16 later.
// These 32 KB per (Q tile, K tile) pair leave the SM at 15-25 bytes per clock, by per-thread atomics and
// shared-memory bulk reductions alike, and the atomics share the load/store unit with the compute warps' dS^T
// stores.  What helps is pausing the drain warps briefly between groups of atomics (see kRedGroup).  Measured and
// rejected, all when this kernel still took head dimension 128 and 64 KB per pair: pacing by spinning on the clock
// (the spin takes issue slots from the compute warps), bulk reductions from a 16 KB staging buffer,
// atomics into an L2-hot block (same time, so the limit is on the SM's side), dK before dQ, and
// staggering the Q walk of neighbouring key blocks.
// dK and dV stay in tensor memory for the whole item and are written once (dK scaled by the
// softmax scale).
//
// The MMA warp runs its loop warp-uniformly and an elected lane issues: a tcgen05.mma issue blocks,
// and a lone diverged thread that also computes descriptors pays 80-100 cycles per instruction, so
// descriptors are built once per item and a k-step is a constant add.  P^T is published in two
// parts (the first 32 query columns of each column group first), so the dV product starts on
// those while the rest is still being exponentiated.
//
// Roles:  warps 0-7 compute (two groups, each owns 64 of the 128 query columns, one key per thread),
//         warp 8 MMA issue, warp 9 scheduler + TMA producer + per-row statistics staging
//         (warps 10-11 idle: the control group of four gives most of its registers away),
//         warps 12-15 dQ drain (tensor memory -> global atomics).
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "attn_kernels.h"
#include "launch.h"
#include "sched.cuh"
#include "sm100_ptx.cuh"

namespace dcp {

// The drain warps pause after every kRedGroup vector atomics, and warp k of the four starts k pauses
// late.  Issued back to back, a tile's atomics fill the SM's queue towards L2, and the TMA
// requests and shared-memory stores of the other warps wait behind them; short sleeps (which, unlike
// a spin on the clock, take no issue slots) let those through.  __nanosleep rounds down to steps of
// about 128 ns here (100 ns had no effect, 150-250 ns the same effect), so the values sit in the
// middle of a step.  Chosen at head dimension 128, which the pair kernel has since taken over (video batch, this kernel
// alone: 60.2 ms without any pause, 58.3 with the pauses, 55.8 with the stagger as well; two steps per pause or per
// stagger, or a pause after every second atomic, 57-85 ms); at 64 other pauses and groups give 0 to + 3 %.
constexpr int kRedGroup = 4;
constexpr unsigned kRedSleepNs = 192;        // one step
constexpr unsigned kRedStaggerNs = 128;      // per drain warp, plus half a step
constexpr int kBwdThreads = 512;
constexpr float kLog2e = 1.4426950408889634f;

constexpr int kD = 64;                       // columns of a tile (head dimensions above have the pair kernel)

struct BwdCfg {
    static constexpr int kTileBytes = kTile * kD * 2;    // K, V, Q or dO tile: one box of 64 columns
    static constexpr int kDsBytes = kTile * kTile * 2;   // dS^T tile, bf16
    // shared-memory map (offsets from a 1024-byte aligned base)
    static constexpr int kOffK = 0;
    static constexpr int kOffV = kTileBytes;
    static constexpr int kQStages = 2;                     // Q is needed early (S^T) and late (dK)
    // K and V have two slots: the next item's (and, behind them in the producer's order, its first Q, terms and dO) load
    // while this item still runs; with one slot they waited for its last product, a load latency per item.  Backward, 65536
    // tokens, 16 heads, us with one slot and with two: of 64 150 tokens 738 and 730, causal 693 and 672, 256 556 and 549, 300 735
    // and 726; of 40 256 548 and 509, causal 495 and 467; causal 16384 of 40, 56 and 64 within 0.5 %.
    static constexpr int kKvBytes = 2 * kTileBytes;
    static constexpr int kOffQ = 2 * kKvBytes;
    static constexpr int kOffDo = (4 + kQStages) * kTileBytes;          // dO lives only from dP^T to dV: one stage
    static constexpr int kOffDs = (5 + kQStages) * kTileBytes;
    static constexpr int kStatBytes = kTile * 16 * 2;      // [128 x 16] bf16 tile, K-contiguous, no swizzle
    static constexpr int kOffOnes = kOffDs + kDsBytes;     // two constant tiles: ones in columns 0-2 / 8-10
    static constexpr int kOffStat = kOffOnes + 2 * kStatBytes;   // 2 slots of per-query terms
    static constexpr int kOffCtl = kOffStat + 2 * kStatBytes;
    static constexpr int kSmemBytes = kOffCtl + 320;
    static_assert(kSmemBytes <= 232448, "exceeds the 227 KB a CTA may use");
    // tensor-memory columns
    static constexpr uint32_t kSt = 0, kDp = 128, kDv = 256, kDk = 384;
};

struct BwdControl {
    uint64_t work_full[2], work_empty[2];
    uint64_t kv_full[2], kv_empty[2];
    uint64_t q_full[2], q_empty[2], do_full, do_empty, stat_full[2], stat_empty[2];
    uint64_t s_full, p_half, p_full, dp_full, ds_full, ds_free, dq_full, dq_free, dkv_full, dkv_free;
    WorkItem work[2];
    uint32_t tmem_base;
    uint32_t abort_flag;
};
static_assert(sizeof(BwdControl) <= 320, "control block must fit its slot");

__device__ __forceinline__ void red_add_v4(float* addr, float a, float b, float c, float d) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

__device__ __forceinline__ void bwd_load_tile(uint8_t* dst, const CUtensorMap* map, uint64_t* bar, int head, int row) {
    tma_load_3d(dst, map, bar, 0, head, row);
}

// Compute-warp work of an item that is a single tile pair (a virtual sequence of at most 128 tokens,
// in which short sequences may have been merged): P^T and dS^T with a key seen only by the queries at
// the positions of its own sequence, which the per-token table gives.  Kept out of line so that the
// loop of the common case is compiled exactly as it would be without this path.  `g` is the running
// tile-pair count of the calling thread (it selects the barrier phases).
template <bool CAUSAL>
__device__ __noinline__ void compute_single_tile_item(BwdControl& sh, const BwdParams& p, const WorkItem w, uint32_t st_tmem,
                                                      uint32_t dp_tmem, uint8_t* ds_row, int half, int key_in_tile,
                                                      uint32_t g, const WaitGuard guard) {
    const int lane = threadIdx.x & 31;
    const bool key_valid = key_in_tile < w.len;
    int q_lo = 0, q_hi = 0;
    if (key_valid) {
        const uint32_t b = p.bounds[(size_t)w.tok0 + key_in_tile];
        q_lo = (int)(b & 0xffu);
        q_hi = (int)(b >> 8);
    }
    if (CAUSAL && key_in_tile > q_lo) q_lo = key_in_tile;     // a key is seen from its own position on
    float pf[64];
    mbar_wait_warp(&sh.s_full, g & 1u, guard);
    tc_fence_after();
    {
        uint32_t sr[64];
        tmem_ld_x32(st_tmem, *reinterpret_cast<uint32_t(*)[32]>(&sr[0]));
        tmem_ld_x32(st_tmem + 32, *reinterpret_cast<uint32_t(*)[32]>(&sr[32]));
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int q_first = half * 64 + c * 32;
#pragma unroll
            for (int e = 0; e < 32; ++e) {
                const int qi = q_first + e;
                const float x = fast_exp2(__uint_as_float(sr[c * 32 + e]) * p.scale_log2);
                pf[c * 32 + e] = (qi >= q_lo && qi < q_hi) ? x : 0.f;
            }
            uint32_t pk[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) pk[e] = pack_bf16x2(pf[c * 32 + 2 * e], pf[c * 32 + 2 * e + 1]);
            tmem_st_x16(st_tmem + c * 16, pk);
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(c == 0 ? &sh.p_half : &sh.p_full);
        }
    }
    mbar_wait_warp(&sh.dp_full, g & 1u, guard);
    if (g >= 1) mbar_wait_warp(&sh.ds_free, (g - 1) & 1u, guard);
    tc_fence_after();
    {
        uint32_t dr[64];
        tmem_ld_x32(dp_tmem, *reinterpret_cast<uint32_t(*)[32]>(&dr[0]));
        tmem_ld_x32(dp_tmem + 32, *reinterpret_cast<uint32_t(*)[32]>(&dr[32]));
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            uint32_t pk[4];
#pragma unroll
            for (int e = 0; e < 4; ++e)
                pk[e] = pack_bf16x2(pf[c * 8 + 2 * e] * __uint_as_float(dr[c * 8 + 2 * e]),
                                    pf[c * 8 + 2 * e + 1] * __uint_as_float(dr[c * 8 + 2 * e + 1]));
            *reinterpret_cast<uint4*>(ds_row + sw128_offset(key_in_tile, c)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
        }
    }
    fence_async_smem();
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(&sh.ds_full);
}

template <bool CAUSAL>
__global__ void __launch_bounds__(kBwdThreads, 1)
attn_bwd_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ CUtensorMap tmap_do,
                const __grid_constant__ BwdParams p) {
    using Cfg = BwdCfg;
    extern __shared__ __align__(1024) uint8_t smem[];
    BwdControl& sh = *reinterpret_cast<BwdControl*>(smem + Cfg::kOffCtl);

    const int tid = threadIdx.x;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);     // via a shuffle: provably uniform within the warp
    const int lane = tid & 31;
    const WaitGuard guard{&sh.abort_flag, &p.sched.hdr->status};

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh.work_full[i], 1);
            mbar_init(&sh.work_empty[i], 13);   // 8 compute warps + 4 drain warps + the MMA thread
            mbar_init(&sh.stat_full[i], 1);
            mbar_init(&sh.stat_empty[i], 1);
        }
        for (int i = 0; i < Cfg::kQStages; ++i) {
            mbar_init(&sh.q_full[i], 1);
            mbar_init(&sh.q_empty[i], 1);
        }
        mbar_init(&sh.do_full, 1);
        mbar_init(&sh.do_empty, 1);
        for (int i = 0; i < 2; ++i) {
            mbar_init(&sh.kv_full[i], 1);
            mbar_init(&sh.kv_empty[i], 1);
        }
        mbar_init(&sh.s_full, 1);
        mbar_init(&sh.p_half, 8);     // first 32 query columns of each group's P^T written
        mbar_init(&sh.p_full, 8);
        mbar_init(&sh.dp_full, 1);
        mbar_init(&sh.ds_full, 8);
        mbar_init(&sh.ds_free, 1);
        mbar_init(&sh.dq_full, 1);
        mbar_init(&sh.dq_free, 4);
        mbar_init(&sh.dkv_full, 1);
        mbar_init(&sh.dkv_free, 8);
        sh.abort_flag = 0;
        fence_mbar_init();
        // the swizzled tile layout needs a 1024-byte aligned base; refuse to run otherwise
        if ((smem_u32(smem) & 1023u) != 0) sh.abort_flag = 1;
    }
    __syncwarp();
    if (warp == 0) {
        tmem_alloc(&sh.tmem_base, 512);
        tmem_relinquish();
    }
    {   // constant A operands of the rank-1 MMAs: [128 keys x 16] with ones in columns 0-2 (adds the lse
        // term to S^T) and in columns 8-10 (adds the D term to dP^T).  Layout: 8x8 core matrices of
        // 128 bytes, row groups 128 bytes apart, the two column halves 2048 bytes apart.
        uint32_t* ones = reinterpret_cast<uint32_t*>(smem + Cfg::kOffOnes);
        for (int i = tid; i < 2 * Cfg::kStatBytes / 4; i += kBwdThreads) {
            const int tile = i / (Cfg::kStatBytes / 4), w32 = i % (Cfg::kStatBytes / 4);
            const int half = w32 / 512, in_row = w32 % 4;            // 32-bit word inside a 16-byte row chunk
            const bool on = half == tile;                            // tile 0: first column half, tile 1: second
            ones[i] = !on ? 0u : in_row == 0 ? 0x3f803f80u : in_row == 1 ? 0x00003f80u : 0u;   // 1,1 | 1,0 | 0..
        }
        fence_async_smem();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh.tmem_base;
    grid_trigger();
    grid_wait();
    if (tid == 0 && sh.abort_flag) atomicMax(&p.sched.hdr->status, (uint32_t)kStatusBadSmemAlign);
    if (tid == 0) span_begin(p.sched, 1);

    // Q tiles that see key block `blk`: [first_q, n_q)
    auto q_range = [](const WorkItem& w, int& first_q, int& n_q) {
        n_q = (w.len + kTile - 1) / kTile;
        first_q = CAUSAL ? w.blk : 0;
    };

    if (warp >= 8 && warp < 12) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 104;");
    if (warp == 9) {
        // ------------------------------------------------- scheduler, TMA producer, statistics staging
        if (lane == 0) {
            tma_prefetch_desc(&tmap_q);
            tma_prefetch_desc(&tmap_k);
            tma_prefetch_desc(&tmap_v);
            tma_prefetch_desc(&tmap_do);
        }
        const uint32_t n_items = p.split ? p.sched.hdr->n_long_items : p.sched.hdr->n_items;
        uint32_t n_work = 0, g = 0;
        SeqCursor cur;
        while (true) {
            const uint32_t slot = n_work & 1u;
            uint32_t item = 0;
            if (lane == 0) {
                if (n_work >= 2) mbar_wait(&sh.work_empty[slot], ((n_work >> 1) - 1) & 1u, guard);
                item = claim_item(p.sched.hdr, n_work, blockIdx.x, gridDim.x, sh.abort_flag);
            }
            item = __shfl_sync(0xffffffffu, item, 0);
            WorkItem w{0, -1, 0, 0, 0};
            if (item < n_items) w = decode_item(p.sched, p.cu_seqlens, item, kTile, p.n_heads, gridDim.x, CAUSAL, false, cur);
            if (lane == 0) {
                sh.work[slot] = w;
                mbar_arrive(&sh.work_full[slot]);
            }
            __syncwarp();
            if (w.len < 0) break;
            int first_q, n_q;
            q_range(w, first_q, n_q);
            if (lane == 0) {
                uint8_t* kv = smem + slot * Cfg::kKvBytes;
                if (n_work >= 2) mbar_wait(&sh.kv_empty[slot], ((n_work >> 1) - 1) & 1u, guard);
                mbar_expect_tx(&sh.kv_full[slot], Cfg::kKvBytes);
                bwd_load_tile(kv + Cfg::kOffK, &tmap_k, &sh.kv_full[slot], w.head, w.tok0 + w.blk * kTile);
                bwd_load_tile(kv + Cfg::kOffV, &tmap_v, &sh.kv_full[slot], w.head, w.tok0 + w.blk * kTile);
            }
            ++n_work;
            for (int i = first_q; i < n_q; ++i, ++g) {
                const uint32_t stage = g % Cfg::kQStages, fill = g / Cfg::kQStages;
                const int row = w.tok0 + i * kTile;
                if (lane == 0) {
                    if (fill >= 1) mbar_wait(&sh.q_empty[stage], (fill - 1) & 1u, guard);
                    mbar_expect_tx(&sh.q_full[stage], Cfg::kTileBytes);
                    bwd_load_tile(smem + Cfg::kOffQ + stage * Cfg::kTileBytes, &tmap_q, &sh.q_full[stage], w.head, row);
                    // per-query terms (2 slots): slot g&1 is free once the rank-1 MMAs of tile g-2 are done.
                    // The 4 KB block of this (tile, head) comes by bulk copy in the layout the MMA reads.
                    if (g >= 2) mbar_wait(&sh.stat_empty[g & 1u], ((g >> 1) - 1) & 1u, guard);
                    mbar_expect_tx(&sh.stat_full[g & 1u], Cfg::kStatBytes);
                    tma_load_bulk(smem + Cfg::kOffStat + (g & 1u) * Cfg::kStatBytes,
                                  p.stats + (((size_t)w.tile0 + i) * p.n_heads + w.head) * (Cfg::kStatBytes / 2),
                                  Cfg::kStatBytes, &sh.stat_full[g & 1u]);
                    if (g >= 1) mbar_wait(&sh.do_empty, (g - 1) & 1u, guard);
                    mbar_expect_tx(&sh.do_full, Cfg::kTileBytes);
                    bwd_load_tile(smem + Cfg::kOffDo, &tmap_do, &sh.do_full, w.head, row);
                }
            }
        }
    } else if (warp == 8) {
        // ------------------------------------------------- MMA issue
        // All 32 lanes run the loop in lock step and only `leader` issues, so that every operand is
        // warp-uniform and an MMA costs a couple of adds: each instruction between two MMAs is pipe idle time.
        {
            const bool leader = elect_one();
            // Shared-memory descriptors are built once; a k-step only adds a constant to the address
            // field (the issuing thread is on the critical path: MMA issue blocks while the pipe is busy).
            constexpr uint32_t idesc_abt = make_idesc_bf16(128, 128, false, false);  // both operands K-contiguous
            constexpr uint32_t idesc_nd_kb = make_idesc_bf16(128, kD, false, true);   // A K-contig / tmem, B N-contig
            constexpr uint32_t idesc_nd_mm = make_idesc_bf16(128, kD, true, true);    // A M-contig, B N-contig
            constexpr uint32_t kStageStep = Cfg::kTileBytes >> 4;
            const uint64_t k_km0 = make_sdesc_sw128(smem_u32(smem + Cfg::kOffK), 16, 1024);
            const uint64_t k_mn0 = make_sdesc_sw128(smem_u32(smem + Cfg::kOffK), Cfg::kTileBytes, 1024);
            const uint64_t v_km0 = make_sdesc_sw128(smem_u32(smem + Cfg::kOffV), 16, 1024);
            const uint64_t q_km0 = make_sdesc_sw128(smem_u32(smem + Cfg::kOffQ), 16, 1024);
            const uint64_t q_mn0 = make_sdesc_sw128(smem_u32(smem + Cfg::kOffQ), Cfg::kTileBytes, 1024);
            const uint64_t do_km = make_sdesc_sw128(smem_u32(smem + Cfg::kOffDo), 16, 1024);
            const uint64_t do_mn = make_sdesc_sw128(smem_u32(smem + Cfg::kOffDo), Cfg::kTileBytes, 1024);
            const uint64_t ds_km = make_sdesc_sw128(smem_u32(smem + Cfg::kOffDs), 16, 1024);
            const uint64_t ds_mn = make_sdesc_sw128(smem_u32(smem + Cfg::kOffDs), 16384, 1024);
            const uint64_t ones_s = make_sdesc_nosw(smem_u32(smem + Cfg::kOffOnes), 2048, 128);
            const uint64_t ones_d = make_sdesc_nosw(smem_u32(smem + Cfg::kOffOnes + Cfg::kStatBytes), 2048, 128);
            const uint64_t stat0 = make_sdesc_nosw(smem_u32(smem + Cfg::kOffStat), 2048, 128);
            constexpr uint32_t kStatStep = Cfg::kStatBytes >> 4;
            // address-field increments (16-byte units) of k-step ks
            auto km_step = [](int ks, int box_bytes) -> uint64_t { return (uint64_t)(((ks / 4) * box_bytes + (ks % 4) * 32) >> 4); };
            auto mn_step = [](int ks) -> uint64_t { return (uint64_t)((ks * 2048) >> 4); };
            // D[128 x 128] = A B^T, both [128 x 64] tiles with head_dim contiguous
            auto issue_abt = [&](uint32_t d_tmem, uint64_t a, uint64_t b) {
#pragma unroll
                for (int ks = 0; ks < kD / 16; ++ks)
                    if (leader)
                        tc_mma_ss(d_tmem, a + km_step(ks, Cfg::kTileBytes), b + km_step(ks, Cfg::kTileBytes), idesc_abt, ks > 0);
            };
            // Up to three barriers, each polled by a lane of its own (the others poll the first) and the loop left by a vote:
            // the time to see a barrier is spent once and not one barrier after the other, while the tensor pipe idles.
            // 65536 tokens, 16 heads of 64, one barrier after the other -> together: 300 tokens 494 -> 487 us, causal 404 ->
            // 391; 1200 causal 690 -> 667; 4096 3176 -> 3154, causal 1718 -> 1679.  Waits that are always for a single barrier
            // stay with mbar_wait_warp (by the vote 0 to 2 % slower); that for P^T's first half, with dkv_free in an item's first
            // tile, is by the vote in every tile (a branch to mbar_wait_warp in the others: 0 to 1 % slower).
            auto wait = [&](int n, uint64_t* b0, uint32_t p0, uint64_t* b1, uint32_t p1, uint64_t* b2, uint32_t p2) {
                uint64_t* b = n > 1 && lane == 1 ? b1 : n > 2 && lane == 2 ? b2 : b0;
                const uint32_t par = n > 1 && lane == 1 ? p1 : n > 2 && lane == 2 ? p2 : p0;
                mbar_wait_all(b, par & 1u, guard);
                tc_fence_after();
            };
            uint32_t n_work = 0, g = 0;
            while (true) {
                const uint32_t slot = n_work & 1u;
                const bool got = mbar_wait_warp(&sh.work_full[slot], (n_work >> 1) & 1u, guard);
                if (!__all_sync(0xffffffffu, got)) break;
                const WorkItem w = sh.work[slot];
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.work_empty[slot]);
                if (w.len < 0) break;
                int first_q, n_q;
                q_range(w, first_q, n_q);
                const int N = n_q - first_q;
                const uint64_t kv_step = (uint64_t)(slot * (Cfg::kKvBytes >> 4));
                const uint64_t k_km = k_km0 + kv_step, k_mn = k_mn0 + kv_step, v_km = v_km0 + kv_step;
                // S^T and dP^T of the first tile
                uint32_t stage = g % Cfg::kQStages;
                wait(3, &sh.kv_full[slot], n_work >> 1, &sh.q_full[stage], g / Cfg::kQStages, &sh.stat_full[g & 1u], g >> 1);
                issue_abt(tmem + Cfg::kSt, k_km, q_km0 + stage * kStageStep);
                if (leader) tc_mma_ss(tmem + Cfg::kSt, ones_s, stat0 + (g & 1u) * kStatStep, idesc_abt, true);
                if (leader) tc_commit(&sh.s_full);
                wait(g >= 1 ? 2 : 1, &sh.do_full, g, &sh.dq_free, g - 1, &sh.do_full, g);
                issue_abt(tmem + Cfg::kDp, v_km, do_km);
                if (leader) tc_mma_ss(tmem + Cfg::kDp, ones_d, stat0 + (g & 1u) * kStatStep, idesc_abt, true);
                if (leader) tc_commit(&sh.dp_full);
                if (leader) tc_commit(&sh.stat_empty[g & 1u]);
                for (int n = 0; n < N; ++n, ++g) {
                    const uint32_t nstage = stage + 1 == Cfg::kQStages ? 0 : stage + 1;
                    const bool has_next = n + 1 < N;
                    // dV += P^T dO
                    wait(n == 0 && n_work >= 1 ? 2 : 1, &sh.p_half, g, &sh.dkv_free, n_work - 1, &sh.p_half, g);
#pragma unroll
                    for (int part = 0; part < 2; ++part) {
                        if (part == 1) {
                            mbar_wait_warp(&sh.p_full, g & 1u, guard);
                            tc_fence_after();
                        }
#pragma unroll
                        for (int k4 = 0; k4 < 4; ++k4) {
                            const int ks = (k4 / 2) * 4 + part * 2 + (k4 % 2);     // k-steps {0,1,4,5} then {2,3,6,7}
                            if (leader) tc_mma_ts(tmem + Cfg::kDv, tmem + Cfg::kSt + (ks / 4) * 64 + (ks % 4) * 8, do_mn + mn_step(ks),
                                      idesc_nd_kb, n > 0 || part > 0 || k4 > 0);
                        }
                    }
                    if (leader) tc_commit(&sh.do_empty);
                    // S^T of the next tile
                    if (has_next) {
                        wait(2, &sh.q_full[nstage], (g + 1) / Cfg::kQStages, &sh.stat_full[(g + 1) & 1u], (g + 1) >> 1, &sh.q_full[nstage], 0);
                        issue_abt(tmem + Cfg::kSt, k_km, q_km0 + nstage * kStageStep);
                        if (leader) tc_mma_ss(tmem + Cfg::kSt, ones_s, stat0 + ((g + 1) & 1u) * kStatStep, idesc_abt, true);
                        if (leader) tc_commit(&sh.s_full);
                    }
                    // dQ tile = dS K  (A: dS^T read M-contiguous; B: K with head_dim contiguous)
                    mbar_wait_warp(&sh.ds_full, g & 1u, guard);
                    tc_fence_after();
#pragma unroll
                    for (int ks = 0; ks < kTile / 16; ++ks)
                        if (leader) tc_mma_ss(tmem + Cfg::kDp, ds_mn + mn_step(ks), k_mn + mn_step(ks), idesc_nd_mm, ks > 0);
                    if (leader) tc_commit(&sh.dq_full);
                    // dK += dS^T Q
#pragma unroll
                    for (int ks = 0; ks < kTile / 16; ++ks)
                        if (leader) tc_mma_ss(tmem + Cfg::kDk, ds_km + km_step(ks, 16384), q_mn0 + stage * kStageStep + mn_step(ks),
                                  idesc_nd_kb, n > 0 || ks > 0);
                    if (leader) tc_commit(&sh.q_empty[stage]);
                    if (leader) tc_commit(&sh.ds_free);
                    // dP^T of the next tile (its columns hold dQ until the drain warps have read it)
                    if (has_next) {
                        wait(2, &sh.do_full, g + 1, &sh.dq_free, g, &sh.do_full, 0);
                        issue_abt(tmem + Cfg::kDp, v_km, do_km);
                        if (leader) tc_mma_ss(tmem + Cfg::kDp, ones_d, stat0 + ((g + 1) & 1u) * kStatStep, idesc_abt, true);
                        if (leader) tc_commit(&sh.dp_full);
                        if (leader) tc_commit(&sh.stat_empty[(g + 1) & 1u]);
                    }
                    stage = nstage;
                }
                if (leader) tc_commit(&sh.dkv_full);
                if (leader) tc_commit(&sh.kv_empty[slot]);
                ++n_work;
            }
        }
    }
    } else if (warp < 8) {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 136;");
        // ------------------------------------------------- compute: P^T, dS^T, final dK / dV
        const int half = warp >> 2;                                  // which 64 query columns
        const int key_in_tile = (warp & 3) * 32 + lane;              // tensor-memory lane = key
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t st_tmem = tmem + lane_base + Cfg::kSt + half * 64;
        const uint32_t pt_tmem = tmem + lane_base + Cfg::kSt + half * 64;   // bf16 pairs, inside this group's own S^T columns
        const uint32_t dp_tmem = tmem + lane_base + Cfg::kDp + half * 64;
        uint8_t* ds_row = smem + Cfg::kOffDs + half * 16384;
        const uint64_t sc2 = pack_f32x2(p.scale_log2, p.scale_log2);
        uint32_t n_work = 0, g = 0;
        while (true) {
            const uint32_t slot = n_work & 1u;
            const bool got = mbar_wait_warp(&sh.work_full[slot], (n_work >> 1) & 1u, guard);
            if (!__all_sync(0xffffffffu, got)) break;
            const WorkItem w = sh.work[slot];
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.work_empty[slot]);
            if (w.len < 0) break;
            int first_q, n_q;
            q_range(w, first_q, n_q);
            const int key = w.blk * kTile + key_in_tile;
            const bool key_valid = key < w.len;
            const bool key_tail = (w.blk + 1) * kTile > w.len;

            if (p.bounds != nullptr && w.len <= kTile) {     // one tile pair, possibly several merged sequences
                compute_single_tile_item<CAUSAL>(sh, p, w, st_tmem, dp_tmem, ds_row, half, key_in_tile, g, guard);
                ++g;
                first_q = n_q;                                // nothing left for the loop below
            }
            for (int i = first_q; i < n_q; ++i, ++g) {
                const bool diag = CAUSAL && i == w.blk;
                float pf[64];
                mbar_wait_warp(&sh.s_full, g & 1u, guard);
                tc_fence_after();
                {
                    // all 64 scores of this thread's key row are requested before the single wait
                    uint32_t sr[64];
                    tmem_ld_x32(st_tmem, *reinterpret_cast<uint32_t(*)[32]>(&sr[0]));
                    tmem_ld_x32(st_tmem + 32, *reinterpret_cast<uint32_t(*)[32]>(&sr[32]));
                    tmem_wait_ld();
                    // the key is seen by the queries from `lo` of this thread's 64 on
                    const int lo = !key_valid ? 64 : diag ? key - (i * kTile + half * 64) : -64;
                    auto form_p = [&](auto masked) {
#pragma unroll
                        for (int c = 0; c < 2; ++c) {
                            // 32 query columns at a time: the dV product starts on the first chunk while the
                            // second is still being exponentiated
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
                            if (c == 0) {
                                tmem_wait_st();
                                tc_fence_before();
                                __syncwarp();
                                if (lane == 0) mbar_arrive(&sh.p_half);
                            }
                        }
                    };
                    // Masked tiles have a copy of the loop, with one select per element (before: a test of (key_valid, diag, key >
                    // query) on every element, in the one loop).  65536 tokens, 16 heads of 64: causal 300-token sequences 435 ->
                    // 408 us, 1200 736 -> 708, 4096 1802 -> 1768; without a causal mask 1200 1201 -> 1190, 4096 3352 -> 3295.  Scaling two
                    // scores per instruction: another 1 % (causal 512 402 -> 399, 1200 689 -> 680; dS formed that way: nothing).
                    if (key_tail || diag) form_p(std::true_type{});
                    else form_p(std::false_type{});
                }
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.p_full);

                // dS^T = P^T o (dP^T - D)
                mbar_wait_warp(&sh.dp_full, g & 1u, guard);
                if (g >= 1) mbar_wait_warp(&sh.ds_free, (g - 1) & 1u, guard);
                tc_fence_after();
                {
                    uint32_t dr[64];
                    tmem_ld_x32(dp_tmem, *reinterpret_cast<uint32_t(*)[32]>(&dr[0]));
                    tmem_ld_x32(dp_tmem + 32, *reinterpret_cast<uint32_t(*)[32]>(&dr[32]));
                    tmem_wait_ld();
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        uint32_t pk[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            pk[e] = pack_bf16x2(pf[c * 8 + 2 * e] * __uint_as_float(dr[c * 8 + 2 * e]),
                                                pf[c * 8 + 2 * e + 1] * __uint_as_float(dr[c * 8 + 2 * e + 1]));
                        *reinterpret_cast<uint4*>(ds_row + sw128_offset(key_in_tile, c)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    }
                }
                fence_async_smem();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.ds_full);
            }

            // item epilogue: dV and dK rows of this key block (each group writes half the columns)
            mbar_wait_warp(&sh.dkv_full, n_work & 1u, guard);
            tc_fence_after();
            const size_t tok = (size_t)w.tok0 + (size_t)key;
            const size_t out_off = tok * p.row_stride + w.head * p.head_dim + half * (kD / 2);
#pragma unroll
            for (int which = 0; which < 2; ++which) {
                const uint32_t src = tmem + lane_base + (which == 0 ? Cfg::kDv : Cfg::kDk) + half * (kD / 2);
                __nv_bfloat16* dst = (which == 0 ? p.dv : p.dk) + out_off;
                const float mul = which == 0 ? 1.0f : p.scale;
#pragma unroll
                for (int c = 0; c < kD / 64; ++c) {
                    uint32_t acc[32];
                    tmem_ld_x32(src + c * 32, acc);
                    tmem_wait_ld();
                    if (key_valid) {
#pragma unroll
                        for (int v4 = 0; v4 < 4; ++v4) {
                            uint4 val;
                            val.x = pack_bf16x2(__uint_as_float(acc[v4 * 8 + 0]) * mul, __uint_as_float(acc[v4 * 8 + 1]) * mul);
                            val.y = pack_bf16x2(__uint_as_float(acc[v4 * 8 + 2]) * mul, __uint_as_float(acc[v4 * 8 + 3]) * mul);
                            val.z = pack_bf16x2(__uint_as_float(acc[v4 * 8 + 4]) * mul, __uint_as_float(acc[v4 * 8 + 5]) * mul);
                            val.w = pack_bf16x2(__uint_as_float(acc[v4 * 8 + 6]) * mul, __uint_as_float(acc[v4 * 8 + 7]) * mul);
                            if (half * (kD / 2) + c * 32 + v4 * 8 < p.head_dim) *reinterpret_cast<uint4*>(dst + c * 32 + v4 * 8) = val;
                        }
                    }
                    __syncwarp();    // the next load is warp-wide
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.dkv_free);
            ++n_work;
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 136;");
        // ------------------------------------------------- dQ drain: tensor memory -> fp32 atomics
        const int q_in_tile = (warp & 3) * 32 + lane;               // warps 12-15 -> lane quarters 0-3
        const uint32_t dq_tmem = tmem + ((uint32_t)((warp & 3) * 32) << 16) + Cfg::kDp;
        uint32_t n_work = 0, g = 0;
        while (true) {
            const uint32_t slot = n_work & 1u;
            const bool got = mbar_wait_warp(&sh.work_full[slot], (n_work >> 1) & 1u, guard);
            if (!__all_sync(0xffffffffu, got)) break;
            const WorkItem w = sh.work[slot];
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.work_empty[slot]);
            if (w.len < 0) break;
            ++n_work;
            int first_q, n_q;
            q_range(w, first_q, n_q);
            for (int i = first_q; i < n_q; ++i, ++g) {
                mbar_wait_warp(&sh.dq_full, g & 1u, guard);
                tc_fence_after();
                // accumulator block of (tile, head) is [16][128 rows][4]: the 32 rows of a warp are
                // contiguous for a fixed column group, so each vector atomic covers whole sectors
                const int qrow = i * kTile + q_in_tile;
                float* dst = p.dq_acc + (((size_t)w.tile0 + i) * p.n_heads + w.head) * (size_t)(kTile * kD) + q_in_tile * 4;
                // read the whole tile first and release tensor memory at once: dP^T of the next tile waits
                // on it, while the atomics below may take as long as they like
                uint32_t acc[kD];
#pragma unroll
                for (int c = 0; c < kD / 32; ++c) tmem_ld_x32(dq_tmem + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&acc[c * 32]));
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sh.dq_free);
                if (w.len <= kTile) {
                    // the sequence's only tile pair: this is the whole dQ, no accumulation needed
                    if (qrow < w.len) {
                        __nv_bfloat16* out = p.dq + ((size_t)w.tok0 + qrow) * p.row_stride + w.head * p.head_dim;
#pragma unroll
                        for (int c = 0; c < kD / 8; ++c) {
                            uint4 val;
                            val.x = pack_bf16x2(__uint_as_float(acc[c * 8 + 0]) * p.scale, __uint_as_float(acc[c * 8 + 1]) * p.scale);
                            val.y = pack_bf16x2(__uint_as_float(acc[c * 8 + 2]) * p.scale, __uint_as_float(acc[c * 8 + 3]) * p.scale);
                            val.z = pack_bf16x2(__uint_as_float(acc[c * 8 + 4]) * p.scale, __uint_as_float(acc[c * 8 + 5]) * p.scale);
                            val.w = pack_bf16x2(__uint_as_float(acc[c * 8 + 6]) * p.scale, __uint_as_float(acc[c * 8 + 7]) * p.scale);
                            if (c * 8 < p.head_dim) *reinterpret_cast<uint4*>(out + c * 8) = val;
                        }
                    }
                } else {
                    const bool live = qrow < w.len;
                    if ((warp & 3) > 0) __nanosleep((warp & 3) * kRedStaggerNs + 64);
#pragma unroll
                    for (int c = 0; c < kD / 4; ++c) {
                        // only the columns that hold data are zeroed before and read afterwards (all 64 for head dimension 40: 1200
                        // tokens 1372 -> 1299 us, causal 16384 7523 -> 6533; 56 7588 -> 7217; 64 unchanged)
                        if (c * 4 >= p.head_dim) break;
                        if (live) red_add_v4(dst + c * (kTile * 4), __uint_as_float(acc[c * 4]), __uint_as_float(acc[c * 4 + 1]),
                                   __uint_as_float(acc[c * 4 + 2]), __uint_as_float(acc[c * 4 + 3]));
                        if ((c % kRedGroup) == kRedGroup - 1) __nanosleep(kRedSleepNs);
                    }
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (tid == 0) span_end(p.sched, 1);
    __syncwarp();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

template <bool CAUSAL>
static cudaError_t launch_one(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tdo,
                              const BwdParams& p, int n_ctas, cudaStream_t stream) {
    if (cudaError_t e = allow_smem<attn_bwd_kernel<CAUSAL>>(BwdCfg::kSmemBytes)) return e;
    return launch_dependent(attn_bwd_kernel<CAUSAL>, n_ctas, kBwdThreads, BwdCfg::kSmemBytes, stream, tq, tk, tv, tdo, p);
}

cudaError_t launch_attn_bwd(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& tdo,
                            const BwdParams& p, bool causal, int n_ctas, cudaStream_t stream) {
    return causal ? launch_one<true>(tq, tk, tv, tdo, p, n_ctas, stream) : launch_one<false>(tq, tk, tv, tdo, p, n_ctas, stream);
}

}  // namespace dcp
