// Forward and backward for work items that are a single tile: a (virtual) sequence of at most 128 tokens and one head.
//
// Such an item is a chain (load, S, softmax, product, store) with nothing to overlap inside it, a few microseconds long
// for 0.1-0.2 us of memory traffic per SM: what it needs is other items in flight on the same SM.  The multi-tile kernels
// hold one CTA per SM (all of tensor memory, 200 KB of shared memory), so they ran such items one after the other.
// Here a CTA is small: one compute thread per row (two in the backward); tensor memory is reused within the item, so that
//
//     forward,  head_dim <= 64:   128 columns,  48 KB  -> 4 CTAs per SM         head_dim > 64:  256 columns,  96 KB -> 2 CTAs
//     backward, head_dim <= 64:   256 columns, 112 KB  -> 2 CTAs per SM         head_dim > 64:  512 columns, 192 KB -> 1 CTA
//
// and the next item's loads start as soon as an operand's buffer is free.  Queries are rows (lanes) in both directions.
// The backward's per-query terms, -lse/scale and -D_i = -sum_c dO_ic O_ic, enter S and dP as in the multi-tile kernels: by
// a K = 16 product of a [128 x 16] tile of bf16 parts with a tile of ones.  The compute warps form that tile from O and dO in
// shared memory while the products that S and dP begin with run, so these items need no pre kernel, no fp32 accumulator
// and no conversion pass: q, k, v, o, dO in, dq, dk, dv out.  (D_i = sum_j P_ij dP_ij from registers would save reading o: 512
// texts of 16-200 tokens, 16 heads of 64, training step 417 us instead of 427.  But it is another number wherever o
// is not this call's own P V: rounded to bf16, or the output over more keys than these, with the lse to match.)
//
// Several short sequences may share the tile: row i sees the keys [first, end) of its own sequence, and
// a warp skips the 32-key chunks that none of its rows sees.
//
// Roles (forward, 192 threads): warps 0-3 compute, warp 4 TMA producer, warp 5 MMA issue; backward: see there.  Items are
// dealt round robin: they cost about the same, the longest first.
//
// Backward in tensor memory: S and dP (128 columns each); one pass over both gives P and dS -> shared memory; then
// dV = P^T dO, dK = dS^T Q, dQ = dS K overwrite S and dP (P^T and dS^T are the same bytes read with keys contiguous as the
// M dimension).
//
// Every sum here has the order that the multi-tile kernels give it, so an item's results are the same bits whichever kernel
// the batch sends it to.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "attn_kernels.h"
#include "launch.h"
#include "row_terms.cuh"
#include "sched.cuh"
#include "sm100_ptx.cuh"

namespace dcp {
namespace {

constexpr int kTileThreads = 192;
constexpr int kBoxBytes = kTile * 128;               // 128 rows of 64 bf16 columns

struct TileItem {
    int tok0, len, head, seq;
};

// Item i of the single-tile part of the work list: its sequences come after the longer ones, n_heads items each.
__device__ __forceinline__ TileItem tile_item(const SchedView& s, const int32_t* cu, uint32_t first_seq, uint32_t i, int n_heads) {
    TileItem w;
    w.seq = s.order[first_seq + i / (uint32_t)n_heads];
    w.head = (int)(i % (uint32_t)n_heads);
    w.tok0 = cu[w.seq];
    w.len = cu[w.seq + 1] - w.tok0;
    return w;
}

// Keys [lo, hi) that a row sees; none for rows past the end.  A row of a merged sequence (`members` = the caller's
// boundaries) finds its own sequence by bisection among the members: a few cached loads while the item's products run.
// (A table of every token's range, as the multi-tile kernels read it, takes a launch to fill.)
__device__ __forceinline__ void row_keys(const TileItem& w, int row, const SchedView& s, const int32_t* __restrict__ members, bool causal,
                                         int& lo, int& hi) {
    lo = hi = 0;
    if (row < w.len) {
        hi = w.len;
        if (members) {
            int a = s.vfirst[w.seq], b = s.vfirst[w.seq + 1];
            if (b - a > 1) {                         // the last member that starts at or before this token: it is not empty
                while (b - a > 1) {
                    const int mid = (a + b) >> 1;
                    if (members[mid] <= w.tok0 + row) a = mid;
                    else b = mid;
                }
                lo = members[a] - w.tok0;
                hi = members[a + 1] - w.tok0;
            }
        }
        if (causal && hi > row + 1) hi = row + 1;
    }
}
// the keys lo..hi-1 of chunk c as bits
__device__ __forceinline__ uint32_t chunk_bits(int lo, int hi, int c) {
    const int a = max(lo - c * 32, 0), b = min(hi - c * 32, 32);
    return b <= a ? 0u : (0xffffffffu >> (32 - b)) & (0xffffffffu << a);
}

template <int D>
__device__ __forceinline__ void load_tile(uint8_t* dst, const CUtensorMap* map, uint64_t* bar, int head, int row) {
#pragma unroll
    for (int b = 0; b < D / 64; ++b) tma_load_3d(dst + b * kBoxBytes, map, bar, b * 64, head, row);
}

// 32 rows of an accumulator (this warp's lanes), W columns: tensor memory -> x mul -> bf16 -> 2 KB of staging in shared
// memory (rows of 64 bytes, 16-byte chunks swizzled) -> global memory, eight rows per instruction.  The accumulator has
// been read when it returns.
template <int W>
__device__ __forceinline__ void store_rows(__nv_bfloat16* out, int64_t row_stride, int cols, uint8_t* stage, uint32_t tmem, float mul,
                                           int rows_left) {
    const int lane = threadIdx.x & 31;
    const int sub = lane >> 2, chunk = lane & 3;
#pragma unroll
    for (int c = 0; c < W / 32; ++c) {
        uint32_t acc[32];
        tmem_ld_x32(tmem + c * 32, acc);
        tmem_wait_ld();
#pragma unroll
        for (int v4 = 0; v4 < 4; ++v4) {
            uint4 val;
            val.x = pack_bf16x2(__uint_as_float(acc[v4 * 8 + 0]) * mul, __uint_as_float(acc[v4 * 8 + 1]) * mul);
            val.y = pack_bf16x2(__uint_as_float(acc[v4 * 8 + 2]) * mul, __uint_as_float(acc[v4 * 8 + 3]) * mul);
            val.z = pack_bf16x2(__uint_as_float(acc[v4 * 8 + 4]) * mul, __uint_as_float(acc[v4 * 8 + 5]) * mul);
            val.w = pack_bf16x2(__uint_as_float(acc[v4 * 8 + 6]) * mul, __uint_as_float(acc[v4 * 8 + 7]) * mul);
            *reinterpret_cast<uint4*>(stage + lane * 64 + ((v4 ^ ((lane >> 1) & 3)) << 4)) = val;
        }
        __syncwarp();
        const int col = c * 32 + chunk * 8;
        __nv_bfloat16* dst = out + (size_t)sub * row_stride + col;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int row = i * 8 + sub;
            const uint4 val = *reinterpret_cast<const uint4*>(stage + row * 64 + ((chunk ^ ((row >> 1) & 3)) << 4));
            if (row < rows_left && col < cols) *reinterpret_cast<uint4*>(dst + (size_t)(i * 8) * row_stride) = val;
        }
        __syncwarp();                                // the staging rows have been read
    }
}

// ------------------------------------------------------------------------------------------------- forward
struct FwdTileShared {
    uint64_t qk_full, v_full, s_full, p_full, o_full, v_free, o_free;
    uint32_t tmem_base, abort_flag;
};

template <int D>
__global__ void __launch_bounds__(kTileThreads, D == 64 ? 4 : 2)
tile_fwd_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ FwdParams p, bool causal) {
    constexpr int kTileBytes = kTile * D * 2;
    constexpr uint32_t kCols = D == 64 ? 128 : 256, kColO = 64;      // P (packed) in columns 0-63 of S, O from 64 on
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t *sQ = smem, *sK = smem + kTileBytes, *sV = smem + 2 * kTileBytes;
    FwdTileShared& sh = *reinterpret_cast<FwdTileShared*>(smem + 3 * kTileBytes);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const WaitGuard guard{&sh.abort_flag, &p.sched.hdr->status};
    if (tid == 0) {
        for (uint64_t* b : {&sh.qk_full, &sh.v_full, &sh.s_full, &sh.o_full}) mbar_init(b, 1);
        for (uint64_t* b : {&sh.p_full, &sh.v_free, &sh.o_free}) mbar_init(b, 4);
        sh.abort_flag = (smem_u32(smem) & 1023u) != 0 ? 1u : 0u;     // the swizzled layouts need an aligned base
        fence_mbar_init();
    }
    if (warp == 4) {
        tmem_alloc(&sh.tmem_base, kCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh.tmem_base;
    grid_trigger();
    grid_wait();
    if (tid == 0 && sh.abort_flag) atomicMax(&p.sched.hdr->status, (uint32_t)kStatusBadSmemAlign);
    const uint32_t first_seq = p.sched.hdr->n_long_seqs;
    const uint32_t n = sh.abort_flag ? 0u : p.sched.hdr->n_items - p.sched.hdr->n_long_items;
    if (tid == 0) span_merge_begin(p.sched, 0);

    if (warp == 4) {
        if (lane == 0) {
            uint32_t k = 0;
            for (uint32_t i = blockIdx.x; i < n; i += gridDim.x, ++k) {
                const TileItem w = tile_item(p.sched, p.cu_seqlens, first_seq, i, p.n_heads);
                if (k >= 1) mbar_wait(&sh.s_full, (k - 1) & 1u, guard);
                mbar_expect_tx(&sh.qk_full, 2 * kTileBytes);
                load_tile<D>(sQ, &tmap_q, &sh.qk_full, w.head, w.tok0);
                load_tile<D>(sK, &tmap_k, &sh.qk_full, w.head, w.tok0);
                if (k >= 1) mbar_wait(&sh.v_free, (k - 1) & 1u, guard);
                mbar_expect_tx(&sh.v_full, kTileBytes);
                load_tile<D>(sV, &tmap_v, &sh.v_full, w.head, w.tok0);
            }
        }
    } else if (warp == 5) {
        const bool leader = elect_one();
        const int n_ks = (p.head_dim + 15) >> 4;                     // steps of 16 columns that hold data
        constexpr uint32_t idesc_s = make_idesc_bf16(128, 128, false, false);
        const uint32_t idesc_o = make_idesc_bf16(128, n_ks * 16, false, true);
        const uint64_t q_km = make_sdesc_sw128(smem_u32(sQ), 16, 1024), k_km = make_sdesc_sw128(smem_u32(sK), 16, 1024);
        const uint64_t v_mn = make_sdesc_sw128(smem_u32(sV), kBoxBytes, 1024);
        uint32_t k = 0;
        for (uint32_t i = blockIdx.x; i < n; i += gridDim.x, ++k) {
            mbar_wait_all(&sh.qk_full, k & 1u, guard);
            if (k >= 1) mbar_wait_all(&sh.o_free, (k - 1) & 1u, guard);
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks) {
                const uint64_t off = (uint64_t)(((ks / 4) * kBoxBytes + (ks % 4) * 32) >> 4);
                if (leader && ks < n_ks) tc_mma_ss(tmem, q_km + off, k_km + off, idesc_s, ks > 0);
            }
            if (leader) tc_commit(&sh.s_full);
            mbar_wait_all(&sh.v_full, k & 1u, guard);
            mbar_wait_all(&sh.p_full, k & 1u, guard);
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
                if (leader) tc_mma_ts(tmem + kColO, tmem + ks * 8, v_mn + (uint64_t)((ks * 2048) >> 4), idesc_o, ks > 0);
            if (leader) tc_commit(&sh.o_full);
        }
    } else {
        const uint32_t my = tmem + ((uint32_t)(warp * 32) << 16);
        const int row = tid;                                         // query row
        const uint64_t sc2 = pack_f32x2(p.scale_log2, p.scale_log2);
        TileItem w{0, 0, 0, 0};
        int lo = 0, hi = 0;
        if (blockIdx.x < n) {
            w = tile_item(p.sched, p.cu_seqlens, first_seq, blockIdx.x, p.n_heads);
            row_keys(w, row, p.sched, p.members, causal, lo, hi);
        }
        uint32_t k = 0;
        for (uint32_t i = blockIdx.x; i < n; i += gridDim.x, ++k) {
            // chunks that some row of the warp sees
            const int wlo = __reduce_min_sync(0xffffffffu, hi > lo ? lo : kTile), whi = __reduce_max_sync(0xffffffffu, hi);
            mbar_wait_warp(&sh.s_full, k & 1u, guard);
            tc_fence_after();
            float m = -INFINITY;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (c * 32 < whi && c * 32 + 32 > wlo) {
                    uint32_t s[32];
                    tmem_ld_x32(my + c * 32, s);
                    tmem_wait_ld();
                    const uint32_t bits = chunk_bits(lo, hi, c);
                    float mx[4] = {m, m, m, m};
#pragma unroll
                    for (int e = 0; e < 32; ++e)
                        if (bits & (1u << e)) mx[e & 3] = fmaxf(mx[e & 3], __uint_as_float(s[e]));
                    m = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
                }
            }
            if (hi <= lo) m = 0.f;
            const float neg_m = -m * p.scale_log2;
            const uint64_t nm2 = pack_f32x2(neg_m, neg_m);
            uint64_t sum2[2] = {0ull, 0ull};         // keys 0, 4, .. | 1, 5, .. and 2, 6, .. | 3, 7, ..
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                uint32_t pk[16];
                if (c * 32 < whi && c * 32 + 32 > wlo) {
                    uint32_t s[32];
                    tmem_ld_x32(my + c * 32, s);
                    tmem_wait_ld();
                    const uint32_t bits = chunk_bits(lo, hi, c);
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        float x0, x1;
                        unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(s[2 * e]), __uint_as_float(s[2 * e + 1])), sc2, nm2), x0, x1);
                        const float p0 = bits & (1u << (2 * e)) ? fast_exp2(x0) : 0.f;
                        const float p1 = bits & (2u << (2 * e)) ? fast_exp2(x1) : 0.f;
                        sum2[e & 1] = add_f32x2(sum2[e & 1], pack_f32x2(p0, p1));
                        pk[e] = pack_bf16x2(p0, p1);
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 16; ++e) pk[e] = 0u;
                }
                tmem_st_x16(my + c * 16, pk);        // over columns of S that have been read
            }
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.p_full);
            const TileItem cur = w;
            const bool valid = row < cur.len;
            float l;
            {
                float a0, a1, b0, b1;
                unpack_f32x2(sum2[0], a0, a1);
                unpack_f32x2(sum2[1], b0, b1);
                l = (a0 + a1) + (b0 + b1);
            }
            const float inv_l = l > 0.f ? 1.0f / l : 0.f;
            if (valid) p.lse[(size_t)cur.head * p.total_tokens + cur.tok0 + row] = m * p.scale + __logf(l);
            if (i + gridDim.x < n) {                 // the next item's keys, while the product runs
                w = tile_item(p.sched, p.cu_seqlens, first_seq, i + gridDim.x, p.n_heads);
                row_keys(w, row, p.sched, p.members, causal, lo, hi);
            }
            mbar_wait_warp(&sh.o_full, k & 1u, guard);
            tc_fence_after();
            // a row's 1 / l goes with its thread: scaled here, so the rows leave unscaled from the staging buffer
            uint8_t* stage = sV + warp * 4096;       // V has been read by the product
#pragma unroll
            for (int half = 0; half < D / 64; ++half) {
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    uint32_t acc[32];
                    tmem_ld_x32(my + kColO + half * 64 + c * 32, acc);
                    tmem_wait_ld();
#pragma unroll
                    for (int v4 = 0; v4 < 4; ++v4) {
                        uint4 val;
                        val.x = pack_bf16x2(__uint_as_float(acc[v4 * 8 + 0]) * inv_l, __uint_as_float(acc[v4 * 8 + 1]) * inv_l);
                        val.y = pack_bf16x2(__uint_as_float(acc[v4 * 8 + 2]) * inv_l, __uint_as_float(acc[v4 * 8 + 3]) * inv_l);
                        val.z = pack_bf16x2(__uint_as_float(acc[v4 * 8 + 4]) * inv_l, __uint_as_float(acc[v4 * 8 + 5]) * inv_l);
                        val.w = pack_bf16x2(__uint_as_float(acc[v4 * 8 + 6]) * inv_l, __uint_as_float(acc[v4 * 8 + 7]) * inv_l);
                        *reinterpret_cast<uint4*>(stage + half * kBoxBytes + sw128_offset((uint32_t)lane, (uint32_t)(c * 4 + v4))) = val;
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.o_free);
            const int chunk = lane & 7, rows_left = cur.len - warp * 32;
            __nv_bfloat16* out = p.o + ((size_t)cur.tok0 + warp * 32 + (lane >> 3)) * p.row_stride + cur.head * p.head_dim + chunk * 8;
#pragma unroll
            for (int half = 0; half < D / 64; ++half) {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int r = j * 4 + (lane >> 3);
                    const uint4 val = *reinterpret_cast<const uint4*>(stage + half * kBoxBytes + sw128_offset((uint32_t)r, (uint32_t)chunk));
                    if (r < rows_left && half * 64 + chunk * 8 < p.head_dim)
                        *reinterpret_cast<uint4*>(out + half * 64 + (size_t)(j * 4) * p.row_stride) = val;
                }
            }
            fence_async_smem();                      // the next V is written by TMA after these reads
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.v_free);
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (tid == 0) span_merge_end(p.sched, 0);
    if (warp == 4) tmem_dealloc(tmem, kCols);
}

// ------------------------------------------------------------------------------------------------- backward
// 320 threads: warps 0-3 take the keys (and output columns) of the first half, warps 4-7 those of the second, so that a
// thread holds half a row; warp 8 TMA producer, warp 9 MMA issue.  An item is one chain per CTA, and tensor memory allows
// two CTAs per SM: with whole rows and four warps it took 10 us, half of it in this arithmetic and in the stores, and V,
// loaded only after the stores had staged through its buffer, another 1.5 us (512 texts of 16-200 tokens, 16 heads of 64:
// this kernel 124 -> 101 us, the training step 441 -> 422; 112 and 427 since it reads o).
constexpr int kTileBwdThreads = 320;

struct BwdTileShared {
    uint64_t in_full, o_full, terms_full, s_full, ds_full, dv_full, dk_full, dq_full, item_free;
    uint32_t tmem_base, abort_flag;
};

template <int D>
struct BwdTileCfg {
    static constexpr int kTileBytes = kTile * D * 2;
    static constexpr int kOffQ = 0, kOffK = kTileBytes, kOffDo = 2 * kTileBytes;
    static constexpr int kOffP = 3 * kTileBytes;             // V (and O) until dP is there, then P (32 KB)
    static constexpr int kOffDs = kOffP + 32768;             // dS, then staging (2 KB per warp)
    // until S and dP are there, dS's buffer holds the per-query terms and the ones beside the staging
    static constexpr int kOffTerms = kOffDs + 16384;
    static constexpr int kOffOnes = kOffTerms + kTermTileBytes;      // ones, zeros, ones (2 KB each), see the pair kernel
    // O: in the half of P's buffer that V leaves free (two CTAs per SM have no other room), or beside
    static constexpr int kOffO = D == 64 ? kOffP + kTileBytes : kOffDs + 32768;
    static constexpr int kOffCtl = kOffDs + 32768 + (D == 64 ? 0 : kTileBytes);
    static constexpr int kSmemBytes = kOffCtl + 128;
    static constexpr uint32_t kCols = D == 64 ? 256 : 512;
    static constexpr uint32_t kColS = 0, kColDp = 128, kColDv = 0, kColDk = D, kColDq = 2 * D;
};
static_assert(sizeof(BwdTileShared) <= 128, "control block must fit its slot");

template <int D>
__global__ void __launch_bounds__(kTileBwdThreads, D == 64 ? 2 : 1)
tile_bwd_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ CUtensorMap tmap_o,
                const __grid_constant__ CUtensorMap tmap_do, const __grid_constant__ BwdParams p, bool causal) {
    using Cfg = BwdTileCfg<D>;
    extern __shared__ __align__(1024) uint8_t smem[];
    BwdTileShared& sh = *reinterpret_cast<BwdTileShared*>(smem + Cfg::kOffCtl);
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const WaitGuard guard{&sh.abort_flag, &p.sched.hdr->status};
    if (tid == 0) {
        for (uint64_t* b : {&sh.in_full, &sh.o_full, &sh.s_full, &sh.dv_full, &sh.dk_full, &sh.dq_full}) mbar_init(b, 1);
        for (uint64_t* b : {&sh.terms_full, &sh.ds_full, &sh.item_free}) mbar_init(b, 8);
        sh.abort_flag = (smem_u32(smem) & 1023u) != 0 ? 1u : 0u;
        fence_mbar_init();
    }
    if (warp == 8) {
        tmem_alloc(&sh.tmem_base, Cfg::kCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sh.tmem_base;
    grid_trigger();
    grid_wait();
    if (tid == 0 && sh.abort_flag) atomicMax(&p.sched.hdr->status, (uint32_t)kStatusBadSmemAlign);
    const uint32_t first_seq = p.sched.hdr->n_long_seqs;
    const uint32_t n = sh.abort_flag ? 0u : p.sched.hdr->n_items - p.sched.hdr->n_long_items;
    if (tid == 0) span_merge_begin(p.sched, 1);

    if (warp == 8) {
        if (lane == 0) {
            uint32_t k = 0;
            for (uint32_t i = blockIdx.x; i < n; i += gridDim.x, ++k) {
                const TileItem w = tile_item(p.sched, p.cu_seqlens, first_seq, i, p.n_heads);
                if (k >= 1) mbar_wait(&sh.dv_full, (k - 1) & 1u, guard);     // (and the previous item's loads have completed)
                mbar_expect_tx(&sh.o_full, 2 * Cfg::kTileBytes);
                load_tile<D>(smem + Cfg::kOffO, &tmap_o, &sh.o_full, w.head, w.tok0);
                load_tile<D>(smem + Cfg::kOffDo, &tmap_do, &sh.o_full, w.head, w.tok0);
                mbar_expect_tx(&sh.in_full, 3 * Cfg::kTileBytes);
                load_tile<D>(smem + Cfg::kOffP, &tmap_v, &sh.in_full, w.head, w.tok0);      // the product has read P
                if (k >= 1) mbar_wait(&sh.dk_full, (k - 1) & 1u, guard);
                load_tile<D>(smem + Cfg::kOffQ, &tmap_q, &sh.in_full, w.head, w.tok0);
                if (k >= 1) mbar_wait(&sh.dq_full, (k - 1) & 1u, guard);
                load_tile<D>(smem + Cfg::kOffK, &tmap_k, &sh.in_full, w.head, w.tok0);
            }
        }
    } else if (warp == 9) {
        const bool leader = elect_one();
        const int n_ks = (p.head_dim + 15) >> 4;
        constexpr uint32_t idesc_s = make_idesc_bf16(128, 128, false, false);
        const uint32_t idesc_mm = make_idesc_bf16(128, n_ks * 16, true, true);      // dV, dK: A with M contiguous
        const uint32_t idesc_km = make_idesc_bf16(128, n_ks * 16, false, true);     // dQ
        const uint64_t q_km = make_sdesc_sw128(smem_u32(smem + Cfg::kOffQ), 16, 1024);
        const uint64_t k_km = make_sdesc_sw128(smem_u32(smem + Cfg::kOffK), 16, 1024);
        const uint64_t v_km = make_sdesc_sw128(smem_u32(smem + Cfg::kOffP), 16, 1024);
        const uint64_t do_km = make_sdesc_sw128(smem_u32(smem + Cfg::kOffDo), 16, 1024);
        const uint64_t q_mn = make_sdesc_sw128(smem_u32(smem + Cfg::kOffQ), kBoxBytes, 1024);
        const uint64_t k_mn = make_sdesc_sw128(smem_u32(smem + Cfg::kOffK), kBoxBytes, 1024);
        const uint64_t do_mn = make_sdesc_sw128(smem_u32(smem + Cfg::kOffDo), kBoxBytes, 1024);
        const uint64_t p_mn = make_sdesc_sw128(smem_u32(smem + Cfg::kOffP), kBoxBytes, 1024);
        const uint64_t ds_mn = make_sdesc_sw128(smem_u32(smem + Cfg::kOffDs), kBoxBytes, 1024);
        const uint64_t ds_km = make_sdesc_sw128(smem_u32(smem + Cfg::kOffDs), 16, 1024);
        const uint64_t terms = make_sdesc_nosw(smem_u32(smem + Cfg::kOffTerms), 2048, 128);
        const uint64_t ones_s = make_sdesc_nosw(smem_u32(smem + Cfg::kOffOnes), 2048, 128);
        const uint64_t ones_d = make_sdesc_nosw(smem_u32(smem + Cfg::kOffOnes + 2048), 2048, 128);
        auto km_step = [](int ks) -> uint64_t { return (uint64_t)(((ks / 4) * kBoxBytes + (ks % 4) * 32) >> 4); };
        auto mn_step = [](int ks) -> uint64_t { return (uint64_t)((ks * 2048) >> 4); };
        uint32_t k = 0;
        for (uint32_t i = blockIdx.x; i < n; i += gridDim.x, ++k) {
            // The operands, dO and the accumulators' columns (of the item before, once they have been read), each polled by a
            // lane of its own: the time to see a barrier is spent once.  One after the other: 1 to 2.5 % slower at head
            // dimension 64, 3 to 4 % at 72, the same at 128.  (The forward's two waits together: + 4 % on causal items of 128
            // tokens, - 3 to 0 % otherwise; left as they are.)
            const bool dout = lane == 1, free_cols = lane == 2 && k >= 1;
            mbar_wait_all(dout ? &sh.o_full : free_cols ? &sh.item_free : &sh.in_full, (free_cols ? k - 1 : k) & 1u, guard);
            tc_fence_after();
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks)
                if (leader && ks < n_ks) tc_mma_ss(tmem + Cfg::kColS, q_km + km_step(ks), k_km + km_step(ks), idesc_s, ks > 0);
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks)
                if (leader && ks < n_ks) tc_mma_ss(tmem + Cfg::kColDp, do_km + km_step(ks), v_km + km_step(ks), idesc_s, ks > 0);
            mbar_wait_all(&sh.terms_full, k & 1u, guard);
            if (leader) tc_mma_ss(tmem + Cfg::kColS, terms, ones_s, idesc_s, true);
            if (leader) tc_mma_ss(tmem + Cfg::kColDp, terms, ones_d, idesc_s, true);
            if (leader) tc_commit(&sh.s_full);
            mbar_wait_all(&sh.ds_full, k & 1u, guard);
            tc_fence_after();
#pragma unroll
            for (int k8 = 0; k8 < 8; ++k8) {                 // k-steps {0,1,4,5} then {2,3,6,7}, as the multi-tile kernel adds them
                const int ks = (k8 / 2 % 2) * 4 + (k8 / 4) * 2 + k8 % 2;
                if (leader) tc_mma_ss(tmem + Cfg::kColDv, p_mn + mn_step(ks), do_mn + mn_step(ks), idesc_mm, k8 > 0);
            }
            if (leader) tc_commit(&sh.dv_full);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
                if (leader) tc_mma_ss(tmem + Cfg::kColDk, ds_mn + mn_step(ks), q_mn + mn_step(ks), idesc_mm, ks > 0);
            if (leader) tc_commit(&sh.dk_full);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
                if (leader) tc_mma_ss(tmem + Cfg::kColDq, ds_km + km_step(ks), k_mn + mn_step(ks), idesc_km, ks > 0);
            if (leader) tc_commit(&sh.dq_full);
        }
    } else {
        const int half = warp >> 2, quarter = warp & 3;      // of the columns, of the rows
        const uint32_t my = tmem + ((uint32_t)(quarter * 32) << 16);
        const int row = quarter * 32 + lane;                 // query row
        uint8_t *p_row = smem + Cfg::kOffP + half * kBoxBytes, *ds_row = smem + Cfg::kOffDs + half * kBoxBytes;
        uint8_t* stage = smem + Cfg::kOffDs + warp * 2048;
        const uint64_t sc2 = pack_f32x2(p.scale_log2, p.scale_log2);
        const int t_row = warp * 16 + (lane & 15), t_role = lane >> 4;   // the row and which of its terms this thread stores
        TileItem w{0, 0, 0, 0};
        int lo = 0, hi = 0;
        float lse = 0.f;                                     // of t_row
        auto fetch = [&](uint32_t i) {
            w = tile_item(p.sched, p.cu_seqlens, first_seq, i, p.n_heads);
            row_keys(w, row, p.sched, p.members, causal, lo, hi);
            lse = t_row < w.len ? p.lse[(size_t)w.head * p.total_tokens + w.tok0 + t_row] : 0.f;
        };
        if (blockIdx.x < n) fetch(blockIdx.x);
        uint32_t k = 0;
        for (uint32_t i = blockIdx.x; i < n; i += gridDim.x, ++k) {
            // The buffer of dS is free here: this thread has seen dQ of the item before, the last product that reads it.
            for (int c = tid; c < 6144 / 16; c += 256)
                *reinterpret_cast<uint4*>(smem + Cfg::kOffOnes + c * 16) =
                    c / 128 == 1 ? make_uint4(0u, 0u, 0u, 0u) : make_uint4(0x3f803f80u, 0x00003f80u, 0u, 0u);   // 1,1 | 1,0 | 0..
            mbar_wait_warp(&sh.o_full, k & 1u, guard);
            {
                // the even (odd) chunks of eight columns of this row, added as the pre kernel's lanes add theirs
                float part[D / 16];
#pragma unroll
                for (int c = 0; c < D / 16; ++c) {
                    const int chunk = 2 * c + t_role;
                    const uint32_t at = (uint32_t)(chunk / 8) * kBoxBytes + sw128_offset((uint32_t)t_row, (uint32_t)(chunk % 8));
                    part[c] = chunk_dot(*reinterpret_cast<const uint4*>(smem + Cfg::kOffO + at),
                                        *reinterpret_cast<const uint4*>(smem + Cfg::kOffDo + at));
                }
#pragma unroll
                for (int s = D / 32; s > 0; s >>= 1) {
#pragma unroll
                    for (int c = 0; c < s; ++c) part[c] += part[c + s];
                }
                const float sum = part[0] + __shfl_xor_sync(0xffffffffu, part[0], 16);
                const bool live = t_row < w.len;
                const float none = t_role == 0 ? kNoRow : 0.f;
                store_term(smem + Cfg::kOffTerms, t_row, t_role, !live ? none : t_role == 0 ? -lse * p.inv_scale : -sum);
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.terms_full);
            const int wlo = __reduce_min_sync(0xffffffffu, hi > lo ? lo : kTile), whi = __reduce_max_sync(0xffffffffu, hi);
            mbar_wait_warp(&sh.s_full, k & 1u, guard);            // (the products have read V, the terms and the ones)
            tc_fence_after();
#pragma unroll 1
            for (int u = 0; u < 2; ++u) {
                const int c = half * 2 + u;
                const bool seen = c * 32 < whi && c * 32 + 32 > wlo;
                auto put = [&](int v4, const uint32_t (&pk)[4], const uint32_t (&ds)[4]) {
                    const uint32_t at = sw128_offset((uint32_t)row, (uint32_t)(u * 4 + v4));
                    *reinterpret_cast<uint4*>(p_row + at) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    *reinterpret_cast<uint4*>(ds_row + at) = make_uint4(ds[0], ds[1], ds[2], ds[3]);
                };
                if (seen) {
                    uint32_t s[32], dp[32];
                    tmem_ld_x32(my + Cfg::kColS + c * 32, s);
                    tmem_ld_x32(my + Cfg::kColDp + c * 32, dp);
                    tmem_wait_ld();
                    const uint32_t bits = chunk_bits(lo, hi, c);
                    // Of 64 columns every element is exponentiated and the mask selects afterwards: no branch around the
                    // exponential (- 1 to - 3 %; of 128 columns, one CTA per SM, + 0 to 1 %: there the mask comes first).
#pragma unroll
                    for (int v4 = 0; v4 < 4; ++v4) {
                        uint32_t pk[4], ds[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const int j = v4 * 8 + 2 * e;
                            float x0, x1;
                            unpack_f32x2(mul_f32x2(pack_f32x2(__uint_as_float(s[j]), __uint_as_float(s[j + 1])), sc2), x0, x1);
                            if constexpr (D == 64) {
                                x0 = fast_exp2(x0);
                                x1 = fast_exp2(x1);
                            }
                            const float p0 = bits & (1u << j) ? (D == 64 ? x0 : fast_exp2(x0)) : 0.f;
                            const float p1 = bits & (2u << j) ? (D == 64 ? x1 : fast_exp2(x1)) : 0.f;
                            pk[e] = pack_bf16x2(p0, p1);
                            ds[e] = pack_bf16x2(p0 * __uint_as_float(dp[j]), p1 * __uint_as_float(dp[j + 1]));
                        }
                        put(v4, pk, ds);
                    }
                } else {
                    const uint32_t zero[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                    for (int v4 = 0; v4 < 4; ++v4) put(v4, zero, zero);
                }
            }
            fence_async_smem();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.ds_full);
            const TileItem cur = w;
            if (i + gridDim.x < n) fetch(i + gridDim.x);
            constexpr int W = D / 2;                         // output columns of this warp
            const int rows_left = cur.len - quarter * 32, cols = p.head_dim - half * W;
            const size_t off = ((size_t)cur.tok0 + quarter * 32) * p.row_stride + (size_t)cur.head * p.head_dim + half * W;
            // (dV, dK: rows are keys.)  dS has been read when dQ is there, so its buffer stages what leaves; the next item's
            // operands are on their way meanwhile.
            mbar_wait_warp(&sh.dq_full, k & 1u, guard);
            tc_fence_after();
            store_rows<W>(p.dv + off, p.row_stride, cols, stage, my + Cfg::kColDv + half * W, 1.0f, rows_left);
            store_rows<W>(p.dk + off, p.row_stride, cols, stage, my + Cfg::kColDk + half * W, p.scale, rows_left);
            store_rows<W>(p.dq + off, p.row_stride, cols, stage, my + Cfg::kColDq + half * W, p.scale, rows_left);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh.item_free);
        }
    }
    __syncwarp();
    tc_fence_before();
    __syncthreads();
    if (tid == 0) span_merge_end(p.sched, 1);
    if (warp == 8) tmem_dealloc(tmem, Cfg::kCols);
}

template <int D>
cudaError_t launch_fwd(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const FwdParams& p, bool causal,
                       unsigned n_ctas, cudaStream_t stream) {
    constexpr int kSmem = 3 * kTile * D * 2 + 128;
    if (cudaError_t e = allow_smem<tile_fwd_kernel<D>>(kSmem)) return e;
    return launch_dependent(tile_fwd_kernel<D>, n_ctas, kTileThreads, kSmem, stream, tq, tk, tv, p, causal);
}
template <int D>
cudaError_t launch_bwd(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& to,
                       const CUtensorMap& tdo, const BwdParams& p, bool causal, unsigned n_ctas, cudaStream_t stream) {
    if (cudaError_t e = allow_smem<tile_bwd_kernel<D>>(BwdTileCfg<D>::kSmemBytes)) return e;
    return launch_dependent(tile_bwd_kernel<D>, n_ctas, kTileBwdThreads, BwdTileCfg<D>::kSmemBytes, stream, tq, tk, tv, to, tdo, p,
                            causal);
}

unsigned tile_grid(int n_sms, int per_sm, int32_t n_seqs, int32_t n_heads) {
    const long long most = (long long)n_seqs * n_heads, full = (long long)n_sms * per_sm;
    return (unsigned)(most < full ? most : full);
}

}  // namespace

cudaError_t launch_tile_fwd(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const FwdParams& p, bool causal,
                            int n_sms, cudaStream_t stream) {
    return p.head_dim > 64 ? launch_fwd<128>(tq, tk, tv, p, causal, tile_grid(n_sms, 2, p.sched.n_seqs, p.n_heads), stream)
                           : launch_fwd<64>(tq, tk, tv, p, causal, tile_grid(n_sms, 4, p.sched.n_seqs, p.n_heads), stream);
}

cudaError_t launch_tile_bwd(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const CUtensorMap& to,
                            const CUtensorMap& tdo, const BwdParams& p, bool causal, int n_sms, cudaStream_t stream) {
    return p.head_dim > 64 ? launch_bwd<128>(tq, tk, tv, to, tdo, p, causal, tile_grid(n_sms, 1, p.sched.n_seqs, p.n_heads), stream)
                           : launch_bwd<64>(tq, tk, tv, to, tdo, p, causal, tile_grid(n_sms, 2, p.sched.n_seqs, p.n_heads), stream);
}

}  // namespace dcp
