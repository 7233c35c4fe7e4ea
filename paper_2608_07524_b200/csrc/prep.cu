// Work-list construction and the two small memory-bound backward helpers.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "attn_kernels.h"
#include "launch.h"
#include "row_terms.cuh"
#include "sched.cuh"
#include "sm100_ptx.cuh"

namespace dcp {

constexpr int kRankInKernelMax = 256;     // above this many sequences the rank sort runs over several CTAs (rank_kernel)
// The one-CTA kernels below have NT threads: 256 for batches of at most 256 sequences, whose time is the barriers and
// dependent loads of a CTA (fewer warps, cheaper barriers), 1024 for larger ones.

template <int NT> __device__ inline uint32_t block_exclusive_scan(uint32_t v, uint32_t* scratch, uint32_t* total);
template <int NT> __device__ inline int block_exclusive_max_scan(int v, int* scratch);

// Merging of short sequences into virtual sequences of at most 128 tokens.  One CTA.
//
// A sequence is "short" if length <= max_short (empty ones included).  Two local rules say when a short
// sequence joins the virtual sequence of its short predecessor:
//   rule 0: both START in the same window of `window` = 129 - max_short packed positions, so a virtual
//           sequence spans at most (window - 1) + max_short = 128 tokens;
//   rule 1: the predecessor's first and this sequence's last token lie in the same ALIGNED window of 128
//           positions, so a virtual sequence lies inside one such window (sequences that cross a window
//           boundary stay alone).
// Rule 0 fills tiles well when sequences are much shorter than 64 tokens, rule 1 when they are close to
// 64 and aligned (64-token sequences pair up exactly, which their start windows of 65 almost never allow).
// Both are local (whether a sequence starts a virtual sequence depends on it and its predecessor only),
// so heads are found in parallel and compacted with a scan; the kernel counts the heads under both rules
// and keeps the rule that gives fewer (rule 1 only if the batch has no empty sequence, which keeps the
// bound on the number of tiles that sizes the workspace: it is derived for rule 0).
// Outputs: vcu[0..n_v] = boundaries of the virtual sequences, vcu[n_v+1..n_seqs] = total_tokens
// (empty padding, so that vcu is a valid boundary array of n_seqs sequences); hdr->n_vseq = n_v;
// hdr->merge_rule = the rule used; vfirst[v] = first input sequence of virtual sequence v, vfirst[n_v] = n_seqs;
// vstart[i] (unless null) = first token of the virtual sequence that input sequence i belongs to (read by
// bounds_kernel, so that no thread there has to walk back over a run, which under rule 0 may hold any number of
// empty sequences).
__device__ __forceinline__ bool merge_is_head(const int32_t* __restrict__ cu, int i, int32_t max_short, uint32_t rule) {
    if (i == 0 || cu[i + 1] - cu[i] > max_short || cu[i] - cu[i - 1] > max_short) return true;
    if (rule == 0) {
        const int window = kTile + 1 - max_short;
        return cu[i - 1] / window != cu[i] / window;
    }
    return cu[i - 1] / kTile != (cu[i + 1] - 1) / kTile;
}

template <int NT>
__global__ void __launch_bounds__(NT) merge_kernel(const int32_t* __restrict__ cu, int32_t n_seqs, int32_t total_tokens,
                                                   int32_t max_short, WorkspaceHeader* hdr, int32_t* vcu, int32_t* vfirst, int32_t* vstart) {
    __shared__ uint32_t scratch[33];
    grid_trigger();
    grid_wait();
    const int tid = threadIdx.x;
    const int per = (n_seqs + NT - 1) / NT;
    const int begin = min(tid * per, n_seqs), end = min(begin + per, n_seqs);
    // The boundaries come from the caller and index everything that follows: they must start at 0, never
    // decrease and end at total_tokens.  If not, the status word says so and every sequence is made empty,
    // which turns the rest of the call into no-ops.  This kernel is the first of a call.
    int bad = (tid == 0 && (cu[0] != 0 || cu[n_seqs] != total_tokens)) ? 1 : 0;
    for (int i = begin; i < end; ++i) bad |= cu[i + 1] < cu[i] ? 1 : 0;
    bad = __syncthreads_or(bad);
    if (tid == 0) header_begin_call(hdr, bad != 0);
    if (bad) {
        for (int i = tid; i <= n_seqs; i += NT) vcu[i] = 0;
        if (tid == 0) hdr->n_vseq = 0;
        return;
    }
    uint32_t local0 = 0, local1 = 0, n_v0 = 0, n_v1 = 0;
    int empty = 0;
    for (int i = begin; i < end; ++i) {
        local0 += merge_is_head(cu, i, max_short, 0) ? 1u : 0u;
        local1 += merge_is_head(cu, i, max_short, 1) ? 1u : 0u;
        empty |= cu[i + 1] == cu[i] ? 1 : 0;
    }
    empty = __syncthreads_or(empty);
    const uint32_t run0 = block_exclusive_scan<NT>(local0, scratch, &n_v0);
    const uint32_t run1 = block_exclusive_scan<NT>(local1, scratch, &n_v1);
    const uint32_t rule = (!empty && n_v1 < n_v0) ? 1u : 0u;
    const uint32_t n_v = rule ? n_v1 : n_v0;
    uint32_t run = rule ? run1 : run0;
    if (tid == 0) {
        hdr->n_vseq = n_v;
        hdr->merge_rule = rule;
        vfirst[n_v] = n_seqs;
    }
    int last_head = -1;
    for (int i = begin; i < end; ++i)
        if (merge_is_head(cu, i, max_short, rule)) {
            vcu[run] = cu[i];
            vfirst[run++] = i;
            last_head = i;
        }
    for (uint32_t i = n_v + tid; i <= (uint32_t)n_seqs; i += NT) vcu[i] = total_tokens;
    if (!vstart) return;
    // head of the run each sequence belongs to: the last head at or before it (sequence 0 is always one)
    int cur = block_exclusive_max_scan<NT>(last_head, reinterpret_cast<int*>(scratch));
    for (int i = begin; i < end; ++i) {
        if (merge_is_head(cu, i, max_short, rule)) cur = i;
        vstart[i] = cu[cur];
    }
}

// One warp per input sequence of at most 128 tokens, over as many CTAs as needed: bounds[t] for
// each of its tokens t = (first, end) position of the sequence relative to the start of its virtual
// sequence, one byte each (the lanes write consecutive tokens).  merge_kernel has left that start in vstart[].
__global__ void __launch_bounds__(256) bounds_kernel(const int32_t* __restrict__ cu, int32_t n_seqs,
                                                     const WorkspaceHeader* __restrict__ hdr,
                                                     const int32_t* __restrict__ vstart, uint16_t* __restrict__ bounds) {
    grid_trigger();
    grid_wait();
    const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= n_seqs || hdr->call_bad) return;      // merge_kernel found the boundaries inconsistent
    const int32_t a = cu[i], b = cu[i + 1];
    if (b == a || b - a > kTile) return;
    const int32_t v0 = vstart[i];
    const uint16_t packed = (uint16_t)((a - v0) | ((b - v0) << 8));
    for (int32_t t = a + lane; t < b; t += 32) bounds[t] = packed;
}

// Rank sort, eight threads per sequence over as many CTAs as needed: order[] = sequence ids sorted by
// (length descending, id ascending).  Used on its own for batches of more than kRankInKernelMax
// sequences (one CTA doing it for a thousand sequences takes 37 us, one thread per sequence 13 us, this 5 us); small
// batches do the same loop inside prep_kernel and save the launch.  Sequences
// from *n_live on (if given) are empty padding: they keep their own index as rank and are not
// compared against.
constexpr int kRankPerCta = 32, kRankSlices = 8;
__global__ void __launch_bounds__(256) rank_kernel(const int32_t* __restrict__ cu, int32_t n_seqs,
                                                  const uint32_t* __restrict__ n_live_ptr, int32_t* order) {
    __shared__ int32_t len_tile[1024];
    grid_trigger();
    grid_wait();
    const int n_live = n_live_ptr ? min((int)*n_live_ptr, n_seqs) : n_seqs;
    const int slice = threadIdx.x & (kRankSlices - 1), i = blockIdx.x * kRankPerCta + threadIdx.x / kRankSlices;
    if ((int)blockIdx.x * kRankPerCta >= n_live) {     // a whole block of padding
        if (slice == 0 && i < n_seqs) order[i] = i;
        return;
    }
    const int32_t len_i = i < n_seqs ? cu[i + 1] - cu[i] : 0;
    int rank = slice == 0 && i > n_live ? i - n_live : 0;      // padding before i, all of length 0 like i itself
    for (int j0 = 0; j0 < n_live; j0 += 1024) {
        const int cnt = min(1024, n_live - j0);
        __syncthreads();
        for (int t = threadIdx.x; t < cnt; t += 256) len_tile[t] = cu[j0 + t + 1] - cu[j0 + t];
        __syncthreads();
        for (int t = slice; t < cnt; t += kRankSlices) {
            const int32_t len_j = len_tile[t];
            rank += (len_j > len_i) || (len_j == len_i && j0 + t < i);
        }
    }
#pragma unroll
    for (int s = 1; s < kRankSlices; s <<= 1) rank += __shfl_xor_sync(0xffffffffu, rank, s);
    if (slice == 0 && i < n_seqs) order[rank] = i;
}

// Exclusive prefix sum of one value per thread over a CTA of NT threads; *total receives
// the sum.  scratch holds 33 words.
template <int NT>
__device__ inline uint32_t block_exclusive_scan(uint32_t v, uint32_t* scratch, uint32_t* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, s);
        if (lane >= s) incl += t;
    }
    __syncthreads();                       // scratch may still be read from an earlier call
    if (lane == 31) scratch[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const uint32_t w = lane < NT / 32 ? scratch[lane] : 0u;
        uint32_t wi = w;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, wi, s);
            if (lane >= s) wi += t;
        }
        scratch[lane] = wi - w;
        if (lane == 31) scratch[32] = wi;
    }
    __syncthreads();
    *total = scratch[32];
    return scratch[warp] + incl - v;
}

// Exclusive running maximum of one value per thread (in thread order) over a CTA of NT
// threads; -1 where nothing precedes.  scratch holds 33 words.
template <int NT>
__device__ inline int block_exclusive_max_scan(int v, int* scratch) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, s);
        if (lane >= s) incl = max(incl, t);
    }
    __syncthreads();                       // scratch may still be read from an earlier scan
    if (lane == 31) scratch[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int wi = lane < NT / 32 ? scratch[lane] : -1;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, wi, s);
            if (lane >= s) wi = max(wi, t);
        }
        scratch[lane] = wi;                // inclusive over warps
    }
    __syncthreads();
    int excl = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) excl = -1;
    if (warp > 0) excl = max(excl, scratch[warp - 1]);
    return excl;
}

// One CTA.  order[] as above (computed here if `ranked` is 0, by rank_kernel if 1; 2 keeps the input
// order, a measurement aid); prefix[i] = number of work items of the
// first i sequences in that order, where a sequence of length L contributes
// ceil(L / rows_per_block) * n_heads items; tile_prefix[b] = 128-row tiles before sequence b.
// Sequences from *n_live_ptr on (if given) are empty padding and sorted last: only the live ones
// are scanned, the rest get the totals.
template <int NT>
__global__ void __launch_bounds__(NT) prep_kernel(const int32_t* __restrict__ cu, int32_t n_seqs,
                                                  const uint32_t* __restrict__ n_live_ptr, int32_t rows_per_block, int32_t n_heads,
                                                  WorkspaceHeader* hdr, int32_t* order, uint32_t* prefix, uint32_t* tile_prefix,
                                                  int ranked, int32_t total_tokens, uint32_t tile_capacity, int32_t long_min_len, int32_t max_len,
                                                  SmSpan* spans, int which, bool clear_spans) {
    __shared__ uint32_t scratch[33];
    __shared__ int32_t len_sh[NT];
    unsigned long long now = 0;
    if (threadIdx.x == 0) now = global_timer_ns();    // before the wait: reading the timer takes long enough to see in a small call
    grid_trigger();
    grid_wait();
    const int tid = threadIdx.x;
    const int n_live = n_live_ptr ? min((int)*n_live_ptr, n_seqs) : n_seqs;
    if (clear_spans)
        for (int i = tid; i < kMaxSms; i += NT) spans[which * kMaxSms + i] = SmSpan{~0ull, 0ull};
    if (!n_live_ptr) {
        // no merge_kernel ran before: check the caller's boundaries here (see merge_kernel)
        int bad = (tid == 0 && (cu[0] != 0 || cu[n_seqs] != total_tokens)) ? 1 : 0;
        for (int i = tid; i < n_seqs; i += NT) bad |= cu[i + 1] < cu[i] ? 1 : 0;
        bad = __syncthreads_or(bad);
        if (tid == 0) header_begin_call(hdr, bad != 0);
        if (bad) {
            for (int i = tid; i <= n_seqs; i += NT) { prefix[i] = 0; tile_prefix[i] = 0; }
            for (int i = tid; i < n_seqs; i += NT) order[i] = i;
            if (tid == 0) hdr->n_items = hdr->n_long_items = hdr->n_long_seqs = hdr->work_counter = 0;
            return;
        }
    }
    if (ranked == 2) {
        // input order: the long sequences, the others, the empty ones
        const int chunk = (n_live + NT - 1) / NT;
        const int from = min(tid * chunk, n_live), to = min(from + chunk, n_live);
        auto kind = [&](int i) { const int32_t len = cu[i + 1] - cu[i]; return len >= long_min_len ? 0 : len > 0 ? 1 : 2; };
        uint32_t cnt[2] = {0, 0}, all[2], at[3];
        for (int i = from; i < to; ++i)
            if (kind(i) < 2) ++cnt[kind(i)];
        at[0] = block_exclusive_scan<NT>(cnt[0], scratch, &all[0]);
        at[1] = block_exclusive_scan<NT>(cnt[1], scratch, &all[1]);
        at[2] = all[0] + all[1] + (uint32_t)from - at[0] - at[1];
        at[1] += all[0];
        for (int i = from; i < to; ++i) order[at[kind(i)]++] = i;
        for (int i = n_live + tid; i < n_seqs; i += NT) order[i] = i;
    } else if (!ranked) {                             // n_seqs <= kRankInKernelMax: one sequence per thread
        len_sh[tid] = tid < n_seqs ? cu[tid + 1] - cu[tid] : -1;
        __syncthreads();
        if (tid < n_seqs) {
            const int32_t len_i = len_sh[tid];
            int rank = 0;
            for (int j = 0; j < n_seqs; ++j) {
                const int32_t len_j = len_sh[j];
                rank += (len_j > len_i) || (len_j == len_i && j < tid);
            }
            order[rank] = tid;
        }
    }
    __syncthreads();
    // exclusive scan of item counts over the sorted order: contiguous chunk per thread
    const int per = (n_live + NT - 1) / NT;
    const int begin = min(tid * per, n_live), end = min(begin + per, n_live);
    auto items_of = [&](int pos) -> uint32_t {
        const int s = order[pos];
        const int32_t len = cu[s + 1] - cu[s];
        return (uint32_t)((len + rows_per_block - 1) / rows_per_block) * (uint32_t)n_heads;
    };
    uint32_t local = 0, total = 0;
    int unforeseen = 0;
    for (int i = begin; i < end; ++i) {
        local += items_of(i);
        unforeseen |= cu[order[i] + 1] - cu[order[i]] > max_len ? 1 : 0;
    }
    uint32_t run = block_exclusive_scan<NT>(local, scratch, &total);
    if (tid == 0) {
        hdr->spans_from[which] = now;
        hdr->n_items = total;
        hdr->work_counter = 0;
        hdr->n_long_items = hdr->n_long_seqs = 0;
    }
    __syncthreads();
    auto is_long = [&](int pos) { return pos < n_live && cu[order[pos] + 1] - cu[order[pos]] >= long_min_len; };
    for (int i = begin; i < end; ++i) {
        prefix[i] = run;
        run += items_of(i);
        if (is_long(i) && !is_long(i + 1)) {              // they come first in the order
            hdr->n_long_items = run;
            hdr->n_long_seqs = i + 1;
        }
    }
    for (int i = n_live + tid; i <= n_seqs; i += NT) prefix[i] = total;
    // tile_prefix[b] = number of 128-row tiles of sequences 0..b-1 (input order): same two-level scan
    auto tiles_of = [&](int b) -> uint32_t { return (uint32_t)((cu[b + 1] - cu[b] + kTile - 1) / kTile); };
    local = 0;
    for (int i = begin; i < end; ++i) local += tiles_of(i);
    run = block_exclusive_scan<NT>(local, scratch, &total);
    unforeseen = __syncthreads_or(unforeseen);
    if (total > tile_capacity || unforeseen) {
        // more tiles than the workspace was sized for, or a sequence longer than the launched kernels take: max_seqlen was
        // understated (the bound on merged runs relies on it).  Nothing may index the per-tile storage: no items, no tiles.
        for (int i = tid; i <= n_seqs; i += NT) tile_prefix[i] = 0;
        if (tid == 0) {
            hdr->n_items = hdr->n_long_items = 0;
            atomicMax(&hdr->status, (uint32_t)kStatusBadLengths);
        }
        return;
    }
    for (int i = begin; i < end; ++i) {
        tile_prefix[i] = run;
        run += tiles_of(i);
    }
    for (int i = n_live + tid; i <= n_seqs; i += NT) tile_prefix[i] = total;
}

int prep_launches(int32_t n_seqs, bool merge, bool table, bool input_order) {
    return (n_seqs > kRankInKernelMax && !input_order ? 2 : 1) + (merge ? 1 : 0) + (merge && table && n_seqs > 0 ? 1 : 0);
}

cudaError_t launch_prep(const int32_t* cu_seqlens, int32_t n_seqs, int32_t total_tokens, int32_t max_seqlen,
                        int32_t rows_per_block, int32_t n_heads, const SchedView& sched, bool merge, uint16_t* bounds,
                        uint32_t tile_capacity, bool input_order, int32_t long_min_len, int32_t max_len, int which, bool clear_spans,
                        cudaStream_t stream) {
    const int32_t* cu = cu_seqlens;
    const uint32_t* n_live = nullptr;
    const bool small = n_seqs <= 256;
    if (merge) {                                        // merge short sequences; everything below sees vcu
        const int32_t max_short = max_seqlen < kMergeMaxLen ? (max_seqlen > 0 ? max_seqlen : 1) : kMergeMaxLen;
        // order[] is not needed until the ranking below: until then it carries each sequence's run start, which the
        // table's kernel reads.  That launch is 4 us of a call's chain, so only calls whose kernels read the table have it
        int32_t* vstart = bounds ? const_cast<int32_t*>(sched.order) : nullptr;
        if (cudaError_t e = launch_dependent(small ? merge_kernel<256> : merge_kernel<1024>, 1, small ? 256 : 1024, 0, stream, cu_seqlens,
                                             n_seqs, total_tokens, max_short, sched.hdr, const_cast<int32_t*>(sched.vcu),
                                             const_cast<int32_t*>(sched.vfirst), vstart))
            return e;
        if (bounds && n_seqs > 0)
            if (cudaError_t e = launch_dependent(bounds_kernel, (n_seqs + 7) / 8, 256, 0, stream, cu_seqlens, n_seqs, sched.hdr, vstart,
                                                 bounds))
                return e;
        cu = sched.vcu;
        n_live = &sched.hdr->n_vseq;
    }
    const int ranked = input_order ? 2 : (n_seqs > kRankInKernelMax ? 1 : 0);
    if (ranked == 1)
        if (cudaError_t e = launch_dependent(rank_kernel, (n_seqs + kRankPerCta - 1) / kRankPerCta, 256, 0, stream, cu, n_seqs, n_live,
                                             const_cast<int32_t*>(sched.order)))
            return e;
    return launch_dependent(small ? prep_kernel<256> : prep_kernel<1024>, 1, small ? 256 : 1024, 0, stream, cu, n_seqs, n_live,
                            rows_per_block, n_heads, sched.hdr, const_cast<int32_t*>(sched.order), const_cast<uint32_t*>(sched.prefix),
                            const_cast<uint32_t*>(sched.tile_prefix), ranked, total_tokens, tile_capacity, long_min_len, max_len,
                            sched.spans, which, clear_spans);
}

// A (128-row tile, head) block of the backward helpers.
struct BlockRef {
    uint32_t tile, head;
    int row0, len, tok0;        // first row inside the sequence, the sequence's length and first token
};

// Where the helpers find their blocks.  tiles_per_item > 0: in the work list's sequences of more than one tile, which come
// first in it, tiles_per_item tiles to an item; heads vary fastest, so that CTAs running at the same time share memory
// pages.  0: in all tiles of the batch, in input order.  Going through all tiles of a batch of short sequences, nine
// tenths of them to be skipped after a search, took longer than the work (512 sequences of 16-200 tokens, head_dim 64: pre
// kernel 51 -> 40 us, post 33 -> 29; with only the rows inside the sequences zeroed and read, 35 and 25).
struct BlockList {
    const int32_t* cu;
    const int32_t* order;
    const uint32_t* prefix;
    const uint32_t* tile_prefix;
    const WorkspaceHeader* hdr;
    int32_t n_seqs, n_heads, tiles_per_item;

    __device__ __forceinline__ uint32_t size() const {
        return tiles_per_item > 0 ? hdr->n_long_items * (uint32_t)tiles_per_item : tile_prefix[n_seqs] * (uint32_t)n_heads;
    }
    // Called by converged warps: the lanes probe 32 places at a time, two rounds of loads for a thousand sequences where a
    // binary search by every thread took ten dependent ones (512 sequences of 16-200 tokens: pre kernel 55 -> 47 us, post
    // 41 -> 30).  The post kernel looks the NEXT block up while the current block's loads are in flight.
    __device__ __forceinline__ BlockRef find(uint32_t idx) const {
        const int lane = threadIdx.x & 31;
        const bool listed = tiles_per_item > 0;
        const uint32_t* const start = listed ? prefix : tile_prefix;
        const uint32_t scale = listed ? (uint32_t)tiles_per_item : (uint32_t)n_heads;
        int lo = 0, hi = listed ? (int)hdr->n_long_seqs : n_seqs;   // the last place whose blocks start at or before idx
        while (hi - lo > 1) {
            const int step = (hi - lo + 31) >> 5, probe = lo + lane * step;
            const uint32_t below = __ballot_sync(0xffffffffu, probe < hi && start[probe] * scale <= idx);
            lo += (__popc(below) - 1) * step;   // lane 0 probes lo itself, which is below
            hi = min(lo + step, hi);
        }
        const int seq = listed ? order[lo] : lo;
        const uint32_t local = idx - start[lo] * scale, in_seq = local / (uint32_t)n_heads;
        BlockRef r;
        r.head = local % (uint32_t)n_heads;
        r.tile = tile_prefix[seq] + in_seq;
        r.row0 = (int)in_seq * kTile;
        r.tok0 = cu[seq];
        r.len = cu[seq + 1] - r.tok0;
        return r;
    }
};

// ---------------------------------------------------------------------------------------------
// Backward helper 1.  For every (128-row tile, head) it writes a [128 rows x 16] bf16 tile holding,
// per query row, -lse/scale (columns 0-2) and -D_i = -sum_c dO_ic O_ic (columns 8-10), each split
// into three bf16 parts whose sum carries 24 bits; the main kernel adds them to its score and dP
// accumulators with a K=16 MMA against a tile of ones.  Rows past the sequence end get -1e30 and 0,
// which makes their probabilities vanish without masking.  The tile is stored in the MMA's shared-
// memory layout (8x8 core matrices; column halves 2048 bytes apart) and is 4 KB-aligned, so one bulk
// copy fetches it.  Also zeroes the fp32 dQ accumulator blocks of sequences longer than direct_len, one key block of the main
// kernel (shorter ones get their dQ written directly by it), the columns that hold data.  HBM-bound.  Zeroing behind a
// pass's loads, head_dim's columns instead of D, and the loads in flight below (us before and after, 65536 tokens x 16 heads): 64
// columns 112 -> 101, 72 columns 195 -> 140, 128 columns 215 -> 190 (5.8 TB/s); text batch 251 -> 227, 2-D model's spatial axis
// 386 -> 353, of 72 370 -> 267.
constexpr int kPreCtas = 6;      // per SM: 40 registers a thread
template <int D>
__global__ void __launch_bounds__(256, kPreCtas) bwd_pre_kernel(const __nv_bfloat16* __restrict__ o,
                                                      const __nv_bfloat16* __restrict__ d_o, const float* __restrict__ lse,
                                                      const BlockList list, __nv_bfloat16* __restrict__ stats,
                                                      float* __restrict__ dq_acc, size_t dq_acc_vec4,
                                                      int32_t total_tokens, int32_t n_heads, int32_t head_dim,
                                                      int64_t row_stride, float inv_scale, int32_t direct_len) {
    grid_trigger();
    grid_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t n_blocks = list.size();
    for (uint32_t idx = blockIdx.x; idx < n_blocks; idx += gridDim.x) {
        // (looking the next block's tile up while this block's loads are in flight, as the post kernel does, made
        // this kernel slower: 0.39 -> 0.44 ms on 131072 tokens x 16 heads)
        const BlockRef ref = list.find(idx);
        const int row0 = ref.row0, len = ref.len, tok0 = ref.tok0;
        if (row0 >= len) continue;                       // an item's second tile may lie past the end
        const uint32_t t = ref.tile, h = ref.head, blk = t * (uint32_t)n_heads + h;
        // this (tile, head) block of the dQ accumulator; a sequence of a single key block needs none (the main kernel holds
        // its whole dQ and writes it directly).  The main kernel adds to no other rows or columns than these.
        float4* acc_blk = reinterpret_cast<float4*>(dq_acc) + (size_t)blk * (kTile * D / 4);
        const bool zero = len > direct_len && (size_t)(blk + 1) * (kTile * D / 4) <= dq_acc_vec4;
        {
        uint8_t* out = reinterpret_cast<uint8_t*>(stats) + ((size_t)t * n_heads + h) * kTermTileBytes;
        // Half a warp reads a row with 16-byte loads (D = 128; a quarter warp for D = 64), so that a warp
        // instruction covers 2 (4) rows; a warp takes 4 (8) rows per pass with four loads of 16 bytes in flight per
        // lane.  The kernel waits on HBM latency: bytes in flight are what it runs on, and six CTAs of 40 registers have more
        // of them than four of 64 with twice the loads per lane (eight loads, four CTAs: 7 to 14 % slower; 16, two: 38 %;
        // two, eight: 7 %).
        constexpr int kLanesPerRow = D / 8;                 // 16 or 8
        constexpr int kRowsPerInst = 32 / kLanesPerRow;     // 2 or 4
        constexpr int kU = 2;                               // row groups in flight per lane
        const int sub = lane / kLanesPerRow, col = (lane % kLanesPerRow) * 8;
        const bool lane_live = col < head_dim;
        const int lane_col = lane_live ? col : 0;
        for (int r0 = warp * kRowsPerInst * kU; r0 < kTile; r0 += 8 * kRowsPerInst * kU) {
            uint4 a[kU], b[kU];
            float nl[kU], acc[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                const int r = r0 + u * kRowsPerInst + sub;
                a[u] = make_uint4(0u, 0u, 0u, 0u);
                b[u] = make_uint4(0u, 0u, 0u, 0u);
                nl[u] = kNoRow;
                if (row0 + r < len) {
                    const size_t tok = (size_t)tok0 + row0 + r;
                    // rows hold head_dim <= D columns; lanes past them re-read column 0 and drop it, so that the
                    // loads stay unconditional
                    const size_t row = tok * (size_t)row_stride + (size_t)h * head_dim + lane_col;
                    a[u] = *reinterpret_cast<const uint4*>(o + row);
                    b[u] = *reinterpret_cast<const uint4*>(d_o + row);
                    if (!lane_live) a[u] = make_uint4(0u, 0u, 0u, 0u);
                    if (lane % kLanesPerRow == 0) nl[u] = -lse[(size_t)h * total_tokens + tok] * inv_scale;
                }
            }
            // Behind the loads, which would queue behind these stores.  (Unrolled, the loop costs registers, and with them
            // resident CTAs: + 70 %.)
            if (zero) {
                constexpr int kPer = 8 * kRowsPerInst * kU * D / 4;
                const int z0 = (r0 - warp * kRowsPerInst * kU) * D / 4;
                for (int e = z0 + threadIdx.x; e < z0 + kPer; e += blockDim.x)
                    if (e % kTile < len - row0 && e / kTile * 4 < head_dim) acc_blk[e] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
                float sum = chunk_dot(a[u], b[u]);
#pragma unroll
                for (int sft = kLanesPerRow / 2; sft > 0; sft >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, sft);
                acc[u] = sum;
            }
            // the first lane of a row's group writes its lse chunk, the second its D chunk
            const int role = lane % kLanesPerRow;
            if (role < 2) {
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    const int r = r0 + u * kRowsPerInst + sub;
                    store_term(out, r, role, role == 0 ? nl[u] : -acc[u]);     // every lane of the group holds the row's sum
                }
            }
        }
        }
    }
}

cudaError_t launch_bwd_pre(const __nv_bfloat16* o, const __nv_bfloat16* d_o, const float* lse, const int32_t* cu_seqlens,
                           const SchedView& sched, __nv_bfloat16* stats, float* dq_acc, size_t dq_acc_elems,
                           int32_t total_tokens, int32_t n_heads, int32_t head_dim, int64_t row_stride, float scale,
                           int32_t tiles_per_item, int32_t direct_len, int n_sms, cudaStream_t stream) {
    // as many CTAs as are resident, or twice as many (ragged batches, whose blocks are not alike: text batch 0.977 -> 0.970 of
    // the time before), no more than (tile, head) blocks the batch can have
    const size_t most = max_tiles(total_tokens, sched.n_seqs) * (size_t)n_heads, full = (size_t)n_sms * kPreCtas * (head_dim > 64 ? 2 : 1);
    const unsigned blocks = (unsigned)(most < full ? most : full);
    const BlockList list{cu_seqlens, sched.order, sched.prefix, sched.tile_prefix, sched.hdr, sched.n_seqs, n_heads, tiles_per_item};
    return launch_dependent(head_dim > 64 ? bwd_pre_kernel<128> : bwd_pre_kernel<64>, blocks, 256, 0, stream, o, d_o, lse, list, stats,
                            dq_acc, dq_acc_elems / 4, total_tokens, n_heads, head_dim, row_stride, 1.0f / scale, direct_len);
}

// Backward helper 2: dq[T, H, d] = bf16(scale * dq_acc).  dq_acc holds, per (tile, head), a block
// [d/4][128 rows][4 floats]; a CTA reads one block with coalesced 16-byte loads, transposes it in
// shared memory as bf16 and writes whole rows.  Rows past the sequence end are skipped, and so are
// sequences of at most direct_len tokens, whose dQ the main kernel has already written.  A thread's eight loads of a pass lie
// a constant distance apart, columns past head_dim are not read, and the grid is one wave of resident CTAs (us before and after,
// 65536 tokens x 16 heads): 64 columns 75 -> 68, 72 columns 127 -> 91, 128 columns 148 -> 130; text batch 178 -> 160, 2-D
// model's spatial axis 253 -> 222.
constexpr int kPostCtas = 4;     // per SM: 64 registers a thread, 35 KB of shared memory
template <int D>
__global__ void __launch_bounds__(256, kPostCtas) bwd_post_kernel(const float* __restrict__ dq_acc, __nv_bfloat16* __restrict__ dq,
                                                       const BlockList list, int32_t n_heads, int32_t head_dim, int64_t row_stride,
                                                       float scale, int32_t direct_len) {
    constexpr int kRowBytes = D * 2 + 16;                    // padded row of bf16
    __shared__ __align__(16) uint8_t tile[kTile * kRowBytes];
    grid_trigger();
    grid_wait();
    const uint32_t n_blocks = list.size();
    if (blockIdx.x >= n_blocks) return;
    BlockRef ref = list.find(blockIdx.x), ref_next = ref;
    for (uint32_t idx = blockIdx.x; idx < n_blocks; idx += gridDim.x, ref = ref_next) {
        const uint32_t t = ref.tile, h = ref.head;
        const bool more = idx + gridDim.x < n_blocks;
        const int row0 = ref.row0, len = ref.len;
        const int rows = min(kTile, len - row0);
        if (len <= direct_len || row0 >= len) {          // a single key block: the main kernel has written dq itself
            if (more) ref_next = list.find(idx + gridDim.x);
            continue;
        }
        const float4* src = reinterpret_cast<const float4*>(dq_acc + ((size_t)t * n_heads + h) * (kTile * D));
        // eight 16-byte loads in flight per thread before the first use (the kernel waits on HBM latency), and the
        // next block's tile is looked up while the first eight are in flight; columns past head_dim hold nothing
        const int r = threadIdx.x % kTile, half = threadIdx.x / kTile;
#pragma unroll
        for (int i0 = 0; i0 < D / 8; i0 += 8) {
            if (i0 * 8 >= head_dim) break;
            float4 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (r < rows && (2 * (i0 + u) + half) * 4 < head_dim) v[u] = src[(i0 + u) * 256 + threadIdx.x];
            if (i0 == 0 && more) ref_next = list.find(idx + gridDim.x);
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int c4 = 2 * (i0 + u) + half;
                if (r >= rows || c4 * 4 >= head_dim) continue;
                __nv_bfloat162 lo2 = __floats2bfloat162_rn(v[u].x * scale, v[u].y * scale);
                __nv_bfloat162 hi2 = __floats2bfloat162_rn(v[u].z * scale, v[u].w * scale);
                uint2 pk;
                pk.x = *reinterpret_cast<uint32_t*>(&lo2);
                pk.y = *reinterpret_cast<uint32_t*>(&hi2);
                *reinterpret_cast<uint2*>(tile + r * kRowBytes + c4 * 8) = pk;
            }
        }
        __syncthreads();
        const int kChunks = head_dim * 2 / 16;               // 16-byte chunks per stored row (head_dim <= D columns)
        for (int e = threadIdx.x; e < rows * kChunks; e += blockDim.x) {
            const int r = e / kChunks, c = e % kChunks;
            const uint4 v = *reinterpret_cast<const uint4*>(tile + r * kRowBytes + c * 16);
            __nv_bfloat16* out = dq + ((size_t)ref.tok0 + row0 + r) * (size_t)row_stride + (size_t)h * head_dim;
            reinterpret_cast<uint4*>(out)[c] = v;
        }
        __syncthreads();
    }
}

cudaError_t launch_bwd_post(const float* dq_acc, __nv_bfloat16* dq, const int32_t* cu_seqlens, const SchedView& sched,
                            int32_t total_tokens, int32_t n_heads, int32_t head_dim, int64_t row_stride, float scale,
                            int32_t tiles_per_item, int32_t direct_len, int n_sms, cudaStream_t stream) {
    const size_t most = max_tiles(total_tokens, sched.n_seqs) * (size_t)n_heads;
    const unsigned blocks = most < (size_t)n_sms * kPostCtas ? (unsigned)most : (unsigned)n_sms * kPostCtas;
    const BlockList list{cu_seqlens, sched.order, sched.prefix, sched.tile_prefix, sched.hdr, sched.n_seqs, n_heads, tiles_per_item};
    return launch_dependent(head_dim > 64 ? bwd_post_kernel<128> : bwd_post_kernel<64>, blocks, 256, 0, stream, dq_acc, dq, list,
                            n_heads, head_dim, row_stride, scale, direct_len);
}

}  // namespace dcp
