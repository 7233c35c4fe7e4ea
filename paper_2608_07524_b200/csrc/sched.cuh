// Workspace layout and the length-aware work list shared by the forward and backward kernels.
//
// The paper's subject is load imbalance caused by widely varying sequence lengths (Section 2.3);
// on one GPU the same problem shows up as SMs idling while one long sequence finishes.  The work
// list therefore orders sequences longest first, and persistent CTAs pull items from it through a
// global atomic counter, so the cheap items of short sequences fill the tail.
//
// Very short sequences (a 2-D model's temporal axis has 1-13 tokens per sequence) would each
// occupy a whole 128-row tile.  Runs of consecutive short sequences are therefore merged into
// "virtual sequences" of at most 128 tokens that the kernels treat as one tile with a
// block-diagonal mask: the work list is built over the virtual boundaries `vcu` (a subsequence of
// cu_seqlens, padded with empty sequences), and a per-token table gives, for tokens of virtual
// sequences of at most 128 tokens, the range of positions the token's own sequence covers.  (Only the multi-tile
// kernels read that table, and only when they take such items: the single-tile kernels search cu_seqlens, see attn_tile.cu.)
#pragma once
#include <cstdint>

#include "item_order.h"

namespace dcp {

constexpr int kTile = 128;            // rows of a Q tile / keys of a K,V tile
constexpr int kFwdRowsPerItem = 256;  // a forward work item is two Q tiles of one (sequence, head), or one where items are few
constexpr int kMergeMaxLen = 64;      // sequences longer than this are never merged with their neighbours

// Status codes a kernel may leave in the workspace's status word (0 = no error).
enum : uint32_t {
    kStatusOk = 0,
    kStatusWaitTimeout = 1,
    kStatusBadSmemAlign = 2,
    kStatusBadLengths = 3     // cu_seqlens disagrees with the sizes the caller declared; nothing was computed
};

// First bytes of every workspace.  `status` must stay at offset 0 (dcp_query_status reads it).
// The status word is sticky: kernels only ever raise it (atomicMax), so a failure of any call on this
// workspace stays visible until dcp_query_status has reported and cleared it.  A workspace needs no
// initialisation by the caller: the first kernel of a call that does not find `magic` treats the
// header as fresh memory and clears the status word itself.
constexpr uint32_t kHeaderMagic0 = 0x64637031u, kHeaderMagic1 = 0x9e3779b9u;
constexpr int kCheckCtas = 16;        // CTAs of the short-sequence path's check kernel, at most
constexpr int kMaxSms = 256;          // SMs whose time span the header area can record
struct WorkspaceHeader {
    uint32_t status;        // 0 = ok, else the highest kStatus* code a kernel has left since the last query
    uint32_t work_counter;  // items claimed beyond the workers' first ones
    uint32_t n_items;       // items in the list
    uint32_t n_vseq;        // virtual sequences that are not padding
    uint32_t merge_rule;    // which of the two merging rules built them (see merge_kernel)
    uint32_t call_bad;      // this call's boundaries were inconsistent (reset by every call)
    uint32_t magic[2];      // kHeaderMagic0/1 once the header has been initialised
    uint32_t n_long_items;  // items of the sequences of more than one tile, which come first in the list; the single-tile
    uint32_t n_long_seqs;   // kernels take the rest.  (Both 0 where one kernel takes the whole list.)  And those sequences
    uint32_t check_bad[16]; // short-sequence path: whether a CTA of the check kernel found this call's boundaries inconsistent
    unsigned long long spans_from[2];     // when the list of the last forward / backward was built; 0: it recorded no spans
    uint32_t pad[34];
};
static_assert(sizeof(WorkspaceHeader) == 256, "header is 256 bytes");

#ifdef __CUDACC__
// Run by one thread of the first kernel of every call: a header that does not carry the magic words is
// fresh memory, whose status word means nothing yet.  Afterwards the status word is only ever raised.
__device__ __forceinline__ void header_begin_call(WorkspaceHeader* hdr, bool bad) {
    if (hdr->magic[0] != kHeaderMagic0 || hdr->magic[1] != kHeaderMagic1) {
        hdr->status = kStatusOk;
        hdr->spans_from[0] = hdr->spans_from[1] = 0ull;
        hdr->magic[0] = kHeaderMagic0;
        hdr->magic[1] = kHeaderMagic1;
    }
    hdr->call_bad = bad ? 1u : 0u;
    if (bad) atomicMax(&hdr->status, (uint32_t)kStatusBadLengths);
}
#endif

// When the first persistent CTA of the forward (slot 0) or the backward's main kernels (slot 1) on an SM started and when the
// last one there ran out of work, in nanoseconds of the GPU's global timer (what begins before spans_from is not this
// call's).  Their spread over the SMs is the single-GPU form of the paper's imbalance ratio (Section 2.3, Section 4.2): with
// a good work order every SM ends within one item of the others.  By SM, because a call may have two main kernels, of one to
// four CTAs per SM: the multi-tile kernels, one CTA on every SM, store; the single-tile kernels that follow them merge theirs
// in, and where these are alone prep_kernel has cleared the slot.
struct SmSpan {
    unsigned long long begin_ns, end_ns;
};
constexpr size_t kSpanBytes = 2 * kMaxSms * sizeof(SmSpan);      // 8 KB right after the header

// After the header and the span table: int32 order[n_seqs] (sequence ids, longest first, ties by id),
// uint32 prefix[n_seqs + 1] (items before the i-th sequence of `order`),
// uint32 tile_prefix[n_seqs + 1] (128-row tiles before sequence b, in input order) and
// int32 vcu[n_seqs + 1] (virtual sequence boundaries) and int32 vfirst[n_seqs + 1] (first input sequence of each virtual
// one); the last two are unused when sequences are not merged.
// All of these are indexed by VIRTUAL sequence; `cu` is the boundary array the kernels read
// (vcu, or the caller's cu_seqlens when merging is off).
struct SchedView {
    WorkspaceHeader* hdr;
    SmSpan* spans;          // [2][kMaxSms]
    const int32_t* order;
    const uint32_t* prefix;
    const uint32_t* tile_prefix;
    const int32_t* vcu;
    const int32_t* vfirst;
    int32_t n_seqs;
};

__host__ __device__ constexpr size_t sched_bytes(int32_t n_seqs) {
    return (sizeof(WorkspaceHeader) + kSpanBytes + sizeof(int32_t) * (size_t)n_seqs +
            4 * sizeof(uint32_t) * ((size_t)n_seqs + 1) + 255) & ~(size_t)255;
}

// Per-token table of the merged path: low byte = first position, high byte = one past the last
// position of the token's own sequence, both relative to the start of its virtual sequence.
__host__ __device__ constexpr size_t bounds_bytes(int32_t total_tokens) {
    return (sizeof(uint16_t) * (size_t)total_tokens + 255) & ~(size_t)255;
}

// Upper bound on the number of 128-row tiles of a packed batch: every (virtual) sequence may end in
// a partial tile.  After merging there are at most n_seqs virtual sequences and also at most
// 3 T / 65 + 2: one starts at sequence 0, at a sequence longer than kMergeMaxLen (at most T / 65 of
// those), right after such a sequence, or where the window changes (a window has >= 65 positions).
__host__ __device__ inline size_t max_tiles(int32_t total_tokens, int32_t n_seqs) {
    const size_t by_windows = 3 * ((size_t)total_tokens / (kTile + 1 - kMergeMaxLen)) + 3;
    return (size_t)total_tokens / kTile + ((size_t)n_seqs < by_windows ? (size_t)n_seqs : by_windows);
}

// A decoded work item.  len < 0 marks the end of the list.
struct WorkItem {
    int32_t tok0;   // first token of the sequence in the packed batch
    int32_t len;    // sequence length
    int32_t head;
    int32_t blk;    // block inside the sequence: 256 or 128 query rows forward, 128 keys backward (256 on CTA pairs)
    int32_t tile0;  // index of the sequence's first 128-row tile among all tiles of the batch
};

// The n-th item of a worker (persistent CTA or pair): the first is its own number, the counter hands out the rest (one
// round trip less before a short call's only item: five short requests forward 23.1 -> 22.4 us).
__device__ __forceinline__ uint32_t claim_item(WorkspaceHeader* hdr, uint32_t n, uint32_t worker, uint32_t n_workers, uint32_t abort_flag) {
    if (abort_flag) return 0xffffffffu;
    return n == 0 ? worker : n_workers + atomicAdd(&hdr->work_counter, 1u);
}

// Map item index -> (sequence, head, block); the order inside a sequence is item_place's.
//
// Called by a whole warp.  `cur` keeps the sequence of the item before, which the next item of a worker usually shares (a
// sequence has n_heads or more items in a row); otherwise the lanes probe 32 places of the list at a time.  One thread's
// binary search, eight or nine dependent loads for every item, kept the backward kernels waiting for their next item
// (main kernel: 300 sequences of 200 tokens, head_dim 64: 376 -> 355 us; 600 of 256, head_dim 128: 1073 -> 1050; 32
// causal texts of 512-8192: 2633 -> 2548).  The forward, whose items are claimed further ahead, is within 1 %.
struct SeqCursor {
    uint32_t begin = 0, end = 0;            // its items
    int32_t tok0 = 0, len = 0, tile0 = 0;
};
__device__ inline WorkItem decode_item(const SchedView& s, const int32_t* cu_seqlens, uint32_t item, int rows_per_blk,
                                       int n_heads, int n_workers, bool causal, bool heavy_is_last, SeqCursor& cur) {
    if (item - cur.begin >= cur.end - cur.begin) {
        const int lane = threadIdx.x & 31;
        int lo = 0, hi = s.n_seqs;          // largest i with prefix[i] <= item
        while (hi - lo > 1) {
            const int step = (hi - lo + 31) >> 5, probe = lo + lane * step;
            const uint32_t below = __ballot_sync(0xffffffffu, probe < hi && s.prefix[probe] <= item);
            lo += (__popc(below) - 1) * step;       // lane 0 probes lo itself, which is below
            hi = min(lo + step, hi);
        }
        const int seq = s.order[lo];
        cur.begin = s.prefix[lo];
        cur.end = s.prefix[lo + 1];
        cur.tok0 = cu_seqlens[seq];
        cur.len = cu_seqlens[seq + 1] - cur.tok0;
        cur.tile0 = (int32_t)s.tile_prefix[seq];
    }
    WorkItem w;
    w.tok0 = cur.tok0;
    w.len = cur.len;
    w.tile0 = cur.tile0;
    const uint32_t local = item - cur.begin;
    const uint32_t nblk = (uint32_t)(w.len + rows_per_blk - 1) / (uint32_t)rows_per_blk;
    const ItemPlace at = item_place(local, nblk, (uint32_t)n_heads, (uint32_t)n_workers, causal, heavy_is_last);
    w.head = (int32_t)at.head;
    w.blk = (int32_t)at.blk;
    return w;
}

}  // namespace dcp
