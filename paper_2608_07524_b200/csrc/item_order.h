// Order of a sequence's work items: which head and row block the n-th one is.  Plain arithmetic, also compiled for the host.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define DCP_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define DCP_HOST_DEVICE inline
#endif

namespace dcp {

struct ItemPlace {
    uint32_t head, blk;
};

// Without a mask the items of a sequence are alike and blocks vary fastest, so that CTAs running at the same time share one
// head's K and V in L2.  Under a causal mask the heaviest blocks come first (forward, heavy_is_last: last rows see the most
// keys; backward: first keys are seen by the most rows), of as many heads together as give every worker two items: one head
// at a time, the last head's heaviest block, up to a hundred times the lightest, started when most of the work was done (one
// 15904-token sequence beside nine short ones, 4 heads: backward main kernel 813 us, 656 with its heads together); all heads
// together, sequences of many blocks lose the sharing in L2 (131072 tokens, 8 heads: forward 28.1 ms one head at a time,
// 32.9 together).
DCP_HOST_DEVICE ItemPlace item_place(uint32_t local, uint32_t nblk, uint32_t n_heads, uint32_t n_workers, bool causal,
                                     bool heavy_is_last) {
    ItemPlace w;
    uint32_t b;
    if (causal) {
        // groups of `least` or more heads, as equal as they come (a small last group would be the tail all over again)
        const uint32_t heads = n_heads, least = (2u * n_workers + nblk - 1) / nblk;
        const uint32_t groups = least < heads ? heads / least : 1u, size = heads / groups, larger = heads % groups;
        const uint32_t in_larger = larger * (size + 1) * nblk;       // items of the groups of one head more, which come first
        const uint32_t g_size = local < in_larger ? size + 1 : size, rest = local < in_larger ? local : local - in_larger;
        const uint32_t head0 = (local < in_larger ? 0u : larger * (size + 1)) + rest / (g_size * nblk) * g_size;
        const uint32_t in_group = rest % (g_size * nblk);
        w.head = head0 + in_group % g_size;
        b = in_group / g_size;
    } else {
        w.head = local / nblk;
        b = local % nblk;
    }
    w.blk = heavy_is_last ? nblk - 1 - b : b;
    return w;
}

}  // namespace dcp
