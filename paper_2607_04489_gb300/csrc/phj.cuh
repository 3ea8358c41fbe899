// Work items and row access shared by the partitioned join's kernels (phj.cu,
// phj_sum.cu).
#pragma once

#include "common.cuh"
#include "keygroup.cuh"

#ifndef EIGER_PROBE_CHUNK
#define EIGER_PROBE_CHUNK 32768
#endif

namespace eiger {

constexpr int kJoinThreads = EIGER_JOIN_THREADS;
constexpr uint32_t kBuildCap = EIGER_BUILD_CAP;      // build rows per shared-memory table
constexpr uint32_t kProbeChunk = EIGER_PROBE_CHUNK;  // probe rows per work item, at most

// Direct-addressed tables: the partition's bits and the kbits - pbits bits
// below them name a mixed key completely, so those low bits are its slot and no
// key is stored or compared. Used while the slots are few enough
// (kDirectBits) and the build rows fill at least an eighth of them.
//
// A further row of a key that is already in the table goes to a chain entry of
// the item (in a launch for such items): the slot then holds the entry's code
// instead of a row, the entry its row and what the slot held before (a row or
// another code). Codes are the kPieceRows words below kHole, so rows stay below
// them (kDirectMaxRows).
constexpr int kDirectBits = 14;     // 4-byte slots: 64 KB, and 8 KB of chains: three CTAs per SM
constexpr uint32_t kChainMax = 1024;              // further rows of repeated keys an item holds
constexpr uint32_t kPieceRows = 4096;             // build rows of a piece of an item with more: all may be chained
constexpr uint32_t kChainTop = 0xFFFFFFFEu;       // code of entry e: kChainTop - e
constexpr int64_t kDirectMaxRows = (int64_t)kChainTop - (kPieceRows - 1);  // build rows, for matches
struct ChainEntry {
    uint32_t row, next;
};
constexpr int kDirectSumBits = 13;  // 12-byte slots: 96 KB beside the sum's row stages
constexpr uint32_t kDirectProbeChunk = 65536;  // probe rows per work item then: one table serves more
// Build rows per work item of the direct sum, at most: a table takes any number of
// rows, but with few keys a partition has many rows for one CTA, all on a few slots
// (2^24 rows of two keys: 5.96 ms by one CTA a key, 0.16 in chunks).
// The items of a partition's chunks add up. Beyond twice the probe chunk, more
// build rows save little of the probe rows read again per chunk.
constexpr uint32_t kDirectSumChunk = 2 * kDirectProbeChunk;
__device__ __forceinline__ uint32_t direct_slot(uint32_t k, int pbits, int sbits) {
    return (k << pbits) >> (32 - sbits);
}

template <typename KeyT>
struct JoinIn {
    const KeyT* bkey;
    const uint32_t* bidx;
    const uint32_t* bstart;
    const KeyT* pkey;
    const uint32_t* pidx;
    const uint32_t* pstart;
    const unsigned long long* item_prefix;
    uint32_t P;
    uint32_t bcap, pcap;  // build and probe rows per work item, at most
    int pbits, sbits;     // partition bits; direct-addressed tables: bits of the slot below them
    uint32_t* chained;         // direct-addressed tables: the items left to tables with chains
    unsigned long long* redo;  // and those with too many repeats for these, left to pieces (redo_entry)
};

// Items with more repeats than their chains hold, cut into pieces of at most
// kPieceRows build rows. Ctrl::nredo counts the items (upper 24 bits) and
// their pieces (lower 40) in one atomic, so the list is in the order of its
// items' first pieces; an entry holds an item's first piece and the item.
constexpr int kRedoItemBits = 24, kRedoPieceBits = 40;
__host__ __device__ __forceinline__ unsigned long long redo_entry(unsigned long long first, unsigned long long item) {
    return (first << kRedoItemBits) | item;
}

__host__ __device__ __forceinline__ uint32_t chunks_of(uint32_t rows, uint32_t cap) {
    return rows / cap + (rows % cap != 0);
}

// A work item's rows: partition p's build chunk [bs0, bs0 + bn) and probe chunk
// [ps0, ps0 + pn). The chunks of a partition are balanced (sizes differ by at
// most one row), so no item joins a full table with a sliver of probe rows.
struct ItemRows {
    uint32_t bs0, bn, ps0, pn;
};

template <typename KeyT>
__device__ __forceinline__ ItemRows item_rows(const JoinIn<KeyT>& a, unsigned long long item, uint32_t p) {
    const uint32_t b0 = a.bstart[p], bsz = a.bstart[p + 1] - b0;
    const uint32_t p0 = a.pstart[p], psz = a.pstart[p + 1] - p0;
    const uint32_t npc = chunks_of(psz, a.pcap), nbc = chunks_of(bsz, a.bcap);
    const uint32_t local = (uint32_t)(item - a.item_prefix[p]);  // < items of one partition
    const uint32_t bc = local / npc, pc = local - bc * npc;
    ItemRows r;
    const uint32_t b_lo = (uint32_t)((unsigned long long)bc * bsz / nbc);
    const uint32_t p_lo = (uint32_t)((unsigned long long)pc * psz / npc);
    r.bs0 = b0 + b_lo;
    r.bn = (uint32_t)((unsigned long long)(bc + 1) * bsz / nbc) - b_lo;
    r.ps0 = p0 + p_lo;
    r.pn = (uint32_t)((unsigned long long)(pc + 1) * psz / npc) - p_lo;
    return r;
}

// Build rows per work item of a join (a partition's at most this many at a time);
// the pieces of an item of direct matches are its later launch's business.
inline uint32_t build_chunk(int direct, bool carried_sum) {
    return !direct ? kBuildCap : carried_sum ? kDirectSumChunk : 0xFFFFFFFFu;
}

__device__ __forceinline__ uint32_t slot_hash(uint32_t k) { return k * 0x9E3779B1u; }
__device__ __forceinline__ uint32_t slot_hash(uint64_t k) {
    return (uint32_t)((k * 0x9E3779B97F4A7C15ull) >> 32);
}

__device__ __forceinline__ uint32_t next_slot(uint32_t s, uint32_t tsize) {
    return s + 1 == tsize ? 0u : s + 1;
}

// The 128-byte lines of rows [0, n) of a partitioned side (keys, then tuple
// IDs unless rows are identified by position) asked into L2, one line per
// participating thread and step (thread t of `threads`). A hint: no register
// waits on it.
template <bool POS, typename KeyT>
__device__ __forceinline__ void prefetch_rows_l2(const KeyT* key, const uint32_t* idx, uint32_t n, uint32_t t,
                                                 uint32_t threads) {
    const uint32_t klines = (uint32_t)((n * sizeof(KeyT) + 127) / 128);
    const uint32_t ilines = POS ? 0u : (n * 4u + 127) / 128;
    for (uint32_t l = t; l < klines + ilines; l += threads) {
        const char* p = l < klines ? reinterpret_cast<const char*>(key) + (size_t)l * 128
                                   : reinterpret_cast<const char*>(idx) + (size_t)(l - klines) * 128;
        asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
    }
}

// Warp-collective: the partition of a work item (prefix[0] = 0).
__device__ __forceinline__ uint32_t find_partition(const unsigned long long* __restrict__ prefix,
                                                   uint32_t P, unsigned long long item) {
    return warp_last_le(P, item, [&](uint32_t i) { return prefix[i]; });
}

// The fused sum over positions (phj_sum.cu): out.b.src[0] and out.p.src[0] are
// the carried payload columns, indexed like the keys of `a`; distinct: the
// estimated share of the build rows that differ in their key.
template <typename KeyT>
cudaError_t phj_sum_launch(const JoinIn<KeyT>& a, int direct, double distinct, const JoinOut& out, Ctrl* ctrl,
                           const DevInfo& di, cudaStream_t stream, int64_t nb, int64_t np);

}  // namespace eiger
