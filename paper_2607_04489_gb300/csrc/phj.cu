// Partitioned hash join (Sec. 3.2): after both sides are radix-partitioned on
// the same hash bits, partition p of R can only match partition p of S. Each
// build partition fits a hash table in shared memory, so every probe is a
// shared-memory access instead of a random global one.
//
// Work item = (partition p, build chunk c_R, probe chunk c_S). A build
// partition larger than one shared-memory table (duplicate-heavy keys) is cut
// into chunks of at most kBuildCap rows, each joined with the whole probe
// partition; a large probe partition (skew) is cut into chunks of at most
// kProbeChunk rows so that hot partitions spread over many CTAs. The chunks of
// a partition are balanced in size. A persistent grid pulls
// items from a global counter. Per item a CTA clears a table of about three
// slots per build row (load factor <= 1/3), inserts the build chunk with
// shared-memory CAS, then streams the probe chunk, walking linear-probe chains;
// or, where the build keys are dense and distinct, fills a direct-addressed
// table (phj.cuh) that takes the whole build partition and reads one word per
// probe row (later launches take the partitions with repeated keys, see JoinKind).
// Index pairs leave through per-warp output runs (chunks.cuh), so the probe
// loop has no CTA barrier; columns through one CTA reservation per round, column
// by column; the matches of repeated build keys through the CTA stage
// (emit.cuh).
//
// What bounds it: direct-addressed pairs read one shared word and write 8 bytes
// per probe row (28M rows of dense keys: 0.23 ms with hash tables, 0.17 ms);
// columns wait on the gathers of the build side's values (114M rows, two 4-byte
// columns a side: 1.79 ms row by row through hash tables and the stage, 1.29 ms).
// Equal build keys in a hash table are inserted past one another by reads: 2^25 x
// 2^27 rows with one key on 5 % of the build rows, 57 -> 28 ms.
#include <algorithm>

#include "chunks.cuh"
#include "emit.cuh"
#include "kernels.cuh"
#include "phj.cuh"

namespace eiger {

size_t part_counts_len(int64_t n, int b1, int b2, int passes);
size_t part_scan_blocks(size_t counts_len);

namespace {

// How matches leave the kernel: index pairs through per-warp output runs
// (chunks.cuh), columns (and indices beside them) through a CTA reservation per
// round, or summed.
enum JoinMode { kPairs, kColumns, kSum };

// Rows each thread keeps in flight per round (the current round and the next
// one's loads) and CTAs per SM. Index pairs of 32-bit keys: 4 rows, three
// 512-thread CTAs per SM (40 registers), so that while one CTA clears or builds
// its table the others probe theirs (measured on GB300: 16 % faster than two
// CTAs of 8 rows). Columns and sums keep more live state per match and 64-bit
// keys larger tables: two CTAs per SM (64 registers), 8 rows for the sums of
// 32-bit keys and 4 otherwise.
template <typename KeyT, int MODE>
struct Rows {
    static constexpr bool kLean = sizeof(KeyT) == 4 && MODE == kPairs;
    static constexpr int kN = sizeof(KeyT) == 4 && MODE == kSum ? 8 : 4;
    static constexpr int kMinBlocks = (kLean ? 1536 : 1024) / kJoinThreads;
    static constexpr uint32_t kRound = kJoinThreads * kN;
};
constexpr int kJoinStage = kJoinThreads * 4;  // matches staged between two flushes (duplicate build keys)
constexpr uint32_t kTableMax = 2 * kBuildCap;
constexpr uint32_t kEmptyRow = 0xFFFFFFFFu;

// Work items of partition p: build chunks x probe chunks (none if a side is empty).
__global__ void items_count_kernel(const uint32_t* __restrict__ bstart, const uint32_t* __restrict__ pstart,
                                   uint32_t P, uint32_t bcap, uint32_t pcap, unsigned long long* __restrict__ count) {
    for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < P; p += gridDim.x * blockDim.x) {
        const uint32_t bs = bstart[p + 1] - bstart[p];
        const uint32_t ps = pstart[p + 1] - pstart[p];
        count[p] = (bs && ps) ? (unsigned long long)chunks_of(bs, bcap) * chunks_of(ps, pcap) : 0ull;
    }
}

// One block: exclusive scan of the item counts in place, 4096 per chunk with
// coalesced loads and stores; prefix[P] and ctrl->nitems get the total.
__global__ void __launch_bounds__(1024)
    items_scan_kernel(unsigned long long* __restrict__ prefix, uint32_t P, Ctrl* ctrl) {
    constexpr int kPer = 4;
    constexpr uint32_t kChunk = 1024 * kPer;
    __shared__ unsigned long long s_buf[kChunk];
    __shared__ unsigned long long s_warp[1024 / kWarp];
    const unsigned lane = lane_id();
    const int warp = threadIdx.x / kWarp;
    unsigned long long carry = 0;
    for (uint32_t base = 0; base < P; base += kChunk) {
        for (uint32_t i = threadIdx.x; i < kChunk; i += blockDim.x)
            s_buf[i] = base + i < P ? prefix[base + i] : 0ull;
        __syncthreads();
        unsigned long long local = 0;
#pragma unroll
        for (int j = 0; j < kPer; ++j) local += s_buf[threadIdx.x * kPer + j];
        unsigned long long x = local;
#pragma unroll
        for (int o = 1; o < kWarp; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
            if ((int)lane >= o) x += y;
        }
        if ((int)lane == kWarp - 1) s_warp[warp] = x;
        __syncthreads();
        if (warp == 0) {
            unsigned long long v = s_warp[lane];
#pragma unroll
            for (int o = 1; o < kWarp; o <<= 1) {
                const unsigned long long y = __shfl_up_sync(0xffffffffu, v, o);
                if ((int)lane >= o) v += y;
            }
            s_warp[lane] = v;
        }
        __syncthreads();
        unsigned long long run = carry + (warp ? s_warp[warp - 1] : 0ull) + x - local;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const unsigned long long c = s_buf[threadIdx.x * kPer + j];
            s_buf[threadIdx.x * kPer + j] = run;
            run += c;
        }
        carry += s_warp[kWarp - 1];
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < kChunk && base + i < P; i += blockDim.x) prefix[base + i] = s_buf[i];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        prefix[P] = carry;
        ctrl->nitems = carry;
    }
}

template <typename KeyT>
struct SmemTable;

// Home slot of a key in a table of `tsize` slots. The partition was chosen by
// the top bits of a mixed key, so the keys of one partition are a scattered
// subset of the key space; a Fibonacci (multiplicative) hash of the key itself
// spreads them over the table, and a multiply-shift range reduction maps its
// top bits onto [0, tsize).
// Slots come in aligned pairs: the home slot is even, so a probe reads its
// first two candidates with one 16-byte shared load (inserts are ordinary
// linear probing from the same home slot, filling a pair's first slot first).
template <typename KeyT>
__device__ __forceinline__ uint32_t home_slot(KeyT k, uint32_t tsize) {
    return 2u * (uint32_t)(((unsigned long long)slot_hash(k) * (tsize >> 1)) >> 32);
}

// 32-bit keys: one packed 64-bit word per slot, claimed by CAS.
template <>
struct SmemTable<uint32_t> {
    static constexpr size_t kSlotBytes = 8;
    unsigned long long* slot;
    __device__ void bind(unsigned char* smem) { slot = reinterpret_cast<unsigned long long*>(smem); }
    // every slot of a table of tsize (a multiple of 2) slots, two per 16-byte store
    __device__ void clear_all(uint32_t tsize) {
        ulonglong2* p = reinterpret_cast<ulonglong2*>(slot);
        for (uint32_t i = threadIdx.x; i < tsize / 2; i += blockDim.x) p[i] = make_ulonglong2(kEmptySlot, kEmptySlot);
    }
    // 1: inserted; 0: slot taken by another key; -1: slot taken by the same key
    __device__ int insert(uint32_t s, uint32_t k, uint32_t row) {
        const unsigned long long prev = atomicCAS(slot + s, kEmptySlot, ((unsigned long long)k << 32) | row);
        if (prev == kEmptySlot) return 1;
        return (uint32_t)(prev >> 32) == k ? -1 : 0;
    }
    // whether slot s is taken (dup: by key k)
    __device__ bool taken(uint32_t s, uint32_t k, int& dup) const {
        const unsigned long long v = *(volatile unsigned long long*)(slot + s);
        if (v != kEmptySlot && (uint32_t)(v >> 32) == k) dup = 1;
        return v != kEmptySlot;
    }
    // the aligned pair of slots starting at even slot s
    __device__ ulonglong2 pair(uint32_t s) const { return *reinterpret_cast<const ulonglong2*>(slot + s); }
    // 0: empty (chain ends), 1: occupied, other key, 2: match
    __device__ int probe(uint32_t s, uint32_t k, uint32_t& row) const {
        const unsigned long long v = slot[s];
        if (v == kEmptySlot) return 0;
        row = (uint32_t)v;
        return (uint32_t)(v >> 32) == k ? 2 : 1;
    }
};

// 64-bit keys: key array plus row array; the row word is claimed by CAS.
template <>
struct SmemTable<uint64_t> {
    static constexpr size_t kSlotBytes = 12;
    unsigned long long* key;
    uint32_t* row;
    __device__ void bind(unsigned char* smem) {
        key = reinterpret_cast<unsigned long long*>(smem);
        row = reinterpret_cast<uint32_t*>(smem + (size_t)kTableMax * 8);
    }
    __device__ void clear_all(uint32_t tsize) {
        for (uint32_t i = threadIdx.x; i < tsize; i += blockDim.x) row[i] = kEmptyRow;
    }
    // 1: inserted; 0: slot taken (its key may still be in flight, so equal
    // keys are not detected here but by has_equal_keys after the build)
    __device__ int insert(uint32_t s, uint64_t k, uint32_t r) {
        if (atomicCAS(row + s, kEmptyRow, r) != kEmptyRow) return 0;
        key[s] = k;
        return 1;
    }
    __device__ bool taken(uint32_t s, uint64_t, int&) const { return *(volatile uint32_t*)(row + s) != kEmptyRow; }
    // After every insert has completed: 1 when an occupied slot of this
    // thread's share finds its own key earlier in its probe chain, i.e. the
    // table holds a key twice. Linear probing leaves no empty slot between a
    // key's home slot and its slot, so each walk is short and bounded.
    __device__ int has_equal_keys(uint32_t tsize) const;
    __device__ int probe(uint32_t s, uint64_t k, uint32_t& r) const {
        const uint32_t v = row[s];
        if (v == kEmptyRow) return 0;
        r = v;
        return key[s] == k ? 2 : 1;
    }
};

__device__ int SmemTable<uint64_t>::has_equal_keys(uint32_t tsize) const {
    for (uint32_t s = threadIdx.x; s < tsize; s += blockDim.x) {
        if (row[s] == kEmptyRow) continue;
        const uint64_t k = key[s];
        uint32_t t = home_slot(k, tsize);
        for (uint32_t n = 0; t != s && n < tsize; ++n, t = next_slot(t, tsize))
            if (key[t] == k) return 1;
    }
    return 0;
}

// Rows of a probe round: kRows per thread, strided by the block size so every
// load instruction of a warp reads 32 consecutive rows.
template <typename KeyT, int N>
struct RoundRegs {
    KeyT k[N];
    uint32_t id[N];
};

// POS (GFTR): a row is identified by its position in the partitioned arrays
// (pos0 + i), not by the tuple ID stored beside its key.
template <bool POS, typename KeyT, int N>
__device__ __forceinline__ void load_round(RoundRegs<KeyT, N>& r, const KeyT* __restrict__ key,
                                           const uint32_t* __restrict__ idx, uint32_t base,
                                           uint32_t n, uint32_t pos0) {
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const uint32_t i = base + j * kJoinThreads + threadIdx.x;
        if (i < n) {
            r.k[j] = __ldcs(key + i);
            r.id[j] = POS ? pos0 + i : __ldcs(idx + i);
        }
    }
}

constexpr int kJoinWarps = kJoinThreads / kWarp;

// kHash: one hash table per item. The rest for dense, hardly repeated 32-bit
// build keys, one launch after the other:
// kDirect: direct-addressed tables, slot -> build row. An item whose build keys
// repeat (a slot taken twice) is left to the next launch.
// kChained: such items, the further rows of a key in chains (phj.cuh); one with
// more than the chains hold is left to the last launch. Chains in the first
// launch, for all items, cost unique keys their registers (2^25 x 2^27 rows:
// pairs 2163 -> 2254 us, two columns a side 3908 -> 4196).
// kPieces: those, each piece of at most kPieceRows build rows an item of its own
// with chains for all of them, so that one heavily repeated key (a default value)
// spreads over the chip and no other key meets its rows (2^25 x 2^27 rows, one key
// on 2 % of the build rows, pairs: 180 ms with hash tables, whose equal keys half
// of the probes walked, 2.2 ms; two columns a side 127 and 4.3).
enum JoinKind { kHash, kDirect, kChained, kPieces };

// Bytes of a direct-addressed table, a multiple of 16.
__host__ __device__ constexpr size_t direct_table_bytes(int sbits) { return ((size_t)4 << sbits) / 16 * 16 + 16; }

// Warp-collective: the rest of the chains at[j] of probe rows id[j], with their
// columns. One reservation for the warp, then each lane walks its chains.
template <int N, uint32_t CHAINS>
__device__ __forceinline__ void emit_chains(const uint32_t (&at)[N], const uint32_t (&id)[N], const ChainEntry* chain,
                                            const JoinOut& out, unsigned long long* cursor) {
    auto next = [&](uint32_t v) { return kChainTop - v < CHAINS ? chain[kChainTop - v].next : kHole; };
    uint32_t count = 0;
#pragma unroll
    for (int j = 0; j < N; ++j)
        for (uint32_t v = at[j]; v != kHole; v = next(v)) ++count;
    __syncwarp();
    uint32_t x = count;
#pragma unroll
    for (int o = 1; o < kWarp; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if ((int)lane_id() >= o) x += y;
    }
    unsigned long long base = 0;
    if (lane_id() == kWarp - 1 && x) base = atomicAdd(cursor, (unsigned long long)x);
    unsigned long long pos = __shfl_sync(0xffffffffu, base, kWarp - 1) + x - count;
#pragma unroll
    for (int j = 0; j < N; ++j)
        for (uint32_t v = at[j]; v != kHole; v = next(v))
            write_match(out, pos++, kChainTop - v < CHAINS ? chain[kChainTop - v].row : v, id[j]);
    __syncwarp();
}

template <typename KeyT, int MODE, bool POS, int KIND>
__global__ void __launch_bounds__(kJoinThreads, (Rows<KeyT, MODE>::kMinBlocks))
    phj_join_kernel(JoinIn<KeyT> a, const __grid_constant__ JoinOut out, PairSink sink, Ctrl* ctrl) {
    extern __shared__ __align__(16) unsigned char smem[];
    constexpr bool PAIRS = MODE == kPairs, AGG = MODE == kSum;
    constexpr bool kSlots = KIND != kHash;                // direct-addressed
    constexpr bool kLater = kSlots && KIND != kDirect;    // goes on with an earlier launch's output runs
    constexpr uint32_t kChains = KIND == kPieces ? kPieceRows : kChainMax;
    // the stage follows the table in dynamic shared memory; index pairs and
    // aggregates use none, so none is allocated for them (shared memory left
    // unreserved serves as L1 cache, which the payload gathers of the
    // aggregate need)
    Stage<kJoinStage>& st = *reinterpret_cast<Stage<kJoinStage>*>(smem + (size_t)kTableMax * SmemTable<KeyT>::kSlotBytes);
    constexpr int kN = Rows<KeyT, MODE>::kN;
    constexpr uint32_t kRound = Rows<KeyT, MODE>::kRound;
    __shared__ uint32_t s_grp[2][MODE == kColumns ? kN * kJoinWarps : 1];
    __shared__ unsigned long long s_base[2];
    __shared__ unsigned long long s_next_item;
    __shared__ unsigned long long s_item;
    __shared__ uint32_t s_next_part, s_piece, s_chained;
    SmemTable<KeyT> tab;
    tab.bind(smem);
    uint32_t* dtab = reinterpret_cast<uint32_t*>(smem);
    ChainEntry* chain = reinterpret_cast<ChainEntry*>(smem + direct_table_bytes(a.sbits));
    // (without items left to it, a later launch leaves the warp records as they are)
    const unsigned long long left = KIND == kPieces ? ctrl->nredo : KIND == kChained ? ctrl->nchained : 0ull;
    if (kLater && left == 0) return;
    if (MODE == kColumns && !kSlots && threadIdx.x == 0) st.count = 0;
    AggState agg{0ull, 0ull};
    const uint32_t gwarp = blockIdx.x * kJoinWarps + threadIdx.x / kWarp;
    WarpChunk wc;
    wc.init(sink.run);
    if (PAIRS && kLater) warp_chunk_resume(wc, sink, gwarp);
    uint32_t flushes = 0;
    const unsigned long long nitems = KIND == kPieces      ? left & ((1ull << kRedoPieceBits) - 1)
                                      : KIND == kChained ? left
                                                         : ctrl->nitems;
    unsigned long long* const next = KIND == kPieces      ? &ctrl->next_redo
                                     : KIND == kChained ? &ctrl->next_chained
                                                        : &ctrl->next_item;

    // Work items are claimed one ahead: the claim for the next item is issued
    // when an item starts, and its partition is looked up by warp 0 after the
    // build, so neither round trip sits between two items.
    auto look_up = [&](unsigned long long claim) {  // warp 0
        unsigned long long item = claim;
        uint32_t piece = 0, p = 0;
        if (claim < nitems) {
            if constexpr (KIND == kPieces) {
                const uint32_t e = warp_last_le((uint32_t)(left >> kRedoPieceBits), claim,
                                                [&](uint32_t i) { return a.redo[i] >> kRedoItemBits; });
                piece = (uint32_t)(claim - (a.redo[e] >> kRedoItemBits));
                item = a.redo[e] & ((1ull << kRedoItemBits) - 1);
            }
            if (KIND == kChained) item = a.chained[claim];
            p = find_partition(a.item_prefix, a.P, item);
        }
        if (threadIdx.x == 0) {
            s_next_item = claim;
            s_next_part = p;
            if (kLater) s_item = item;
            if (KIND == kPieces) s_piece = piece;
        }
        return p;
    };
    if (threadIdx.x < kWarp) {
        unsigned long long it0 = 0;
        if (threadIdx.x == 0) it0 = atomicAdd(next, 1ull);
        look_up(__shfl_sync(0xffffffffu, it0, 0));
    }
    __syncthreads();

    for (;;) {
        const unsigned long long cur_item = s_next_item;
        const uint32_t p = s_next_part;
        if (cur_item >= nitems) break;
        const unsigned long long item = kLater ? s_item : cur_item;
        unsigned long long claim = 0;
        if (threadIdx.x == 0) claim = atomicAdd(next, 1ull);

        ItemRows ir = item_rows(a, item, p);
        if constexpr (KIND == kPieces) {  // the piece's share of the build rows
            const uint32_t pieces = chunks_of(ir.bn, kPieceRows);
            const uint32_t lo = (uint32_t)((unsigned long long)s_piece * ir.bn / pieces);
            const uint32_t hi = (uint32_t)((unsigned long long)(s_piece + 1) * ir.bn / pieces);
            ir.bs0 += lo;
            ir.bn = hi - lo;
        }
        const uint32_t bn = ir.bn, pn = ir.pn;
        const KeyT* bkey = a.bkey + ir.bs0;
        const uint32_t* bidx = a.bidx + ir.bs0;
        const KeyT* pkey = a.pkey + ir.ps0;
        const uint32_t* pidx = a.pidx + ir.ps0;
        const uint32_t bpos0 = ir.bs0, ppos0 = ir.ps0;

        // Issue the first build and probe loads before clearing the table, so
        // their latency overlaps the clear.
        RoundRegs<KeyT, kN> cur, nxt;
        load_round<POS>(nxt, bkey, bidx, 0, bn, bpos0);
        if (!kSlots) load_round<POS>(cur, pkey, pidx, 0, pn, ppos0);

        // Looks up the next item while the probes run, and asks L2 for the
        // start of its partition's build rows and its first probe round, so
        // that it starts on cache hits.
        auto next_item = [&] {
            if (threadIdx.x >= kWarp) return;
            const unsigned long long cl = __shfl_sync(0xffffffffu, claim, 0);
            const uint32_t pn2 = look_up(cl);
            if (cl < nitems) {
                const uint32_t nb0 = a.bstart[pn2], nbn = min(a.bstart[pn2 + 1] - nb0, kBuildCap);
                const uint32_t np0 = a.pstart[pn2], npn = min(a.pstart[pn2 + 1] - np0, kRound);
                prefetch_rows_l2<POS>(a.bkey + nb0, a.bidx + nb0, nbn, threadIdx.x, kWarp);
                prefetch_rows_l2<POS>(a.pkey + np0, a.pidx + np0, npn, threadIdx.x, kWarp);
            }
        };
        // Probe rows round by round: the next round's loads are in flight while
        // this round probes, and the round after it is on its way into L2.
        auto probe_rounds = [&](auto&& round) {
            for (uint32_t base = 0; base < pn; base += kRound) {
                if (base + kRound < pn) load_round<POS>(nxt, pkey, pidx, base + kRound, pn, ppos0);
                if (base + 2 * kRound < pn)
                    prefetch_rows_l2<POS>(pkey + base + 2 * kRound, pidx + base + 2 * kRound,
                                          min(pn - (base + 2 * kRound), kRound), threadIdx.x, kJoinThreads);
                round(base);
                cur = nxt;
            }
        };
        // A round with at most one match per row: brow[j] or kHole.
        auto emit_round = [&](const uint32_t(&brow)[kN]) {
            if constexpr (PAIRS) {
#pragma unroll
                for (int j = 0; j < kN; ++j) warp_emit(wc, sink, brow[j] != kHole, brow[j], cur.id[j]);
            } else if constexpr (AGG) {
#pragma unroll
                for (int j = 0; j < kN; ++j)
                    if (brow[j] != kHole) {
                        agg.sum += (unsigned long long)read_pay(out.b.src[0], out.b.bytes[0], brow[j]) +
                                   (unsigned long long)read_pay(out.p.src[0], out.p.bytes[0], cur.id[j]);
                        agg.count += 1;
                    }
            } else {
                const uint32_t h = flushes++ & 1;
                flush_matches<kN, kJoinThreads>(brow, cur.id, s_grp[h], &s_base[h], out, &ctrl->cursor);
            }
        };

        if constexpr (kSlots) {
            const uint32_t slots = 1u << a.sbits;
            // more build rows than slots and chains together hold: no use trying
            const bool over = KIND == kDirect && bn > slots + kChainMax;
            uint4* d4 = reinterpret_cast<uint4*>(dtab);
            if (!over)
                for (uint32_t i = threadIdx.x; i < slots / 4 + 1; i += kJoinThreads)
                    d4[i] = make_uint4(kHole, kHole, kHole, kHole);
            if (kLater && threadIdx.x == 0) s_chained = 0;
            __syncthreads();
            int dup = 0;
            // Build rows a round ahead (a partition's build takes several);
            // behind the last round, the first probe rows. 10M x 120M rows with
            // two columns a side: 1285 -> 1187 us.
            for (uint32_t bb = 0; bb < bn && !over; bb += kRound) {
                const bool more = bb + kRound < bn;
                if (more)
                    load_round<POS>(cur, bkey, bidx, bb + kRound, bn, bpos0);
                else
                    load_round<POS>(cur, pkey, pidx, 0, pn, ppos0);
#pragma unroll
                for (int j = 0; j < kN; ++j)
                    if (bb + j * kJoinThreads + threadIdx.x < bn) {
                        const uint32_t s = direct_slot(nxt.k[j], a.pbits, a.sbits);
                        const uint32_t old = atomicExch(dtab + s, nxt.id[j]);
                        if constexpr (KIND == kDirect) {
                            dup |= old != kHole;
                        } else if (old != kHole) {  // a repeated key: its earlier row leaves the slot
                            const uint32_t e = atomicAdd(&s_chained, 1u);
                            if (e < kChains) chain[e] = ChainEntry{old, s};
                        }
                    }
                if (more) nxt = cur;
            }
            const bool repeats = __syncthreads_or(dup) != 0;
            const uint32_t chained = kLater ? s_chained : 0u;
            next_item();
            if (over || chained > kChains) {  // (never a piece)
                if (threadIdx.x == 0) {
                    const unsigned long long at =
                        atomicAdd(&ctrl->nredo, (1ull << kRedoPieceBits) | chunks_of(bn, kPieceRows));
                    a.redo[at >> kRedoPieceBits] = redo_entry(at & ((1ull << kRedoPieceBits) - 1), item);
                }
            } else if (repeats) {
                if (threadIdx.x == 0) a.chained[atomicAdd(&ctrl->nchained, 1u)] = (uint32_t)item;
            } else {
                if constexpr (kLater) {  // hang the displaced rows before the rows that stayed
                    for (uint32_t e = threadIdx.x; e < chained; e += kJoinThreads)
                        chain[e].next = atomicExch(dtab + chain[e].next, kChainTop - e);
                    __syncthreads();
                }
                probe_rounds([&](uint32_t base) {
                    uint32_t at[kN];
#pragma unroll
                    for (int j = 0; j < kN; ++j)
                        at[j] = base + j * kJoinThreads + threadIdx.x < pn
                                    ? dtab[direct_slot(cur.k[j], a.pbits, a.sbits)]
                                    : kHole;
                    if constexpr (KIND == kDirect) {
                        emit_round(at);
                    } else {  // every row's first match, then their second ones, and so on
                        for (int level = 0;; ++level) {
                            bool more = false;
                            uint32_t brow[kN];
#pragma unroll
                            for (int j = 0; j < kN; ++j) {
                                brow[j] = at[j];
                                const uint32_t e = kChainTop - at[j];
                                at[j] = kHole;
                                if (e < kChains) {
                                    brow[j] = chain[e].row;
                                    at[j] = chain[e].next;
                                    more = true;
                                }
                            }
                            emit_round(brow);
                            if constexpr (MODE == kColumns) {
                                if (!__syncthreads_or(more)) break;
                                if (level == 1) {  // third matches and on are few, or all of a few rows
                                    emit_chains<kN, kChains>(at, cur.id, chain, out, &ctrl->cursor);
                                    break;
                                }
                            } else {
                                if (!__any_sync(0xffffffffu, more)) break;
                            }
                        }
                    }
                });
            }
        } else {  // hash tables
            // about three slots per build row (load <= 1/3), at most kTableMax
            uint32_t tsize = (3 * bn + 31) & ~31u;
            if (tsize < 64) tsize = 64;
            if (tsize > kTableMax) tsize = kTableMax;
            tab.clear_all(tsize);
            __syncthreads();
            // Build. An insert that meets its own key proves a duplicate in this
            // chunk; without one, every probe key has at most one match here.
            int dup = 0;
            for (uint32_t bb = 0; bb < bn; bb += kRound) {
                if (bb) load_round<POS>(nxt, bkey, bidx, bb, bn, bpos0);
#pragma unroll
                for (int j = 0; j < kN; ++j) {
                    if (bb + j * kJoinThreads + threadIdx.x < bn) {
                        uint32_t s = home_slot(nxt.k[j], tsize);
                        for (uint32_t step = 0;;) {
                            const int r = tab.insert(s, nxt.k[j], nxt.id[j]);
                            if (r > 0) break;
                            if (r < 0) dup = 1;
                            // past the taken slots by reads: the rows of one
                            // key would all queue for each slot's atomic
                            do {
                                s = next_slot(s, tsize);
                            } while (++step < tsize && tab.taken(s, nxt.k[j], dup));
                            if (step >= tsize) {
                                atomicOr(&ctrl->err, kErrTableFull);
                                break;
                            }
                        }
                    }
                    __syncwarp();
                }
            }
            if constexpr (sizeof(KeyT) != 4) {
                __syncthreads();  // every key of the table is written
                dup = tab.has_equal_keys(tsize);
            }
            const bool unique = __syncthreads_or(dup) == 0;
            next_item();
            if (unique) {
                // Fast path: stop at the first match, no collectives per step.
                probe_rounds([&](uint32_t base) {
                    uint32_t brow[kN];
#pragma unroll
                    for (int j = 0; j < kN; ++j) {
                        brow[j] = kHole;
                        if (base + j * kJoinThreads + threadIdx.x < pn) {
                            const KeyT k = cur.k[j];
                            uint32_t s = home_slot(k, tsize);
                            if constexpr (sizeof(KeyT) == 4) {
                                for (uint32_t step = 0; step < tsize; step += 2) {
                                    const ulonglong2 v = tab.pair(s);
                                    if (v.x == kEmptySlot) break;
                                    if ((uint32_t)(v.x >> 32) == (uint32_t)k) {
                                        brow[j] = (uint32_t)v.x;
                                        break;
                                    }
                                    if (v.y == kEmptySlot) break;
                                    if ((uint32_t)(v.y >> 32) == (uint32_t)k) {
                                        brow[j] = (uint32_t)v.y;
                                        break;
                                    }
                                    s = s + 2 == tsize ? 0u : s + 2;
                                }
                            } else {
                                for (uint32_t step = 0; step < tsize; ++step) {
                                    uint32_t r;
                                    const int q = tab.probe(s, k, r);
                                    if (q == 0) break;
                                    if (q == 2) {
                                        brow[j] = r;
                                        break;
                                    }
                                    s = next_slot(s, tsize);
                                }
                            }
                        }
                        __syncwarp();
                    }
                    emit_round(brow);
                });
            } else {
                // General path (duplicate keys): every match of every chain,
                // emitted through the warp-aggregated stage.
                probe_rounds([&](uint32_t base) {
#pragma unroll 1
                    for (int j = 0; j < kN; ++j) {
                        bool active = base + j * kJoinThreads + threadIdx.x < pn;
                        const KeyT k = cur.k[j];
                        const uint32_t id = cur.id[j];
                        uint32_t s = active ? home_slot(k, tsize) : 0u;
                        uint32_t steps = 0;
                        while (__any_sync(0xffffffffu, active)) {
                            bool hit = false;
                            uint32_t brow = 0;
                            if (active) {
                                const int r = tab.probe(s, k, brow);
                                if (r == 0) {
                                    active = false;
                                } else {
                                    hit = r == 2;
                                    s = next_slot(s, tsize);
                                    if (++steps == tsize) active = false;
                                }
                            }
                            if constexpr (PAIRS)
                                warp_emit(wc, sink, hit, brow, id);
                            else
                                emit<AGG, kJoinStage>(st, agg, hit, brow, id, out, &ctrl->cursor);
                        }
                        if constexpr (MODE == kColumns) stage_flush<AGG, kJoinStage>(st, out, &ctrl->cursor);
                    }
                });
            }
        }
        __syncthreads();
    }
    if (AGG) agg_commit(agg, ctrl);
    if constexpr (PAIRS) warp_chunk_commit(wc, sink, gwarp);
}

// Launches of one join, as many CTAs per SM as fit. Each warp writes a record of
// the pairs sink; a later launch is no larger than the one before it, so that its
// warps go on with that one's runs.
template <typename KeyT>
struct JoinLaunch {
    const JoinIn<KeyT>& a;
    const JoinOut& out;
    const PairSink& sink;
    Ctrl* ctrl;
    const DevInfo& di;
    cudaStream_t stream;
    double bytes;  // of the first launch, but for the matches
    uint32_t grid = kMaxOutWarps / kJoinWarps;

    template <int MODE, bool POS, int KIND>
    cudaError_t run() {
        auto kern = phj_join_kernel<KeyT, MODE, POS, KIND>;
        const size_t smem = KIND == kHash ? (size_t)kTableMax * SmemTable<KeyT>::kSlotBytes +
                                                (MODE == kColumns ? sizeof(Stage<kJoinStage>) : 0)
                                          : direct_table_bytes(a.sbits) +
                                                (KIND == kChained  ? kChainMax
                                                 : KIND == kPieces ? kPieceRows
                                                                   : 0) * sizeof(ChainEntry);
        cudaError_t e = allow_smem(kern);
        if (e != cudaSuccess) return e;
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kJoinThreads, smem) != cudaSuccess ||
            per_sm < 1)
            per_sm = 1;
        grid = std::min(grid, (uint32_t)(di.sms * per_sm));
        constexpr bool kFirst = KIND == kHash || KIND == kDirect;
        ProfScope ps(kFirst ? "phj_join" : KIND == kChained ? "phj_join.chained" : "phj_join.pieces", kFirst ? bytes : 0.0,
                     stream, kFirst ? match_bytes(out) : 0.0);
        kern<<<grid, kJoinThreads, smem, stream>>>(a, out, sink, ctrl);
        return cudaGetLastError();
    }
    template <int KIND>
    cudaError_t run_as(bool pairs, int gftr) {
        return out.aggregate ? run<kSum, false, KIND>()
               : pairs       ? run<kPairs, false, KIND>()
               : gftr        ? run<kColumns, true, KIND>()
                             : run<kColumns, false, KIND>();
    }
    uint32_t warps() const { return grid * kJoinWarps; }  // of the last launch
};

template <typename KeyT>
cudaError_t launch_join(const PhjScratch& s, const PlanDev& plan, const JoinOut& out, Ctrl* ctrl,
                        const DevInfo& di, cudaStream_t stream, int64_t nb, int64_t np) {
    const int passes = plan.variant == 3 ? 2 : 1;
    const int buf = passes - 1;
    JoinIn<KeyT> a;
    a.bkey = static_cast<const KeyT*>(s.side[0].key[buf]);
    a.bidx = s.side[0].idx[buf];
    a.bstart = s.side[0].part_start;
    a.pkey = static_cast<const KeyT*>(s.side[1].key[buf]);
    a.pidx = s.side[1].idx[buf];
    a.pstart = s.side[1].part_start;
    a.item_prefix = s.item_prefix;
    a.P = 1u << (plan.bits1 + (passes == 2 ? plan.bits2 : 0));
    const bool pairs = !out.aggregate && out.bidx && out.pidx && out.b.n == 0 && out.p.n == 0 && !out.b.rowmap &&
                       !out.p.rowmap;
    a.bcap = build_chunk(plan.direct, out.aggregate && plan.gftr);
    a.pcap = plan.direct ? kDirectProbeChunk : kProbeChunk;
    a.pbits = plan.bits1 + (passes == 2 ? plan.bits2 : 0);
    a.sbits = plan.kbits - a.pbits > 1 ? plan.kbits - a.pbits : 1;
    // the sum with carried payloads has its own kernel (phj_sum.cu)
    if (out.aggregate && plan.gftr) return phj_sum_launch<KeyT>(a, plan.direct, plan.distinct, out, ctrl, di, stream, nb, np);
    PairSink sink{};
    sink.run = plan.direct ? kDirectRun : kHashRun;
    if (pairs) {
        sink.bidx = out.bidx;
        sink.pidx = out.pidx;
        sink.capacity = out.capacity;
        sink.ovf_b = s.ovf[0];
        sink.ovf_p = s.ovf[1];
        sink.cursor = &ctrl->cursor;
        sink.rec = static_cast<ChunkRec*>(s.rec);
    }
    a.redo = s.redo;
    a.chained = s.chained;
    // reads every partitioned (key', row) of both sides once, writes the matches
    const double bytes = (double)(sizeof(KeyT) + sizeof(uint32_t)) * (double)(nb + np);
    JoinLaunch<KeyT> l{a, out, sink, ctrl, di, stream, bytes};
    cudaError_t e;
    if constexpr (sizeof(KeyT) == 4) {
        if (plan.direct) {
            e = l.template run_as<kDirect>(pairs, plan.gftr);
            const uint32_t warps = l.warps();
            if (e == cudaSuccess) e = l.template run_as<kChained>(pairs, plan.gftr);
            if (e == cudaSuccess) e = l.template run_as<kPieces>(pairs, plan.gftr);
            if (e != cudaSuccess || !pairs) return e;
            return chunk_fix_run(sink, warps, s.fix, &ctrl->err, di, stream);
        }
    }
    e = l.template run_as<kHash>(pairs, plan.gftr);
    if (e != cudaSuccess || !pairs) return e;
    return chunk_fix_run(sink, l.warps(), s.fix, &ctrl->err, di, stream);
}

}  // namespace

PhjScratch phj_layout(Carve& c, int64_t nb, int64_t np, const PlanDev& plan) {
    PhjScratch s;
    const int passes = plan.variant == 3 ? 2 : 1;
    const int b1 = plan.bits1, b2 = passes == 2 ? plan.bits2 : 0;
    const size_t kb = plan.key32 ? 4 : 8;
    const size_t P = (size_t)1 << (b1 + b2);
    part_side_layout(c, s.side[0], nb, b1, b2, passes, false, kb, plan, 0);
    part_side_layout(c, s.side[1], np, b1, b2, passes, false, kb, plan, 1);
    s.item_prefix = c.take<unsigned long long>(P + 1);
    s.rec = c.take<ChunkRec>(kMaxOutWarps);
    s.ovf[0] = c.take<uint32_t>((size_t)kMaxOutWarps * kMaxRun);
    s.ovf[1] = c.take<uint32_t>((size_t)kMaxOutWarps * kMaxRun);
    s.fix = chunk_fix_layout(c);
    s.redo = c.take<unsigned long long>(P + (size_t)np / kDirectProbeChunk + 1);
    s.chained = c.take<uint32_t>(P + (size_t)np / kDirectProbeChunk + 1);
    return s;
}

cudaError_t phj_run(const JoinArgs& a, const PlanDev& plan, const PhjScratch& s, const JoinOut& out,
                    Ctrl* ctrl, cudaStream_t stream) {
    if (a.nb == 0 || a.np == 0) return cudaSuccess;  // no partition pair can match
    DevInfo di;
    cudaError_t e = current_device_info(&di);
    if (e != cudaSuccess) return e;
    // the two sides are partitioned concurrently: build on a second stream
    cudaStream_t side;
    if ((e = fork_side(stream, &side)) != cudaSuccess) return e;
    if ((e = partition_side(a.bkeys, a.nb, 0, plan, s.side[0], &out.b, &ctrl->err, side)) != cudaSuccess)
        return e;
    if ((e = partition_side(a.pkeys, a.np, 1, plan, s.side[1], &out.p, &ctrl->err, stream)) != cudaSuccess)
        return e;
    if ((e = join_side(stream, side)) != cudaSuccess) return e;
    const int passes = plan.variant == 3 ? 2 : 1;
    // GFTR: gather from the partitioned copies at the positions the join emits
    const JoinOut o = plan.gftr ? gftr_out(out, s.side[0], s.side[1], passes - 1) : out;
    const uint32_t P = 1u << (plan.bits1 + (passes == 2 ? plan.bits2 : 0));
    {
        ProfScope ps("phj_items", 32.0 * P, stream, 0.0, 2);
        items_count_kernel<<<(P + 255) / 256, 256, 0, stream>>>(
            s.side[0].part_start, s.side[1].part_start, P, build_chunk(plan.direct, out.aggregate && plan.gftr),
            plan.direct ? kDirectProbeChunk : kProbeChunk, s.item_prefix);
        items_scan_kernel<<<1, 1024, 0, stream>>>(s.item_prefix, P, ctrl);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    return plan.key32 ? launch_join<uint32_t>(s, plan, o, ctrl, di, stream, a.nb, a.np)
                      : launch_join<uint64_t>(s, plan, o, ctrl, di, stream, a.nb, a.np);
}

}  // namespace eiger
