// Group-by with aggregates (Sec. 3.3), chosen and sized from the HyperLogLog++
// estimate of the number of groups (Sec. 4.2: the group cardinality picks the
// algorithm and sizes the hash table).
//
// Keys travel as 32- or 64-bit offsets from the key minimum (frame of
// reference, Sec. 4.3). Aggregates are 64-bit: SUM modulo 2^64, COUNT, signed
// MIN and MAX, so every result is exact and independent of the order rows
// arrive in.
//
// HASH: one global open-addressing table (linear probing, slots a power of two
// sized from the estimate), keys claimed by CAS and aggregates updated by
// global atomics. While the groups fit shared memory, every CTA first aggregates
// its rows in a table of its own (CtaTable), then merges its groups into the
// global table; compaction writes the occupied slots out.
//
// PARTITION: the keys are radix-partitioned on hash bits (Sec. 3.3 hashes
// before partitioning so partitions are even) with the value columns carried
// along (gather from transformed relations), so that each partition's groups
// fit one shared-memory table; a persistent grid takes partitions from a
// global counter, aggregates each in shared memory and writes its groups out.
//
// What bounds the CTA tables' row loop: the shared-memory latency and
// wavefronts of a row's key group, its sums' atomics and its MIN / MAX read,
// about 26 wavefronts per 32 rows in the hash variant (2^26 rows, 3000 groups) and
// 31 in the partitions' (2^20 groups), with their clearing and writing out.
// Measured on GB300, int32 keys, SUM and MAX of
// int32 columns: 2^27 rows, 3000 groups, 4.27 ms (global atomics) -> 0.62 ms;
// 2^28 rows in 4096 partitions of 1024 groups, 3.97 -> 1.30 ms (64-bit words,
// lanes of equal slots combined by __match_any_sync and a leader's loop, one
// row per thread per round before).
//
// A key whose offset equals the empty-slot pattern (all ones: only possible
// when the key span is the whole 32- or 64-bit range) is aggregated in one
// extra slot past the table.
#include "kernels.cuh"
#include "keygroup.cuh"

namespace eiger {

namespace {

constexpr int kGbThreads = 512;
constexpr uint32_t kPartSlots = 4096;      // most slots of a partition's shared-memory table
constexpr size_t kGbSmemMax = 200 * 1024;   // most bytes of a CTA table of the hash variant
constexpr int kProbeCap = 1 << 20;         // probe steps before a global insert gives up

template <typename KeyT>
struct Empty;
template <>
struct Empty<uint32_t> {
    static constexpr uint32_t v = 0xFFFFFFFFu;
};
template <>
struct Empty<uint64_t> {
    static constexpr unsigned long long v = ~0ull;
};

__device__ __forceinline__ long long agg_init(int op) {
    return op == EIGER_AGG_MIN ? (long long)INT64_MAX : op == EIGER_AGG_MAX ? (long long)INT64_MIN : 0ll;
}

__device__ __forceinline__ long long agg_combine(int op, long long a, long long b) {
    switch (op) {
        case EIGER_AGG_SUM:
        case EIGER_AGG_COUNT:
            return (long long)((unsigned long long)a + (unsigned long long)b);
        case EIGER_AGG_MIN:
            return a < b ? a : b;
        default:
            return a > b ? a : b;
    }
}

// Adds v into *p (global memory) under op.
__device__ __forceinline__ void agg_atomic(int op, long long* p, long long v) {
    switch (op) {
        case EIGER_AGG_SUM:
        case EIGER_AGG_COUNT:
            atomicAdd(reinterpret_cast<unsigned long long*>(p), (unsigned long long)v);
            break;
        case EIGER_AGG_MIN:
            atomicMin(p, v);
            break;
        default:
            atomicMax(p, v);
    }
}

// The aggregates of a group-by: per aggregate its op, value column (of the
// caller, or carried through the partitioning) and width.
struct AggSpec {
    int n;
    int op[kMaxCols];
    const void* vals[kMaxCols];
    int bytes[kMaxCols];
};

__device__ __forceinline__ long long agg_value(const AggSpec& s, int a, uint32_t row) {
    if (s.op[a] == EIGER_AGG_COUNT) return 1;
    return s.bytes[a] == 4 ? (long long)__ldcs(static_cast<const int*>(s.vals[a]) + row)
                           : __ldcs(static_cast<const long long*>(s.vals[a]) + row);
}

// ------------------------------------------------------------------ hash variant

template <typename KeyT>
struct GbTable {
    KeyT* keys;         // [slots + 1]; keys[slots] unused (the special slot is flagged below)
    long long* aggs;    // [naggs][stride]
    unsigned* special;  // 1 when the all-ones key has been seen
    unsigned long long slots;
    unsigned long long stride;                // >= slots + 1
    const unsigned long long* slots_dev;      // when set, kernels read the slot count here
};

// Kernels that get a table whose size was decided on the device read it first.
template <typename KeyT>
__device__ __forceinline__ void resolve_slots(GbTable<KeyT>& t) {
    if (t.slots_dev) t.slots = *t.slots_dev;
}

template <typename KeyT>
__global__ void gb_init_kernel(GbTable<KeyT> t, AggSpec s) {
    resolve_slots(t);
    const unsigned long long total = t.slots + 1;
    for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; i < total;
         i += (unsigned long long)gridDim.x * blockDim.x) {
        t.keys[i] = Empty<KeyT>::v;
        for (int a = 0; a < s.n; ++a) t.aggs[(size_t)a * t.stride + i] = agg_init(s.op[a]);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *t.special = 0;
}

// Global slot of key k (claimed if new); t.slots for the all-ones key; or
// ~0ull when the probe cap is exhausted (error flagged).
template <typename KeyT>
__device__ __forceinline__ unsigned long long gb_global_slot(const GbTable<KeyT>& t, KeyT k, unsigned* err) {
    if (k == Empty<KeyT>::v) {
        atomicOr(t.special, 1u);
        return t.slots;
    }
    const unsigned long long mask = t.slots - 1;
    unsigned long long s = (unsigned long long)KeyCodec<KeyT>::hash(k) & mask;
    for (int step = 0; step < kProbeCap && (unsigned long long)step <= mask; ++step) {
        KeyT cur = t.keys[s];
        if (cur == k) return s;
        if (cur == Empty<KeyT>::v) {
            const KeyT prev = cas_key(t.keys + s, Empty<KeyT>::v, k);
            if (prev == Empty<KeyT>::v || prev == k) return s;
        }
        s = (s + 1) & mask;
    }
    atomicOr(err, kErrTableFull);
    return ~0ull;
}

template <typename InKey, typename KeyT>
__global__ void __launch_bounds__(kGbThreads)
    gb_hash_global_kernel(const InKey* __restrict__ keys, uint32_t n, uint64_t offset, GbTable<KeyT> t, AggSpec s,
                          unsigned* err) {
    const unsigned long long total = t.stride;
    for (unsigned long long rr = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; rr < n;
         rr += (unsigned long long)gridDim.x * blockDim.x) {
        const uint32_t r = (uint32_t)rr;
        const KeyT k = KeyCodec<KeyT>::encode((int64_t)__ldcs(keys + r), offset);
        const unsigned long long slot = gb_global_slot(t, k, err);
        if (slot == ~0ull) continue;
        for (int a = 0; a < s.n; ++a) agg_atomic(s.op[a], t.aggs + (size_t)a * total + slot, agg_value(s, a, r));
    }
}

// ------------------------------------------------------------------ CTA tables

// Aggregates of a CTA's shared-memory table, held in 32-bit words wherever the
// type allows: native shared-memory atomics are 32 bits wide, and a MIN or MAX
// is read first and updated only by a row that improves it (reads of one hot
// group are broadcast, its atomics would be serial).
//   kSum     two words (low, high): the low word's atomic returns the old value,
//            the high word takes the value's high half plus the carry, when
//            that is not zero;
//   kCount   one word (a CTA sees fewer than 2^32 rows);
//   kMin32.. one word: MIN and MAX of 4-byte columns;
//   kMin64.. 8 bytes: of 8-byte columns.
enum AggKind { kSum, kCount, kMin32, kMax32, kMin64, kMax64 };

// Layout of a CTA table: keys[slots + 1] (slots a multiple of 4), then per aggregate one cell per slot
// and copy. Every slot has 2^rlog copies of its aggregates, one per lane class,
// so that few groups do not serialise a warp's atomics; readers combine them.
// Slot `slots` is the special one.
struct CtaLayout {
    uint32_t slots;
    int rlog;
    int n;
    int kind[kMaxCols];
    uint32_t off[kMaxCols];  // bytes
    uint32_t bytes;
};

inline CtaLayout cta_layout(const AggSpec& s, uint32_t slots, int rlog, size_t key_bytes) {
    CtaLayout l{};
    l.slots = slots;
    l.rlog = rlog;
    l.n = s.n;
    size_t o = align_up((size_t)(slots + 1) * key_bytes, 16);
    const size_t cells = (size_t)(slots + 1) << rlog;
    for (int a = 0; a < s.n; ++a) {
        const bool wide = s.bytes[a] == 8;
        l.kind[a] = s.op[a] == EIGER_AGG_SUM     ? kSum
                    : s.op[a] == EIGER_AGG_COUNT ? kCount
                    : s.op[a] == EIGER_AGG_MIN   ? (wide ? kMin64 : kMin32)
                                                 : (wide ? kMax64 : kMax32);
        l.off[a] = (uint32_t)o;
        o = align_up(o + cells * (l.kind[a] == kCount || l.kind[a] == kMin32 || l.kind[a] == kMax32 ? 4 : 8), 16);
    }
    l.bytes = (uint32_t)o;
    return l;
}

template <typename KeyT>
struct CtaTable {
    KeyT* keys;
    unsigned char* base;
    const CtaLayout& l;
    uint32_t cells;

    __device__ CtaTable(unsigned char* smem, const CtaLayout& layout)
        : keys(reinterpret_cast<KeyT*>(smem)), base(smem), l(layout), cells((layout.slots + 1) << layout.rlog) {}

    __device__ void clear() {
        for (uint32_t i = threadIdx.x; i <= l.slots; i += blockDim.x) keys[i] = Empty<KeyT>::v;
        for (int a = 0; a < l.n; ++a) {
            uint32_t* w = reinterpret_cast<uint32_t*>(base + l.off[a]);
            long long* d = reinterpret_cast<long long*>(base + l.off[a]);
            switch (l.kind[a]) {
                case kSum:
                    for (uint32_t i = threadIdx.x; i < 2 * cells; i += blockDim.x) w[i] = 0;
                    break;
                case kCount:
                    for (uint32_t i = threadIdx.x; i < cells; i += blockDim.x) w[i] = 0;
                    break;
                case kMin32:
                    for (uint32_t i = threadIdx.x; i < cells; i += blockDim.x) w[i] = 0x7FFFFFFFu;
                    break;
                case kMax32:
                    for (uint32_t i = threadIdx.x; i < cells; i += blockDim.x) w[i] = 0x80000000u;
                    break;
                case kMin64:
                    for (uint32_t i = threadIdx.x; i < cells; i += blockDim.x) d[i] = INT64_MAX;
                    break;
                default:
                    for (uint32_t i = threadIdx.x; i < cells; i += blockDim.x) d[i] = INT64_MIN;
            }
        }
    }
    // Slots of J rows' keys (hashes h), claimed if new; the special slot for the
    // all-ones key; ~0u for a row without one (!ok, or the table is full). The
    // home groups of all rows are read first, which settles nearly every row;
    // the warp is brought together after each of the others.
    template <int J>
    __device__ __forceinline__ void slots_of(const KeyT (&k)[J], const uint32_t (&h)[J], const bool (&ok)[J],
                                             uint32_t (&slot)[J]) {
        KeyGroup<KeyT> g[J];
#pragma unroll
        for (int j = 0; j < J; ++j) {
            slot[j] = group_home<KeyT>(h[j], l.slots);
            g[j].load(keys + slot[j]);
        }
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const uint32_t i = g[j].first(k[j]);
            if (ok[j] && i < KeyGroup<KeyT>::kN && k[j] != Empty<KeyT>::v) {
                slot[j] += i;
            } else if (!ok[j]) {
                slot[j] = ~0u;
            } else if (k[j] == Empty<KeyT>::v) {
                keys[l.slots] = 0;  // taken
                slot[j] = l.slots;
            } else {
                bool fresh;
                slot[j] = claim_slot(keys, l.slots, k[j], slot[j], fresh);
            }
            __syncwarp();
        }
    }
    // Adds J rows' values (halves lo, hi) into the cells of aggregate a.
    template <int J>
    __device__ __forceinline__ void update(int a, const uint32_t (&cell)[J], const uint32_t (&lo)[J],
                                           const uint32_t (&hi)[J]) {
        uint32_t* w = reinterpret_cast<uint32_t*>(base + l.off[a]);
        int* si = reinterpret_cast<int*>(w);
        long long* d = reinterpret_cast<long long*>(w);
        switch (l.kind[a]) {
            case kSum:
#pragma unroll
                for (int j = 0; j < J; ++j)
                    if (cell[j] != ~0u) {
                        const uint32_t old = atomicAdd(w + cell[j], lo[j]);
                        const uint32_t h = hi[j] + (old + lo[j] < lo[j] ? 1u : 0u);
                        if (h) atomicAdd(w + cells + cell[j], h);
                    }
                break;
            case kCount:
#pragma unroll
                for (int j = 0; j < J; ++j)
                    if (cell[j] != ~0u) atomicAdd(w + cell[j], 1u);
                break;
            case kMin32:
#pragma unroll
                for (int j = 0; j < J; ++j)
                    if (cell[j] != ~0u && (int)lo[j] < *(volatile int*)(si + cell[j])) atomicMin(si + cell[j], (int)lo[j]);
                break;
            case kMax32:
#pragma unroll
                for (int j = 0; j < J; ++j)
                    if (cell[j] != ~0u && (int)lo[j] > *(volatile int*)(si + cell[j])) atomicMax(si + cell[j], (int)lo[j]);
                break;
            case kMin64:
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    const long long v = (long long)(((unsigned long long)hi[j] << 32) | lo[j]);
                    if (cell[j] != ~0u && v < *(volatile long long*)(d + cell[j])) atomicMin(d + cell[j], v);
                }
                break;
            default:
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    const long long v = (long long)(((unsigned long long)hi[j] << 32) | lo[j]);
                    if (cell[j] != ~0u && v > *(volatile long long*)(d + cell[j])) atomicMax(d + cell[j], v);
                }
        }
    }
    // Aggregate a of a slot, its copies combined.
    __device__ long long value(int a, int op, uint32_t slot) const {
        const uint32_t* w = reinterpret_cast<const uint32_t*>(base + l.off[a]);
        long long acc = agg_init(op);
        for (uint32_t c = slot << l.rlog, e = c + (1u << l.rlog); c < e; ++c) {
            long long v;
            switch (l.kind[a]) {
                case kSum: v = (long long)(((unsigned long long)w[cells + c] << 32) | w[c]); break;
                case kCount: v = (long long)w[c]; break;
                case kMin32:
                case kMax32: v = (long long)(int)w[c]; break;
                default: v = reinterpret_cast<const long long*>(w)[c];
            }
            acc = agg_combine(op, acc, v);
        }
        return acc;
    }
    __device__ bool taken(uint32_t slot) const { return keys[slot] != Empty<KeyT>::v; }
};

constexpr int kGbRows = 4;  // rows per thread per round

// Every warp of the CTA: aggregates rows [lo, hi) into the table, in rounds of
// kGbRows x 32 rows claimed from the counter *next (0 before): equal shares
// instead left the warps the scheduler favours waiting a third of the time for
// the others. key(r)
// gives a row's key, hash(k) its 32-bit hash; a row whose key finds the table
// full goes to full(k, r). N: aggregates held (at least s.n); W8: some value
// column is 8 bytes wide. A round's keys and values are all loaded before the
// first table access, so a row costs one round trip to memory.
template <typename KeyT, int N, bool W8, typename KeyF, typename HashF, typename FullF>
__device__ __forceinline__ void aggregate_rows(CtaTable<KeyT>& tab, const AggSpec& s, unsigned long long lo,
                                               unsigned long long hi, uint32_t* next, KeyF key, HashF hash,
                                               FullF full) {
    constexpr int J = kGbRows;
    const unsigned lane = lane_id();
    const uint32_t copy = lane & ((1u << tab.l.rlog) - 1u);
    for (;;) {
        uint32_t round = 0;
        if (lane == 0) round = atomicAdd(next, 1u);
        round = __shfl_sync(0xffffffffu, round, 0);
        const unsigned long long base = lo + (unsigned long long)round * (J * kWarp);
        if (base >= hi) break;
        KeyT k[J];
        uint32_t v[N][J], vh[W8 ? N : 1][J];
        bool ok[J];
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const unsigned long long r = base + j * kWarp + lane;
            ok[j] = r < hi;
            if (ok[j]) k[j] = key((uint32_t)r);
        }
#pragma unroll
        for (int a = 0; a < N; ++a) {
            if (a >= s.n || s.op[a] == EIGER_AGG_COUNT) continue;
            const uint32_t r0 = (uint32_t)base + lane;
            if (W8 && s.bytes[a] == 8) {
                const uint2* p = static_cast<const uint2*>(s.vals[a]) + r0;
#pragma unroll
                for (int j = 0; j < J; ++j)
                    if (ok[j]) {
                        const uint2 x = __ldcs(p + j * kWarp);
                        v[a][j] = x.x;
                        vh[W8 ? a : 0][j] = x.y;
                    }
            } else {
                const uint32_t* p = static_cast<const uint32_t*>(s.vals[a]) + r0;
#pragma unroll
                for (int j = 0; j < J; ++j)
                    if (ok[j]) {
                        v[a][j] = __ldcs(p + j * kWarp);
                        if (W8) vh[W8 ? a : 0][j] = (uint32_t)((int)v[a][j] >> 31);
                    }
            }
        }
        // (left to itself the warp drifts apart in the searches and stays so for
        // the rest of the round: 3 lanes per instruction, the value loads sunk
        // into the divergent code, a fourteenth of the speed)
        __syncwarp();
        uint32_t h[J], cell[J];
#pragma unroll
        for (int j = 0; j < J; ++j) h[j] = hash(k[j]);
        tab.template slots_of<J>(k, h, ok, cell);
#pragma unroll
        for (int j = 0; j < J; ++j) {
            if (cell[j] != ~0u)
                cell[j] = (cell[j] << tab.l.rlog) + copy;
            else if (ok[j])
                full(k[j], (uint32_t)(base + j * kWarp + lane));
        }
        __syncwarp();
#pragma unroll
        for (int a = 0; a < N; ++a) {
            if (a >= s.n) continue;
            if constexpr (W8) {
                tab.update<J>(a, cell, v[a], vh[a]);
            } else {
                uint32_t sign[J];
#pragma unroll
                for (int j = 0; j < J; ++j) sign[j] = (uint32_t)((int)v[a][j] >> 31);
                tab.update<J>(a, cell, v[a], sign);
            }
            __syncwarp();
        }
    }
}

// Adds the CTA table's groups into a global table.
template <typename KeyT>
__device__ __forceinline__ void merge_groups(const CtaTable<KeyT>& tab, const AggSpec& s, const GbTable<KeyT>& t,
                                             unsigned* err) {
    for (uint32_t i = threadIdx.x; i <= tab.l.slots; i += blockDim.x) {
        if (!tab.taken(i)) continue;
        const unsigned long long g = gb_global_slot(t, i == tab.l.slots ? KeyT(Empty<KeyT>::v) : tab.keys[i], err);
        if (g == ~0ull) continue;
        for (int a = 0; a < s.n; ++a) agg_atomic(s.op[a], t.aggs + (size_t)a * t.stride + g, tab.value(a, s.op[a], i));
    }
}

// Hash variant with CTA tables: a contiguous row range per CTA; rows whose key
// finds the CTA's table full (an estimate far too low) go to the global table.
template <typename InKey, typename KeyT, int N, bool W8>
__global__ void __launch_bounds__(1024, 1)
    gb_hash_smem_kernel(const InKey* __restrict__ keys, uint32_t n, uint64_t offset, GbTable<KeyT> t,
                        const __grid_constant__ AggSpec s, const __grid_constant__ CtaLayout layout, unsigned* err) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_next;
    CtaTable<KeyT> tab(smem, layout);
    tab.clear();
    if (threadIdx.x == 0) s_next = 0;
    __syncthreads();
    const unsigned long long per = ((unsigned long long)n + gridDim.x - 1) / gridDim.x;
    const unsigned long long lo = blockIdx.x * per;
    const unsigned long long hi = lo + per < n ? lo + per : n;
    aggregate_rows<KeyT, N, W8>(
        tab, s, lo, hi, &s_next, [&](uint32_t r) { return KeyCodec<KeyT>::encode((int64_t)__ldcs(keys + r), offset); },
        [&](KeyT k) {
            return (uint32_t)(KeyCodec<KeyT>::mix(k, KeyCodec<KeyT>::kBits) >> (KeyCodec<KeyT>::kBits - 32));
        },
        [&](KeyT k, uint32_t r) {
            const unsigned long long g = gb_global_slot(t, k, err);
            if (g != ~0ull)
                for (int a = 0; a < s.n; ++a) agg_atomic(s.op[a], t.aggs + (size_t)a * t.stride + g, agg_value(s, a, r));
        });
    __syncthreads();
    merge_groups(tab, s, t, err);
}

// Output of a group-by: keys in the caller's dtype and one int64 column per aggregate.
struct GbOut {
    void* keys;
    int key_bytes;
    long long* aggs[kMaxCols];
    unsigned long long capacity;
};

__device__ __forceinline__ void write_group(const GbOut& o, unsigned long long pos, int64_t key, const long long* v,
                                            int naggs) {
    if (pos >= o.capacity) return;
    if (o.key_bytes == 4)
        static_cast<int32_t*>(o.keys)[pos] = (int32_t)key;
    else
        static_cast<int64_t*>(o.keys)[pos] = key;
    for (int a = 0; a < naggs; ++a) o.aggs[a][pos] = v[a];
}

// Occupied slots of the global table -> output, reserved per warp. mixed_bits:
// the table holds partitioned (mixed) keys; 0: encoded keys.
template <typename KeyT>
__global__ void gb_compact_kernel(GbTable<KeyT> t, AggSpec s, uint64_t offset, int mixed_bits, GbOut o, Ctrl* ctrl) {
    resolve_slots(t);
    const unsigned long long total = t.slots + 1;
    const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
    const unsigned long long start = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    const unsigned long long rounds = (total + stride - 1) / stride;
    for (unsigned long long it = 0; it < rounds; ++it) {
        const unsigned long long i = start + it * stride;
        bool has = false;
        if (i < t.slots)
            has = t.keys[i] != Empty<KeyT>::v;
        else if (i == t.slots)
            has = *t.special != 0;
        const unsigned m = __ballot_sync(0xffffffffu, has);
        if (!m) continue;
        const int leader = __ffs(m) - 1;
        unsigned long long base = 0;
        if ((int)lane_id() == leader) base = atomicAdd(&ctrl->cursor, (unsigned long long)__popc(m));
        base = __shfl_sync(0xffffffffu, base, leader);
        if (has) {
            KeyT k = i == t.slots ? Empty<KeyT>::v : t.keys[i];
            if (mixed_bits) k = KeyCodec<KeyT>::unmix(k, mixed_bits);
            long long v[kMaxCols];
            for (int a = 0; a < s.n; ++a) v[a] = t.aggs[(size_t)a * t.stride + i];
            write_group(o, base + __popc(m & lanemask_lt()), (int64_t)((uint64_t)k + offset), v, s.n);
        }
    }
}

// ------------------------------------------------------------------ partition variant

// Rows per work item of the partition variant: one and a half average
// partitions while the partitions alone fill the chip several times over, so
// that an ordinary partition is one item and writes its groups straight out
// (2^28 rows over 4096 partitions cut at 65536 rows each, their average: half
// of them merged through the spill table, 0.47 ms more); else the rows over
// eight items per SM. At least gb_min_chunk: the spill table is sized for it.
inline uint32_t gb_min_chunk(unsigned long long n) { return n >= (1ull << 24) ? 65536u : 16384u; }

inline uint32_t gb_chunk(unsigned long long n, uint32_t P, int sms) {
    unsigned long long c = P >= (uint32_t)(8 * sms) ? 3 * n / (2ull * P) : n / (8ull * sms);
    const unsigned long long lo = gb_min_chunk(n);
    return (uint32_t)(c < lo ? lo : c > (1u << 20) ? (1u << 20) : c);
}

template <typename KeyT>
struct GbPartIn {
    const KeyT* key;                          // partitioned keys
    const uint32_t* start;                    // [P + 1]
    const unsigned long long* item_prefix;    // [P + 1] work items before each partition
    uint32_t P;
    uint32_t chunk;                           // rows per work item
    int pbits;                                // partition bits (the top bits of the mixed keys)
    AggSpec s;                                // value columns: the partitioned copies
    CtaLayout layout;
};

// One block: work items per partition (row chunks of `chunk`), their
// exclusive prefix, the item total (ctrl->nitems) and the slots of the spill
// table for the groups of partitions that span several items: at most
// kPartSlots groups each, at load <= 1/2, capped at spill_max.
__global__ void __launch_bounds__(1024)
    gb_items_kernel(const uint32_t* __restrict__ start, uint32_t P, unsigned long long* __restrict__ prefix,
                    Ctrl* ctrl, unsigned long long* spill_slots, unsigned long long spill_max, uint32_t chunk) {
    __shared__ unsigned long long s_w[1024 / kWarp];
    __shared__ unsigned long long s_m[1024 / kWarp];
    const unsigned lane = lane_id();
    const int w = threadIdx.x / kWarp;
    unsigned long long carry = 0, multi = 0;
    for (uint32_t base = 0; base < P; base += blockDim.x) {
        const uint32_t p = base + threadIdx.x;
        unsigned long long items = 0;
        if (p < P) {
            const uint32_t rows = start[p + 1] - start[p];
            items = (rows + (unsigned long long)chunk - 1) / chunk;
        }
        unsigned long long x = items, m = items > 1;
#pragma unroll
        for (int o = 1; o < kWarp; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
            const unsigned long long z = __shfl_up_sync(0xffffffffu, m, o);
            if ((int)lane >= o) {
                x += y;
                m += z;
            }
        }
        if ((int)lane == kWarp - 1) {
            s_w[w] = x;
            s_m[w] = m;
        }
        __syncthreads();
        if (w == 0) {
            unsigned long long t = s_w[lane], u = s_m[lane];
#pragma unroll
            for (int o = 1; o < kWarp; o <<= 1) {
                const unsigned long long y = __shfl_up_sync(0xffffffffu, t, o);
                const unsigned long long z = __shfl_up_sync(0xffffffffu, u, o);
                if ((int)lane >= o) {
                    t += y;
                    u += z;
                }
            }
            s_w[lane] = t;
            s_m[lane] = u;
        }
        __syncthreads();
        if (p < P) prefix[p] = carry + (w ? s_w[w - 1] : 0ull) + x - items;
        carry += s_w[kWarp - 1];
        multi += s_m[kWarp - 1];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        prefix[P] = carry;
        ctrl->nitems = carry;
        unsigned long long sl = 64;
        while (sl < 2ull * kPartSlots * multi && sl < spill_max) sl <<= 1;
        *spill_slots = multi ? (sl < spill_max ? sl : spill_max) : 0ull;
    }
}

// A persistent grid takes work items (a partition's chunk of rows) from a
// global counter and aggregates each in a shared-memory table. A partition
// that is one item writes its groups out directly; the items of a larger
// partition (few groups, many rows) merge their groups into the spill table,
// which is compacted afterwards.
template <typename KeyT, int N, bool W8>
__global__ void __launch_bounds__(kGbThreads, 2)
    gb_part_kernel(const __grid_constant__ GbPartIn<KeyT> a, GbTable<KeyT> spill, uint64_t offset, int kbits,
                   const __grid_constant__ GbOut o, Ctrl* ctrl) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_warp[kGbThreads / kWarp];
    __shared__ unsigned long long s_item;
    __shared__ uint32_t s_part;
    __shared__ unsigned long long s_base;
    __shared__ int s_full;
    __shared__ uint32_t s_next;
    resolve_slots(spill);
    CtaTable<KeyT> tab(smem, a.layout);
    const unsigned long long nitems = ctrl->nitems;
    const unsigned lane = lane_id();
    const int w = threadIdx.x / kWarp;
    for (;;) {
        if (threadIdx.x < kWarp) {
            unsigned long long it = 0;
            if (threadIdx.x == 0) it = atomicAdd(&ctrl->next_item, 1ull);
            it = __shfl_sync(0xffffffffu, it, 0);
            const uint32_t p =
                it < nitems ? warp_last_le(a.P, it, [&](uint32_t i) { return a.item_prefix[i]; }) : 0u;
            if (threadIdx.x == 0) {
                s_item = it;
                s_part = p;
                s_full = 0;
                s_next = 0;
            }
        }
        tab.clear();
        __syncthreads();
        const unsigned long long item = s_item;
        if (item >= nitems) break;
        const uint32_t p = s_part;
        const unsigned long long c = item - a.item_prefix[p];
        const bool multi = a.item_prefix[p + 1] - a.item_prefix[p] > 1;
        const uint32_t pend = a.start[p + 1];
        const unsigned long long beg = (unsigned long long)a.start[p] + c * a.chunk;
        const unsigned long long end = beg + a.chunk < pend ? beg + a.chunk : pend;
        aggregate_rows<KeyT, N, W8>(
            tab, a.s, beg, end, &s_next, [&](uint32_t r) { return __ldcs(a.key + r); },
            [&](KeyT k) { return (uint32_t)((KeyT)(k << a.pbits) >> (KeyCodec<KeyT>::kBits - 32)); },
            [&](KeyT, uint32_t) { s_full = 1; });
        __syncthreads();
        if (s_full) {  // more groups than one table: the host repartitions with more bits
            if (threadIdx.x == 0) atomicOr(&ctrl->err, kErrTableFull);
            __syncthreads();
            continue;
        }
        if (multi) {
            merge_groups(tab, a.s, spill, &ctrl->err);
            __syncthreads();
            continue;
        }
        // Compact: each warp owns a run of slots; the warps' counts are scanned,
        // one global reservation, then the warps write their groups in slot
        // order, lane by lane on consecutive output positions.
        const uint32_t per = ((a.layout.slots + 1 + kGbThreads - 1) / kGbThreads) * kWarp;  // slots per warp
        const uint32_t s0 = w * per, s1 = min(s0 + per, a.layout.slots + 1);
        uint32_t cnt = 0;
        for (uint32_t i = s0 + lane; i < s1; i += kWarp) cnt += tab.taken(i);
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (lane == 0) s_warp[w] = cnt;
        __syncthreads();
        if (w == 0) {
            uint32_t v = (int)lane < kGbThreads / kWarp ? s_warp[lane] : 0u;
            const uint32_t own = v;
#pragma unroll
            for (int off = 1; off < kWarp; off <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, v, off);
                if ((int)lane >= off) v += y;
            }
            if ((int)lane < kGbThreads / kWarp) s_warp[lane] = v - own;
            if (lane == kWarp - 1) s_base = v ? atomicAdd(&ctrl->cursor, (unsigned long long)v) : 0ull;
        }
        __syncthreads();
        unsigned long long pos = s_base + s_warp[w];
        for (uint32_t i0 = s0; i0 < s1; i0 += kWarp) {
            const uint32_t i = i0 + lane;
            const bool has = i < s1 && tab.taken(i);
            const unsigned m = __ballot_sync(0xffffffffu, has);
            if (has) {
                const KeyT k = i == a.layout.slots ? Empty<KeyT>::v : tab.keys[i];
                long long v[kMaxCols];
                for (int b = 0; b < a.s.n; ++b) v[b] = tab.value(b, a.s.op[b], i);
                write_group(o, pos + __popc(m & lanemask_lt()),
                            (int64_t)((uint64_t)KeyCodec<KeyT>::unmix(k, kbits) + offset), v, a.s.n);
            }
            pos += __popc(m);
        }
        __syncthreads();
    }
}

// Whether some value column is 8 bytes wide.
inline bool wide_values(const AggSpec& s) {
    for (int a = 0; a < s.n; ++a)
        if (s.op[a] != EIGER_AGG_COUNT && s.bytes[a] == 8) return true;
    return false;
}

template <typename KeyT>
size_t gb_global_bytes(unsigned long long slots, int naggs) {
    return align_up((size_t)(slots + 1) * sizeof(KeyT), 256) + (size_t)naggs * (slots + 1) * 8 + 256;
}

constexpr size_t kGbHalfSm = 112 * 1024;  // table bytes that let two CTAs share an SM

// CTA table of the hash variant: copies of the aggregates while they fit 48 KB
// (several CTAs per SM), at most one per lane.
template <typename KeyT>
CtaLayout hash_cta_layout(const AggSpec& s, uint32_t slots) {
    int rlog = 0;
    while (rlog < 5 && cta_layout(s, slots, rlog + 1, sizeof(KeyT)).bytes <= 48 * 1024) ++rlog;
    return cta_layout(s, slots, rlog, sizeof(KeyT));
}

template <typename InKey, typename KeyT>
cudaError_t gb_hash_run(const GbArgs& g, const GbPlanDev& plan, const GbScratch& sc, const AggSpec& s,
                        const GbOut& o, Ctrl* ctrl, const DevInfo& di, cudaStream_t stream) {
    GbTable<KeyT> t;
    Carve c{static_cast<char*>(sc.table), 0};
    t.keys = c.take<KeyT>(plan.slots + 1);
    t.aggs = c.take<long long>((size_t)s.n * (plan.slots + 1));
    t.special = c.take<unsigned>(1);
    t.slots = plan.slots;
    t.stride = plan.slots + 1;
    t.slots_dev = nullptr;
    cudaError_t e;
    const double kb = (double)sizeof(KeyT);
    {
        ProfScope ps("gb_init", (kb + 8.0 * s.n) * (double)(plan.slots + 1), stream);
        const unsigned long long blocks = (plan.slots + 1 + 255) / 256;
        gb_init_kernel<KeyT><<<(int)(blocks < 4096 ? blocks : 4096), 256, 0, stream>>>(t, s);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    double vbytes = 0;
    for (int a = 0; a < s.n; ++a) vbytes += s.op[a] == EIGER_AGG_COUNT ? 0 : s.bytes[a];
    const uint32_t n = (uint32_t)g.n;
    if (plan.smem_slots) {
        const bool w8 = wide_values(s);
        auto kern = s.n <= 1   ? (w8 ? gb_hash_smem_kernel<InKey, KeyT, 1, true> : gb_hash_smem_kernel<InKey, KeyT, 1, false>)
                    : s.n == 2 ? (w8 ? gb_hash_smem_kernel<InKey, KeyT, 2, true> : gb_hash_smem_kernel<InKey, KeyT, 2, false>)
                               : (w8 ? gb_hash_smem_kernel<InKey, KeyT, 4, true> : gb_hash_smem_kernel<InKey, KeyT, 4, false>);
        const CtaLayout l = hash_cta_layout<KeyT>(s, plan.smem_slots);
        if ((e = allow_smem(kern)) != cudaSuccess) return e;
        // a table that leaves room for a second CTA runs 512 threads each, a
        // larger one 1024; no more CTAs than rounds of rows
        const int threads = l.bytes <= kGbHalfSm ? 512 : 1024;
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, l.bytes) != cudaSuccess || per_sm < 1)
            per_sm = 1;
        const unsigned long long want = ((unsigned long long)n + threads * kGbRows - 1) / (threads * kGbRows);
        const int grid = want < (unsigned long long)di.sms * per_sm ? (int)want : di.sms * per_sm;
        ProfScope ps("gb_hash_smem", ((double)sizeof(InKey) + vbytes) * (double)n, stream);
        kern<<<grid, threads, l.bytes, stream>>>(static_cast<const InKey*>(g.keys), n, plan.offset, t, s, l, &ctrl->err);
    } else {
        ProfScope ps("gb_hash_global", ((double)sizeof(InKey) + vbytes) * (double)n, stream);
        gb_hash_global_kernel<InKey, KeyT><<<di.sms * 4, kGbThreads, 0, stream>>>(
            static_cast<const InKey*>(g.keys), n, plan.offset, t, s, &ctrl->err);
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    ProfScope ps("gb_compact", (kb + 8.0 * s.n) * (double)(plan.slots + 1), stream,
                 (double)sizeof(InKey) + 8.0 * s.n);
    const unsigned long long blocks = (plan.slots + 1 + 255) / 256;
    gb_compact_kernel<KeyT><<<(int)(blocks < 8192 ? blocks : 8192), 256, 0, stream>>>(t, s, plan.offset, 0, o, ctrl);
    return cudaGetLastError();
}

template <typename InKey, typename KeyT>
cudaError_t gb_part_run(const GbArgs& g, const GbPlanDev& plan, const GbScratch& sc, const AggSpec& s,
                        const GbOut& o, Ctrl* ctrl, const DevInfo& di, cudaStream_t stream) {
    // partition the keys with the value columns carried along
    PlanDev pd{};
    pd.variant = plan.bits2 ? EIGER_PHJ2 : EIGER_PHJ1;
    pd.bits1 = plan.bits1;
    pd.bits2 = plan.bits2;
    pd.narrow = sizeof(KeyT) == 4;
    pd.key32 = sizeof(KeyT) == 4;
    pd.dtype = sizeof(InKey) == 4 ? EIGER_I32 : EIGER_I64;
    pd.range.lo = INT64_MIN;
    pd.range.hi = INT64_MAX;
    pd.range.offset = plan.offset;
    pd.check_range = 0;
    pd.kbits = plan.kbits;
    pd.no_rows = 1;  // groups are aggregated from the carried columns by position
    ColSide carry{};
    int nc = 0;
    int col_of[kMaxCols];
    for (int a = 0; a < s.n; ++a) {
        col_of[a] = -1;
        if (s.op[a] == EIGER_AGG_COUNT) continue;
        carry.src[nc] = s.vals[a];
        carry.bytes[nc] = s.bytes[a];
        col_of[a] = nc++;
    }
    carry.n = nc;
    pd.gftr = nc > 0;
    pd.ncols[0] = nc;
    for (int q = 0; q < nc; ++q) pd.col_bytes[0][q] = carry.bytes[q];
    cudaError_t e = partition_side(g.keys, g.n, 0, pd, sc.part, &carry, &ctrl->err, stream);
    if (e != cudaSuccess) return e;
    const int buf = plan.bits2 ? 1 : 0;
    const uint32_t P = 1u << (plan.bits1 + plan.bits2);
    const uint32_t chunk = gb_chunk((unsigned long long)g.n, P, di.sms);
    GbTable<KeyT> spill;
    {
        Carve c{static_cast<char*>(sc.spill), 0};
        spill.keys = c.take<KeyT>(sc.spill_max + 1);
        spill.aggs = c.take<long long>((size_t)s.n * (sc.spill_max + 1));
        spill.special = c.take<unsigned>(1);
        spill.slots = sc.spill_max;
        spill.stride = sc.spill_max + 1;
        spill.slots_dev = sc.spill_slots;
    }
    {
        ProfScope ps("gb_items", 8.0 * P, stream, 0.0, 2);
        gb_items_kernel<<<1, 1024, 0, stream>>>(sc.part.part_start, P, sc.item_prefix, ctrl, sc.spill_slots,
                                                sc.spill_max, chunk);
        gb_init_kernel<KeyT><<<di.sms * 2, 256, 0, stream>>>(spill, s);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    GbPartIn<KeyT> in;
    in.key = static_cast<const KeyT*>(sc.part.key[buf]);
    in.start = sc.part.part_start;
    in.item_prefix = sc.item_prefix;
    in.P = P;
    in.chunk = chunk;
    in.pbits = plan.bits1 + plan.bits2;
    in.s = s;
    for (int a = 0; a < s.n; ++a)
        if (col_of[a] >= 0) in.s.vals[a] = sc.part.col[buf][col_of[a]];
    in.layout = cta_layout(s, plan.part_slots, 0, sizeof(KeyT));
    const bool w8 = wide_values(s);
    auto kern = s.n <= 1   ? (w8 ? gb_part_kernel<KeyT, 1, true> : gb_part_kernel<KeyT, 1, false>)
                : s.n == 2 ? (w8 ? gb_part_kernel<KeyT, 2, true> : gb_part_kernel<KeyT, 2, false>)
                           : (w8 ? gb_part_kernel<KeyT, 4, true> : gb_part_kernel<KeyT, 4, false>);
    const size_t smem = in.layout.bytes;
    if ((e = allow_smem(kern)) != cudaSuccess) return e;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kGbThreads, smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    double vbytes = 0;
    for (int a = 0; a < s.n; ++a) vbytes += s.op[a] == EIGER_AGG_COUNT ? 0 : s.bytes[a];
    {
        ProfScope ps("gb_part", ((double)sizeof(KeyT) + vbytes) * (double)g.n, stream,
                     (double)sizeof(InKey) + 8.0 * s.n);
        kern<<<di.sms * per_sm, kGbThreads, smem, stream>>>(in, spill, plan.offset, plan.kbits, o, ctrl);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    // the groups of multi-item partitions (an empty spill table when there are none)
    ProfScope ps("gb_spill_compact", 0.0, stream);
    gb_compact_kernel<KeyT><<<di.sms * 2, 256, 0, stream>>>(spill, s, plan.offset, plan.kbits, o, ctrl);
    return cudaGetLastError();
}

}  // namespace

uint32_t gb_part_slots(double groups) {
    const double want = 3.75 * groups + 64.0;
    return want < (double)kPartSlots ? (uint32_t)want & ~3u : kPartSlots;
}

uint32_t gb_hash_slots(double groups, const GbAggs& aggs, bool key32) {
    AggSpec s{};
    s.n = aggs.n;
    for (int a = 0; a < aggs.n; ++a) {
        s.op[a] = aggs.op[a];
        s.bytes[a] = aggs.bytes[a];
    }
    const size_t kb = key32 ? 4 : 8;
    const double per_slot = (double)cta_layout(s, 4096, 0, kb).bytes / 4097.0;
    const double most = (double)(kGbSmemMax - 1024) / per_slot - 8.0;
    double want = 3.5 * groups + 64.0;
    if (want > most) want = most;
    return want >= 1.6 * groups + 64.0 ? (uint32_t)want & ~3u : 0;
}

GbScratch gb_layout(Carve& c, int64_t n, const GbPlanDev& plan, const int* col_bytes, int ncols) {
    GbScratch s{};
    if (plan.variant == EIGER_GB_HASH) {
        const size_t b = plan.key32 ? gb_global_bytes<uint32_t>(plan.slots, plan.naggs)
                                    : gb_global_bytes<uint64_t>(plan.slots, plan.naggs);
        s.table = c.take<unsigned char>(b);
    } else {
        PlanDev pd{};
        pd.gftr = ncols > 0;
        pd.ncols[0] = ncols;
        for (int q = 0; q < ncols; ++q) pd.col_bytes[0][q] = col_bytes[q];
        const int passes = plan.bits2 ? 2 : 1;
        part_side_layout(c, s.part, n, plan.bits1, plan.bits2, passes, false, plan.key32 ? 4 : 8, pd, 0);
        // spill table: each multi-item partition has more than a chunk's rows and
        // at most kPartSlots groups; load <= 1/2
        const unsigned long long nn = n > 0 ? (unsigned long long)n : 1ull;
        unsigned long long groups = (nn / gb_min_chunk(nn) + 1) * kPartSlots;
        if (groups > nn) groups = nn;
        unsigned long long sl = 64;
        while (sl < 2 * groups) sl <<= 1;
        s.spill_max = sl;
        s.spill = c.take<unsigned char>(plan.key32 ? gb_global_bytes<uint32_t>(sl, plan.naggs)
                                                   : gb_global_bytes<uint64_t>(sl, plan.naggs));
        s.spill_slots = c.take<unsigned long long>(1);
        s.item_prefix = c.take<unsigned long long>(((size_t)1 << (plan.bits1 + plan.bits2)) + 1);
    }
    return s;
}

cudaError_t gb_run(const GbArgs& g, const GbPlanDev& plan, const GbScratch& sc, const GbAggs& aggs, void* out_keys,
                   unsigned long long capacity, Ctrl* ctrl, cudaStream_t stream) {
    if (g.n == 0) return cudaSuccess;
    DevInfo di;
    cudaError_t e = current_device_info(&di);
    if (e != cudaSuccess) return e;
    AggSpec s{};
    s.n = aggs.n;
    GbOut o{};
    o.keys = out_keys;
    o.key_bytes = g.dtype == EIGER_I32 ? 4 : 8;
    o.capacity = capacity;
    for (int a = 0; a < aggs.n; ++a) {
        s.op[a] = aggs.op[a];
        s.vals[a] = aggs.vals[a];
        s.bytes[a] = aggs.bytes[a];
        o.aggs[a] = aggs.out[a];
    }
    const bool i32 = g.dtype == EIGER_I32;
    if (plan.variant == EIGER_GB_HASH) {
        if (plan.key32)
            return i32 ? gb_hash_run<int32_t, uint32_t>(g, plan, sc, s, o, ctrl, di, stream)
                       : gb_hash_run<int64_t, uint32_t>(g, plan, sc, s, o, ctrl, di, stream);
        return gb_hash_run<int64_t, uint64_t>(g, plan, sc, s, o, ctrl, di, stream);
    }
    if (plan.key32)
        return i32 ? gb_part_run<int32_t, uint32_t>(g, plan, sc, s, o, ctrl, di, stream)
                   : gb_part_run<int64_t, uint32_t>(g, plan, sc, s, o, ctrl, di, stream);
    return gb_part_run<int64_t, uint64_t>(g, plan, sc, s, o, ctrl, di, stream);
}

}  // namespace eiger
