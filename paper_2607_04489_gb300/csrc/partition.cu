// Radix partitioning for the partitioned hash join (Sec. 3.2, the PHJ the
// paper adopts; partitions are taken on bits of a hash of the key so their
// sizes are even, as Sec. 3.3 does before partitioning).
//
// Each pass splits every input segment by `bits` further bits of the mixed key:
// pass 1 by the top b1 bits, pass 2 by the next b2 bits within each pass-1
// partition. A pass runs three steps over fixed tiles of kPartTile rows:
//   hist    per tile, a shared-memory histogram of the digits, written to a
//           counts array laid out [segment][digit][tile-in-segment];
//   scan    one device-wide exclusive scan of that array, which turns every
//           (tile, digit) count into the global output offset of that tile's
//           run of the digit (segments stay contiguous and in order);
//   scatter per tile, place each row behind its digit's run with a
//           shared-memory atomic, staging the tile in shared memory grouped by
//           digit, then write each digit run to its global offset with
//           consecutive threads on consecutive addresses (coalesced runs
//           instead of one scattered 8-byte store per row).
// The first pass reads the raw key column (row ids are implicit), applies the
// probe-side range test (a probe key outside [min_R, max_R] cannot match and
// is dropped here), the frame-of-reference narrowing and the key mix; later
// passes read the (mixed key', row) pairs of the previous pass.
#include <cstdio>
#include <type_traits>

#include "kernels.cuh"

namespace eiger {

namespace {

#ifndef EIGER_PART_THREADS
#define EIGER_PART_THREADS 512
#endif
constexpr int kPartThreads = EIGER_PART_THREADS;
constexpr int kPartItems = kPartTile / kPartThreads;  // rows per thread per tile
constexpr uint32_t kNoDigit = 0xFFFFFFFFu;

constexpr int kScanThreads = 512;
constexpr int kScanItems = 16;
constexpr int kScanChunk = kScanThreads * kScanItems;

// Payload columns that travel with the keys (GFTR): read at the tile rows of
// `in`, written to the same output positions as the keys.
struct ColCarry {
    const void* in[kMaxCols];
    void* out[kMaxCols];
    int bytes[kMaxCols];
    int n;
};

template <typename InKey, typename KeyT>
struct PartPass {
    const InKey* raw;        // pass 1 input: raw key column
    const KeyT* in_key;      // later passes: previous pass output
    const uint32_t* in_idx;
    KeyT* out_key;
    uint32_t* out_idx;
    uint32_t n;              // pass 1: rows
    uint64_t offset;         // pass 1: key' = key - offset (modulo the key's width),
    uint64_t span;           // rows with key' > span are dropped
    int dshift;              // digit = (key' >> dshift) & dmask
    uint32_t dmask;
    int bits;
    int kbits;               // hash partitioning: bits of the key mix
    uint32_t* counts;
    uint32_t* scan_done;     // chunks the scan has summed; the histogram clears it
    const Tile* tiles;       // nullptr: pass-1 tiling of [0, n)
    const uint32_t* ntiles_dev;
    uint32_t ntiles_fixed;
    ColCarry cc;
    int col_apart;           // hash scatter: the first column batch has a stage of its own
    // Exclusive ends of the memory a tile load may read around its rows (key
    // source, tuple-ID source); the arrays' bases are the starts. A tile whose
    // 16-byte aligned cover [align_down(first), align_up(last + 1)) lies
    // inside is loaded by one bulk copy of the cover; nullptr: never.
    const void* src_end[2];
};

template <typename InKey, typename KeyT>
__device__ __forceinline__ Tile get_tile(const PartPass<InKey, KeyT>& a, uint32_t t) {
    if (a.tiles) return a.tiles[t];
    Tile tl;
    tl.start = t * (uint32_t)kPartTile;
    const uint32_t rest = a.n - tl.start;
    tl.len = rest < (uint32_t)kPartTile ? rest : (uint32_t)kPartTile;
    tl.seg = 0;
    tl.tile_base = 0;
    tl.ntiles_seg = a.ntiles_fixed;
    return tl;
}

__device__ __forceinline__ size_t count_index(const Tile& tl, uint32_t t, uint32_t d, int bits) {
    return ((size_t)tl.tile_base << bits) + (size_t)d * tl.ntiles_seg + (t - tl.tile_base);
}

// Partition digit: bits of the carried key (mixed by pass 1 for hash
// partitioning, the encoded key itself for the sort).
template <typename KeyT>
__device__ __forceinline__ uint32_t digit_of(KeyT k, int dshift, uint32_t dmask) {
    return (uint32_t)(k >> dshift) & dmask;
}

// Exclusive scan of in[0, n) into out[0, n), n <= kPartItems * blockDim.x.
// Block-collective; returns the total. s_warp: blockDim.x / 32 words. With
// `rebase`, also rebase[i] -= out[i] for every i (by the thread that wrote
// out[i], so no barrier is needed in between).
__device__ uint32_t block_scan_smem(const uint32_t* in, uint32_t* out, uint32_t n, uint32_t* s_warp,
                                    uint32_t* rebase = nullptr) {
    const uint32_t per = (n + blockDim.x - 1) / blockDim.x;
    uint32_t beg = threadIdx.x * per;
    if (beg > n) beg = n;
    uint32_t end = beg + per;
    if (end > n) end = n;
    uint32_t local = 0;
    for (uint32_t i = beg; i < end; ++i) local += in[i];
    uint32_t x = local;
    const unsigned lane = lane_id();
#pragma unroll
    for (int o = 1; o < kWarp; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if ((int)lane >= o) x += y;
    }
    const int warp = threadIdx.x / kWarp;
    const int nw = blockDim.x / kWarp;
    __syncthreads();
    if ((int)lane == kWarp - 1) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t v = (int)lane < nw ? s_warp[lane] : 0u;
#pragma unroll
        for (int o = 1; o < kWarp; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
            if ((int)lane >= o) v += y;
        }
        if ((int)lane < nw) s_warp[lane] = v;
    }
    __syncthreads();
    uint32_t prefix = (warp ? s_warp[warp - 1] : 0u) + x - local;
    const uint32_t total = s_warp[nw - 1];
    for (uint32_t i = beg; i < end; ++i) {
        out[i] = prefix;
        if (rebase) rebase[i] -= prefix;
        prefix += in[i];
    }
    return total;
}

// Input element type of a pass: raw keys in pass 1, (key', row) later.
template <typename InKey, typename KeyT, bool FIRST>
struct PassIn {
    using E = typename std::conditional<FIRST, InKey, KeyT>::type;
    static constexpr uint32_t kPad = 32 / sizeof(E);  // room for the 16-byte lead and tail of a cover copy
    static constexpr size_t kKeyBytes = align_up((kPartTile + kPad) * sizeof(E), 16);
    static constexpr size_t kIdxBytes = FIRST ? 0 : align_up((kPartTile + 8) * sizeof(uint32_t), 16);
    // one ring buffer, with or without the tuple IDs of a later pass
    __host__ __device__ static constexpr size_t buf_bytes(bool rows) { return kKeyBytes + (rows ? kIdxBytes : 0); }
};

// Shared-memory tile ring: two input buffers, each filled by TMA bulk copies
// one tile ahead of the one being processed, each with its mbarrier.
template <typename InKey, typename KeyT, bool FIRST>
struct TileRing {
    using P = PassIn<InKey, KeyT, FIRST>;
    using E = typename P::E;
    uint64_t* bar;          // [2]
    unsigned char* buf;     // [2] of `stride` bytes: keys, then (later passes) rows
    uint32_t stride;

    __device__ E* keys(int b) const { return reinterpret_cast<E*>(buf + b * stride); }
    __device__ uint32_t* rows(int b) const { return reinterpret_cast<uint32_t*>(buf + b * stride + P::kKeyBytes); }

    __device__ static const E* key_src(const PartPass<InKey, KeyT>& a, uint32_t start) {
        if constexpr (FIRST)
            return a.raw + start;
        else
            return a.in_key + start;
    }

    // Warp 0 only: start loading tile `tl` into buffer b (with its tuple IDs
    // when ROWS). Lane 0 declares the bulk bytes on the buffer's barrier and
    // issues the bulk copies first; the lanes then copy the few unaligned
    // head and tail elements in parallel while the bulk copies are in flight,
    // and lane 0 arrives once they are written, so waiters see both.
    template <bool ROWS>
    __device__ void issue(const PartPass<InKey, KeyT>& a, const Tile& tl, int b) const {
        const unsigned lane = lane_id();
        const E* kf = key_src(a, tl.start);
        {
            // The aligned cover of the tile inside the source arrays: one bulk
            // copy per array, no element copies, no wait in this warp.
            const E* kbase = FIRST ? reinterpret_cast<const E*>(a.raw) : reinterpret_cast<const E*>(a.in_key);
            uint32_t kb = 0, ib = 0;
            const char* kc = cover(kf, tl.len, kbase, a.src_end[0], kb);
            const char* ic = nullptr;
            bool ok = kc != nullptr;
            if constexpr (ROWS) {
                ic = cover(a.in_idx + tl.start, tl.len, a.in_idx, a.src_end[1], ib);
                ok = ok && ic != nullptr;
            }
            if (ok) {
                if (lane == 0) {
                    fence_proxy_async_smem();
                    mbar_arrive_expect_tx(&bar[b], kb + ib);
                    bulk_load(keys(b), kc, kb, &bar[b]);
                    if constexpr (ROWS) bulk_load(rows(b), ic, ib, &bar[b]);
                }
                return;
            }
        }
        uint32_t klead, klo, khi;
        uint32_t bytes = tile_copy_plan(kf, tl.len, klead, klo, khi);
        uint32_t ilead = 0, ilo = 0, ihi = 0;
        const uint32_t* rf = nullptr;
        if constexpr (ROWS) {
            rf = a.in_idx + tl.start;
            bytes += tile_copy_plan(rf, tl.len, ilead, ilo, ihi);
        }
        if (lane == 0) {
            fence_proxy_async_smem();
            mbar_expect_tx(&bar[b], bytes);
            tile_copy_body(keys(b), kf, klead, klo, khi, &bar[b]);
            if constexpr (ROWS) tile_copy_body(rows(b), rf, ilead, ilo, ihi, &bar[b]);
        }
        edges_warp(keys(b), kf, tl.len, klead, klo, khi, lane);
        if constexpr (ROWS) edges_warp(rows(b), rf, tl.len, ilead, ilo, ihi, lane);
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar[b]);
    }

    // Start of the 16-byte aligned cover of [first, first + len) and its bytes
    // (a multiple of 16), or nullptr when the cover leaves [base, end).
    template <typename T>
    __device__ static const char* cover(const T* first, uint32_t len, const T* base, const void* end,
                                        uint32_t& bytes) {
        if (!end) return nullptr;
        const uintptr_t lo = reinterpret_cast<uintptr_t>(first) & ~(uintptr_t)15;
        const uintptr_t hi = (reinterpret_cast<uintptr_t>(first + len) + 15) & ~(uintptr_t)15;
        if (lo < reinterpret_cast<uintptr_t>(base) || hi > reinterpret_cast<uintptr_t>(end)) return nullptr;
        bytes = (uint32_t)(hi - lo);
        return reinterpret_cast<const char*>(lo);
    }

    // Lane l of the issuing warp copies head element l and tail element l.
    template <typename T>
    __device__ static void edges_warp(T* dst, const T* first, uint32_t len, uint32_t lead, uint32_t lo,
                                      uint32_t hi, unsigned lane) {
        if (lane < lo) dst[lead + lane] = first[lane];
        if (hi + lane < len) dst[lead + hi + lane] = first[hi + lane];
    }
};

template <typename E>
__device__ __forceinline__ uint32_t lead_of(const E* first) {
    return (uint32_t)((reinterpret_cast<uintptr_t>(first) & 15u) / sizeof(E));
}

// Warp 0: start loading tile `tl` of a scatter pass into buffer b. Later passes
// load the tile's tuple IDs too, unless the side keeps none (in_idx == nullptr:
// its consumer reads rows by position only).
template <typename InKey, typename KeyT, bool FIRST>
__device__ __forceinline__ void issue_tile(const TileRing<InKey, KeyT, FIRST>& ring,
                                           const PartPass<InKey, KeyT>& a, const Tile& tl, int b) {
    if constexpr (FIRST) {
        ring.template issue<false>(a, tl, b);
    } else {
        if (a.in_idx)
            ring.template issue<true>(a, tl, b);
        else
            ring.template issue<false>(a, tl, b);
    }
}

// Decodes an input key: applies the range test, the narrowing and (hash
// partitioning) the mix in pass 1. Returns false for a dropped row.
template <typename InKey, typename KeyT, bool FIRST, bool SORTM>
__device__ __forceinline__ bool decode_key(const PartPass<InKey, KeyT>& a,
                                           typename PassIn<InKey, KeyT, FIRST>::E in, KeyT& k) {
    if constexpr (FIRST) {
        // offset from the build minimum; a key outside [min, max] has one
        // beyond the span (compared in the input's width)
        using U = typename std::conditional<sizeof(InKey) == 4, uint32_t, uint64_t>::type;
        const U d = (U)in - (U)a.offset;
        k = (KeyT)d;
        if constexpr (!SORTM) k = KeyCodec<KeyT>::mix(k, a.kbits);
        return d <= (U)a.span;
    } else {
        k = in;
    }
    return true;
}

// Element e of the current tile, decoded.
template <typename InKey, typename KeyT, bool FIRST, bool SORTM>
__device__ __forceinline__ bool tile_key(const PartPass<InKey, KeyT>& a,
                                         const typename PassIn<InKey, KeyT, FIRST>::E* kbuf, uint32_t e,
                                         KeyT& k) {
    return decode_key<InKey, KeyT, FIRST, SORTM>(a, kbuf[e], k);
}

template <typename InKey, typename KeyT, bool FIRST>
__device__ __forceinline__ TileRing<InKey, KeyT, FIRST> ring_setup(unsigned char* smem, size_t off, bool rows) {
    using P = PassIn<InKey, KeyT, FIRST>;
    TileRing<InKey, KeyT, FIRST> r;
    r.bar = reinterpret_cast<uint64_t*>(smem);
    r.buf = smem + off;
    r.stride = (uint32_t)P::buf_bytes(rows);
    if (threadIdx.x == 0) {
        mbar_init(&r.bar[0], 1);
        mbar_init(&r.bar[1], 1);
        fence_mbar_init();
    }
    return r;
}

// After a failed bounded wait: record the error and wait (bounded) for the
// copy into the other buffer, so no TMA write lands after the CTA exits.
template <typename InKey, typename KeyT, bool FIRST>
__device__ void ring_abort(const TileRing<InKey, KeyT, FIRST>& r, int other, uint32_t parity,
                           bool other_pending, unsigned* err) {
    if (threadIdx.x == 0) {
        atomicOr(err, kErrInternal);
        if (other_pending) mbar_wait(&r.bar[other], parity);
    }
}

constexpr int kHistThreads = 256;
constexpr int kHistWarps = kHistThreads / kWarp;
constexpr int kHistPad = 4;  // words behind a warp's counters: a tile's counts lie in other banks than its neighbours'
constexpr int kHistLoads = 4;  // 16-byte loads in flight per lane

constexpr size_t hist_smem_bytes(int bits) {
    return kHistWarps * (((size_t)1 << bits) + kHistPad) * sizeof(uint32_t);
}

// Warp-collective: counts elements [beg, end) of the pass's input by digit into
// the warp's counters. The 16-byte words inside are loaded whole, the elements
// before and behind them one by one.
template <typename InKey, typename KeyT, bool FIRST, bool SORTM>
__device__ __forceinline__ void warp_count(const PartPass<InKey, KeyT>& a,
                                           const typename PassIn<InKey, KeyT, FIRST>::E* src, uint32_t n,
                                           uint32_t* cnt) {
    using E = typename PassIn<InKey, KeyT, FIRST>::E;
    constexpr uint32_t V = 16 / sizeof(E);
    const uint32_t lane = lane_id();
    const auto count = [&](E e) {
        KeyT k;
        if (decode_key<InKey, KeyT, FIRST, SORTM>(a, e, k)) atomicAdd(&cnt[digit_of(k, a.dshift, a.dmask)], 1u);
    };
    uint32_t head = (V - lead_of(src)) % V;
    if (head > n) head = n;
    const uint32_t nv = (n - head) / V, tail = head + nv * V;
    if (lane < head) count(src[lane]);
    if (tail + lane < n) count(src[tail + lane]);
    const uint4* v = reinterpret_cast<const uint4*>(src + head);
    for (uint32_t base = lane; base < nv; base += kWarp * kHistLoads) {
        union {
            uint4 w;
            E e[V];
        } x[kHistLoads];
#pragma unroll
        for (int j = 0; j < kHistLoads; ++j)
            if (base + j * kWarp < nv) x[j].w = __ldg(v + base + j * kWarp);
#pragma unroll
        for (int j = 0; j < kHistLoads; ++j)
            if (base + j * kWarp < nv) {
#pragma unroll
                for (uint32_t q = 0; q < V; ++q) count(x[j].e[q]);
            }
    }
}

// Digit counts of every tile. A warp takes a tile (with `split`, an eighth of
// one, for inputs of few tiles) and counts it into shared memory of its own, so
// nothing waits inside a tile; the CTA then stores the counts of its eight
// neighbouring tiles together, a 32-byte sector per digit. Bound by
// instructions (21 per 32 rows in pass 1, with the mix; 7 in pass 2, which
// reads at 0.77 of DRAM's rate) and the shared-memory atomics. Against a CTA per 4096-row tile fed by
// bulk copies, two barriers and a store of lone counts per tile: 600M 32-bit
// keys 750 -> 484 us (7 bits, pass 1) and 556 -> 352 us (8 bits, pass 2); 60M
// 64-bit keys, 12 bits, 622 -> 310 us; 20M 64-bit keys, near HBM already,
// 41 -> 42 us. Five CTAs per SM: four cost 4 %, six no less.
template <typename InKey, typename KeyT, bool FIRST, bool SORTM>
__global__ void __launch_bounds__(kHistThreads, 5) part_hist_kernel(PartPass<InKey, KeyT> a, bool split) {
    using Ring = TileRing<InKey, KeyT, FIRST>;
    extern __shared__ __align__(16) uint32_t s_hist[];
    __shared__ size_t s_index[kHistWarps];     // of the tile's count of digit 0
    __shared__ uint32_t s_stride[kHistWarps];  // from one digit to the next; 0: no tile
    const uint32_t nd = 1u << a.bits, lane = lane_id(), w = threadIdx.x / kWarp;
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.scan_done = 0u;
    uint32_t* cnt = s_hist + w * (nd + kHistPad);
    const uint32_t ntiles = a.tiles ? *a.ntiles_dev : a.ntiles_fixed;
    const uint32_t per = split ? 1u : (uint32_t)kHistWarps;  // tiles per CTA and round
    for (uint32_t t0 = blockIdx.x * per; t0 < ntiles; t0 += gridDim.x * per) {
        const uint32_t t = split ? t0 : t0 + w;
        for (uint32_t d = lane; d < nd; d += kWarp) cnt[d] = 0;
        __syncwarp();
        if (t < ntiles) {
            const Tile tl = get_tile(a, t);
            uint32_t beg = 0, end = tl.len;
            if (split) {
                beg = w * (kPartTile / kHistWarps);
                end = beg + kPartTile / kHistWarps < tl.len ? beg + kPartTile / kHistWarps : tl.len;
            }
            if (beg < end)
                warp_count<InKey, KeyT, FIRST, SORTM>(a, Ring::key_src(a, tl.start) + beg, end - beg, cnt);
            if (lane == 0) {
                s_index[w] = count_index(tl, t, 0, a.bits);
                s_stride[w] = tl.ntiles_seg;
            }
        } else if (lane == 0) {
            s_stride[w] = 0;
        }
        __syncthreads();
        if (split) {
            for (uint32_t d = threadIdx.x; d < nd; d += kHistThreads) {
                uint32_t c = 0;
#pragma unroll
                for (int q = 0; q < kHistWarps; ++q) c += s_hist[q * (nd + kHistPad) + d];
                a.counts[s_index[0] + (size_t)d * s_stride[0]] = c;
            }
        } else {
            const uint32_t q = threadIdx.x % kHistWarps;
            const size_t at = s_index[q], stride = s_stride[q];
            if (stride)
                for (uint32_t d = threadIdx.x / kHistWarps; d < nd; d += kHistThreads / kHistWarps)
                    a.counts[at + d * stride] = s_hist[q * (nd + kHistPad) + d];
        }
        __syncthreads();
    }
}

// A dropped row (outside the range, or behind a short tile) counts under a digit
// of its lane's own and is staged behind the tile, where nothing is read: the loops
// over a thread's rows then have no branches.
constexpr uint32_t kDropped = kPartTile;     // its stage position
constexpr uint32_t kStageRows = kPartTile + 8;
constexpr uint32_t kPosPad = kWarp;          // words behind the digits' positions: the dropped rows' counters

// Words of the digit positions and offsets of two tiles.
__host__ __device__ constexpr size_t scatter_counters(int bits) {
    return 4 * ((size_t)1 << bits) + 2 * kPosPad;
}

// Ring and stage of the hash scatter: keys, with tuple IDs beside them (pass 1:
// as 16-bit rows of the tile), and a batch of carried columns (8 bytes per
// row), apart from the keys or in their place.
template <typename InKey, typename KeyT, bool FIRST>
__host__ __device__ constexpr size_t scatter_smem_bytes(int bits, bool rows, bool cols, bool col_apart) {
    const size_t key_stage = sizeof(KeyT) + (rows ? (FIRST ? 2 : 4) : 0);
    const size_t stage = !cols ? key_stage : col_apart ? key_stage + 8 : key_stage > 8 ? key_stage : 8;
    return align_up(16 + scatter_counters(bits) * sizeof(uint32_t), 16) +
           2 * PassIn<InKey, KeyT, FIRST>::buf_bytes(rows) + (size_t)kStageRows * stage;
}

// Shared memory that lets two CTAs of a kernel share an SM.
constexpr size_t kTwoPerSm = 113 * 1024;

// Digits a thread owns in the per-tile offset table (prefetched one tile ahead).
constexpr int kGoffPerThread = (1 << kMaxBits) / kPartThreads;

constexpr int kPartWarps = kPartThreads / kWarp;
constexpr int kDigitBits1 = 9;  // radix bits with one digit per thread
static_assert((1 << kDigitBits1) == kPartThreads, "one digit per thread");
constexpr int kWarpRows = kPartTile / kPartWarps;  // sort scatter: consecutive rows per warp
static_assert(kWarpRows == kPartItems * kWarp, "sort tiles are warp-blocked");

// Block-collective (sort scatter): moves one carried column of the current
// tile to the output positions of its rows. Row j of this thread (tile element
// w * kWarpRows + j * 32 + lane, digit and rank in dr[j]) is staged at its tile
// position start[d] + (rows of digit d in earlier warps) + rank, then every
// digit run is written out with consecutive threads on consecutive addresses,
// like the keys.
template <typename V, typename DigT>
__device__ __forceinline__ void carry_column(const V* __restrict__ src, V* __restrict__ dst,
                                             const uint32_t (&dr)[kPartItems], const uint16_t* s_wc, uint32_t nd,
                                             const uint32_t* s_start, const uint32_t* s_goff, const DigT* s_dig,
                                             uint32_t nk, V* s_col) {
    const unsigned lane = lane_id();
    const uint32_t w = threadIdx.x / kWarp;
#pragma unroll
    for (int j = 0; j < kPartItems; ++j) {
        if (dr[j] != kNoDigit) {
            const uint32_t d = dr[j] & 0xFFFu;
            const uint32_t e = w * kWarpRows + j * kWarp + lane;
            s_col[s_start[d] + s_wc[w * nd + d] + (dr[j] >> 12)] = __ldcs(src + e);
        }
    }
    __syncthreads();
    for (uint32_t q = threadIdx.x; q < nk; q += blockDim.x) {
        const uint32_t d = s_dig[q];
        dst[s_goff[d] + q] = s_col[q];
    }
    __syncthreads();
}

// Carried columns travel in batches of at most 8 bytes per row: one 8-byte
// column, or one or two 4-byte ones. Returns the first column after the batch
// that starts at c.
__host__ __device__ __forceinline__ int batch_end(const ColCarry& cc, int c) {
    return c + 1 < cc.n && cc.bytes[c] == 4 && cc.bytes[c + 1] == 4 ? c + 2 : c + 1;
}

// Columns [c, ce) of the current tile: a thread's rows read in tile order into
// registers (issued before the barrier that precedes their staging), staged at
// their tile positions, and written to the output positions g of the stage
// entries. v[0], v[1]: the halves of an 8-byte value, or two 4-byte columns.
template <bool FULL>
__device__ __forceinline__ void load_batch_rows(const ColCarry& cc, int c, int ce, const Tile& tl,
                                                uint32_t (&v)[2][kPartItems]) {
    if (cc.bytes[c] == 8) {
        const uint2* src = static_cast<const uint2*>(cc.in[c]) + tl.start + threadIdx.x;
#pragma unroll
        for (int j = 0; j < kPartItems; ++j)
            if (FULL || j * kPartThreads + threadIdx.x < tl.len) {
                const uint2 x = __ldcs(src + j * kPartThreads);
                v[0][j] = x.x;
                v[1][j] = x.y;
            }
        return;
    }
    const uint32_t* s0 = static_cast<const uint32_t*>(cc.in[c]) + tl.start + threadIdx.x;
    const uint32_t* s1 = static_cast<const uint32_t*>(cc.in[ce - 1]) + tl.start + threadIdx.x;
#pragma unroll
    for (int j = 0; j < kPartItems; ++j)
        if (FULL || j * kPartThreads + threadIdx.x < tl.len) v[0][j] = __ldcs(s0 + j * kPartThreads);
    if (ce - c == 2) {
#pragma unroll
        for (int j = 0; j < kPartItems; ++j)
            if (FULL || j * kPartThreads + threadIdx.x < tl.len) v[1][j] = __ldcs(s1 + j * kPartThreads);
    }
}

__device__ __forceinline__ void load_batch(const ColCarry& cc, int c, int ce, const Tile& tl,
                                           uint32_t (&v)[2][kPartItems]) {
    if (tl.len == (uint32_t)kPartTile)
        load_batch_rows<true>(cc, c, ce, tl, v);
    else
        load_batch_rows<false>(cc, c, ce, tl, v);
}

__device__ __forceinline__ void stage_batch(const ColCarry& cc, int c, int ce, const uint32_t (&pos)[kPartItems],
                                            const uint32_t (&v)[2][kPartItems], unsigned char* stage) {
    if (cc.bytes[c] == 8) {
        uint2* s = reinterpret_cast<uint2*>(stage);
#pragma unroll
        for (int j = 0; j < kPartItems; ++j) s[pos[j]] = make_uint2(v[0][j], v[1][j]);
        return;
    }
    uint32_t* s = reinterpret_cast<uint32_t*>(stage);
#pragma unroll
    for (int j = 0; j < kPartItems; ++j) s[pos[j]] = v[0][j];
    if (ce - c == 2) {
        s += kStageRows;
#pragma unroll
        for (int j = 0; j < kPartItems; ++j) s[pos[j]] = v[1][j];
    }
}

template <bool FULL>
__device__ __forceinline__ void write_batch_rows(const ColCarry& cc, int c, int ce, const uint32_t (&g)[kPartItems],
                                                 uint32_t nk, const unsigned char* stage) {
    if (cc.bytes[c] == 8) {
        const uint2* s = reinterpret_cast<const uint2*>(stage) + threadIdx.x;
        uint2* dst = static_cast<uint2*>(cc.out[c]);
#pragma unroll
        for (int i = 0; i < kPartItems; ++i)
            if (FULL || i * kPartThreads + threadIdx.x < nk) dst[g[i]] = s[i * kPartThreads];
        return;
    }
    const uint32_t* s = reinterpret_cast<const uint32_t*>(stage) + threadIdx.x;
#pragma unroll 1
    for (; c < ce; ++c, s += kStageRows) {
        uint32_t* dst = static_cast<uint32_t*>(cc.out[c]);
#pragma unroll
        for (int i = 0; i < kPartItems; ++i)
            if (FULL || i * kPartThreads + threadIdx.x < nk) dst[g[i]] = s[i * kPartThreads];
    }
}

__device__ __forceinline__ void write_batch(const ColCarry& cc, int c, int ce, const uint32_t (&g)[kPartItems],
                                            uint32_t nk, const unsigned char* stage) {
    if (nk == (uint32_t)kPartTile)
        write_batch_rows<true>(cc, c, ce, g, nk, stage);
    else
        write_batch_rows<false>(cc, c, ce, g, nk, stage);
}

// One thread: asks L2 to fetch the carried columns of tile `tl`, a tile ahead
// of its loads (the 16-byte aligned part of each column's rows).
__device__ __forceinline__ void prefetch_columns(const ColCarry& cc, const Tile& tl) {
#pragma unroll 1
    for (int c = 0; c < cc.n; ++c) {
        const uintptr_t a = reinterpret_cast<uintptr_t>(cc.in[c]) + (size_t)tl.start * cc.bytes[c];
        const uintptr_t lo = (a + 15) & ~(uintptr_t)15, hi = (a + tl.len * (uint32_t)cc.bytes[c]) & ~(uintptr_t)15;
        if (hi > lo)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(lo), "r"((uint32_t)(hi - lo)) : "memory");
    }
}

template <typename DigT>
__device__ __forceinline__ void carry_columns(const ColCarry& cc, uint32_t tstart, const uint32_t (&dr)[kPartItems],
                                              const uint16_t* s_wc, uint32_t nd, const uint32_t* s_start,
                                              const uint32_t* s_goff, const DigT* s_dig, uint32_t nk,
                                              void* s_stage) {
#pragma unroll 1
    for (int c = 0; c < cc.n; ++c) {
        if (cc.bytes[c] == 4)
            carry_column(static_cast<const uint32_t*>(cc.in[c]) + tstart, static_cast<uint32_t*>(cc.out[c]), dr, s_wc,
                         nd, s_start, s_goff, s_dig, nk, static_cast<uint32_t*>(s_stage));
        else
            carry_column(static_cast<const unsigned long long*>(cc.in[c]) + tstart,
                         static_cast<unsigned long long*>(cc.out[c]), dr, s_wc, nd, s_start, s_goff, s_dig, nk,
                         static_cast<unsigned long long*>(s_stage));
    }
}

// Global offset and row count of a tile's digits, DPT consecutive groups of 32
// digits per warp (lane l of warp w owns digits (w * DPT + q) * 32 + l). The
// count is the distance to the next entry of the scanned counts: the next
// tile's run of the digit, the next digit's first tile, the next segment, or
// the total behind the last entry.
template <int DPT>
struct TileDigits {
    uint32_t goff[DPT], cnt[DPT];
    __device__ static uint32_t digit(int q) {
        return ((threadIdx.x / kWarp) * DPT + q) * kWarp + lane_id();
    }
    __device__ __forceinline__ void load(const uint32_t* __restrict__ counts, const Tile& tl, uint32_t t, int bits) {
#pragma unroll
        for (int q = 0; q < DPT; ++q) {
            const uint32_t d = digit(q);
            goff[q] = cnt[q] = 0;
            if (d >> bits) continue;
            const uint32_t* p = counts + count_index(tl, t, d, bits);
            goff[q] = p[0];
            cnt[q] = p[1] - goff[q];
        }
    }
    // Before the barrier: this warp's rows, for the warps behind it.
    __device__ __forceinline__ void warp_total(uint32_t* s_wtot) const {
        uint32_t v = 0;
#pragma unroll
        for (int q = 0; q < DPT; ++q) v += cnt[q];
        v = __reduce_add_sync(0xffffffffu, v);
        if (lane_id() == 0) s_wtot[threadIdx.x / kWarp] = v;
    }
    // After it: the tile position of every digit's first row into s_pos, global
    // offset minus tile position into s_goff; returns the tile's rows.
    __device__ __forceinline__ uint32_t place(const uint32_t* s_wtot, uint32_t* s_pos, uint32_t* s_goff,
                                              int bits) const {
        const unsigned lane = lane_id();
        const int w = threadIdx.x / kWarp;
        const uint32_t v = lane < kPartWarps ? s_wtot[lane] : 0u;
        const uint32_t total = __reduce_add_sync(0xffffffffu, v);
        uint32_t run = __reduce_add_sync(0xffffffffu, (int)lane < w ? v : 0u);
#pragma unroll
        for (int q = 0; q < DPT; ++q) {
            uint32_t x = cnt[q];
#pragma unroll
            for (int o = 1; o < kWarp; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if ((int)lane >= o) x += y;
            }
            const uint32_t d = digit(q), pos = run + x - cnt[q];
            if (!(d >> bits)) {
                s_pos[d] = pos;
                s_goff[d] = goff[q] - pos;
            }
            run += __shfl_sync(0xffffffffu, x, kWarp - 1);
        }
        return total;
    }
};

// Scatter of one hash-partitioning pass. The scanned counts already hold every
// tile's digit runs, so the tile positions of the runs are known before its
// rows are read: one shared-memory atomic per row gives the row's place in the
// digit-sorted stage, and two CTA barriers separate a tile's staging from its
// write-out (plus two per further batch of carried columns). The positions of
// the next tile are laid out (double-buffered) while this one is written. A
// row's digit is read back from the staged key, whose mix already happened in
// pass 1; the global positions of a thread's rows are computed once and serve
// the tuple IDs and every carried column.
//
// What bounds it: the output runs, short pieces of as many places as there are
// digits (DRAM moves 4.5 to 5.4 TB/s, of 6.8 for a copy), and close behind them
// shared-memory wavefronts, about 22 per 32 rows with one 8-byte column: the
// rank atomics, and staging at random positions. It had taken about 38 (the
// rank's start looked up per use, a digit array beside the keys) and eight
// barriers per tile; then issue slots (126 and 100 instructions per 32 rows
// in passes 1 and 2: a branch per row and step, ring buffers behind an indexed
// array in local memory, spills; now 90 and 65).
// Measured on GB300, first written -> two barriers -> without branches: 2^28
// rows with two 4-byte columns, 6 + 6 bits, 2.13 + 1.93 -> 1.60 + 1.60 -> 1.39 +
// 1.35 ms; 30M 64-bit keys with a 4-byte column, 6 + 6 bits, 322 + 297 -> 229 +
// 186 -> 142 + 143 us; 20M random 64-bit keys with tuple IDs, 5 + 6 bits, 164 +
// 174 -> 90 + 125 -> 86 + 115 us; 600M 32-bit keys with an 8-byte column, 7 + 8
// bits, 3.68 + 3.25 -> 2.65 + 3.19 ms.
//
// At most 64 registers: two CTAs per SM wherever shared memory allows.
template <typename InKey, typename KeyT, bool FIRST, int DPT, bool COLS>
__global__ void __launch_bounds__(kPartThreads, 2) part_scatter_kernel(PartPass<InKey, KeyT> a, unsigned* err) {
    using Ring = TileRing<InKey, KeyT, FIRST>;
    using P = PassIn<InKey, KeyT, FIRST>;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_wtot[kPartWarps];
    const uint32_t nd = 1u << a.bits;
    const bool rows = a.out_idx != nullptr;  // tuple IDs travel with the keys
    uint32_t* s_pos2 = reinterpret_cast<uint32_t*>(smem + 16);  // [2][nd + kPosPad]
    uint32_t* s_goff2 = s_pos2 + 2 * (nd + kPosPad);            // [2][nd]
    const size_t ring_off = align_up(16 + scatter_counters(a.bits) * 4, 16);
    const Ring ring = ring_setup<InKey, KeyT, FIRST>(smem, ring_off, rows);
    KeyT* s_key = reinterpret_cast<KeyT*>(smem + ring_off + 2 * P::buf_bytes(rows));
    static_assert(kPartTile <= 65536, "a row of a tile fits 16 bits");
    using RowT = typename std::conditional<FIRST, uint16_t, uint32_t>::type;  // pass 1: row in the tile
    RowT* s_idx = reinterpret_cast<RowT*>(s_key + kStageRows);
    unsigned char* col_stage =
        reinterpret_cast<unsigned char*>(s_key) + (a.col_apart ? (size_t)kStageRows * sizeof(KeyT) : 0);
    __syncthreads();

    const uint32_t ntiles = a.tiles ? *a.ntiles_dev : a.ntiles_fixed;
    uint32_t t = blockIdx.x;
    if (t >= ntiles) return;
    Tile tl = get_tile(a, t);
    Tile tl_next{};
    TileDigits<DPT> dg;
    dg.load(a.counts, tl, t, a.bits);
    if (threadIdx.x < kWarp) issue_tile(ring, a, tl, 0);
    dg.warp_total(s_wtot);
    __syncthreads();
    uint32_t nk = dg.place(s_wtot, s_pos2, s_goff2, a.bits);
    if (t + gridDim.x < ntiles) {
        tl_next = get_tile(a, t + gridDim.x);
        dg.load(a.counts, tl_next, t + gridDim.x, a.bits);
    }
    __syncthreads();

    for (uint32_t it = 0; t < ntiles; t += gridDim.x, ++it) {
        const int b = it & 1;
        const uint32_t tn = t + gridDim.x;
        const bool more = tn < ntiles;
        if (threadIdx.x < kWarp && more) issue_tile(ring, a, tl_next, b ^ 1);
        if constexpr (COLS)
            if (threadIdx.x == kWarp && more) prefetch_columns(a.cc, tl_next);
        uint32_t* s_pos = s_pos2 + b * (nd + kPosPad);
        const uint32_t* s_goff = s_goff2 + b * nd;
        int c = 0, ce = 0;
        uint32_t val[2][kPartItems];  // a batch of column values of this thread's tile rows
        if constexpr (COLS) {
            ce = batch_end(a.cc, 0);
            if (a.col_apart) load_batch(a.cc, 0, ce, tl, val);
        }
        const bool ok = mbar_wait(&ring.bar[b], (it >> 1) & 1);
        const auto* kbuf = ring.keys(b) + lead_of(Ring::key_src(a, tl.start));
        uint32_t pos[kPartItems];  // tile position, kDropped for a dropped row
        if (ok) {
            const uint32_t* rbuf = nullptr;
            if constexpr (!FIRST)
                if (rows) rbuf = ring.rows(b) + lead_of(a.in_idx + tl.start);
            KeyT kk[kPartItems];
#pragma unroll
            for (int j = 0; j < kPartItems; ++j) {
                // (behind a short tile the ring buffer is read as it lies)
                const uint32_t e = j * kPartThreads + threadIdx.x;
                const bool in = decode_key<InKey, KeyT, FIRST, false>(a, kbuf[e], kk[j]);
                const bool kept = in & (e < tl.len);
                const uint32_t d = kept ? digit_of(kk[j], a.dshift, a.dmask) : nd + lane_id();
                pos[j] = atomicAdd(&s_pos[d], 1u);
                if (!kept) pos[j] = kDropped;
            }
#pragma unroll
            for (int j = 0; j < kPartItems; ++j) {
                s_key[pos[j]] = kk[j];
                if (rows) {
                    const uint32_t e = j * kPartThreads + threadIdx.x;
                    s_idx[pos[j]] = FIRST ? (RowT)e : (RowT)rbuf[e];
                }
            }
        }
        if (more) dg.warp_total(s_wtot);
        if constexpr (COLS) {
            if (a.col_apart) {
                if (ok) stage_batch(a.cc, 0, ce, pos, val, col_stage);
            } else {
                load_batch(a.cc, 0, ce, tl, val);
            }
        }
        if (__syncthreads_or(!ok)) {
            ring_abort(ring, b ^ 1, ((it + 1) >> 1) & 1, more, err);
            return;
        }
        uint32_t nk_next = 0;
        Tile tl_after{};
        if (more) {
            nk_next = dg.place(s_wtot, s_pos2 + (b ^ 1) * (nd + kPosPad), s_goff2 + (b ^ 1) * nd, a.bits);
            if (tn + gridDim.x < ntiles) {
                tl_after = get_tile(a, tn + gridDim.x);
                dg.load(a.counts, tl_after, tn + gridDim.x, a.bits);
            }
        }
        uint32_t g[kPartItems];  // output positions of stage entries tid, tid + threads, ...
        const auto write_keys = [&](auto full) {
#pragma unroll
            for (int i = 0; i < kPartItems; ++i) {
                const uint32_t q = i * kPartThreads + threadIdx.x;
                if (decltype(full)::value || q < nk) {
                    const KeyT k = s_key[q];
                    g[i] = s_goff[digit_of(k, a.dshift, a.dmask)] + q;
                    a.out_key[g[i]] = k;
                    if (rows) a.out_idx[g[i]] = (FIRST ? tl.start : 0u) + s_idx[q];
                }
            }
        };
        if (nk == (uint32_t)kPartTile)
            write_keys(std::true_type{});
        else
            write_keys(std::false_type{});
        if constexpr (COLS) {
            if (a.col_apart) {
                write_batch(a.cc, c, ce, g, nk, col_stage);
                c = ce;
                ce = c < a.cc.n ? batch_end(a.cc, c) : c;
                if (ce > c) load_batch(a.cc, c, ce, tl, val);
            }
#pragma unroll 1
            while (c < ce) {
                __syncthreads();  // the stage's last contents are written out
                stage_batch(a.cc, c, ce, pos, val, col_stage);
                const int c0 = c, c1 = ce;
                c = ce;
                ce = c < a.cc.n ? batch_end(a.cc, c) : c;
                if (ce > c) load_batch(a.cc, c, ce, tl, val);
                __syncthreads();
                write_batch(a.cc, c0, c1, g, nk, col_stage);
            }
        }
        tl = tl_next;
        tl_next = tl_after;
        nk = nk_next;
        __syncthreads();  // the stage and this tile's ring buffer are free
    }
}

// ------------------------------------------------------------ stable sort scatter

template <typename InKey, typename KeyT, bool FIRST>
__host__ __device__ constexpr size_t sort_scatter_smem_bytes(int bits) {
    return align_up(16 + 3 * ((size_t)1 << bits) * sizeof(uint32_t), 16) +
           2 * PassIn<InKey, KeyT, FIRST>::buf_bytes(true) + align_up((size_t)kPartTile * sizeof(KeyT), 16) +
           (size_t)kPartTile * sizeof(uint32_t) + (size_t)kPartTile * sizeof(uint8_t) +
           (size_t)kPartWarps * ((size_t)1 << bits) * sizeof(uint16_t);
}

// One pass of the stable LSD radix sort (the sort of the sort-merge join,
// Sec. 3.2). Same three steps as a partitioning pass, but the digit is taken
// from the key itself and the scatter is stable: every warp owns kWarpRows
// consecutive rows of the tile and ranks them in order, 32 at a time, with
// __match_any_sync against its own per-digit counters; the counters of the
// warps are then scanned in warp order, so rows of equal digit keep their
// input order within the tile, and the [digit][tile] scan keeps tile order.
template <typename InKey, typename KeyT, bool FIRST>
__global__ void __launch_bounds__(kPartThreads, 2) sort_scatter_kernel(PartPass<InKey, KeyT> a, unsigned* err) {
    using Ring = TileRing<InKey, KeyT, FIRST>;
    using P = PassIn<InKey, KeyT, FIRST>;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_warp[kPartThreads / kWarp];
    __shared__ uint32_t s_kept;
    const uint32_t nd = 1u << a.bits;
    const bool rows = a.out_idx != nullptr;  // tuple IDs travel with the keys
    uint32_t* s_cnt = reinterpret_cast<uint32_t*>(smem + 16);
    uint32_t* s_start = s_cnt + nd;
    uint32_t* s_goff = s_start + nd;
    const size_t ring_off = align_up(16 + 3 * (size_t)nd * 4, 16);
    const Ring ring = ring_setup<InKey, KeyT, FIRST>(smem, ring_off, true);
    KeyT* s_key = reinterpret_cast<KeyT*>(smem + ring_off + 2 * P::buf_bytes(true));
    uint32_t* s_idx = reinterpret_cast<uint32_t*>(reinterpret_cast<unsigned char*>(s_key) +
                                                  align_up((size_t)kPartTile * sizeof(KeyT), 16));
    uint8_t* s_dig = reinterpret_cast<uint8_t*>(s_idx + kPartTile);
    uint16_t* s_wc = reinterpret_cast<uint16_t*>(s_dig + kPartTile);  // [warp][digit]
    __syncthreads();

    const unsigned lane = lane_id();
    const uint32_t w = threadIdx.x / kWarp;
    const uint32_t ntiles = a.tiles ? *a.ntiles_dev : a.ntiles_fixed;
    uint32_t t = blockIdx.x;
    uint32_t goff[kGoffPerThread] = {};
    Tile tl_cur;
    if (t < ntiles) {
        tl_cur = get_tile(a, t);
#pragma unroll
        for (int q = 0; q < kGoffPerThread; ++q) {
            const uint32_t d = threadIdx.x + q * kPartThreads;
            if (d < nd) goff[q] = a.counts[count_index(tl_cur, t, d, a.bits)];
        }
    }
    Tile d_next{};  // warp 0: descriptor of the next tile to issue, loaded one tile early
    if (threadIdx.x < kWarp) {
        if (t < ntiles) issue_tile(ring, a, tl_cur, 0);
        if (t + gridDim.x < ntiles) d_next = get_tile(a, t + gridDim.x);
    }
    for (uint32_t it = 0; t < ntiles; t += gridDim.x, ++it) {
        const int b = it & 1;
        const uint32_t tn = t + gridDim.x;
        if (threadIdx.x < kWarp && tn < ntiles) {
            issue_tile(ring, a, d_next, b ^ 1);
            if (tn + gridDim.x < ntiles) d_next = get_tile(a, tn + gridDim.x);
        }
        for (uint32_t d = lane; d < nd; d += kWarp) s_wc[w * nd + d] = 0;
#pragma unroll
        for (int q = 0; q < kGoffPerThread; ++q) {
            const uint32_t d = threadIdx.x + q * kPartThreads;
            if (d < nd) s_goff[d] = goff[q];
        }
        const bool ok = mbar_wait(&ring.bar[b], (it >> 1) & 1);
        if (__syncthreads_or(!ok)) {
            ring_abort(ring, b ^ 1, ((it + 1) >> 1) & 1, tn < ntiles, err);
            return;
        }
        const Tile tl = tl_cur;
        if (tn < ntiles) {
            tl_cur = get_tile(a, tn);
            if constexpr (!FIRST)
                if (threadIdx.x == 0 && a.cc.n) prefetch_columns(a.cc, tl_cur);
#pragma unroll
            for (int q = 0; q < kGoffPerThread; ++q) {
                const uint32_t d = threadIdx.x + q * kPartThreads;
                if (d < nd) goff[q] = a.counts[count_index(tl_cur, tn, d, a.bits)];
            }
        }
        const auto* kbuf = ring.keys(b) + lead_of(Ring::key_src(a, tl.start));
        const uint32_t* rbuf = nullptr;
        if constexpr (!FIRST)
            if (rows) rbuf = ring.rows(b) + lead_of(a.in_idx + tl.start);

        KeyT kk[kPartItems];
        uint32_t dr[kPartItems];  // (rank within this warp's rows << 12) | digit, or kNoDigit
#pragma unroll
        for (int j = 0; j < kPartItems; ++j) {
            const uint32_t e = w * kWarpRows + j * kWarp + lane;
            const bool v = e < tl.len && tile_key<InKey, KeyT, FIRST, true>(a, kbuf, e, kk[j]);
            const uint32_t d = v ? digit_of(kk[j], a.dshift, a.dmask) : kNoDigit;
            const unsigned peers = __match_any_sync(0xffffffffu, d);
            const uint32_t before = v ? s_wc[w * nd + d] : 0u;
            __syncwarp();
            if (v && (int)lane == __ffs(peers) - 1) s_wc[w * nd + d] = (uint16_t)(before + __popc(peers));
            __syncwarp();
            dr[j] = v ? ((before + __popc(peers & lanemask_lt())) << 12) | d : kNoDigit;
        }
        __syncthreads();
        // per digit: exclusive prefix over the warps in order, and the tile count
        for (uint32_t d = threadIdx.x; d < nd; d += blockDim.x) {
            uint32_t run = 0;
#pragma unroll
            for (int q = 0; q < kPartWarps; ++q) {
                const uint32_t c = s_wc[q * nd + d];
                s_wc[q * nd + d] = (uint16_t)run;
                run += c;
            }
            s_cnt[d] = run;
        }
        __syncthreads();
        // s_goff becomes (global offset - tile offset) of each digit
        const uint32_t kept = block_scan_smem(s_cnt, s_start, nd, s_warp, s_goff);
        if (threadIdx.x == 0) s_kept = kept;
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kPartItems; ++j) {
            if (dr[j] != kNoDigit) {
                const uint32_t e = w * kWarpRows + j * kWarp + lane;
                const uint32_t d = dr[j] & 0xFFFu;
                const uint32_t pos = s_start[d] + s_wc[w * nd + d] + (dr[j] >> 12);
                s_key[pos] = kk[j];
                s_dig[pos] = (uint8_t)d;
                if (rows) s_idx[pos] = FIRST ? tl.start + e : rbuf[e];
            }
        }
        __syncthreads();
        const uint32_t nk = s_kept;
        for (uint32_t pos = threadIdx.x; pos < nk; pos += blockDim.x) {
            const uint32_t d = s_dig[pos];
            const uint32_t g = s_goff[d] + pos;
            a.out_key[g] = s_key[pos];
            if (rows) a.out_idx[g] = s_idx[pos];
        }
        __syncthreads();
        if (a.cc.n) carry_columns(a.cc, tl.start, dr, s_wc, nd, s_start, s_goff, s_dig, nk, s_key);
    }
}

// ------------------------------------------------------------ device-wide scan

struct ScanLen {
    size_t fixed;
    const uint32_t* ntiles_dev;  // when set: length = *ntiles_dev << bits
    int bits;
    __device__ __forceinline__ size_t get() const {
        return ntiles_dev ? ((size_t)*ntiles_dev << bits) : fixed;
    }
};

// Exclusive scan of a warp's sums: returns the prefix of `v`, the warp's total
// in *total.
__device__ __forceinline__ uint32_t warp_exscan(uint32_t v, uint32_t* total) {
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < kWarp; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if ((int)lane_id() >= o) x += y;
    }
    *total = __shfl_sync(0xffffffffu, x, kWarp - 1);
    return x - v;
}

// The prefix of this warp's `mine` among the CTA's warps; *total: their sum.
__device__ __forceinline__ uint32_t warps_exscan(uint32_t mine, uint32_t* s_warp, uint32_t* total) {
    constexpr int kWarps = kScanThreads / kWarp;
    const int warp = threadIdx.x / kWarp;
    if (lane_id() == 0) s_warp[warp] = mine;
    __syncthreads();
    const uint32_t v = lane_id() < kWarps ? s_warp[lane_id()] : 0u;
    *total = __reduce_add_sync(0xffffffffu, v);
    return __reduce_add_sync(0xffffffffu, (int)lane_id() < warp ? v : 0u);
}

// A thread's entries of a chunk of m: kScanItems / 4 words of 16 bytes, a warp's
// words side by side (entries at or past m read as 0).
constexpr int kScanVec = kScanItems / 4;
static_assert(kScanItems % 4 == 0 && kScanThreads / kWarp <= kWarp, "layout of a chunk");

__device__ __forceinline__ uint32_t scan_first() {
    return (threadIdx.x / kWarp) * (kWarp * kScanItems) + lane_id() * 4;
}

__device__ __forceinline__ void scan_load(const uint32_t* p, uint32_t m, uint4 (&v)[kScanVec]) {
#pragma unroll
    for (int r = 0; r < kScanVec; ++r) {
        const uint32_t i = scan_first() + r * (kWarp * 4);
        if (i + 4 <= m) {
            v[r] = *reinterpret_cast<const uint4*>(p + i);
        } else {
            v[r].x = i < m ? p[i] : 0u;
            v[r].y = i + 1 < m ? p[i + 1] : 0u;
            v[r].z = i + 2 < m ? p[i + 2] : 0u;
            v[r].w = 0u;
        }
    }
}

// Scan of the counts in two launches: chunk sums, whose prefixes the CTA that
// finishes last computes (no CTA waits for another), then the chunks in place.
// Bound by reading the counts twice, the second time mostly from L2. 146,484
// tiles x 256 digits: 242 -> 76 us; 4,883 tiles x 64: 24.5 -> 12.3 us, against
// three launches with strided shared-memory access. One launch, with the
// scatter adding the chunk prefixes as it loads the offsets, takes 51 and 8 us
// but costs the scatters that carry columns 4 % (3253 -> 3426 us), in registers.
__global__ void __launch_bounds__(kScanThreads)
    scan_sums_kernel(const uint32_t* __restrict__ data, ScanLen L, uint32_t* sums, uint32_t* done, uint32_t* total) {
    __shared__ uint32_t s_warp[kScanThreads / kWarp];
    __shared__ uint32_t s_last;
    const size_t len = L.get();
    const size_t beg = (size_t)blockIdx.x * kScanChunk;
    if (len == 0 && blockIdx.x == 0 && threadIdx.x == 0) *total = 0u;
    if (beg >= len) return;
    uint4 v[kScanVec];
    scan_load(data + beg, (uint32_t)(len - beg < (size_t)kScanChunk ? len - beg : (size_t)kScanChunk), v);
    uint32_t mine = 0, chunk;
#pragma unroll
    for (int r = 0; r < kScanVec; ++r) mine += v[r].x + v[r].y + v[r].z + v[r].w;
    warps_exscan(__reduce_add_sync(0xffffffffu, mine), s_warp, &chunk);
    const uint32_t nchunks = (uint32_t)((len + kScanChunk - 1) / kScanChunk);
    if (threadIdx.x == 0) {
        sums[blockIdx.x] = chunk;
        __threadfence();
        s_last = atomicAdd(done, 1u) + 1 == nchunks;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    uint32_t carry = 0;
    for (uint32_t base = 0; base < nchunks; base += kScanThreads) {
        const uint32_t i = base + threadIdx.x;
        uint32_t wt, t;
        const uint32_t x = warp_exscan(i < nchunks ? __ldcg(sums + i) : 0u, &wt);
        const uint32_t w = warps_exscan(wt, s_warp, &t);
        if (i < nchunks) sums[i] = carry + w + x;
        carry += t;
        __syncthreads();  // s_warp is read
    }
    if (threadIdx.x == 0) *total = carry;
}

__global__ void __launch_bounds__(kScanThreads)
    scan_apply_kernel(uint32_t* __restrict__ data, ScanLen L, const uint32_t* __restrict__ sums,
                      const uint32_t* __restrict__ total) {
    __shared__ uint32_t s_warp[kScanThreads / kWarp];
    const size_t len = L.get();
    const size_t beg = (size_t)blockIdx.x * kScanChunk;
    if (beg >= len) return;
    const uint32_t m = (uint32_t)(len - beg < (size_t)kScanChunk ? len - beg : (size_t)kScanChunk);
    uint32_t* p = data + beg;
    uint4 v[kScanVec];
    scan_load(p, m, v);
    uint32_t pre[kScanVec], mine = 0, chunk;
#pragma unroll
    for (int r = 0; r < kScanVec; ++r) {
        uint32_t t;
        pre[r] = mine + warp_exscan(v[r].x + v[r].y + v[r].z + v[r].w, &t);
        mine += t;
    }
    const uint32_t before = sums[blockIdx.x] + warps_exscan(mine, s_warp, &chunk);
#pragma unroll
    for (int r = 0; r < kScanVec; ++r) {
        const uint32_t i = scan_first() + r * (kWarp * 4);
        uint4 o;
        o.x = before + pre[r];
        o.y = o.x + v[r].x;
        o.z = o.y + v[r].y;
        o.w = o.z + v[r].z;
        if (i + 4 <= m) {
            *reinterpret_cast<uint4*>(p + i) = o;
        } else {
            if (i < m) p[i] = o.x;
            if (i + 1 < m) p[i + 1] = o.y;
            if (i + 2 < m) p[i + 2] = o.z;
        }
    }
    if (threadIdx.x == 0 && beg + m == len) p[m] = *total;  // the end of the last run
}

// ------------------------------------------------------------ pass-2 tiling

// From the scanned pass-1 counts, the pass-1 partitions become the pass-2
// segments; each is cut into tiles of kPartTile rows. Every block scans the
// (at most 2^kMaxBits) segment tile counts in shared memory itself; block 0
// writes the segments and the tile count, and the blocks fill the tiles
// grid-stride.
__global__ void __launch_bounds__(1024)
    seg_tiles_kernel(const uint32_t* __restrict__ counts1, uint32_t ntiles1, int b1,
                     const uint32_t* __restrict__ total1, SegInfo* __restrict__ segs,
                     Tile* __restrict__ tiles, uint32_t* __restrict__ ntiles2) {
    __shared__ uint32_t s_nt[1u << kMaxBits];
    __shared__ uint32_t s_base[1u << kMaxBits];
    __shared__ uint32_t s_warp[1024 / kWarp];
    const uint32_t nseg = 1u << b1;
    for (uint32_t s = threadIdx.x; s < nseg; s += blockDim.x) {
        const uint32_t st = ntiles1 ? counts1[(size_t)s * ntiles1] : 0u;
        const uint32_t en = s + 1 < nseg ? (ntiles1 ? counts1[(size_t)(s + 1) * ntiles1] : 0u) : *total1;
        const uint32_t sz = en - st;
        if (blockIdx.x == 0) {
            segs[s].start = st;
            segs[s].size = sz;
        }
        s_nt[s] = (sz + kPartTile - 1) / kPartTile;
    }
    __syncthreads();
    const uint32_t total = block_scan_smem(s_nt, s_base, nseg, s_warp);
    __syncthreads();
    if (blockIdx.x == 0)
        for (uint32_t s = threadIdx.x; s < nseg; s += blockDim.x) {
            segs[s].tile_base = s_base[s];
            segs[s].ntiles = s_nt[s];
        }
    // the segment of tile k is the last s with s_base[s] <= k among segments
    // that have tiles (binary search in shared memory)
    for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < total; k += gridDim.x * blockDim.x) {
        uint32_t lo = 0, hi = nseg;
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (s_base[mid] <= k) lo = mid; else hi = mid;
        }
        // (an empty segment shares its base with the next one, so the last
        // segment whose base is <= k always has tiles)
        const uint32_t j = k - s_base[lo];
        const uint32_t st = ntiles1 ? counts1[(size_t)lo * ntiles1] : 0u;
        const uint32_t sz = (lo + 1 < nseg ? (ntiles1 ? counts1[(size_t)(lo + 1) * ntiles1] : 0u) : *total1) - st;
        Tile tl;
        tl.start = st + j * kPartTile;
        const uint32_t rest = sz - j * kPartTile;
        tl.len = rest < (uint32_t)kPartTile ? rest : (uint32_t)kPartTile;
        tl.seg = lo;
        tl.tile_base = s_base[lo];
        tl.ntiles_seg = s_nt[lo];
        tiles[k] = tl;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *ntiles2 = total;
}

// Blocks of seg_tiles_kernel for at most `max_tiles` pass-2 tiles.
inline int seg_tiles_grid(size_t max_tiles, const DevInfo& di) {
    const size_t g = (max_tiles + 4095) / 4096;
    const size_t cap = (size_t)di.sms * 2;
    return (int)(g < 1 ? 1 : g > cap ? cap : g);
}

// Start of every final partition, plus part_start[P] = rows kept.
__global__ void part_start_kernel(const uint32_t* __restrict__ counts, int passes, uint32_t ntiles1,
                                  int b1, int b2, const SegInfo* __restrict__ segs,
                                  const uint32_t* __restrict__ total, uint32_t* __restrict__ part_start) {
    const uint32_t P = 1u << (b1 + b2);
    for (uint32_t p = blockIdx.x * blockDim.x + threadIdx.x; p <= P; p += gridDim.x * blockDim.x) {
        uint32_t v;
        if (p == P) {
            v = *total;
        } else if (passes == 1) {
            v = ntiles1 ? counts[(size_t)p * ntiles1] : 0u;
        } else {
            const SegInfo sg = segs[p >> b2];
            const uint32_t d2 = p & ((1u << b2) - 1u);
            v = sg.ntiles ? counts[((size_t)sg.tile_base << b2) + (size_t)d2 * sg.ntiles] : sg.start;
        }
        part_start[p] = v;
    }
}

template <typename K>
int occupancy_grid(K kern, int threads, size_t smem, const DevInfo& di, size_t work) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess ||
        per_sm < 1)
        per_sm = 1;
    size_t g = (size_t)di.sms * per_sm;
    if (work < g) g = work;
    return (int)(g < 1 ? 1 : g);
}

cudaError_t scan_counts(uint32_t* counts, ScanLen L, size_t max_len, uint32_t* block_sums, uint32_t* done,
                        uint32_t* total, cudaStream_t stream) {
    const uint32_t nblocks = (uint32_t)((max_len + kScanChunk - 1) / kScanChunk);
    const uint32_t g = nblocks ? nblocks : 1;
    scan_sums_kernel<<<g, kScanThreads, 0, stream>>>(counts, L, block_sums, done, total);
    scan_apply_kernel<<<g, kScanThreads, 0, stream>>>(counts, L, block_sums, total);
    return cudaGetLastError();
}

// Carried-column bytes per row (each is read once and written once per pass).
inline double carry_bytes(const ColCarry& cc) {
    double b = 0;
    for (int c = 0; c < cc.n; ++c) b += cc.bytes[c];
    return b;
}

// One partitioning (or sort) pass over n rows. Algorithmic bytes per launch:
// the histogram reads each key once; the scatter reads each (key, row) once
// and writes each kept (key', row) once (keys alone when the side keeps no
// tuple IDs), plus the carried columns; the scan reads and writes the counts.
template <typename InKey, typename KeyT, bool FIRST, bool SORTM>
cudaError_t run_pass(PartPass<InKey, KeyT> a, size_t max_tiles, const PartSide& s, uint32_t* total,
                     unsigned* err, const DevInfo& di, cudaStream_t stream, const char* side_name, int pass_no) {
    cudaError_t e;
    a.scan_done = s.total + 3;
    const size_t hsmem = hist_smem_bytes(a.bits);
    // The first batch of carried columns is staged beside the keys, and written
    // with them, when no tuple IDs travel, two CTAs still fit an SM, and the
    // digits' runs of the keys and of the batch lie in at most 256 places; over
    // more, keys and columns do better one after the other. Apart against
    // after, 600M rows with an 8-byte column: 7 bits (256 places) 2.65 against
    // 3.00 ms in pass 1 and 2.58 against 2.68 in pass 2, 8 bits (512) 3.83
    // against 3.23 and 3.20 against 2.80; 2^28 rows with two 4-byte columns: 6
    // bits (192) 1.34 against 1.30 and 1.34 against 1.36, 7 bits (384) 1.78
    // against 1.39 and 1.52 against 1.41; 120M rows, 5 and 6 bits: 0.54 against
    // 0.58 and 0.57 against 0.58.
    const int places = a.cc.n ? 1 + batch_end(a.cc, 0) : 1;
    a.col_apart = !SORTM && a.cc.n && !a.out_idx && ((size_t)places << a.bits) <= 256 &&
                  scatter_smem_bytes<InKey, KeyT, FIRST>(a.bits, false, true, true) <= kTwoPerSm;
    const size_t ssmem = SORTM ? sort_scatter_smem_bytes<InKey, KeyT, FIRST>(a.bits)
                               : scatter_smem_bytes<InKey, KeyT, FIRST>(a.bits, a.out_idx != nullptr, a.cc.n > 0, a.col_apart);
    auto hist = part_hist_kernel<InKey, KeyT, FIRST, SORTM>;
    auto scat = SORTM ? sort_scatter_kernel<InKey, KeyT, FIRST>
                : a.bits <= kDigitBits1
                    ? (a.cc.n ? part_scatter_kernel<InKey, KeyT, FIRST, 1, true>
                              : part_scatter_kernel<InKey, KeyT, FIRST, 1, false>)
                    : (a.cc.n ? part_scatter_kernel<InKey, KeyT, FIRST, kGoffPerThread, true>
                              : part_scatter_kernel<InKey, KeyT, FIRST, kGoffPerThread, false>);
    if ((e = allow_smem(hist)) != cudaSuccess || (e = allow_smem(scat)) != cudaSuccess) return e;
    const double n = (double)a.n;
    const double in_key = FIRST ? (double)sizeof(InKey) : (double)sizeof(KeyT);
    const double row = a.out_idx ? (double)sizeof(uint32_t) : 0.0;  // tuple IDs, when the side keeps them
    const double tuple = (double)sizeof(KeyT) + row;
    const double in_tuple = FIRST ? (double)sizeof(InKey) : tuple;
    const char* kind = SORTM ? "sort" : "part";
    char name[32];
    {
        snprintf(name, sizeof name, "%s_hist.p%d.%s", kind, pass_no, side_name);
        ProfScope ps(name, n * in_key, stream);
        // fewer tiles than about two warps' worth of the chip: a CTA per tile,
        // or the last wave of whole tiles is nearly empty (4,883 tiles of 64-bit
        // keys: 42 us split, 53 whole; 12,208 of 32-bit keys: 122 split, 88 whole)
        const bool split = max_tiles < (size_t)di.sms * 64;
        const size_t work = split ? max_tiles : (max_tiles + kHistWarps - 1) / kHistWarps;
        hist<<<occupancy_grid(hist, kHistThreads, hsmem, di, work), kHistThreads, hsmem, stream>>>(a, split);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    ScanLen L{max_tiles << a.bits, a.tiles ? a.ntiles_dev : nullptr, a.bits};
    {
        snprintf(name, sizeof name, "%s_scan.p%d.%s", kind, pass_no, side_name);
        ProfScope ps(name, 12.0 * (double)(max_tiles << a.bits), stream, 0.0, 2);
        if ((e = scan_counts(a.counts, L, max_tiles << a.bits, s.block_sums, a.scan_done, total, stream)) !=
            cudaSuccess)
            return e;
    }
    snprintf(name, sizeof name, "%s_scatter.p%d.%s", kind, pass_no, side_name);
    ProfScope ps(name, n * (in_tuple + tuple + 2.0 * carry_bytes(a.cc)), stream);
    scat<<<occupancy_grid(scat, kPartThreads, ssmem, di, max_tiles), kPartThreads, ssmem, stream>>>(a, err);
    return cudaGetLastError();
}

// Carried columns of pass `pass` (0-based) of one side: pass 0 reads the
// caller's columns, later passes the previous pass's copies.
ColCarry carry_for(const PlanDev& plan, int side, const ColSide* carry, const PartSide& s, int pass) {
    ColCarry cc{};
    cc.n = plan.gftr && carry ? plan.ncols[side] : 0;
    for (int c = 0; c < cc.n; ++c) {
        cc.in[c] = pass == 0 ? carry->src[c] : s.col[(pass - 1) & 1][c];
        cc.out[c] = s.col[pass & 1][c];
        cc.bytes[c] = plan.col_bytes[side][c];
    }
    return cc;
}

template <typename InKey, typename KeyT>
cudaError_t partition_typed(const InKey* keys, uint32_t n, int side, const PlanDev& plan, const PartSide& s,
                            const ColSide* carry, unsigned* err, const DevInfo& di, cudaStream_t stream) {
    const int passes = plan.variant == 3 ? 2 : 1;
    const int b1 = plan.bits1, b2 = passes == 2 ? plan.bits2 : 0;
    const uint32_t ntiles1 = (n + kPartTile - 1) / kPartTile;
    cudaError_t e;

    PartPass<InKey, KeyT> a{};
    a.raw = keys;
    a.src_end[0] = keys + n;
    a.out_key = static_cast<KeyT*>(s.key[0]);
    a.out_idx = plan.no_rows ? nullptr : s.idx[0];
    a.n = n;
    a.offset = plan.range.offset;
    a.span = side == 1 && plan.check_range ? (uint64_t)plan.range.hi - (uint64_t)plan.range.lo : ~0ull;
    a.dshift = KeyCodec<KeyT>::kBits - b1;
    a.kbits = plan.kbits;
    a.dmask = (1u << b1) - 1u;
    a.bits = b1;
    a.counts = s.counts;
    a.tiles = nullptr;
    a.ntiles_fixed = ntiles1;
    a.cc = carry_for(plan, side, carry, s, 0);
    const char* sn = side == 0 ? "build" : "probe";
    if ((e = run_pass<InKey, KeyT, true, false>(a, ntiles1, s, s.total, err, di, stream, sn, 1)) != cudaSuccess)
        return e;

    if (passes == 2) {
        {
            ProfScope ps("seg_tiles", 0.0, stream);
            const size_t max_tiles2 = (size_t)ntiles1 + ((size_t)1 << b1);
            seg_tiles_kernel<<<seg_tiles_grid(max_tiles2, di), 1024, 0, stream>>>(s.counts, ntiles1, b1, s.total,
                                                                                 s.segs, s.tiles, s.total + 2);
            if ((e = cudaGetLastError()) != cudaSuccess) return e;
        }
        PartPass<InKey, KeyT> b{};
        b.in_key = static_cast<const KeyT*>(s.key[0]);
        b.in_idx = plan.no_rows ? nullptr : s.idx[0];
        b.src_end[0] = static_cast<const char*>(s.key[0]) + (size_t)n * sizeof(KeyT) + 16;
        b.src_end[1] = s.idx[0] + (size_t)n + 4;
        b.out_key = static_cast<KeyT*>(s.key[1]);
        b.out_idx = plan.no_rows ? nullptr : s.idx[1];
        b.n = n;
        b.dshift = KeyCodec<KeyT>::kBits - b1 - b2;
        b.dmask = (1u << b2) - 1u;
        b.bits = b2;
        b.counts = s.counts;
        b.tiles = s.tiles;
        b.ntiles_dev = s.total + 2;
        b.cc = carry_for(plan, side, carry, s, 1);
        const size_t max_tiles2 = (size_t)ntiles1 + ((size_t)1 << b1);
        if ((e = run_pass<InKey, KeyT, false, false>(b, max_tiles2, s, s.total + 1, err, di, stream, sn, 2)) !=
            cudaSuccess)
            return e;
    }
    const uint32_t P = 1u << (b1 + b2);
    const int threads = 256;
    const int blocks = (int)((P + 1 + threads - 1) / threads);
    ProfScope ps("part_start", 8.0 * (P + 1), stream);
    part_start_kernel<<<blocks, threads, 0, stream>>>(s.counts, passes, ntiles1, b1, b2, s.segs, s.total,
                                                      s.part_start);
    return cudaGetLastError();
}

// Stable LSD radix sort of one side (see sort_scatter_kernel): pass 1 reads
// the raw keys (range test and narrowing as in partitioning) with a fixed
// tiling; the kept rows then form one segment, tiled once, which every later
// pass re-reads from the previous pass's buffer.
template <typename InKey, typename KeyT>
cudaError_t sort_typed(const InKey* keys, uint32_t n, int side, const PlanDev& plan, const PartSide& s,
                       const ColSide* carry, unsigned* err, const DevInfo& di, cudaStream_t stream) {
    const int D = plan.bits1, passes = plan.bits2;
    const uint32_t ntiles1 = (n + kPartTile - 1) / kPartTile;
    const char* sn = side == 0 ? "build" : "probe";
    cudaError_t e;
    PartPass<InKey, KeyT> a{};
    a.raw = keys;
    a.src_end[0] = keys + n;
    a.out_key = static_cast<KeyT*>(s.key[0]);
    a.out_idx = plan.no_rows ? nullptr : s.idx[0];
    a.n = n;
    a.offset = plan.range.offset;
    a.span = side == 1 && plan.check_range ? (uint64_t)plan.range.hi - (uint64_t)plan.range.lo : ~0ull;
    a.dshift = 0;
    a.dmask = (1u << D) - 1u;
    a.bits = D;
    a.counts = s.counts;
    a.tiles = nullptr;
    a.ntiles_fixed = ntiles1;
    a.cc = carry_for(plan, side, carry, s, 0);
    if ((e = run_pass<InKey, KeyT, true, true>(a, ntiles1, s, s.total, err, di, stream, sn, 1)) != cudaSuccess)
        return e;
    if (passes < 2) return cudaSuccess;
    {
        ProfScope ps("seg_tiles", 0.0, stream);
        seg_tiles_kernel<<<seg_tiles_grid((size_t)ntiles1 + 1, di), 1024, 0, stream>>>(s.counts, ntiles1, 0, s.total,
                                                                                     s.segs, s.tiles, s.total + 2);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    for (int i = 1; i < passes; ++i) {
        PartPass<InKey, KeyT> b{};
        b.in_key = static_cast<const KeyT*>(s.key[(i - 1) & 1]);
        b.in_idx = plan.no_rows ? nullptr : s.idx[(i - 1) & 1];
        b.src_end[0] = static_cast<const char*>(s.key[(i - 1) & 1]) + (size_t)n * sizeof(KeyT) + 16;
        b.src_end[1] = s.idx[(i - 1) & 1] + (size_t)n + 4;
        b.out_key = static_cast<KeyT*>(s.key[i & 1]);
        b.out_idx = plan.no_rows ? nullptr : s.idx[i & 1];
        b.n = n;
        b.dshift = i * D;
        b.dmask = (1u << D) - 1u;
        b.bits = D;
        b.counts = s.counts;
        b.tiles = s.tiles;
        b.ntiles_dev = s.total + 2;
        b.cc = carry_for(plan, side, carry, s, i);
        if ((e = run_pass<InKey, KeyT, false, true>(b, ntiles1, s, s.total + 1, err, di, stream, sn, i + 1)) !=
            cudaSuccess)
            return e;
    }
    return cudaSuccess;
}

}  // namespace

size_t part_counts_len(int64_t n, int b1, int b2, int passes) {
    const size_t ntiles1 = (size_t)((n + kPartTile - 1) / kPartTile);
    size_t l1 = ntiles1 << b1;
    size_t l2 = passes == 2 ? (ntiles1 + ((size_t)1 << b1)) << b2 : 0;
    return l1 > l2 ? l1 : l2;
}

size_t part_scan_blocks(size_t counts_len) { return (counts_len + kScanChunk - 1) / kScanChunk + 1; }

void part_side_layout(Carve& c, PartSide& ps, int64_t n, int b1, int b2, int passes, bool sort, size_t kb,
                      const PlanDev& plan, int side) {
    const int nbuf = passes < 2 ? passes : 2;
    const int ncols = plan.gftr ? plan.ncols[side] : 0;
    for (int k = 0; k < 2; ++k) {
        // 16 bytes of slack after each buffer: a later pass's tile loads may
        // read the aligned cover of the last rows (see PartPass::src_end)
        ps.key[k] = k < nbuf ? c.take<unsigned char>((size_t)n * kb + 16) : nullptr;
        ps.idx[k] = k < nbuf ? c.take<uint32_t>((size_t)n + 4) : nullptr;
        for (int q = 0; q < kMaxCols; ++q)
            ps.col[k][q] = (k < nbuf && q < ncols) ? c.take<unsigned char>((size_t)n * plan.col_bytes[side][q] + 16)
                                                  : nullptr;
    }
    const size_t ntiles1 = (size_t)((n + kPartTile - 1) / kPartTile);
    ps.counts_len = sort ? ntiles1 << b1 : part_counts_len(n, b1, b2, passes);
    ps.counts = c.take<uint32_t>(ps.counts_len + 1);  // and the total behind the last entry
    ps.block_sums = c.take<uint32_t>(part_scan_blocks(ps.counts_len));
    ps.total = c.take<uint32_t>(4);
    ps.segs = c.take<SegInfo>(sort ? 1 : (size_t)1 << b1);
    ps.tiles = c.take<Tile>(passes >= 2 ? ntiles1 + (sort ? 1 : ((size_t)1 << b1)) : 1);
    ps.part_start = sort ? nullptr : c.take<uint32_t>(((size_t)1 << (b1 + b2)) + 1);
}

int sort_key_bits(const PlanDev& plan) {
    const uint64_t span = (uint64_t)plan.range.hi - (uint64_t)plan.range.lo;
    int b = 0;
    while (b < 64 && (span >> b) != 0) ++b;
    return b;
}

cudaError_t partition_side(const void* keys, int64_t n, int side, const PlanDev& plan, const PartSide& s,
                           const ColSide* carry, unsigned* err, cudaStream_t stream) {
    DevInfo di;
    cudaError_t e = current_device_info(&di);
    if (e != cudaSuccess) return e;
    const uint32_t nn = (uint32_t)n;
    if (plan.key32) {
        if (plan.dtype == 0)
            return partition_typed<int32_t, uint32_t>(static_cast<const int32_t*>(keys), nn, side, plan, s, carry,
                                                      err, di, stream);
        return partition_typed<int64_t, uint32_t>(static_cast<const int64_t*>(keys), nn, side, plan, s, carry,
                                                  err, di, stream);
    }
    return partition_typed<int64_t, uint64_t>(static_cast<const int64_t*>(keys), nn, side, plan, s, carry, err,
                                              di, stream);
}

cudaError_t sort_side(const void* keys, int64_t n, int side, const PlanDev& plan, const PartSide& s,
                      const ColSide* carry, unsigned* err, cudaStream_t stream) {
    DevInfo di;
    cudaError_t e = current_device_info(&di);
    if (e != cudaSuccess) return e;
    const uint32_t nn = (uint32_t)n;
    if (plan.key32) {
        if (plan.dtype == 0)
            return sort_typed<int32_t, uint32_t>(static_cast<const int32_t*>(keys), nn, side, plan, s, carry, err,
                                                 di, stream);
        return sort_typed<int64_t, uint32_t>(static_cast<const int64_t*>(keys), nn, side, plan, s, carry, err, di,
                                             stream);
    }
    return sort_typed<int64_t, uint64_t>(static_cast<const int64_t*>(keys), nn, side, plan, s, carry, err, di,
                                         stream);
}

}  // namespace eiger
