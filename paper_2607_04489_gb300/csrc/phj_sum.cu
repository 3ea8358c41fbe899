// Fused exact sum of the partitioned join with carried payloads (GFTR): per
// work item (phj.cuh) one shared-memory table that maps every distinct build
// key of the chunk to (sum of its build payloads, rows of that key). A probe
// row with payload q then contributes sum + rows * q and `rows` matches from
// one lookup, whatever the key's multiplicity: the sum over matches (i, j) of
// b_i + q_j, taken probe row by probe row. Everything is modulo 2^64, so the
// order of the additions does not matter.
//
// The rows arrive through the CTA's stream (stream.cuh). Hash tables, two CTAs
// per SM (one over full partitions, see big_tables), are bound by shared memory: about 29 wavefronts per 32 probe rows (the
// key group's 16-byte loads at random groups, the sum's 8-byte loads at random
// slots) keep its pipe 87 % busy. Direct-addressed tables need about 11 and run
// near the row streams' rate (5.3 TB/s with 2^12 slots). Measured on GB300,
// 150M x 600M dense int32 keys, int64 payloads: 6.76 ms when every match
// gathered both payloads from global memory by position, 4.76 ms with the sums
// in hash tables, rows in registers one round ahead and one slot per probe,
// 3.92 ms streamed with key groups (3.46 ms on mixed keys), 1.71 ms direct with
// 2^12 slots, 1.91 ms with 2^13 (whose partitions take 1.9 ms less to make);
// 8M x 30M 64-bit keys of six rows each: 2.79 -> 0.21 ms.
#include <algorithm>
#include <cmath>

#include "emit.cuh"
#include "kernels.cuh"
#include "phj.cuh"
#include "stream.cuh"

namespace eiger {

namespace {

constexpr int kStages = 2;

// Slots of {key, sum as two 32-bit halves, rows beyond the first}. The all-ones
// key is the empty pattern; that key itself lives in the extra slot kSlots,
// whose key word turns 0 when it is taken.
template <typename KeyT, bool BIG>
struct SumTable {
    // More than a full build chunk, and two CTAs' tables and rings fit an SM; or,
    // BIG, twice that for one CTA per SM (see big_tables).
    static constexpr uint32_t kSlots = (sizeof(KeyT) == 4 ? 4864 : 4640) * (BIG ? 2 : 1);
    static_assert(kSlots > kBuildCap && kSlots % 4 == 0, "a full build chunk leaves empty slots");
    static constexpr uint32_t kAll = kSlots + 4;  // arrays stay 16-byte aligned
    static constexpr size_t kBytes = kAll * (8 + sizeof(KeyT) + 4);
    static constexpr KeyT kEmpty = ~KeyT(0);
    KeyT* key;
    uint2* sum;
    uint32_t* more;
    __device__ void bind(unsigned char* smem) {
        sum = reinterpret_cast<uint2*>(smem);
        key = reinterpret_cast<KeyT*>(smem + (size_t)kAll * 8);
        more = reinterpret_cast<uint32_t*>(smem + (size_t)kAll * (8 + sizeof(KeyT)));
    }
    __device__ void clear_slot(uint32_t i) {
        sum[i] = make_uint2(0, 0);
        key[i] = kEmpty;
        more[i] = 0;
    }
    template <int THREADS>
    __device__ void clear(uint32_t tsize) {
        for (uint32_t i = threadIdx.x; i < tsize; i += THREADS) clear_slot(i);
        if (threadIdx.x == 0) clear_slot(kSlots);
    }
    using Group = KeyGroup<KeyT>;
    __device__ static uint32_t home(KeyT k, uint32_t tsize) { return group_home<KeyT>(slot_hash(k), tsize); }
    // Adds build row (k, v): 0 for a new key, 1 for a further row of a key, -1
    // when the table is full. 32-bit shared-memory atomics are native: the low
    // half's returns the old value, and the high half takes the addend's high
    // half plus the carry, when that is not zero.
    __device__ int add(KeyT k, uint64_t v, uint32_t tsize) {
        uint32_t s;
        bool again;
        if (k == kEmpty) {
            s = kSlots;
            again = cas_key(key + s, kEmpty, KeyT(0)) != kEmpty;
        } else {
            bool fresh = false;
            s = claim_slot(key, tsize, k, home(k, tsize), fresh);
            if (s == ~0u) return -1;
            again = !fresh;
        }
        const uint32_t lo = (uint32_t)v;
        const uint32_t old = atomicAdd(&sum[s].x, lo);
        const uint32_t hi = (uint32_t)(v >> 32) + (old + lo < lo ? 1u : 0u);
        if (hi) atomicAdd(&sum[s].y, hi);
        if (again) atomicAdd(more + s, 1u);
        return again ? 1 : 0;
    }
    // Slot of k, or ~0u.
    __device__ uint32_t find(KeyT k, uint32_t tsize) const {
        if (k == kEmpty) return key[kSlots] != kEmpty ? kSlots : ~0u;
        uint32_t s = home(k, tsize);
        for (uint32_t step = 0; step < tsize; step += Group::kN) {
            Group g;
            g.load(key + s);
            const uint32_t i = g.first(k);
            if (i < Group::kN) return s + i;
            if (g.last() == kEmpty) return ~0u;
            s = next_group<KeyT>(s, tsize);
        }
        return ~0u;
    }
};

// Direct-addressed form (phj.cuh): slot -> {sum, rows}. No key is stored, no
// search is made, and a key's further rows need no other treatment.
struct SumDirect {
    uint32_t* lo;
    uint32_t* hi;
    uint32_t* rows;
    int pbits, sbits;
    static __host__ __device__ size_t bytes(int sbits) { return (((size_t)1 << sbits) * 3 * 4 + 15) / 16 * 16; }
    __device__ void bind(unsigned char* smem, int pb, int sb) {
        lo = reinterpret_cast<uint32_t*>(smem);
        hi = lo + (1u << sb);
        rows = hi + (1u << sb);
        pbits = pb;
        sbits = sb;
    }
    template <int THREADS>
    __device__ void clear() {
        uint4* p = reinterpret_cast<uint4*>(lo);
        const uint32_t n = (uint32_t)(bytes(sbits) / 16);
        for (uint32_t i = threadIdx.x; i < n; i += THREADS) p[i] = make_uint4(0, 0, 0, 0);
    }
    __device__ void add(uint32_t k, uint64_t v) {
        const uint32_t s = direct_slot(k, pbits, sbits), l = (uint32_t)v;
        const uint32_t old = atomicAdd(lo + s, l);
        const uint32_t h = (uint32_t)(v >> 32) + (old + l < l ? 1u : 0u);
        if (h) atomicAdd(hi + s, h);
        atomicAdd(rows + s, 1u);
    }
};

template <typename KeyT, typename PayT, bool DIRECT, int CONS>
struct SumStream : Stream<2, kStages, 4, DIRECT ? 2 * CONS : 4096 / sizeof(KeyT), ItemRows> {
    static constexpr size_t kBytes = kStages * (SumStream::col_bytes(sizeof(KeyT)) + SumStream::col_bytes(sizeof(PayT)));
};

// CONS consumer threads (plus the stream's two warps): 512, two CTAs per SM, or
// 960 over a table that only one CTA per SM has room for.
template <int CONS>
constexpr bool kBig = CONS > 512;
template <typename KeyT, typename PayT, bool DIRECT, int CONS>
__global__ void __launch_bounds__(CONS + kStreamWarps* kWarp, 1024 / CONS)
    phj_sum_kernel(JoinIn<KeyT> a, const PayT* __restrict__ bpay, const PayT* __restrict__ ppay, Ctrl* ctrl) {
    using S = SumStream<KeyT, PayT, DIRECT, CONS>;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ typename S::Shared s_stream;
    S st;
    st.w[0] = sizeof(KeyT);
    st.w[1] = sizeof(PayT);
    st.setup(&s_stream, smem + (DIRECT ? SumDirect::bytes(a.sbits) : SumTable<KeyT, kBig<CONS>>::kBytes), CONS / kWarp);
    constexpr uint32_t kStageRows = S::kRows;
    typename S::ItemPos q;
    const int warp = threadIdx.x / kWarp;

    if (warp == CONS / kWarp) {  // scheduler
        const unsigned long long nitems = ctrl->nitems;
        for (;;) {
            unsigned long long item = 0;
            if (lane_id() == 0) item = atomicAdd(&ctrl->next_item, 1ull);
            item = __shfl_sync(0xffffffffu, item, 0);
            ItemRows it{};  // no build rows: the end
            if (item < nitems) it = item_rows(a, item, find_partition(a.item_prefix, a.P, item));
            bool ok = true;
            if (lane_id() == 0) ok = st.publish(q, it);
            if (item >= nitems || !__all_sync(0xffffffffu, ok)) break;
        }
        return;
    }
    typename S::StagePos sp;
    if (warp == CONS / kWarp + 1) {  // producer
        if (lane_id() == 0) {
            bool ok = true;
            while (ok) {
                ok = st.wait(&s_stream.ifull[q.i], q.phase);
                if (!ok) break;
                const ItemRows it = s_stream.item[q.i];
                mbar_arrive(&s_stream.iempty[q.i]);
                q.next();
                if (it.bn == 0) break;
                RowCols<2> src;
                src.p[0] = reinterpret_cast<const char*>(a.bkey + it.bs0);
                src.p[1] = reinterpret_cast<const char*>(bpay + it.bs0);
                ok = st.produce(sp, src, it.bn);
                src.p[0] = reinterpret_cast<const char*>(a.pkey + it.ps0);
                src.p[1] = reinterpret_cast<const char*>(ppay + it.ps0);
                ok = ok && st.produce(sp, src, it.pn);
            }
            st.drain(sp);
        }
        return;
    }

    SumTable<KeyT, kBig<CONS>> tab;
    SumDirect dir;
    if constexpr (DIRECT)
        dir.bind(smem, a.pbits, a.sbits);
    else
        tab.bind(smem);
    AggState agg{0ull, 0ull};
    bool dead = false;
    // Every row of n streamed rows: f(key, payload), two rows of a thread at a
    // time; the warp is brought together after each pair.
    auto rows_of = [&](const KeyT* kp, const PayT* vp, uint32_t n, auto&& f) {
        for (uint32_t base = 0; base < n; base += kStageRows) {
            if (!dead && !st.wait(&s_stream.full[sp.i], sp.phase)) dead = true;
            const KeyT* k = st.template rows<KeyT>(sp, 0, reinterpret_cast<const char*>(kp), base);
            const PayT* v = st.template rows<PayT>(sp, 1, reinterpret_cast<const char*>(vp), base);
            const uint32_t len = dead ? 0u : min(n - base, kStageRows);
            f(k, v, len);
            st.release(sp);
        }
    };
    for (;;) {
        if (!st.wait(&s_stream.ifull[q.i], q.phase)) dead = true;
        const ItemRows it = s_stream.item[q.i];
        __syncwarp();
        if (lane_id() == 0) mbar_arrive(&s_stream.iempty[q.i]);
        q.next();
        // (every consumer has left the previous item's table here)
        if (consumers_stop<CONS>(dead, it.bn == 0, &ctrl->err)) break;
        if constexpr (DIRECT) {
            dir.template clear<CONS>();
            consumers_sync<CONS>();
            rows_of(a.bkey + it.bs0, bpay + it.bs0, it.bn, [&](const KeyT* k, const PayT* v, uint32_t len) {
                for (uint32_t i = threadIdx.x; i < len; i += CONS) dir.add((uint32_t)k[i], (uint64_t)(int64_t)v[i]);
            });
            consumers_sync<CONS>();
            rows_of(a.pkey + it.ps0, ppay + it.ps0, it.pn, [&](const KeyT* k, const PayT* v, uint32_t len) {
#pragma unroll 2
                for (uint32_t i = threadIdx.x; i < len; i += CONS) {
                    const uint32_t s = direct_slot((uint32_t)k[i], a.pbits, a.sbits);
                    const uint32_t rows = dir.rows[s];
                    // an empty slot adds sum 0 and rows 0
                    agg.sum += (((uint64_t)dir.hi[s] << 32) | dir.lo[s]) + rows * (uint64_t)(int64_t)v[i];
                    agg.count += rows;
                }
            });
        } else {
            uint32_t tsize = (3 * it.bn + 3) & ~3u;  // load 1/3 while that fits
            if (tsize < 64) tsize = 64;
            if (tsize > SumTable<KeyT, kBig<CONS>>::kSlots) tsize = SumTable<KeyT, kBig<CONS>>::kSlots;
            tab.template clear<CONS>(tsize);
            consumers_sync<CONS>();
            int dup = 0;
            rows_of(a.bkey + it.bs0, bpay + it.bs0, it.bn, [&](const KeyT* k, const PayT* v, uint32_t len) {
                for (uint32_t i = threadIdx.x; i < len; i += CONS) {
                    const int r = tab.add(k[i], (uint64_t)(int64_t)v[i], tsize);
                    if (r < 0) atomicOr(&ctrl->err, kErrTableFull);
                    dup |= r;
                }
            });
            const bool unique = !consumers_or<CONS>(dup != 0);
            rows_of(a.pkey + it.ps0, ppay + it.ps0, it.pn, [&](const KeyT* k, const PayT* v, uint32_t len) {
#pragma unroll 2
                for (uint32_t i = threadIdx.x; i < len; i += CONS) {
                    const uint32_t s = tab.find(k[i], tsize);
                    if (s == ~0u) continue;
                    const uint2 bs = tab.sum[s];
                    const uint64_t b = ((uint64_t)bs.y << 32) | bs.x;
                    const uint64_t q8 = (uint64_t)(int64_t)v[i];
                    const uint32_t rows = unique ? 1u : 1u + tab.more[s];
                    agg.sum += b + (unique ? q8 : rows * q8);
                    agg.count += rows;
                }
            });
        }
    }
    agg_commit(agg, ctrl);
}

template <typename KeyT, typename PayT, bool DIRECT, int CONS>
cudaError_t launch_sum(const JoinIn<KeyT>& a, const JoinOut& out, Ctrl* ctrl, const DevInfo& di, cudaStream_t stream,
                       int64_t nb, int64_t np) {
    auto kern = phj_sum_kernel<KeyT, PayT, DIRECT, CONS>;
    const size_t smem = (DIRECT ? SumDirect::bytes(a.sbits) : SumTable<KeyT, kBig<CONS>>::kBytes) + SumStream<KeyT, PayT, DIRECT, CONS>::kBytes;
    cudaError_t e = allow_smem(kern);
    if (e != cudaSuccess) return e;
    constexpr int kThreads = CONS + kStreamWarps * kWarp;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    // keys and payloads of both sides, each read once
    ProfScope ps("phj_sum", (double)(sizeof(KeyT) + sizeof(PayT)) * (double)(nb + np), stream);
    kern<<<di.sms * per_sm, kThreads, smem, stream>>>(a, static_cast<const PayT*>(out.b.src[0]),
                                                     static_cast<const PayT*>(out.p.src[0]), ctrl);
    return cudaGetLastError();
}

// Whether hash tables want the larger form: where the distinct keys of an ordinary
// work item fill more than about two thirds of the smaller one's slots, whose
// searches then grow long. 2^20 to 2^22 distinct keys in 1024 partitions, four probe
// rows a key, int64 payloads, us in the smaller / larger form: 32-bit keys, 2816
// rows a partition 119 / 135, 3328 162 / 164, 3584 197 / 172, 4096 379 / 203, 4500
// 1024 / 236, 8192 (two items) 1809 / 682; 64-bit ones 2816 170 / 180, 3072 223 / 195,
// 4096 1034 / 270, 4500 6058 / 326, 8192 5729 / 944. The items of a partition hold
// some rows of most of its repeated keys.
template <typename KeyT>
bool big_tables(const JoinIn<KeyT>& a, int64_t nb, double distinct) {
    const double rows = (double)nb / a.P, items = std::max(1.0, std::ceil(rows / kBuildCap));
    const double keys = distinct * rows * (1.0 - std::pow(1.0 - 1.0 / items, 1.0 / std::max(distinct, 1e-9)));
    return keys > (sizeof(KeyT) == 4 ? 3300.0 : 2900.0);
}

template <typename KeyT, typename PayT>
cudaError_t launch_sum_for(const JoinIn<KeyT>& a, int direct, double distinct, const JoinOut& out, Ctrl* ctrl, const DevInfo& di,
                           cudaStream_t stream, int64_t nb, int64_t np) {
    if constexpr (sizeof(KeyT) == 4) {
        if (direct)
            return a.sbits <= 12 ? launch_sum<KeyT, PayT, true, 512>(a, out, ctrl, di, stream, nb, np)
                                 : launch_sum<KeyT, PayT, true, 960>(a, out, ctrl, di, stream, nb, np);
    }
    return big_tables(a, nb, distinct) ? launch_sum<KeyT, PayT, false, 960>(a, out, ctrl, di, stream, nb, np)
                                       : launch_sum<KeyT, PayT, false, 512>(a, out, ctrl, di, stream, nb, np);
}

}  // namespace

template <typename KeyT>
cudaError_t phj_sum_launch(const JoinIn<KeyT>& a, int direct, double distinct, const JoinOut& out, Ctrl* ctrl,
                           const DevInfo& di, cudaStream_t stream, int64_t nb, int64_t np) {
    return out.b.bytes[0] == 4 ? launch_sum_for<KeyT, int32_t>(a, direct, distinct, out, ctrl, di, stream, nb, np)
                               : launch_sum_for<KeyT, int64_t>(a, direct, distinct, out, ctrl, di, stream, nb, np);
}

template cudaError_t phj_sum_launch<uint32_t>(const JoinIn<uint32_t>&, int, double, const JoinOut&, Ctrl*,
                                              const DevInfo&, cudaStream_t, int64_t, int64_t);
template cudaError_t phj_sum_launch<uint64_t>(const JoinIn<uint64_t>&, int, double, const JoinOut&, Ctrl*,
                                              const DevInfo&, cudaStream_t, int64_t, int64_t);

}  // namespace eiger
