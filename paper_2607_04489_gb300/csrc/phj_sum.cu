// Fused exact sum of the partitioned join with carried payloads (GFTR): per
// work item (phj.cuh) one shared-memory table that maps every distinct build
// key of the chunk to (sum of its build payloads, rows of that key). A probe
// row with payload q then contributes sum + rows * q and `rows` matches from
// one lookup, whatever the key's multiplicity: the sum over matches (i, j) of
// b_i + q_j, taken probe row by probe row. Everything is modulo 2^64, so the
// order of the additions does not matter.
//
// The rows arrive through the CTA's stream (stream.cuh), two CTAs per SM. What
// bounds it is shared memory, not the row streams: about 29 shared-memory
// wavefronts per 32 probe rows (the key group's 16-byte loads at random
// groups, the sum's 8-byte loads at random slots) keep its pipe 87 % busy.
// Measured on GB300, 150M x 600M int32 keys, int64 payloads (16-bit
// partitions): 6.76 ms when every match gathered both payloads from global
// memory by position, 4.76 ms with the sums in the table, rows in registers
// one round ahead and one slot per probe, 3.92 ms as it is; 8M x 30M 64-bit
// keys of six rows each: 2.79 -> 0.21 ms (the multiplicity no longer counts).
#include "emit.cuh"
#include "kernels.cuh"
#include "phj.cuh"
#include "stream.cuh"

namespace eiger {

namespace {

constexpr int kConsumers = kJoinThreads;
constexpr int kSumThreads = kConsumers + kStreamWarps * kWarp;
constexpr int kStages = 2;

// Slots of {key, sum as two 32-bit halves, rows beyond the first}. The all-ones
// key is the empty pattern; that key itself lives in the extra slot kSlots,
// whose key word turns 0 when it is taken.
template <typename KeyT>
struct SumTable {
    // More than a full build chunk, and two CTAs' tables and rings fit an SM.
    static constexpr uint32_t kSlots = sizeof(KeyT) == 4 ? 4864 : 4640;
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
    __device__ void clear(uint32_t tsize) {
        for (uint32_t i = threadIdx.x; i < tsize; i += kConsumers) clear_slot(i);
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
            again = cas_smem(key + s, kEmpty, KeyT(0)) != kEmpty;
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

template <typename KeyT, typename PayT>
struct SumStream : Stream<2, kStages, 4, 4096 / sizeof(KeyT), ItemRows> {
    static constexpr size_t kBytes = kStages * (SumStream::col_bytes(sizeof(KeyT)) + SumStream::col_bytes(sizeof(PayT)));
};

template <typename KeyT, typename PayT>
__global__ void __launch_bounds__(kSumThreads, 2)
    phj_sum_kernel(JoinIn<KeyT> a, const PayT* __restrict__ bpay, const PayT* __restrict__ ppay, Ctrl* ctrl) {
    using S = SumStream<KeyT, PayT>;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ typename S::Shared s_stream;
    S st;
    st.w[0] = sizeof(KeyT);
    st.w[1] = sizeof(PayT);
    st.setup(&s_stream, smem + SumTable<KeyT>::kBytes, kConsumers / kWarp);
    constexpr uint32_t kStageRows = S::kRows;
    typename S::ItemPos q;
    const int warp = threadIdx.x / kWarp;

    if (warp == kConsumers / kWarp) {  // scheduler
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
    if (warp == kConsumers / kWarp + 1) {  // producer
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

    SumTable<KeyT> tab;
    tab.bind(smem);
    AggState agg{0ull, 0ull};
    bool dead = false;
    for (;;) {
        if (!st.wait(&s_stream.ifull[q.i], q.phase)) dead = true;
        ItemRows it = s_stream.item[q.i];
        __syncwarp();
        if (lane_id() == 0) mbar_arrive(&s_stream.iempty[q.i]);
        q.next();
        // (every consumer has left the previous item's table here)
        if (consumers_or<kConsumers>(dead) || it.bn == 0) break;
        uint32_t tsize = (3 * it.bn + 3) & ~3u;  // load 1/3 while that fits
        if (tsize < 64) tsize = 64;
        if (tsize > SumTable<KeyT>::kSlots) tsize = SumTable<KeyT>::kSlots;
        tab.clear(tsize);
        consumers_sync<kConsumers>();
        int dup = 0;
        for (uint32_t base = 0; base < it.bn; base += kStageRows) {
            if (!dead && !st.wait(&s_stream.full[sp.i], sp.phase)) dead = true;
            const KeyT* k = st.template rows<KeyT>(sp, 0, reinterpret_cast<const char*>(a.bkey + it.bs0), base);
            const PayT* v = st.template rows<PayT>(sp, 1, reinterpret_cast<const char*>(bpay + it.bs0), base);
            const uint32_t len = dead ? 0u : min(it.bn - base, kStageRows);
            for (uint32_t i = threadIdx.x; i < len; i += kConsumers) {
                const int r = tab.add(k[i], (uint64_t)(int64_t)v[i], tsize);
                if (r < 0) atomicOr(&ctrl->err, kErrTableFull);
                dup |= r;
            }
            st.release(sp);
        }
        const bool unique = !consumers_or<kConsumers>(dup != 0);
        for (uint32_t base = 0; base < it.pn; base += kStageRows) {
            if (!dead && !st.wait(&s_stream.full[sp.i], sp.phase)) dead = true;
            const KeyT* k = st.template rows<KeyT>(sp, 0, reinterpret_cast<const char*>(a.pkey + it.ps0), base);
            const PayT* v = st.template rows<PayT>(sp, 1, reinterpret_cast<const char*>(ppay + it.ps0), base);
            const uint32_t len = dead ? 0u : min(it.pn - base, kStageRows);
#pragma unroll 2
            for (uint32_t i = threadIdx.x; i < len; i += kConsumers) {
                const uint32_t s = tab.find(k[i], tsize);
                if (s == ~0u) continue;
                const uint2 bs = tab.sum[s];
                const uint64_t b = ((uint64_t)bs.y << 32) | bs.x;
                const uint64_t q8 = (uint64_t)(int64_t)v[i];
                const uint32_t rows = unique ? 1u : 1u + tab.more[s];
                agg.sum += b + (unique ? q8 : rows * q8);
                agg.count += rows;
            }
            st.release(sp);
        }
    }
    if (dead && lane_id() == 0) atomicOr(&ctrl->err, kErrInternal);
    agg_commit(agg, ctrl);
}

template <typename KeyT, typename PayT>
cudaError_t launch_sum(const JoinIn<KeyT>& a, const JoinOut& out, Ctrl* ctrl, const DevInfo& di, cudaStream_t stream,
                       int64_t nb, int64_t np) {
    auto kern = phj_sum_kernel<KeyT, PayT>;
    const size_t smem = SumTable<KeyT>::kBytes + SumStream<KeyT, PayT>::kBytes;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kSumThreads, smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    // keys and payloads of both sides, each read once
    ProfScope ps("phj_sum", (double)(sizeof(KeyT) + sizeof(PayT)) * (double)(nb + np), stream);
    kern<<<di.sms * per_sm, kSumThreads, smem, stream>>>(a, static_cast<const PayT*>(out.b.src[0]),
                                                        static_cast<const PayT*>(out.p.src[0]), ctrl);
    return cudaGetLastError();
}

}  // namespace

template <typename KeyT>
cudaError_t phj_sum_launch(const JoinIn<KeyT>& a, const JoinOut& out, Ctrl* ctrl, const DevInfo& di,
                           cudaStream_t stream, int64_t nb, int64_t np) {
    return out.b.bytes[0] == 4 ? launch_sum<KeyT, int32_t>(a, out, ctrl, di, stream, nb, np)
                               : launch_sum<KeyT, int64_t>(a, out, ctrl, di, stream, nb, np);
}

template cudaError_t phj_sum_launch<uint32_t>(const JoinIn<uint32_t>&, const JoinOut&, Ctrl*, const DevInfo&,
                                              cudaStream_t, int64_t, int64_t);
template cudaError_t phj_sum_launch<uint64_t>(const JoinIn<uint64_t>&, const JoinOut&, Ctrl*, const DevInfo&,
                                              cudaStream_t, int64_t, int64_t);

}  // namespace eiger
