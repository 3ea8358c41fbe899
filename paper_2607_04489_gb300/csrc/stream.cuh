// Rows of work items streamed through shared memory, for persistent kernels
// that consume partitioned columns (the partitioned join's fused sum).
//
// Three roles per CTA. A scheduler warp claims items and publishes their
// descriptors in a small queue; a producer warp copies the items' rows, stage
// by stage, with TMA bulk copies into a ring of shared-memory stages; the
// consumer warps take the items from the queue and the rows from the ring. So
// neither the claim and lookup of an item nor the memory latency of its rows
// sits between two items or two stages: the copies run ahead by the depth of
// the ring, whatever phase the consumers are in.
//
// A stage holds up to kStageRows rows of NC columns. Column pieces start
// anywhere, bulk copies on 16-byte boundaries: each copy takes the aligned
// cover of the piece (the columns are workspace buffers with 16 bytes of slack
// behind them), and the rows then begin `address & 15` bytes into it.
//
// Every wait is bounded: when one runs out, the CTA's abort flag goes up, all
// other waits return at once, and the consumers leave together at the end of
// their item (consumers_stop).
#pragma once

#include "common.cuh"

namespace eiger {

constexpr int kStreamWarps = 2;  // scheduler and producer, behind the consumer warps

// Columns of one row source, widths W bytes each.
template <int NC>
struct RowCols {
    const char* p[NC];
};

template <int NC, int STAGES, int QUEUE, uint32_t ROWS, typename Item>
struct Stream {
    static constexpr uint32_t kRows = ROWS;

    struct Shared {
        uint64_t full[STAGES], empty[STAGES];
        uint64_t ifull[QUEUE], iempty[QUEUE];
        Item item[QUEUE];
        int abort;
    };
    // Bytes of a stage for the given column widths.
    __host__ __device__ static constexpr uint32_t col_bytes(uint32_t w) { return ROWS * w + 16; }

    Shared* sh;
    unsigned char* buf;   // STAGES stages
    uint32_t w[NC];       // column widths
    uint32_t off[NC];     // column offsets in a stage
    uint32_t stage_bytes;

    __device__ void setup(Shared* s, unsigned char* b, int consumer_warps) {
        sh = s;
        buf = b;
        uint32_t o = 0;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            off[c] = o;
            o += col_bytes(w[c]);
        }
        stage_bytes = o;
        if (threadIdx.x == 0) {
            for (int i = 0; i < STAGES; ++i) {
                mbar_init(&s->full[i], 1);
                mbar_init(&s->empty[i], consumer_warps);
            }
            for (int i = 0; i < QUEUE; ++i) {
                mbar_init(&s->ifull[i], 1);
                mbar_init(&s->iempty[i], consumer_warps + 1);
            }
            s->abort = 0;
            fence_mbar_init();
        }
        __syncthreads();
    }

    // False when the wait ran out or another one did.
    __device__ bool wait(uint64_t* bar, uint32_t parity) const {
        for (uint32_t i = 0; i < kSpinLimit; ++i) {
            if (mbar_try_wait(bar, parity)) return true;
            if ((i & 63) == 63 && *(volatile int*)&sh->abort) return false;
        }
        *(volatile int*)&sh->abort = 1;
        return false;
    }

    // Position in a ring of N slots.
    template <int N>
    struct Pos {
        uint32_t i = 0, phase = 0;
        __device__ void next() {
            if (++i == N) {
                i = 0;
                phase ^= 1;
            }
        }
    };
    using StagePos = Pos<STAGES>;
    using ItemPos = Pos<QUEUE>;

    // Scheduler, lane 0: publishes an item once its queue slot is free.
    __device__ bool publish(ItemPos& q, const Item& it) const {
        if (!wait(&sh->iempty[q.i], q.phase ^ 1)) return false;
        sh->item[q.i] = it;
        mbar_arrive(&sh->ifull[q.i]);
        q.next();
        return true;
    }

    // Producer, one lane: streams rows [0, n) of the columns at `src`.
    __device__ bool produce(StagePos& st, const RowCols<NC>& src, uint32_t n) const {
        for (uint32_t r = 0; r < n; r += ROWS) {
            const uint32_t len = n - r < ROWS ? n - r : ROWS;
            if (!wait(&sh->empty[st.i], st.phase ^ 1)) return false;
            uintptr_t lo[NC];
            uint32_t bytes[NC], total = 0;
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const uintptr_t a = reinterpret_cast<uintptr_t>(src.p[c]) + (size_t)r * w[c];
                lo[c] = a & ~(uintptr_t)15;
                bytes[c] = (uint32_t)(((a + (size_t)len * w[c] + 15) & ~(uintptr_t)15) - lo[c]);
                total += bytes[c];
            }
            fence_proxy_async_smem();
            mbar_arrive_expect_tx(&sh->full[st.i], total);
#pragma unroll
            for (int c = 0; c < NC; ++c)
                bulk_load(buf + st.i * stage_bytes + off[c], reinterpret_cast<const void*>(lo[c]), bytes[c],
                          &sh->full[st.i]);
            st.next();
        }
        return true;
    }
    // Producer, at the end: no copy may land after the CTA exits.
    __device__ void drain(StagePos st) const {
        for (int i = 0; i < STAGES; ++i) {  // the oldest stage in flight is the next to be refilled
            for (uint32_t k = 0; k < kSpinLimit; ++k)
                if (mbar_try_wait(&sh->full[st.i], st.phase ^ 1)) break;
            st.next();
        }
    }

    // Consumer: column c of the stage, first row at `src_addr` in memory.
    template <typename T>
    __device__ const T* rows(const StagePos& st, int c, const char* src, uint32_t r) const {
        const uint32_t lead = (uint32_t)(reinterpret_cast<uintptr_t>(src) + (size_t)r * sizeof(T)) & 15u;
        return reinterpret_cast<const T*>(buf + st.i * stage_bytes + off[c] + lead);
    }
    // Consumer warp: the stage has been read.
    __device__ void release(StagePos& st) const {
        __syncwarp();
        if (lane_id() == 0) mbar_arrive(&sh->empty[st.i]);
        st.next();
    }
};

// Barriers of the consumer warps alone (barrier 1; barrier 0 is __syncthreads).
template <int THREADS>
__device__ __forceinline__ void consumers_sync() {
    asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
}
template <int THREADS>
__device__ __forceinline__ bool consumers_or(bool v) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.or.pred q, 1, %2, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)v), "n"(THREADS)
        : "memory");
    return r != 0;
}

// Every consumer together, between two items: whether to leave, after the `last`
// item or because some thread's wait ran out (lanes of a warp may differ), which
// raises kErrInternal in *err.
template <int THREADS>
__device__ __forceinline__ bool consumers_stop(bool dead, bool last, unsigned* err) {
    const bool failed = consumers_or<THREADS>(dead);
    if (failed && threadIdx.x == 0) atomicOr(err, kErrInternal);
    return failed || last;
}

}  // namespace eiger
