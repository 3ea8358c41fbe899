// Column statistics on the GPU: signed min/max and the dense HyperLogLog++
// registers of one key column (Sec. 4 "runtime profiling"; Sec. 4.1 HLL++).
//
// One streaming pass. Each CTA keeps a private copy of the 2^14 registers in
// shared memory (as 32-bit words so it can use the native shared-memory
// atomics), reads its share of the column with 16-byte vector loads, and raises
// a register only when the new rank exceeds it: after the first few thousand
// keys almost every update is a plain shared-memory read. Whether it does is
// decided without counting zeros: a register of rank r is kept as 32 - r, and a
// key's rank exceeds r exactly when the top r of its 50 rank bits are all zero.
// A second, short kernel takes the byte-wise max of the per-CTA register arrays
// with __vmaxu4, reduces min/max and counts the ranks, from which the host makes
// the estimate; a column of one CTA needs no second kernel. The results go
// straight into mapped host memory when the caller has some.
//
// What bounds it: the ALU pipe (shifts, logic, compares and selects, most of them
// the 64-bit hash's), 83 % busy before the range took one compare, at 2 x 1024
// threads per SM. (The hash's shifts as multiplications were slower: 270 -> 310
// us at 2^27 int64 keys.) Measured on GB300: 2^27 int64 keys 286 -> 259 us, 2^28
// int32 keys 521 -> 412 us, merge of all partial arrays 24 -> 10 us; a call on
// 1000 keys 64 -> 16 us (the host counted the 2^14 registers).
#include "kernels.cuh"

namespace eiger {

namespace {

constexpr int kThreads = 1024;
constexpr int kKeysPerThread = 16;  // at least, so that a CTA's 64 KB of registers pay
constexpr int kMergeThreads = 512;
constexpr int kMergeWords = 64;     // register words (of 4) per merging CTA
constexpr int kMergeGrid = kHllM / 4 / kMergeWords;
constexpr int kSlices = kMergeThreads / kMergeWords;

// The range of the keys a thread has seen, starting from some key of the column.
// 32-bit: min and max. 64-bit: min and span, so that one subtraction and one
// unsigned compare find a key outside (compares, selects, shifts and logic share
// the ALU pipe, which bounds this kernel).
template <typename K>
struct Seen;
template <>
struct Seen<int32_t> {
    int32_t mn, mx;
    __device__ explicit Seen(int32_t k) : mn(k), mx(k) {}
    __device__ __forceinline__ void visit(int32_t k) {
        mn = k < mn ? k : mn;
        mx = k > mx ? k : mx;
    }
    __device__ int64_t low() const { return mn; }
    __device__ int64_t high() const { return mx; }
};
template <>
struct Seen<int64_t> {
    int64_t mn;
    uint64_t span;
    __device__ explicit Seen(int64_t k) : mn(k), span(0) {}
    __device__ __forceinline__ void visit(int64_t k) {
        if ((uint64_t)k - (uint64_t)mn > span) {
            if (k < mn) {
                span += (uint64_t)mn - (uint64_t)k;
                mn = k;
            } else {
                span = (uint64_t)k - (uint64_t)mn;
            }
        }
    }
    __device__ int64_t low() const { return mn; }
    __device__ int64_t high() const { return (int64_t)((uint64_t)mn + span); }
};

template <typename K>
__device__ __forceinline__ void sketch_visit(K k, Seen<K>& seen, int* sreg) {
    seen.visit(k);
    const uint64_t h = sketch_hash((uint64_t)(int64_t)k);
    const uint32_t hi = (uint32_t)(h >> 32), lo = (uint32_t)h;
    int* reg = sreg + (hi >> (32 - kHllP));
    const uint32_t w = __funnelshift_l(lo, hi, kHllP);  // the upper 32 of the 50 rank bits
    uint32_t head;  // the top r of them; PTX clamps the shift, so r = 0 and r > 32 give 0
    asm("shr.u32 %0, %1, %2;" : "=r"(head) : "r"(w), "r"((uint32_t)*(volatile int*)reg));
    if (head == 0) {
        const uint64_t rest = h << kHllP;
        const int rho = rest ? __clzll((long long)rest) + 1 : kRhoMax;
        atomicMin(reg, 32 - rho);
    }
}

template <typename K>
struct Vec16;
template <>
struct Vec16<int32_t> {
    using T = int4;
    static constexpr int kN = 4;
    __device__ __forceinline__ static int32_t at(const int4& v, int i) {
        return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
    }
};
template <>
struct Vec16<int64_t> {
    using T = longlong2;
    static constexpr int kN = 2;
    __device__ __forceinline__ static int64_t at(const longlong2& v, int i) {
        return i == 0 ? v.x : v.y;
    }
};

// Block-collective min/max of every thread's (mn, mx), in thread 0.
template <int THREADS>
__device__ __forceinline__ void block_minmax(int64_t& mn, int64_t& mx) {
    __shared__ int64_t s_mn[THREADS / kWarp], s_mx[THREADS / kWarp];
#pragma unroll
    for (int o = kWarp / 2; o > 0; o >>= 1) {
        const int64_t a = __shfl_xor_sync(0xffffffffu, mn, o);
        const int64_t b = __shfl_xor_sync(0xffffffffu, mx, o);
        mn = a < mn ? a : mn;
        mx = b > mx ? b : mx;
    }
    if (lane_id() == 0) {
        s_mn[threadIdx.x / kWarp] = mn;
        s_mx[threadIdx.x / kWarp] = mx;
    }
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < THREADS / kWarp; ++w) {
            mn = s_mn[w] < mn ? s_mn[w] : mn;
            mx = s_mx[w] > mx ? s_mx[w] : mx;
        }
}

__device__ __forceinline__ void count_ranks(uint32_t word, uint32_t* s_hist) {
#pragma unroll
    for (int i = 0; i < 4; ++i) atomicAdd(&s_hist[(word >> (8 * i)) & 63u], 1u);
}

// host: mapped host copy of *out, or nullptr; want_regs: it gets the registers too.
template <typename K>
__global__ void __launch_bounds__(kThreads, 2)
    stats_partial_kernel(const K* __restrict__ keys, int64_t n, uint32_t* __restrict__ part_regs,
                         int64_t* __restrict__ part_mm, StatsDev* __restrict__ out, StatsDev* host, int want_regs) {
    using V = Vec16<K>;
    constexpr int kFlight = 4;  // vectors in flight per thread
    extern __shared__ int sreg[];
    __shared__ uint32_t s_hist[kRankBins];

    for (int i = threadIdx.x; i < kHllM / 4; i += kThreads) reinterpret_cast<int4*>(sreg)[i] = make_int4(32, 32, 32, 32);
    if (threadIdx.x < kRankBins) s_hist[threadIdx.x] = 0;
    if (blockIdx.x == 0 && gridDim.x > 1) {  // for the merge
        if (threadIdx.x < kRankBins) out->hist[threadIdx.x] = 0;
        if (threadIdx.x == 0) out->ticket = 0;
    }
    __syncthreads();

    Seen<K> seen(__ldg(keys));

    // Elements before the first 16-byte boundary, then the aligned body with
    // vector loads (several in flight per thread), then the ragged tail.
    const uintptr_t addr = reinterpret_cast<uintptr_t>(keys);
    int64_t head = (int64_t)(((16u - (addr & 15u)) & 15u) / sizeof(K));
    if (head > n) head = n;
    if (blockIdx.x == 0 && (int64_t)threadIdx.x < head) sketch_visit(keys[threadIdx.x], seen, sreg);

    const int64_t nvec = (n - head) / V::kN;
    const typename V::T* vp = reinterpret_cast<const typename V::T*>(keys + head);
    const int64_t stride = (int64_t)gridDim.x * kThreads;
    int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    for (; i + (kFlight - 1) * stride < nvec; i += kFlight * stride) {
        typename V::T a[kFlight];
#pragma unroll
        for (int f = 0; f < kFlight; ++f) a[f] = __ldcs(vp + i + f * stride);
#pragma unroll
        for (int f = 0; f < kFlight; ++f)
#pragma unroll
            for (int j = 0; j < V::kN; ++j) sketch_visit((K)V::at(a[f], j), seen, sreg);
    }
    for (; i < nvec; i += stride) {
        const typename V::T a = __ldcs(vp + i);
#pragma unroll
        for (int j = 0; j < V::kN; ++j) sketch_visit((K)V::at(a, j), seen, sreg);
    }
    const int64_t tail = head + nvec * V::kN;
    if (blockIdx.x == gridDim.x - 1)
        for (int64_t t = tail + threadIdx.x; t < n; t += kThreads) sketch_visit(keys[t], seen, sreg);

    int64_t mn = seen.low(), mx = seen.high();
    block_minmax<kThreads>(mn, mx);  // (and every register is final)
    const bool last = gridDim.x == 1;
    // Registers as bytes, four per 32-bit word (little-endian register order).
    for (int w = threadIdx.x; w < kHllM / 4; w += kThreads) {
        const int4 r = reinterpret_cast<const int4*>(sreg)[w];
        const uint32_t word = (uint32_t)(32 - r.x) | ((uint32_t)(32 - r.y) << 8) | ((uint32_t)(32 - r.z) << 16) |
                              ((uint32_t)(32 - r.w) << 24);
        if (last) {
            out->regs[w] = word;
            if (host && want_regs) host->regs[w] = word;
            count_ranks(word, s_hist);
        } else {
            part_regs[(size_t)blockIdx.x * (kHllM / 4) + w] = word;
        }
    }
    if (!last) {
        if (threadIdx.x == 0) {
            part_mm[2 * blockIdx.x] = mn;
            part_mm[2 * blockIdx.x + 1] = mx;
        }
        return;
    }
    __syncthreads();
    if (threadIdx.x < kRankBins) {
        out->hist[threadIdx.x] = s_hist[threadIdx.x];
        if (host) host->hist[threadIdx.x] = s_hist[threadIdx.x];
    }
    if (threadIdx.x == 0) {
        out->mn = mn;
        out->mx = mx;
        if (host) {
            host->mn = mn;
            host->mx = mx;
        }
    }
}

// kMergeGrid CTAs, each the maximum of kMergeWords register words over all
// `grid` partial arrays (kSlices threads per word, their loads independent);
// CTA 0 also min/max; the last CTA to finish hands the counts of the ranks out.
__global__ void __launch_bounds__(kMergeThreads)
    stats_merge_kernel(const uint32_t* __restrict__ part_regs, const int64_t* __restrict__ part_mm, int grid,
                       StatsDev* out, StatsDev* host, int want_regs) {
    __shared__ uint32_t s_max[kMergeThreads];
    __shared__ uint32_t s_hist[kRankBins];
    __shared__ bool s_last;
    const int word = threadIdx.x % kMergeWords, slice = threadIdx.x / kMergeWords;
    const uint32_t* p = part_regs + blockIdx.x * kMergeWords + word;
    constexpr size_t W = kHllM / 4;
    uint32_t m = 0;
#pragma unroll 8
    for (int g = slice; g < grid; g += kSlices) m = __vmaxu4(m, p[(size_t)g * W]);
    s_max[threadIdx.x] = m;
    if (threadIdx.x < kRankBins) s_hist[threadIdx.x] = 0;
    __syncthreads();
    if (threadIdx.x < kMergeWords) {
#pragma unroll
        for (int s = 1; s < kSlices; ++s) m = __vmaxu4(m, s_max[s * kMergeWords + threadIdx.x]);
        out->regs[blockIdx.x * kMergeWords + threadIdx.x] = m;
        if (host && want_regs) host->regs[blockIdx.x * kMergeWords + threadIdx.x] = m;
        count_ranks(m, s_hist);
    }
    if (blockIdx.x == 0) {
        int64_t mn = INT64_MAX, mx = INT64_MIN;
        for (int g = threadIdx.x; g < grid; g += kMergeThreads) {
            const int64_t a = part_mm[2 * g], b = part_mm[2 * g + 1];
            mn = a < mn ? a : mn;
            mx = b > mx ? b : mx;
        }
        block_minmax<kMergeThreads>(mn, mx);
        if (threadIdx.x == 0) {
            out->mn = mn;
            out->mx = mx;
            if (host) {
                host->mn = mn;
                host->mx = mx;
            }
        }
    }
    __syncthreads();
    if (threadIdx.x < kRankBins && s_hist[threadIdx.x]) atomicAdd(&out->hist[threadIdx.x], s_hist[threadIdx.x]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&out->ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (s_last && host && threadIdx.x < kRankBins) host->hist[threadIdx.x] = __ldcg(&out->hist[threadIdx.x]);
}

}  // namespace

StatsScratch stats_layout(Carve& c) {
    StatsScratch s;
    s.part_regs = c.take<uint32_t>((size_t)kStatsMaxGrid * (kHllM / 4));
    s.part_mm = c.take<int64_t>(2 * (size_t)kStatsMaxGrid);
    s.out = c.take<StatsDev>(1);
    return s;
}

cudaError_t stats_launch(const void* keys, int64_t n, int dtype, const StatsScratch& s, StatsDev* host, bool want_regs,
                         cudaStream_t stream) {
    DevInfo di;
    cudaError_t e = current_device_info(&di);
    if (e != cudaSuccess) return e;
    const int64_t per_cta = (int64_t)kThreads * kKeysPerThread;
    const int64_t want = (n + per_cta - 1) / per_cta;
    const int cap = di.sms * 2 < kStatsMaxGrid ? di.sms * 2 : kStatsMaxGrid;
    const int grid = (int)(want < 1 ? 1 : want > cap ? cap : want);
    const size_t smem = kHllM * sizeof(uint32_t);
    const double kb = dtype == 0 ? 4.0 : 8.0;
    {
        if ((e = dtype == 0 ? allow_smem(stats_partial_kernel<int32_t>, smem)
                            : allow_smem(stats_partial_kernel<int64_t>, smem)) != cudaSuccess)
            return e;
        ProfScope ps("stats_partial", kb * n, stream);
        if (dtype == 0)
            stats_partial_kernel<int32_t><<<grid, kThreads, smem, stream>>>(
                static_cast<const int32_t*>(keys), n, s.part_regs, s.part_mm, s.out, host, want_regs);
        else
            stats_partial_kernel<int64_t><<<grid, kThreads, smem, stream>>>(
                static_cast<const int64_t*>(keys), n, s.part_regs, s.part_mm, s.out, host, want_regs);
    }
    if ((e = cudaGetLastError()) != cudaSuccess || grid == 1) return e;
    ProfScope ps("stats_merge", (double)grid * (kHllM + 16) + kHllM + 16, stream);
    stats_merge_kernel<<<kMergeGrid, kMergeThreads, 0, stream>>>(s.part_regs, s.part_mm, grid, s.out, host, want_regs);
    return cudaGetLastError();
}

}  // namespace eiger
