// Key arrays of hash tables in shared memory (phj_sum.cu, groupby.cu); cas_key
// claims slots in global memory too.
#pragma once

#include "common.cuh"

namespace eiger {

__device__ __forceinline__ uint32_t cas_key(uint32_t* p, uint32_t expect, uint32_t v) {
    return atomicCAS(p, expect, v);
}
__device__ __forceinline__ uint64_t cas_key(uint64_t* p, uint64_t expect, uint64_t v) {
    return atomicCAS(reinterpret_cast<unsigned long long*>(p), (unsigned long long)expect, (unsigned long long)v);
}

// Shared-memory key arrays are probed 16 bytes at a time: a group of four
// 32-bit or two 64-bit keys per load. Home slots are group-aligned and inserts
// fill the groups in order (linear probing), so a key's slot is preceded by no
// empty slot from its home group on. The all-ones pattern marks an empty slot.
template <typename KeyT>
struct KeyGroup;
template <>
struct KeyGroup<uint32_t> {
    static constexpr uint32_t kN = 4;
    uint4 v;
    __device__ __forceinline__ void load(const uint32_t* p) { v = *reinterpret_cast<const uint4*>(p); }
    // index of the first key equal to k, or kN
    __device__ __forceinline__ uint32_t first(uint32_t k) const {
        return v.x == k ? 0u : v.y == k ? 1u : v.z == k ? 2u : v.w == k ? 3u : 4u;
    }
    __device__ __forceinline__ uint32_t first_or_empty(uint32_t k) const {
        return v.x == k || v.x == ~0u ? 0u : v.y == k || v.y == ~0u ? 1u : v.z == k || v.z == ~0u ? 2u
               : v.w == k || v.w == ~0u ? 3u : 4u;
    }
    __device__ __forceinline__ uint32_t last() const { return v.w; }
};
template <>
struct KeyGroup<uint64_t> {
    static constexpr uint32_t kN = 2;
    ulonglong2 v;
    __device__ __forceinline__ void load(const uint64_t* p) { v = *reinterpret_cast<const ulonglong2*>(p); }
    __device__ __forceinline__ uint32_t first(uint64_t k) const { return v.x == k ? 0u : v.y == k ? 1u : 2u; }
    __device__ __forceinline__ uint32_t first_or_empty(uint64_t k) const {
        return v.x == k || v.x == ~0ull ? 0u : v.y == k || v.y == ~0ull ? 1u : 2u;
    }
    __device__ __forceinline__ uint64_t last() const { return v.y; }
};

// Home slot (group-aligned) of hash h in a table of `slots` slots, a multiple
// of the group size.
template <typename KeyT>
__device__ __forceinline__ uint32_t group_home(uint32_t h, uint32_t slots) {
    return KeyGroup<KeyT>::kN * __umulhi(h, slots / KeyGroup<KeyT>::kN);
}
template <typename KeyT>
__device__ __forceinline__ uint32_t next_group(uint32_t s, uint32_t slots) {
    return s + KeyGroup<KeyT>::kN == slots ? 0u : s + KeyGroup<KeyT>::kN;
}

// Slot of k in keys[0, slots), claimed if new (`fresh`), searched from the
// group at `base`; ~0u when the table is full (every group walked once). A lost
// race for a slot reads its group again (at most kN times a group: its slots
// fill up).
template <typename KeyT>
__device__ __forceinline__ uint32_t claim_slot(KeyT* keys, uint32_t slots, KeyT k, uint32_t base, bool& fresh) {
    for (uint32_t left = slots / KeyGroup<KeyT>::kN; left > 0;) {
        KeyGroup<KeyT> g;
        g.load(keys + base);
        const uint32_t i = g.first_or_empty(k);
        if (i == KeyGroup<KeyT>::kN) {
            base = next_group<KeyT>(base, slots);
            --left;
            continue;
        }
        const KeyT cur = cas_key(keys + base + i, ~KeyT(0), k);
        fresh = cur == ~KeyT(0);
        if (fresh || cur == k) return base + i;
    }
    return ~0u;
}

}  // namespace eiger
