// pull.cuh -- Clifford runs as gathers (DevPull) and tile index arithmetic.
#pragma once

#include "device_ops.cuh"
#include "launch.h"

namespace stab {

// A DevPull held by a warp: lane b has column and row b.
struct LanePull {
    uint32_t col, qrow, r0, r1;
};

__device__ __forceinline__ LanePull load_pull(const DevPull *p, int n) {
    const int lane = (int)(threadIdx.x & 31u);
    LanePull L;
    L.col = lane < 2 * n ? p->col[lane] : 0u;
    L.qrow = lane < 2 * n ? p->qrow[lane] : 0u;
    L.r0 = p->r0;
    L.r1 = p->r1;
    return L;
}

// Everything an index i = base ^ off needs of its base (the same in the whole
// warp): j and Q of the base, and in b the bits of off that change Q across.
struct BasePull {
    uint32_t i, j, q, b;
};

__device__ __forceinline__ BasePull base_pull(const LanePull &L, uint32_t base) {
    const bool set = (base >> (threadIdx.x & 31u)) & 1u;
    const uint32_t par = __ballot_sync(0xffffffffu, __popc(L.qrow & base) & 1);
    BasePull B;
    B.i = base;
    B.j = __reduce_xor_sync(0xffffffffu, set ? L.col : 0u);
    B.b = __reduce_xor_sync(0xffffffffu, set ? L.qrow : 0u) ^ par;
    B.q = (uint32_t)__popc(par & base) & 1u;
    return B;
}

// j and Q of a thread's own offset: one bit of it at a time (uniform loop over
// the bits that offsets use).
__device__ __forceinline__ void off_bit(const LanePull &L, int bit, uint32_t off, uint32_t &j,
                                        uint32_t &q) {
    const uint32_t c = __shfl_sync(0xffffffffu, L.col, bit);
    const uint32_t r = __shfl_sync(0xffffffffu, L.qrow, bit);
    if ((off >> bit) & 1u) {
        j ^= c;
        q ^= (uint32_t)__popc(r & off);
    }
}

// Source index and sign of entry base ^ off.
__device__ __forceinline__ uint32_t pull_entry(const LanePull &L, const BasePull &B, int n,
                                               uint32_t off, uint32_t oj, uint32_t oq,
                                               uint32_t &neg) {
    const uint32_t i = B.i ^ off, j = B.j ^ oj, mask = (1u << n) - 1u;
    const uint32_t q = B.q ^ oq ^ (uint32_t)__popc(off & B.b);
    const int e = __popc((i >> n) & i & mask) + __popc(i & L.r0) + 2 * __popc(i & L.r1) +
                  2 * (int)(q & 1u) - __popc((j >> n) & j & mask);
    neg = ((uint32_t)e >> 1) & 1u;
    return j;
}

// A packed integer's bits at their places in the index.
__device__ __forceinline__ uint64_t deposit_runs(uint64_t v, const BitRuns &r) {
    uint64_t out = 0;
    for (int k = 0; k < r.n; ++k)
        out |= ((v >> r.src[k]) & ((1ull << r.len[k]) - 1ull)) << r.dst[k];
    return out;
}

}  // namespace stab
