// Delivery of kept (coordinate, value) pairs to the server: shared by the Top-k and the Random-k kernels.
#pragma once

#include "context.h"

namespace compams {

// A kept (coordinate, value) pair reaches the server: it joins the bucket of its coordinate range at position
// `pos` or, when the bucket is full, the binary64 accumulator.
__device__ __forceinline__ void deliver_pair(const TopkBuffers& b, uint32_t T, uint32_t pos, int32_t j, uint32_t xbits) {
    if (pos < (uint32_t)b.bucket_cap) {
        b.bucket[(size_t)T * (size_t)b.bucket_cap + pos] = make_uint2((uint32_t)j % (uint32_t)kBucketSpan, xbits);
    } else {  // a coordinate range kept by far more entries than average: binary64 atomics instead
        atomicAdd(b.acc + j, (double)__uint_as_float(xbits));
        b.bdirty[T] = 1u;
    }
}

// One pair by one thread.
__device__ __forceinline__ void scatter_one(const TopkBuffers& b, int32_t j, uint32_t xbits) {
    const uint32_t T = (uint32_t)j / (uint32_t)kBucketSpan;
    deliver_pair(b, T, atomicAdd(b.bcount + T, 1u), j, xbits);
}

// One pair per thread in any order, the whole warp together: the lanes whose pairs fall into the same bucket get their
// slots with one atomic.
__device__ __forceinline__ void scatter_warp(const TopkBuffers& b, bool valid, int32_t j, uint32_t xbits) {
    const uint32_t T = valid ? (uint32_t)j / (uint32_t)kBucketSpan : 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned peers = __match_any_sync(0xffffffffu, T);
    uint32_t base = 0;
    const int leader = __ffs(peers) - 1;
    if (valid && lane == leader) base = atomicAdd(b.bcount + T, (uint32_t)__popc(peers));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (!valid) return;
    deliver_pair(b, T, base + (uint32_t)__popc(peers & ((1u << lane) - 1u)), j, xbits);
}

// U entries (coordinate, bits) per thread, the whole warp together, of which the `take`n ones are delivered (`wins`: their
// ballots): neighbouring lanes whose entries fall into the same bucket (taken or not) get their slots with one atomic, and all U
// rounds of atomics are in flight between ask() and put(). The lists that Top-k emits from are grouped by coordinate
// range, so the runs are long; entries in random order cost one atomic each. (Finding all equal buckets of the warp
// with __match_any_sync instead took most of the emission's instructions.)
template <int U>
struct RunSlots {
    uint32_t base[U], head[U], rank[U];
    __device__ __forceinline__ void ask(const TopkBuffers& b, const unsigned (&wins)[U], const uint2 (&cv)[U]) {
        const int lane = threadIdx.x & 31;
        const unsigned below = (1u << lane) - 1u, upto = below | (1u << lane);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t T = cv[u].x / (uint32_t)kBucketSpan;
            const uint32_t left = __shfl_up_sync(0xffffffffu, T, 1);
            const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || left != T);
            head[u] = 31u - (uint32_t)__clz(heads & upto);  // first lane of this lane's run
            const unsigned later = heads & ~upto;           // heads of the runs after it
            const unsigned run = (later ? (later & (0u - later)) - 1u : 0xffffffffu) & ~((1u << head[u]) - 1u);
            rank[u] = (uint32_t)__popc(wins[u] & run & below);
            base[u] = 0;
            if (head[u] == (uint32_t)lane && (wins[u] & run)) base[u] = atomicAdd(b.bcount + T, (uint32_t)__popc(wins[u] & run));
        }
    }
    __device__ __forceinline__ void put(const TopkBuffers& b, const unsigned (&wins)[U], const uint2 (&cv)[U]) const {
        const int lane = threadIdx.x & 31;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t first = __shfl_sync(0xffffffffu, base[u], head[u]);
            if ((wins[u] >> lane) & 1u) deliver_pair(b, cv[u].x / (uint32_t)kBucketSpan, first + rank[u], (int32_t)cv[u].x, cv[u].y);
        }
    }
};
template <int U>
__device__ __forceinline__ void scatter_runs(const TopkBuffers& b, const unsigned (&wins)[U], const uint2 (&cv)[U]) {
    RunSlots<U> slots;
    slots.ask(b, wins, cv);
    slots.put(b, wins, cv);
}

}  // namespace compams
