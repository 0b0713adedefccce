// Random-k path of the COMP-AMS step: every (worker, block) keeps k_b coordinates drawn uniformly at random,
// whatever their values (Section 2.1 lists Random-k beside Top-k among the deterministic sparsifiers; with
// error feedback the dropped coordinates wait in e until they are drawn).
//
// The kept set of (step t, worker i, block b) is { pi(r) : r = 0 .. k_b - 1 }, pi a keyed pseudorandom
// permutation of the block's coordinates: a balanced Feistel network of six rounds over the smallest even
// number of bits that covers d_b, with cycle walking back into [0, d_b). The six 32-bit round keys are the
// halves of the first three words of one Philox4x64-10 block (Salmon, Moraes, Dror, Shaw, SC 2011) at counter
// (0, 0, b, i) under key (seed, t); the round function is the 32-bit finalizer of MurmurHash3 applied to
// (right half xor round key). Being the image of k_b distinct inputs under a bijection, the set has exactly k_b
// members and needs no selection. Two kernels per group of workers: randk_mark, one to eight message slots per thread, computes
// each slot's coordinate and sets its bit in a map of the group's elements; randk_sweep forms x = g + e, and where the bit is
// set x goes to the message and to the server and 0 to E (the residual of a kept coordinate), x to E elsewhere.
//
// The map is what makes the drawn coordinates meet their x in index order: it is small enough for the L2 (64 MB: hence the
// groups), where setting a bit costs a fraction of a visit to DRAM. (A sweep that left x in E, and one atomic exchange per
// slot that fetched it from there and zeroed it, was bound by the rate of scattered accesses, 16 to 18 G per second: step on
// ResNet-18 shapes, n = 16, 1 % 486 -> 429 us, n = 8, d = 2^26, 10 % 4086 -> 2397.)
#include "context.h"
#include "scatter.cuh"

namespace compams {

struct RoundKeys {
    uint32_t k[6];
};

__device__ __forceinline__ RoundKeys randk_round_keys(uint64_t seed, uint64_t step, uint64_t worker, uint64_t block) {
    const uint64_t M0 = 0xD2E7470EE14C6C93ull, M1 = 0xCA5A826395121157ull;
    const uint64_t W0 = 0x9E3779B97F4A7C15ull, W1 = 0xBB67AE8584CAA73Bull;
    uint64_t c0 = 0, c1 = 0, c2 = block, c3 = worker, k0 = seed, k1 = step;
#pragma unroll 1
    for (int round = 0; round < 10; ++round) {
        if (round > 0) {
            k0 += W0;
            k1 += W1;
        }
        const uint64_t hi0 = __umul64hi(M0, c0), lo0 = M0 * c0;
        const uint64_t hi1 = __umul64hi(M1, c2), lo1 = M1 * c2;
        const uint64_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
        c0 = n0;
        c1 = lo1;
        c2 = n2;
        c3 = lo0;
    }
    RoundKeys out;
    out.k[0] = (uint32_t)c0;
    out.k[1] = (uint32_t)(c0 >> 32);
    out.k[2] = (uint32_t)c1;
    out.k[3] = (uint32_t)(c1 >> 32);
    out.k[4] = (uint32_t)c2;
    out.k[5] = (uint32_t)(c2 >> 32);
    return out;
}

__device__ __forceinline__ uint32_t fmix32(uint32_t h) {
    h ^= h >> 16;
    h *= 0x85ebca6bu;
    h ^= h >> 13;
    h *= 0xc2b2ae35u;
    h ^= h >> 16;
    return h;
}

// One application of the network to x, whose domain has 2 w bits.
__device__ __forceinline__ uint32_t randk_network(uint32_t x, int w, const uint32_t (&k)[6]) {
    const uint32_t mask = (1u << w) - 1u;
    uint32_t L = x >> w, R = x & mask;
#pragma unroll
    for (int round = 0; round < 6; ++round) {
        const uint32_t nR = L ^ (fmix32(R ^ k[round]) & mask);
        L = R;
        R = nR;
    }
    return (L << w) | R;
}
__device__ __forceinline__ int randk_half_bits(uint32_t m) {
    int bits = 2;
    while (bits < 32 && (1u << bits) < m) bits += 2;
    return bits >> 1;
}

// The block of a message slot from the slot offsets, by a whole warp (all lanes with the same slot): 32 offsets at a time.
__device__ __forceinline__ int block_of_slot(const Tables& t, const TopkBuffers& b, int64_t q) {
    int lo = 0, count = t.M;  // it is one of the `count` blocks from lo on
    while (count > 1) {
        const int stride = (count + 31) >> 5, at = (threadIdx.x & 31) * stride;
        const int skip = (__popc(__ballot_sync(0xffffffffu, at < count && __ldg(b.seg_off + lo + at) <= q)) - 1) * stride;
        lo += skip;
        count = count - skip < stride ? count - skip : stride;
    }
    return lo;
}

// The block of a slot at or behind the first slot of block `from`, as a rule not far behind: doubling steps, then bisection.
__device__ __forceinline__ int block_of_later_slot(const Tables& t, const TopkBuffers& b, int64_t q, int from) {
    int lo = from, up = 1;
    for (; from + up < t.M && __ldg(b.seg_off + from + up) <= q; up *= 2) lo = from + up;
    int hi = from + up < t.M ? from + up - 1 : t.M - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(b.seg_off + mid) <= q) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Sets the bits of the drawn coordinates. Bit f - origin of the map stands for element f of the flat [n, d] buffers; origin is a
// multiple of 32, so that the map's words are the 128-byte lines of E. A CTA covers `per_thread` x kThreads consecutive message slots
// of one worker; every thread computes the coordinates of its slots. Bound by the instructions of the network (a warp issues in two
// cycles of three): a lane that is back inside the block goes on to its next slot while its neighbours still walk, so that a warp
// waits for the longest sum of walks and not, slot for slot, for the longest walk, and the round keys serve that many more slots
// (one slot per thread took 37 us for 1.8 M slots in blocks of 11.2 M coordinates, two thirds of the domain, this takes 25:
// ResNet-18 shapes, n = 16, 430 -> 418 us per step). With one slot per thread there is nothing to go on to, and the bit is set behind
// the walk (inside it n = 2, d = 300,001, 5 % took 18.9 us per step, now 18.0; n = 16, 1 % 27.4 / 26.4).
__global__ void __launch_bounds__(kThreads) randk_mark_kernel(const __grid_constant__ Tables t, const __grid_constant__ TopkBuffers b,
                                                              int32_t row0, int32_t i0, int64_t origin, uint64_t seed, uint64_t step,
                                                              int per_thread) {
    __shared__ uint32_t keys[kThreads][6];
    const int64_t span = (int64_t)per_thread * kThreads;
    const uint32_t per_worker = (uint32_t)((b.K + span - 1) / span);
    const int tid = threadIdx.x;
    const int il = (int)(blockIdx.x / per_worker);
    const int64_t first = (int64_t)(blockIdx.x % per_worker) * span, last = first + span < b.K ? first + span : b.K;
    const uint64_t worker = (uint64_t)(row0 + i0 + il);
    const int64_t row = (int64_t)(i0 + il) * t.d - origin;
    auto mark = [&](int64_t j) {
        const int64_t f = row + j;
        atomicOr(b.map + (f >> 5), 1u << (f & 31));
    };
    // (bisected by every thread, here and again for its own slot, a CTA over several blocks was slower than one that only does the
    // second: 120 blocks, n = 8, d = 500,000, 3 % 37.0 us per step, then 37.4, now 36.1)
    const int blk0 = block_of_slot(t, b, first);
    if (__ldg(b.seg_off + blk0 + 1) >= last) {  // one block
        if (tid == 0) {
            const RoundKeys rk = randk_round_keys(seed, step, worker, (uint64_t)blk0);
#pragma unroll
            for (int i = 0; i < 6; ++i) keys[0][i] = rk.k[i];
        }
        const int64_t o = __ldg(t.off + blk0);
        const uint32_t len = (uint32_t)(__ldg(t.off + blk0 + 1) - o);
        const int w = randk_half_bits(len);
        const int64_t slot0 = __ldg(b.seg_off + blk0);
        __syncthreads();
        uint32_t k[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) k[i] = keys[0][i];
        dependency_wait();
        allow_dependents();
        if (tid == 0 && first == slot0) b.slots[(size_t)(i0 + il) * t.nseg + blk0] = 0u;  // every block is tiled: segment = block
        int64_t q = first + tid;
        uint32_t x = (uint32_t)(q - slot0);
        if (per_thread == 1) {  // nothing to go on to
            if (q >= last) return;
            do x = randk_network(x, w, k);
            while (x >= len);
            mark(o + x);
            return;
        }
        while (q < last) {
            x = randk_network(x, w, k);
            if (x < len) {
                mark(o + x);
                q += kThreads;
                x = (uint32_t)(q - slot0);
            }
        }
        return;
    }
    dependency_wait();
    allow_dependents();
    // several blocks: the slots of one block are consecutive, so the thread holding a block's first slot (or thread 0, for a
    // block begun before) derives the round keys once and the others read them from shared memory
    for (int64_t q0 = first; q0 < last; q0 += kThreads) {
        const int64_t q = q0 + tid;
        const bool valid = q < last;
        int64_t o = 0;
        uint32_t len = 1, r = 0;
        if (valid) {
            const int blk = block_of_later_slot(t, b, q, blk0);
            o = __ldg(t.off + blk);
            len = (uint32_t)(__ldg(t.off + blk + 1) - o);
            r = (uint32_t)(q - __ldg(b.seg_off + blk));
            if (tid == 0 || r == 0) {
                const RoundKeys rk = randk_round_keys(seed, step, worker, (uint64_t)blk);
#pragma unroll
                for (int i = 0; i < 6; ++i) keys[tid][i] = rk.k[i];
            }
            if (r == 0) b.slots[(size_t)(i0 + il) * t.nseg + blk] = 0u;
        }
        __syncthreads();
        if (valid) {
            const uint32_t* mine = keys[r < (uint32_t)tid ? tid - (int)r : 0];
            const int w = randk_half_bits(len);
            uint32_t k[6];
#pragma unroll
            for (int i = 0; i < 6; ++i) k[i] = mine[i];
            uint32_t x = r;
            do x = randk_network(x, w, k);
            while (x >= len);  // at most a few rounds on average: the domain is less than four times the block
            mark(o + x);
        }
        __syncthreads();  // the keys have been read
    }
}

// A warp's drawn coordinates while it streams: lane l's word of the map for the warp's l-th 32 coordinates, the number of
// drawn ones before it, and room for their x in index order.
// (kRoom of them: the loads in flight need the rest of the SM's memory, 4 KB per warp slowed the kernel by a quarter; an x
// that finds no room stays in E and is fetched from there).
template <int kRoom>
struct Drawing {
    uint32_t word, before;
    float* x;
};
// Element `bit` of the 32 that `word` and `before` describe: a drawn one leaves its x, and its residual is 0.
template <int kRoom>
__device__ __forceinline__ float take_drawn(const Drawing<kRoom>& dr, uint32_t word, uint32_t before, int bit, float x) {
    if (!((word >> bit) & 1u)) return x;
    const uint32_t p = before + (uint32_t)__popc(word & ((1u << bit) - 1u));
    if (p >= (uint32_t)kRoom) return x;
    dr.x[p] = x;
    return 0.0f;  // Algorithm 2, the residual update: e = x - x
}

// One warp's 1024 consecutive coordinates from rw on (relative to the block; at a block's ends some lie outside it): the
// residual of x = g + e written over E. The next iteration's loads are in flight while one is worked on.
template <bool FULL, typename GT, int kRoom>
__device__ __forceinline__ void randk_sweep_span(const GT* __restrict__ g, float* __restrict__ e, int len, int rw, int lane,
                                                 const Drawing<kRoom>& dr) {
    const int cg = align_class(g + rw), ce = align_class(e + rw);
    float4 gv[2], ev[2];
    auto load = [&](int it) {
        const int r = rw + it * 128 + lane * 4;
        if (FULL || (r >= 0 && r + 3 < len)) {
            gv[it & 1] = load4_stream(g + r, cg);
            ev[it & 1] = load4(e + r, ce);
        } else {
            float gt[4], et[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const bool live = (unsigned)(r + k) < (unsigned)len;
                gt[k] = live ? load1_stream(g + r + k) : 0.0f;
                et[k] = live ? e[r + k] : 0.0f;
            }
            gv[it & 1] = make_float4(gt[0], gt[1], gt[2], gt[3]);
            ev[it & 1] = make_float4(et[0], et[1], et[2], et[3]);
        }
    };
    load(0);
#pragma unroll
    for (int it = 0; it < kIters; ++it) {
        if (it + 1 < kIters) load(it + 1);
        const int r = rw + it * 128 + lane * 4, src = it * 4 + (lane >> 3), bit = (lane & 7) * 4;
        const uint32_t word = __shfl_sync(0xffffffffu, dr.word, src), before = __shfl_sync(0xffffffffu, dr.before, src);
        const float4 a = gv[it & 1], b = ev[it & 1];
        // the corrected-gradient step of Algorithm 2
        float4 x = make_float4(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y), __fadd_rn(a.z, b.z), __fadd_rn(a.w, b.w));
        if ((word >> bit) & 15u) {
            x.x = take_drawn(dr, word, before, bit, x.x);
            x.y = take_drawn(dr, word, before, bit + 1, x.y);
            x.z = take_drawn(dr, word, before, bit + 2, x.z);
            x.w = take_drawn(dr, word, before, bit + 3, x.w);
        }
        if (FULL || (r >= 0 && r + 3 < len)) {
            store4(e + r, ce, x);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if ((unsigned)(r + k) < (unsigned)len) e[r + k] = lane_elem(x, k);
        }
    }
}

// The same for bfloat16 gradients where whole spans start on 16-byte boundaries of G and E: 8 coordinates per lane and
// iteration, so that the gradient load is 128 bits wide too.
template <int kRoom>
__device__ __forceinline__ void randk_sweep_span_bf16x8(const bf16_bits* __restrict__ g, float* __restrict__ e, int rw, int lane,
                                                        const Drawing<kRoom>& dr) {
    constexpr int NC = kWarpSpan / 256;
    uint4 gv[2];
    float4 ev[2][2];
    auto load = [&](int c) {
        const int r = rw + c * 256 + lane * 8;
        gv[c & 1] = __ldg(reinterpret_cast<const uint4*>(g + r));
        ev[c & 1][0] = *reinterpret_cast<const float4*>(e + r);
        ev[c & 1][1] = *reinterpret_cast<const float4*>(e + r + 4);
    };
    load(0);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        if (c + 1 < NC) load(c + 1);
        const int r = rw + c * 256 + lane * 8, src = c * 8 + (lane >> 2), bit = (lane & 3) * 8;
        const uint32_t word = __shfl_sync(0xffffffffu, dr.word, src), before = __shfl_sync(0xffffffffu, dr.before, src);
        const uint32_t w[4] = {gv[c & 1].x, gv[c & 1].y, gv[c & 1].z, gv[c & 1].w};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float4 b = ev[c & 1][h];
            float4 x = make_float4(__fadd_rn(__uint_as_float(w[2 * h] << 16), b.x), __fadd_rn(__uint_as_float(w[2 * h] & 0xffff0000u), b.y),
                                   __fadd_rn(__uint_as_float(w[2 * h + 1] << 16), b.z),
                                   __fadd_rn(__uint_as_float(w[2 * h + 1] & 0xffff0000u), b.w));
            if ((word >> (bit + 4 * h)) & 15u) {
                x.x = take_drawn(dr, word, before, bit + 4 * h, x.x);
                x.y = take_drawn(dr, word, before, bit + 4 * h + 1, x.y);
                x.z = take_drawn(dr, word, before, bit + 4 * h + 2, x.z);
                x.w = take_drawn(dr, word, before, bit + 4 * h + 3, x.w);
            }
            *reinterpret_cast<float4*>(e + r + h * 4) = x;
        }
    }
}

// Sum of x over the lanes below this one; *total: over all lanes.
__device__ __forceinline__ uint32_t warp_exclusive_sum(uint32_t x, int lane, uint32_t* total) {
    uint32_t s = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += y;
    }
    *total = __shfl_sync(0xffffffffu, s, 31);
    return s - x;
}

// Grid: tiles x workers of the group. Tiles are shifted to 128-byte lines of G and E as in the Top-k sweep. A warp knows
// from the map how many of its 1024 coordinates are drawn, and asks for their message and bucket slots before it starts on
// g and e; their x wait in shared memory until they do, and every lane then delivers the drawn ones of its 32. The span's
// lines are asked into the L2 before the map is looked at, which lets four CTAs per SM (64 registers) do better than six
// (ResNet-18 shapes 415 us, five 425, six 452; without the prefetch and six 460).
// Drawn coordinates of a warp's 1024 from which on they are taken word by word (a lane per coordinate: stores of neighbours, 32
// rounds however few there are) and not lane by lane (as many rounds as the fullest word has): us per step, lane by lane / word by
// word, n = 4, d = 9 M: 16 % drawn 318 / 321, 20 % 378 / 361, 50 % 986 / 766; n = 16, d = 524,288: 16 % 78 / 79, 50 % 244 / 190.
constexpr uint32_t kByWord = 192;

template <typename GT, int kRoom>
__global__ void __launch_bounds__(kThreads, 4) randk_sweep_kernel(
    const __grid_constant__ Tables t, const __grid_constant__ TopkBuffers b, const GT* __restrict__ G, int32_t i0, int64_t origin,
    int64_t words, int deliver, const __grid_constant__ SegParams sp_) {
    __shared__ float sh_x[kWarps][kRoom];
    __shared__ uint32_t sh_count[kWarps], sh_base;
    dependency_wait();
    allow_dependents();
    const TileInfo ti = sp_.nseg ? find_tile(sp_, blockIdx.x) : load_tile(t.tiles, blockIdx.x);
    const int i = i0 + (int)blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t row0 = (int64_t)i * t.d + ti.o;
    const int rw = ti.r0 - (int)(row0 & 31) + warp * kWarpSpan;
    const GT* g = G + row0;
    float* e = b.E + row0;
    const bool whole = rw >= 0 && rw + kWarpSpan <= ti.len;
    if (whole) {  // on their way to the L2 while the map is looked at: one line of E per lane, one of g for as many
        asm volatile("prefetch.global.L2 [%0];" ::"l"(e + rw + lane * 32));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(g + rw + lane * 32));
    }
    // lane l: the map's word of the warp's l-th 32 coordinates, of which `own` are the block's; the word goes back to 0
    const int64_t q = ((row0 + rw - origin) >> 5) + lane;
    const int w0 = rw + lane * 32;
    uint32_t own = 0xffffffffu;
    if (w0 < 0) own = w0 > -32 ? 0xffffffffu << -w0 : 0u;
    if (w0 + 32 > ti.len) own &= w0 < ti.len ? 0xffffffffu >> (w0 + 32 - ti.len) : 0u;
    uint32_t drawn = own && q < words ? b.map[q] & own : 0u;
    if (drawn) {
        if (own == 0xffffffffu) b.map[q] = 0u;
        else atomicAnd(b.map + q, ~own);  // shared with the neighbouring block or row
    }
    // the coordinates meet at most two server buckets: T and, from `edge` on, the next
    const int64_t j0 = ti.o + (rw < 0 ? 0 : rw);
    const uint32_t T = (uint32_t)(j0 / kBucketSpan);
    const int64_t edge = (int64_t)(T + 1) * kBucketSpan - (ti.o + w0);  // bits of this lane's word from here on are in the next
    const uint32_t late = edge <= 0 ? drawn : edge < 32 ? drawn & (0xffffffffu << (int)edge) : 0u;
    // counts of at most 1024 each: both sums in one word
    uint32_t sums;
    uint32_t rank = warp_exclusive_sum((uint32_t)__popc(drawn) | (uint32_t)__popc(late) << 16, lane, &sums);
    const uint32_t rank_late = rank >> 16, total = sums & 0xffffu, total_late = sums >> 16;
    rank &= 0xffffu;
    uint32_t base = 0;
    if (lane == 1 && deliver && total - total_late) base = atomicAdd(b.bcount + T, total - total_late);
    if (lane == 2 && deliver && total_late) base = atomicAdd(b.bcount + T + 1, total_late);
    // the segment's counter is one word for all of a worker's warps: one atomic per CTA (one per warp made the step twice as long)
    if (lane == 0) sh_count[warp] = total;
    __syncthreads();
    uint32_t pos = rank;
    {
        uint32_t of_cta = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            if (w < warp) pos += sh_count[w];
            of_cta += sh_count[w];
        }
        if (threadIdx.x == 0 && of_cta) sh_base = atomicAdd(b.slots + (size_t)i * t.nseg + ti.seg, of_cta);
    }

    bool wide = false;
    if constexpr (sizeof(GT) == 2)
        wide = whole && ((reinterpret_cast<uintptr_t>(g + rw) | reinterpret_cast<uintptr_t>(e + rw)) & 15u) == 0;
    const Drawing<kRoom> dr{drawn, rank, sh_x[warp]};
    if (wide) {
        if constexpr (sizeof(GT) == 2) randk_sweep_span_bf16x8(g, e, rw, lane, dr);
    } else if (whole) {
        randk_sweep_span<true>(g, e, ti.len, rw, lane, dr);
    } else if (rw < ti.len) {
        randk_sweep_span<false>(g, e, ti.len, rw, lane, dr);
    }

    uint32_t early = __shfl_sync(0xffffffffu, base, 1) + rank - rank_late, next = __shfl_sync(0xffffffffu, base, 2) + rank_late;
    __syncthreads();  // the drawn x and the CTA's first slot are there
    pos += sh_base;
    const SegInfo* si = t.segs + ti.seg;
    const size_t slot0 = (size_t)i * (size_t)b.K + (size_t)si->slot0;
    const uint32_t kb = si->kb;
    if (total > kByWord) {  // the entries of T come before those of the next bucket
        const uint32_t pos0 = pos - rank, in_T = total - total_late;
        const uint32_t b0 = __shfl_sync(0xffffffffu, base, 1), b1 = __shfl_sync(0xffffffffu, base, 2) - in_T;
        for (int u = 0; u < 32; ++u) {
            const uint32_t word = __shfl_sync(0xffffffffu, drawn, u);
            const uint32_t p = __shfl_sync(0xffffffffu, rank, u) + (uint32_t)__popc(word & ((1u << lane) - 1u));
            if (!((word >> lane) & 1u)) continue;
            float* ex = e + rw + u * 32 + lane;
            float x;
            if (p < (uint32_t)kRoom) {
                x = sh_x[warp][p];
            } else {
                x = *ex;
                *ex = 0.0f;
            }
            const int32_t j = (int32_t)(ti.o + rw + u * 32 + lane);
            if (pos0 + p < kb) {
                b.idx[slot0 + pos0 + p] = j;
                b.val[slot0 + pos0 + p] = x;
            } else {
                atomicOr(b.status, 1u);
            }
            if (deliver) deliver_pair(b, p < in_T ? T : T + 1u, (p < in_T ? b0 : b1) + p, j, __float_as_uint(x));
        }
        return;
    }
    while (drawn) {
        const int k = __ffs(drawn) - 1;
        drawn &= drawn - 1;
        const int32_t j = (int32_t)(ti.o + w0 + k);
        const float x = rank < (uint32_t)kRoom ? sh_x[warp][rank] : atomicExch(e + w0 + k, 0.0f);
        ++rank;
        if (pos < kb) {
            b.idx[slot0 + pos] = j;
            b.val[slot0 + pos] = x;
        } else {
            atomicOr(b.status, 1u);
        }
        ++pos;
        if (deliver) {
            const bool l = (late >> k) & 1u;
            deliver_pair(b, T + (l ? 1u : 0u), l ? next : early, j, __float_as_uint(x));
            if (l) ++next;
            else ++early;
        }
    }
}

template <typename GT>
static cudaError_t launch_randk_typed(compams_context* c, const GT* grads) {
    TopkBuffers b = c->tk;  // the kernels see this handle's own rows of the message buffers
    b.idx += (size_t)c->row0 * (size_t)c->K;
    b.val += (size_t)c->row0 * (size_t)c->K;
    cudaError_t e = cudaSuccess;
    for (int32_t i0 = 0; i0 < c->n && e == cudaSuccess; i0 += c->randk_group) {
        const int32_t rows = c->n - i0 < c->randk_group ? c->n - i0 : c->randk_group;
        const int64_t origin = (int64_t)i0 * c->d & ~(int64_t)31;
        // as many slots per thread as leave eight CTAs per SM, an SM full of them, eight at most. us per step with one slot, as many as
        // leave two CTAs, four, eight: n = 8, d = 3 M in 20 blocks, 1 % 81.1, 85.3, 81.0, 81.0; n = 2, d = 2 M in 60, 5 % 38.4, 40.8, 38.3, 38.3;
        // n = 16, d = 6 M in 150, 1 % 261, 273, 267, 262; n = 4, d = 9 M in 100, 5 % 198, 193, 193, 186; ResNet-18 shapes whole, n = 16 431, 420,
        // 418, 420. (n = 3, d = 25 M in 100 blocks, 5 %, eight at most 382, sixteen 410.)
        const int64_t most = c->K * rows / (8 * (int64_t)c->num_sms * kThreads);
        const int per_thread = (int)(most < 1 ? 1 : most > 8 ? 8 : most);
        const int64_t per_worker = (c->K + per_thread * kThreads - 1) / (per_thread * kThreads);
        e = counted(c, launch_after(randk_mark_kernel, dim3((unsigned)(per_worker * rows)), dim3(kThreads), c->stream, c->tab, b, c->row0,
                                    i0, origin, c->seed, c->iter, per_thread));
        if (e != cudaSuccess) break;
        void (*kernel)(const Tables, const TopkBuffers, const GT*, int32_t, int64_t, int64_t, int, const SegParams) =
            c->K * 32 > c->d ? randk_sweep_kernel<GT, 256> : randk_sweep_kernel<GT, 128>;  // mean of a warp: K / d x 1024
        e = counted(c, launch_after(kernel, dim3((unsigned)c->tab.ntiles, (unsigned)rows), dim3(kThreads), c->stream,
                                    c->tab, b, grads, i0, origin, c->randk_words, delivers(c) ? 1 : 0, c->segp));
    }
    return e;
}

cudaError_t launch_randk(compams_context* c, const void* grads) {
    return c->grad_bf16 ? launch_randk_typed(c, (const bf16_bits*)grads) : launch_randk_typed(c, (const float*)grads);
}

}  // namespace compams
