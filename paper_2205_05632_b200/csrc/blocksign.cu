// Block-Sign path (Definition 2) of the COMP-AMS step.
//
// bs_sweep   per (worker, tile): x = g + e (Algorithm 2, the corrected-gradient step), x written over E, sign bits
//            packed, sum |x| of the tile in binary64.
// bs_scales  per (worker, block): adds the tile sums in a fixed order and writes the scale
//            ||x_B||_1 / d_B.
// bs_apply   per coordinate: gbar = (1/n) sum_i sign(x_ij) s_{i,b} from the sign bits and
//            scales (the server's average), fused with the AMSGrad update (the moment, maximum and parameter updates).
//
// The residual e = x - sign(x) s (the residual update) needs the scale, which is known only after the whole
// block has been read. Instead of a second pass over [n, d], E keeps x and the subtraction is
// done when E is next read: by the next step's sweep (with the scale of the step that produced
// x) or by bs_materialize when the caller asks for E. Both evaluate the same single fp32
// subtraction, so the values are those of the residual update bit for bit.
#include <algorithm>

#include "context.h"

namespace compams {

// |x| as a binary64 number without a conversion instruction: for a normal fp32 value the
// binary64 pattern is the same fraction shifted left by 29 bits under an exponent rebiased by 896.
__device__ __forceinline__ double abs_as_double(float x) {
    const uint32_t b = __float_as_uint(x) & 0x7fffffffu;
    if ((b >> 23) == 0u) return (double)__uint_as_float(b);  // zero or subnormal: rare, take the conversion
    return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}

// Four of them added one after the other, with one test for the rare ones: the patterns without sign, counted from the smallest normal
// one up, reach 0xfe000000 where a value is infinite or NaN and, wrapped, where it is zero or subnormal. Those four go by the rule above
// each, so that what a value adds does not depend on its neighbours.
__device__ __forceinline__ void add_abs4(const float (&x)[4], double& acc) {
    uint32_t p[4], most = 0u;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        p[k] = 2u * __float_as_uint(x[k]) - 0x01000000u;
        most = most > p[k] ? most : p[k];
    }
    if (most < 0xfe000000u) {
#pragma unroll
        for (int k = 0; k < 4; ++k) acc += __hiloint2double((int)((p[k] >> 4) + 0x38100000u), (int)(p[k] << 28));
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) acc += abs_as_double(x[k]);
    }
}

// One warp's 1024 consecutive coordinates starting at rw (relative to the block; rw may be negative
// or reach past the block in a tile at either end of it: such coordinates are skipped). The signs come by ballots and are put in
// coordinate order once, at the end (with nibbles that four shuffles per iteration joined into words, and a test per element for
// the values that abs_as_double has to convert: n = 2, d = 1 M 16.4 us per step, now 15.5). A lane keeps its own byte of every ballot,
// one register: with all of the four ballots the build of eight CTAs per SM spilled 52 bytes (n = 2, d = 1 M 15.9 us, n = 8, d = 1.3 M 38.6,
// now 38.1, d = 2^20 27.5 / 27.4). WORDS keeps the four, for the builds of five CTAs per SM, which have registers to spare (n = 16,
// d = 2^23 300 against 306; bfloat16, 80 blocks in d = 3 M, n = 32 210.7 against 213.3).
// CUT: a warp past the end of the block stops.
template <bool FULL, bool WORDS, bool CUT, typename GT>
__device__ __forceinline__ void bs_sweep_tile(const GT* __restrict__ g, float* __restrict__ e, int len, int rw,
                                              int lane, bool deferred, float sp, double& acc, uint32_t& mymask) {
    const int cg = align_class(g + rw), ce = align_class(e + rw);
    // One iteration (4 coordinates per lane) is worked on while the next one's loads are already in flight
    // (two register buffers that alternate; the loop is fully unrolled). Small batches keep the kernel at
    // 32 registers, eight CTAs per SM: measured 0.329 ms against 0.355 ms for two-iteration batches without
    // prefetch at five CTAs per SM (ResNet-18 shapes, n = 16), the rate of a plain device copy.
    constexpr int NB = 1;
    constexpr int NBT = kIters / NB;
    float4 gbuf[2][NB], ebuf[2][NB];
    auto load_batch = [&](int bt, float4 (&gv)[NB], float4 (&ev)[NB]) {
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            const int r = rw + (bt * NB + u) * 128 + lane * 4;
            if (FULL || (r >= 0 && r + 3 < len)) {
                gv[u] = load4_stream(g + r, cg);
                ev[u] = load4(e + r, ce);
            } else {
                float gt[4], et[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const bool live = (unsigned)(r + k) < (unsigned)len;
                    gt[k] = live ? load1_stream(g + r + k) : 0.0f;
                    et[k] = live ? e[r + k] : 0.0f;
                }
                gv[u] = make_float4(gt[0], gt[1], gt[2], gt[3]);
                ev[u] = make_float4(et[0], et[1], et[2], et[3]);
            }
        }
    };
    uint32_t sg[WORDS ? 4 : 1] = {};
    load_batch(0, gbuf[0], ebuf[0]);
#pragma unroll
    for (int bt = 0; bt < NBT; ++bt) {
        if (CUT && rw + bt * NB * 128 >= len) break;
        float4 (&gv)[NB] = gbuf[bt & 1];
        float4 (&ev)[NB] = ebuf[bt & 1];
        if (bt + 1 < NBT) load_batch(bt + 1, gbuf[(bt + 1) & 1], ebuf[(bt + 1) & 1]);
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            const int it = bt * NB + u;
            const int r = rw + it * 128 + lane * 4;
            float xs[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                float xo = lane_elem(ev[u], k);
                // deferred residual: e = x_prev - sign(x_prev) * s_prev (Algorithm 2, the residual update)
                float ee = deferred ? __fsub_rn(xo, copysignf(sp, xo)) : xo;
                float x = __fadd_rn(lane_elem(gv[u], k), ee);  // the corrected-gradient step: x = g + e
                xs[k] = x;
                if (!FULL && (unsigned)(r + k) < (unsigned)len) acc += abs_as_double(x);
            }
            if (FULL) add_abs4(xs, acc);
            if (FULL || (r >= 0 && r + 3 < len)) {
                store4(e + r, ce, make_float4(xs[0], xs[1], xs[2], xs[3]));
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if ((unsigned)(r + k) < (unsigned)len) e[r + k] = xs[k];
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t m = __ballot_sync(0xffffffffu, (int)__float_as_uint(xs[k]) < 0 && (FULL || (unsigned)(r + k) < (unsigned)len));
                if ((lane >> 2) == it) {
                    if constexpr (WORDS) sg[k] = m;
                    else sg[0] |= ((m >> ((lane & 3) * 8)) & 0xffu) << (8 * k);
                }
            }
        }
    }
    // lane l holds the sign ballots of the iteration with the warp's l-th 32 coordinates: bit p of sg[k] is coordinate 4 p + k, and the
    // lane's own 32 are bits 8 (l % 4) ... of each
    mymask = 0u;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        uint32_t y = (WORDS ? sg[WORDS ? k : 0] >> ((lane & 3) * 8) : sg[0] >> (8 * k)) & 0xffu;  // eight bits to every fourth position
        y = (y | (y << 12)) & 0x000f000fu;
        y = (y | (y << 6)) & 0x03030303u;
        y = (y | (y << 3)) & 0x11111111u;
        mymask |= y << k;
    }
}

// The same for bfloat16 gradients on a whole tile whose rows of G and E are 16-byte aligned: 8 coordinates per
// lane and iteration, so that the gradient load is 128 bits wide like the two loads and stores of E (with 4
// coordinates per lane the 64-bit gradient loads leave too few bytes in flight: the sweep ran 8 % slower than
// with fp32 gradients although it reads fewer bytes). A warp's 1024 coordinates are 4 chunks of 256.
__device__ __forceinline__ void bs_sweep_tile_bf16x8(const bf16_bits* __restrict__ g, float* __restrict__ e, int rw, int lane,
                                                     bool deferred, float sp, double& acc, uint32_t& mymask) {
    constexpr int NC = kWarpSpan / 256;
    uint4 gbuf[2];
    float4 ebuf[2][2];
    auto load_chunk = [&](int c, uint4& gv, float4 (&ev)[2]) {
        const int r = rw + c * 256 + lane * 8;
        gv = __ldg(reinterpret_cast<const uint4*>(g + r));
        ev[0] = *reinterpret_cast<const float4*>(e + r);
        ev[1] = *reinterpret_cast<const float4*>(e + r + 4);
    };
    load_chunk(0, gbuf[0], ebuf[0]);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const uint4 gv = gbuf[c & 1];
        float4 (&ev)[2] = ebuf[c & 1];
        if (c + 1 < NC) load_chunk(c + 1, gbuf[(c + 1) & 1], ebuf[(c + 1) & 1]);
        const int r = rw + c * 256 + lane * 8;
        const uint32_t gw[4] = {gv.x, gv.y, gv.z, gv.w};
        uint32_t bits8 = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float xs[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t word = gw[h * 2 + (k >> 1)];
                const float gk = __uint_as_float((k & 1) ? (word & 0xffff0000u) : (word << 16));  // exact widening
                const float xo = lane_elem(ev[h], k);
                // deferred residual: e = x_prev - sign(x_prev) * s_prev (Algorithm 2, the residual update)
                const float ee = deferred ? __fsub_rn(xo, copysignf(sp, xo)) : xo;
                const float x = __fadd_rn(gk, ee);  // the corrected-gradient step: x = g + e
                xs[k] = x;
                acc += abs_as_double(x);
                bits8 |= (__float_as_uint(x) >> 31) << (h * 4 + k);
            }
            *reinterpret_cast<float4*>(e + r + h * 4) = make_float4(xs[0], xs[1], xs[2], xs[3]);
        }
        // 4 lanes make one 32-bit word; word q of the chunk's 8 words sits in lanes 4q .. 4q + 3
        uint32_t w = bits8 << ((lane & 3) * 8);
        w |= __shfl_xor_sync(0xffffffffu, w, 1);
        w |= __shfl_xor_sync(0xffffffffu, w, 2);
        const uint32_t wv = __shfl_sync(0xffffffffu, w, (lane & 7) * 4);
        if ((lane >> 3) == c) mymask = wv;  // lane l ends up holding the sign mask of the warp's l-th 32 coordinates
    }
}

// Tiles are shifted down by s = (i d + o) mod 32, the position of the block's first element within
// a 128-byte line of G and E, so that every warp access covers whole lines (with rows that start
// mid-line a warp's 512 bytes straddle five lines instead of four: measured 7 % slower). The
// sign words stay indexed by coordinate: word q of the block takes its low 32 - s bits from the
// q-th group of 32 shifted coordinates and its high s bits from the next group. The word a tile
// shares with the next tile is put together by bs_scales, or by bs_apply, from the two shares left in `edge`.
// AHEAD: the tile's lines are asked into the L2 first, with five CTAs per SM; CUT: for many tiles that are mostly empty: see
// launch_bs_sweep.
template <typename GT, bool AHEAD, bool CUT>
__global__ void __launch_bounds__(kThreads, sizeof(GT) == 2 || AHEAD ? 5 : 8) bs_sweep_kernel(Tables t, BsBuffers b, const GT* __restrict__ G,
                                                               int deferred, const __grid_constant__ SegParams sp_) {
    __shared__ double red[kWarps];
    __shared__ uint32_t sh_first[kWarps];
    dependency_wait();  // while n d <= kChainMaxElems launched as a programmatic dependent of the step before (whose server
                        // kernel still reads the sign words this kernel is about to overwrite)
    allow_dependents();
    const int tile = blockIdx.x;
    const int i = blockIdx.y;
    const TileInfo ti = sp_.nseg ? find_tile(sp_, tile) : load_tile(t.tiles, tile);
    const int blk = ti.blk;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t row0 = (int64_t)i * t.d + ti.o;
    const int s = (int)(row0 & 31);
    const GT* g = G + row0;
    float* e = b.E + row0;
    const float sp = deferred ? b.scales_prev[(size_t)i * t.M + blk] : 0.0f;
    const int r0s = ti.r0 - s;
    const int rw = r0s + warp * kWarpSpan;

    constexpr bool kWords = sizeof(GT) == 2 || AHEAD;
    double acc = 0.0;
    uint32_t mymask = 0;
    const bool whole = r0s >= 0 && r0s + kTile <= ti.len;
    if (AHEAD && whole) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(e + rw + lane * 32));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(g + rw + lane * 32));
    }
    bool wide = false;
    if constexpr (sizeof(GT) == 2)
        wide = whole && ((reinterpret_cast<uintptr_t>(g + rw) | reinterpret_cast<uintptr_t>(e + rw)) & 15u) == 0;
    if (wide) {
        if constexpr (sizeof(GT) == 2) bs_sweep_tile_bf16x8(g, e, rw, lane, deferred != 0, sp, acc, mymask);
    } else if (whole) {
        bs_sweep_tile<true, kWords, false>(g, e, ti.len, rw, lane, deferred != 0, sp, acc, mymask);
    } else {
        bs_sweep_tile<false, kWords, CUT>(g, e, ti.len, rw, lane, deferred != 0, sp, acc, mymask);
    }

    // tile sum in binary64 (fixed shuffle tree); bs_scales adds the tile sums of a block in a fixed order
    if (lane == 0) sh_first[warp] = mymask;
    const double sum = block_sum_double(acc, red);  // its barriers also publish sh_first
    if (threadIdx.x == 0) b.tile_sum[(size_t)i * t.ntiles + tile] = sum;

    uint32_t next = __shfl_down_sync(0xffffffffu, mymask, 1);
    const bool last = warp == kWarps - 1 && lane == 31;
    if (lane == 31) next = last ? 0u : sh_first[warp + 1];
    const uint32_t word = __funnelshift_r(mymask, next, (uint32_t)s);  // s = 0: the mask itself
    const int q = (ti.r0 >> 5) + warp * 32 + lane;  // word of the block this lane completes
    const int wb = (ti.len + 31) >> 5;
    const int64_t wofs = sp_.nseg ? (int64_t)sp_.wofs[ti.seg] : b.word_off[blk];
    if (!last && q < wb) b.bits[(size_t)i * (size_t)b.W + (size_t)wofs + (size_t)q] = word;
    // shares of the two words in common with the neighbouring tiles: the high bits of the word before
    // this tile's first, the low bits of its last
    if (threadIdx.x == 0 || last) {
        uint32_t* ed = reinterpret_cast<uint32_t*>(b.edge + (size_t)i * t.ntiles + tile);
        if (last) ed[1] = word;
        else ed[0] = s ? (mymask << (32 - s)) : 0u;
    }
}

// Sum of a block's tile sums by one warp, in an order fixed by the tile count (result in lane 0). bs_scales and bs_apply
// add up blocks of at most kWarpTiles tiles this way, so that it does not matter which of them does.
constexpr int kWarpTiles = 256;
__device__ __forceinline__ double tile_sums_by_warp(const double* ts, int nt, int lane) {
    double part = 0.0;
    for (int k = lane; k < nt; k += 32) part += ts[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
    return part;
}
// One division in binary64, one rounding to fp32.
__device__ __forceinline__ float scale_of(double sum, int len) { return __double2float_rn(sum / (double)len); }

// One CTA per (worker, block): scale = ||x_B||_1 / d_B from the tile sums (Definition 2). Built for 256 threads
// (many blocks of a few tiles) and for 1024 with four tile sums requested at a time (a whole-vector block has
// thousands of tiles and only n CTAs to add them: 256 threads took 33 us at d = 2^26, n = 8, most of it waiting
// for one load after the other). The order of the additions is fixed by the tile count and the thread count,
// and every handle of a sharded run makes the same choice, so equal inputs give equal bits.
template <int NT>
__global__ void __launch_bounds__(NT) bs_scales_kernel(Tables t, BsBuffers b) {
    __shared__ double red[NT / 32];
    allow_dependents();
    dependency_wait();  // the sweep's tile sums and word shares
    const int blk = blockIdx.x, i = blockIdx.y;
    const SegInfo* si = t.segs + blk;
    const double* ts = b.tile_sum + (size_t)i * t.ntiles + si->tile0;
    const int nt = si->ntile_b;
    double part = 0.0;
    int k = nt > kWarpTiles ? (int)threadIdx.x : nt;
    for (; k + 3 * NT < nt; k += 4 * NT) {
        const double s0 = ts[k], s1 = ts[k + NT], s2 = ts[k + 2 * NT], s3 = ts[k + 3 * NT];
        part += s0;
        part += s1;
        part += s2;
        part += s3;
    }
    for (; k < nt; k += NT) part += ts[k];
    // the sign word two neighbouring tiles have in common: one share from each
    {
        const uint2* ed = b.edge + (size_t)i * t.ntiles + si->tile0;
        const int wb = (si->len + 31) >> 5;
        uint32_t* words = b.bits + (size_t)i * (size_t)b.W + (size_t)b.word_off[blk];
#pragma unroll 4
        for (int j = threadIdx.x; j < nt; j += NT) {
            const int q = (j + 1) * (kTile / 32) - 1;
            if (q < wb) words[q] = ed[j].y | (j + 1 < nt ? ed[j + 1].x : 0u);
        }
    }
    double S;
    if (nt > kWarpTiles) {
        S = block_sum_double<NT / 32>(part, red);
    } else {
        if (threadIdx.x >= 32) return;
        S = tile_sums_by_warp(ts, nt, threadIdx.x);
    }
    if (threadIdx.x == 0) b.scales_cur[(size_t)i * t.M + blk] = scale_of(S, si->len);
}

// E holds x; turn it into e = x - sign(x) * s in place (Algorithm 2, the residual update).
__global__ void __launch_bounds__(kThreads) bs_materialize_kernel(Tables t, float* __restrict__ E,
                                                                  const float* __restrict__ scales) {
    const int i = blockIdx.y;
    const TileInfo ti = load_tile(t.tiles, blockIdx.x);
    const int blk = ti.blk;
    const int64_t o = ti.o;
    const int64_t len = ti.len;
    const int64_t r0 = ti.r0;
    const float s = scales[(size_t)i * t.M + blk];
    float* e = E + (size_t)i * (size_t)t.d + (size_t)o;
    const int64_t end = (r0 + kTile < len) ? r0 + kTile : len;
    for (int64_t r = r0 + threadIdx.x; r < end; r += kThreads) {
        float x = e[r];
        e[r] = __fsub_rn(x, copysignf(s, x));
    }
}

// Workers whose sign words and scales are staged at a time: with tables of 8 workers' scales, of 4 workers'.
constexpr int kApplyEights = 16, kApplyFours = 32;

// Transposes an 8 x 8 bit matrix whose rows are the bytes of lo (rows 0-3) and hi (rows 4-7): afterwards bit i of byte k
// is what bit k of byte i was. Three rounds of the usual block swap.
__device__ __forceinline__ void transpose8(uint32_t& lo, uint32_t& hi) {
    uint32_t t;
    t = (lo ^ (lo >> 7)) & 0x00aa00aau;
    lo ^= t ^ (t << 7);
    t = (hi ^ (hi >> 7)) & 0x00aa00aau;
    hi ^= t ^ (t << 7);
    t = (lo ^ (lo >> 14)) & 0x0000ccccu;
    lo ^= t ^ (t << 14);
    t = (hi ^ (hi >> 14)) & 0x0000ccccu;
    hi ^= t ^ (t << 14);
    t = (lo & 0x0f0f0f0fu) | ((hi << 4) & 0xf0f0f0f0u);
    hi = ((lo >> 4) & 0x0f0f0f0fu) | (hi & 0xf0f0f0f0u);
    lo = t;
}

constexpr int kApplySpan = 8 * kThreads;  // coordinates per CTA of bs_apply

// Shared memory of one bs_apply CTA.
template <bool FOURS>
struct ApplyShared {
    static constexpr int kChunk = FOURS ? kApplyFours : kApplyEights;
    float state[4][kApplySpan + 4];  // m, v, vhat, theta of the CTA's coordinates, from a 16-byte boundary on
    union {
        struct {
            uint32_t bits[kChunk][kApplySpan / 32];   // [worker][word]
            double four[kChunk / 4][16];              // subset sums of 4 workers' scales
            double eight[FOURS ? 1 : kChunk / 8][FOURS ? 1 : 256];  // ... of 8 workers', not with FOURS
            double scale[kChunk];
        } sum;
        float gbar[kApplySpan + 4];
    };
    uint64_t arrived;  // mbarrier: the state is there
};

// Server side of Block-Sign (Algorithm 2, the server's average and update): one CTA per 2048 consecutive coordinates of a
// block. The tile's block comes from the constant bank, and the optimizer state is on its way to shared memory (four bulk
// copies) before the kernel in front is done.
//
// Per coordinate the sum over workers of +-s_i is (sum of all s_i) - 2 (sum of the s_i whose bit is set). The second sum
// depends only on the coordinate's pattern of sign bits, and all coordinates of the CTA share the workers' scales: for
// every 8 workers a 256-entry table holds the sum of each subset of their scales (exact in binary64 wherever the plain
// sum is), and a coordinate adds one entry per 8 workers. A thread's 8 coordinates are one byte of each worker's sign
// words, so the patterns of 8 workers come from transposing 8 bytes in registers. The averages pass through shared memory,
// and the update runs over groups of 4 coordinates that start on 16-byte boundaries, whatever the block's offset.
//
// Bound by memory from here on (32 B per coordinate and the sign bits); before, with one predicated binary64 add per worker
// and coordinate, or 16-entry tables and a transposition across the warp, by instruction issue (786 instructions per 4
// coordinates at n = 16, half of them the sum), and with blocks off the 16-byte grid by 32-bit accesses: steps of ResNet-18
// shapes, n = 16 429 -> 406 us; d = 6.6 M in 7 ragged blocks, n = 4 105 -> 96; 8 of 32 workers, ResNet-50 shapes 652 -> 627.
// FOURS, from 17 workers on: the words and scales of up to 32 workers come in one round of loads, and a coordinate adds two entries of
// 16-entry tables per 8 workers: all 16 entries of one lie in different banks, where the lanes' lookups in 256 entries met in
// three on average, which is what two rounds of 16 workers were bound by (the shared-memory pipe 73 % busy at n = 32; 8 of 32
// workers, ResNet-50 shapes, this kernel 192 -> 155 us and the step 628 -> 599; n = 32, d = 4.2 M 288 -> 282).
// Tried: 8 consecutive coordinates per thread in the update too, by 256-bit accesses from registers (417 us on the first,
// 142 on the second), three and five CTAs per SM, CTAs of 64 and 128 threads for small vectors (slower than 256; those have
// bs_apply_short).
// OWN: the tile sums have not been added up by bs_scales (small blocks, all workers in this handle): every CTA adds up
// its block's, and completes the sign words that its tile has in common with the next.
template <bool RECORD, bool OWN, bool FOURS>
__global__ void __launch_bounds__(kThreads, 4) bs_apply_kernel(const __grid_constant__ Tables t, const __grid_constant__ BsBuffers b,
                                                               float* __restrict__ theta, const __grid_constant__ HyperParams hp,
                                                               const __grid_constant__ SegParams sp_) {
    constexpr int kApplyChunk = ApplyShared<FOURS>::kChunk;
    __shared__ __align__(128) ApplyShared<FOURS> sh;
    const int tile = blockIdx.x / (kTile / kApplySpan);
    const TileInfo ti = sp_.nseg ? find_tile(sp_, tile) : load_tile(t.tiles, tile);
    const int blk = ti.blk;
    const int len = ti.len;
    const int rs = ti.r0 + (int)(blockIdx.x % (kTile / kApplySpan)) * kApplySpan;  // first coordinate, relative to the block
    if (rs >= len) return;
    const int count = len - rs < kApplySpan ? len - rs : kApplySpan;
    // coordinates j0 .. j1 - 1; positions in shared memory count from the 16-byte boundary g0 (all four vectors are
    // 16-byte aligned at coordinate 0); whole groups of 4 lie in [lo, hi)
    const int64_t j0 = ti.o + rs, g0 = j0 & ~(int64_t)3;
    const int skip = (int)(j0 - g0), end = skip + count;
    const int lo = skip ? 4 : 0, hi = end & ~3;
    float* const vec[4] = {b.m, b.v, b.vhat, theta};
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&sh.arrived);
    if (threadIdx.x == 0) {
        const uint32_t bytes = hi > lo ? (uint32_t)(hi - lo) * 4u : 0u;
        mbar_init(bar);
        mbar_expect(bar, 4u * bytes);
        if (bytes) {
#pragma unroll
            for (int q = 0; q < 4; ++q) bulk_load(&sh.state[q][lo], vec[q] + g0 + lo, bytes, bar);
        }
    }
    dependency_wait();  // the state was last written a step ago; sign words and scales are this step's
    const size_t wbase = (size_t)(sp_.nseg ? (int64_t)sp_.wofs[ti.seg] : b.word_off[blk]) + (size_t)(rs >> 5);
    const int lane = threadIdx.x & 31, wr = threadIdx.x >> 5;
    const int words = (len - rs + 31) >> 5;  // sign words of this CTA's coordinates (possibly more than it has)
    const int edge_word = rs + kApplySpan == ti.r0 + kTile ? kApplySpan / 32 - 1 : -1;
    double a[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0}, all = 0.0;
    for (int i0 = 0; i0 < t.n; i0 += kApplyChunk) {
        const int nc = (t.n - i0 < kApplyChunk) ? t.n - i0 : kApplyChunk;
        const int ng = (nc + 7) >> 3;  // groups of 8 workers in this round; absent workers have sign + and scale 0
        if (i0) __syncthreads();
#pragma unroll
        for (int c = wr; c < kApplyChunk; c += kWarps) {
            uint32_t* src = b.bits + (size_t)(i0 + c) * (size_t)b.W + wbase;
#pragma unroll
            for (int w = lane; w < kApplySpan / 32; w += 32) {
                uint32_t word = 0u;
                if (c < nc && w < words) {
                    if (OWN && w == edge_word) {  // the word in common with the next tile: one share from each
                        const uint2* ed = b.edge + (size_t)(i0 + c) * t.ntiles + tile;
                        word = ed[0].y | (tile + 1 < ti.tile0 + ti.ntile_b ? ed[1].x : 0u);
                        src[w] = word;
                    } else {
                        word = src[w];
                    }
                }
                sh.sum.bits[c][w] = word;
            }
        }
        if (OWN) {
            for (int c = wr; c < nc; c += kWarps) {
                const double s = tile_sums_by_warp(b.tile_sum + (size_t)(i0 + c) * t.ntiles + ti.tile0, ti.ntile_b, lane);
                if (lane == 0) {
                    const float f = scale_of(s, len);
                    sh.sum.scale[c] = (double)f;
                    if (rs == 0) b.scales_cur[(size_t)(i0 + c) * t.M + blk] = f;
                }
            }
        } else if (threadIdx.x < nc) {
            sh.sum.scale[threadIdx.x] = (double)b.scales_cur[(size_t)(i0 + threadIdx.x) * t.M + blk];
        }
        __syncthreads();
        static_assert(kApplyChunk * 4 <= kThreads, "one table entry per thread");
        if (threadIdx.x < kApplyChunk * 4) {  // one table entry per thread: the scales of the subset's members
            const int q = threadIdx.x >> 4, sub = threadIdx.x & 15;
            double e = 0.0;
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (((sub >> j) & 1) && q * 4 + j < nc) e += sh.sum.scale[q * 4 + j];
            sh.sum.four[q][sub] = e;
        }
        __syncthreads();
        if constexpr (!FOURS) {
#pragma unroll
            for (int g = 0; g < kApplyChunk / 8; ++g)
                if (g < ng) sh.sum.eight[g][threadIdx.x] = sh.sum.four[2 * g][threadIdx.x & 15] + sh.sum.four[2 * g + 1][threadIdx.x >> 4];
            __syncthreads();
        }
#pragma unroll
        for (int g = 0; g < kApplyChunk / 8; ++g) {
            if (g < ng) {  // the same for every thread of the CTA
                uint32_t x[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) x[j] = reinterpret_cast<const unsigned char*>(sh.sum.bits[g * 8 + j])[threadIdx.x];
                uint32_t p0 = __byte_perm(__byte_perm(x[0], x[1], 0x0040), __byte_perm(x[2], x[3], 0x0040), 0x5410);
                uint32_t p1 = __byte_perm(__byte_perm(x[4], x[5], 0x0040), __byte_perm(x[6], x[7], 0x0040), 0x5410);
                transpose8(p0, p1);
                if constexpr (FOURS) {
                    all += sh.sum.four[2 * g][15] + sh.sum.four[2 * g + 1][15];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        a[k] += sh.sum.four[2 * g][(p0 >> (8 * k)) & 15u] + sh.sum.four[2 * g + 1][(p0 >> (8 * k + 4)) & 15u];
                        a[4 + k] += sh.sum.four[2 * g][(p1 >> (8 * k)) & 15u] + sh.sum.four[2 * g + 1][(p1 >> (8 * k + 4)) & 15u];
                    }
                } else {
                    all += sh.sum.eight[g][255];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        a[k] += sh.sum.eight[g][(p0 >> (8 * k)) & 255u];
                        a[4 + k] += sh.sum.eight[g][(p1 >> (8 * k)) & 255u];
                    }
                }
            }
        }
    }
    __syncthreads();  // the tables make room for the averages
    {
        float gb[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) gb[k] = mean_from_acc(all - (a[k] + a[k]), hp);
        const int p = skip + (int)threadIdx.x * 8;
        if (skip == 0) {
            *reinterpret_cast<float4*>(sh.gbar + p) = make_float4(gb[0], gb[1], gb[2], gb[3]);
            *reinterpret_cast<float4*>(sh.gbar + p + 4) = make_float4(gb[4], gb[5], gb[6], gb[7]);
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) sh.gbar[p + k] = gb[k];
        }
    }
    __syncthreads();
    if (!mbar_wait(bar)) {  // cannot happen: the copies are this CTA's own
        atomicOr(b.status, 4u);
        return;
    }
    for (int p = (int)threadIdx.x * 4; p < end; p += kThreads * 4) {
        if (p >= lo && p < hi) {
            float4 mm = *reinterpret_cast<const float4*>(&sh.state[0][p]), vv = *reinterpret_cast<const float4*>(&sh.state[1][p]);
            float4 hh = *reinterpret_cast<const float4*>(&sh.state[2][p]), tt = *reinterpret_cast<const float4*>(&sh.state[3][p]);
            const float4 gb = *reinterpret_cast<const float4*>(sh.gbar + p);
            amsgrad_update(gb.x, mm.x, vv.x, hh.x, tt.x, hp);
            amsgrad_update(gb.y, mm.y, vv.y, hh.y, tt.y, hp);
            amsgrad_update(gb.z, mm.z, vv.z, hh.z, tt.z, hp);
            amsgrad_update(gb.w, mm.w, vv.w, hh.w, tt.w, hp);
            if constexpr (RECORD) *reinterpret_cast<float4*>(b.gbar + g0 + p) = gb;
            *reinterpret_cast<float4*>(vec[0] + g0 + p) = mm;
            *reinterpret_cast<float4*>(vec[1] + g0 + p) = vv;
            *reinterpret_cast<float4*>(vec[2] + g0 + p) = hh;
            *reinterpret_cast<float4*>(vec[3] + g0 + p) = tt;
        } else {  // the group that this block's first or last coordinates share with a neighbour
            for (int k = p < skip ? skip : p; k < p + 4 && k < end; ++k) {
                const int64_t j = g0 + k;
                float m1 = b.m[j], v1 = b.v[j], h1 = b.vhat[j], t1 = theta[j];
                amsgrad_update(sh.gbar[k], m1, v1, h1, t1, hp);
                if constexpr (RECORD) b.gbar[j] = sh.gbar[k];
                b.m[j] = m1;
                b.v[j] = v1;
                b.vhat[j] = h1;
                theta[j] = t1;
            }
        }
    }
}

constexpr int kShortChunk = 32;  // workers whose sign words are staged (and transposed) at a time: one per lane

// Transposes four 32 x 32 bit matrices held across a warp: on entry lane i holds x[q] = row i of matrix q
// (bit c = element (i, c)); on return lane c holds column c (bit i = element (i, c)). Five rounds of the
// usual block swap: in round j a lane exchanges with lane ^ j the half of its bits whose position differs
// from its own index in bit j. Shifting the partner's word by +-j and keeping only the positions that
// change is a rotation followed by a bitwise select.
__device__ __forceinline__ void transpose32x4(uint32_t (&x)[4], int lane) {
#pragma unroll
    for (int j = 16; j >= 1; j >>= 1) {
        const uint32_t m = j == 16 ? 0x0000ffffu : j == 8 ? 0x00ff00ffu : j == 4 ? 0x0f0f0f0fu : j == 2 ? 0x33333333u : 0x55555555u;
        const bool up = (lane & j) != 0;
        const uint32_t keep = up ? ~m : m;          // positions whose bit j equals the lane's stay
        const uint32_t rot = up ? 32u - j : (uint32_t)j;  // the partner's bits move down (up) by j
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t y = __shfl_xor_sync(0xffffffffu, x[q], j);
            x[q] = (x[q] & keep) | (__funnelshift_l(y, y, rot) & ~keep);
        }
    }
}

// The same for few tiles: one CTA per 1024 coordinates, one float4 group per thread, so that a vector too short to give
// bs_apply's CTAs of 2048 coordinates an SM each is spread twice as wide and a CTA has half the serial work.
// TABLES = false: one predicated binary64 add per worker and coordinate. TABLES = true: 16-entry tables of 4 workers' scales,
// the patterns from a transposition across the warp: lane i reads worker i's four words of the warp's 128 coordinates,
// transpose32x4 turns them into one word per coordinate, and 16 shuffles hand every lane the patterns of its own 4 coordinates.
// Bound by latency: the words and scales of up to 32 workers come in one round of loads (see launch_bs_apply for the figures).
template <bool TABLES, bool RECORD>
__global__ void __launch_bounds__(kThreads, 5) bs_apply_short_kernel(const __grid_constant__ Tables t, const __grid_constant__ BsBuffers b,
                                                                     float* __restrict__ theta, const __grid_constant__ HyperParams hp,
                                                                     const __grid_constant__ SegParams sp_) {
    __shared__ uint32_t sh_bits[kShortChunk][33];        // [worker][word], rows padded against bank conflicts
    __shared__ double sh_tab[kShortChunk / 4][16];       // TABLES: [group of 4 workers][subset] sum of the subset's
                                                         // scales; else: the workers' scales
    const int tile = blockIdx.x >> 3;
    const TileInfo ti = sp_.nseg ? find_tile(sp_, tile) : load_tile(t.tiles, tile);
    const int blk = ti.blk;
    const int len = ti.len;
    const int rs = ti.r0 + (int)(blockIdx.x & 7) * kWarpSpan;  // first coordinate of this CTA, relative to the block
    if (rs >= len) return;
    const int r = rs + (int)threadIdx.x * 4;
    const int64_t o = ti.o;
    float* gbar = b.gbar + o;
    float* m = b.m + o;
    float* v = b.v + o;
    float* vh = b.vhat + o;
    float* th = theta + o;
    const int cls = align_class(m);  // all five vectors are 16-byte aligned at coordinate 0
    const bool full = r + 3 < len;
    float4 mm = make_float4(0.f, 0.f, 0.f, 0.f), vv = mm, hh = mm, tt = mm;
    if (full) {
        mm = load4(m + r, cls);
        vv = load4(v + r, cls);
        hh = load4(vh + r, cls);
        tt = load4(th + r, cls);
    }
    dependency_wait();  // the state above was last written a step ago; sign words and scales are this step's
    const size_t wbase = (size_t)(sp_.nseg ? (int64_t)sp_.wofs[ti.seg] : b.word_off[blk]) + (size_t)(rs >> 5);
    const int lane = threadIdx.x & 31, wr = threadIdx.x >> 5;  // warp wr owns coordinates 128 wr ... of the CTA's 1024
    const bool word_live = rs + lane * 32 < len;
    double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0, all = 0.0;
    for (int i0 = 0; i0 < t.n; i0 += kShortChunk) {
        const int nc = (t.n - i0 < kShortChunk) ? t.n - i0 : kShortChunk;
        __syncthreads();
        // warp wr stages the words of workers wr, wr + 8, ...: 32 consecutive words each, one per lane
        for (int c = wr; c < nc; c += kWarps)
            sh_bits[c][lane] = word_live ? __ldg(b.bits + (size_t)(i0 + c) * (size_t)b.W + wbase + lane) : 0u;
        if constexpr (TABLES) {
            const int ng = (nc + 3) >> 2;  // groups of 4 workers in this round
            if (threadIdx.x < ng * 16) {   // one table entry per thread: the scales of the subset's members
                const int gq = threadIdx.x >> 4, sub = threadIdx.x & 15;
                double e = 0.0;
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (((sub >> j) & 1) && gq * 4 + j < nc)
                        e += (double)b.scales_cur[(size_t)(i0 + gq * 4 + j) * t.M + blk];
                sh_tab[gq][sub] = e;
            }
            __syncthreads();
            // lane i: worker i's words of this warp's coordinates -> lane c: the workers' bits of coordinate 32 q + c
            uint32_t x[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) x[q] = lane < nc ? sh_bits[lane][wr * 4 + q] : 0u;
            transpose32x4(x, lane);
            // this thread's coordinates 4 lane + k lie in word q = lane / 8 at bit 4 (lane % 8) + k: their patterns
            // sit in lane 4 (lane % 8) + k, matrix lane / 8 (a trip through shared memory instead of these 16
            // shuffles was slower)
            uint4 pat = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint32_t y0 = __shfl_sync(0xffffffffu, x[q], (lane & 7) * 4 + 0);
                const uint32_t y1 = __shfl_sync(0xffffffffu, x[q], (lane & 7) * 4 + 1);
                const uint32_t y2 = __shfl_sync(0xffffffffu, x[q], (lane & 7) * 4 + 2);
                const uint32_t y3 = __shfl_sync(0xffffffffu, x[q], (lane & 7) * 4 + 3);
                if ((lane >> 3) == q) pat = make_uint4(y0, y1, y2, y3);
            }
#pragma unroll
            for (int gq = 0; gq < kShortChunk / 4; ++gq) {
                if (gq < ng) {  // the same for every thread of the CTA
                    all += sh_tab[gq][15];
                    a0 += sh_tab[gq][(pat.x >> (4 * gq)) & 15u];
                    a1 += sh_tab[gq][(pat.y >> (4 * gq)) & 15u];
                    a2 += sh_tab[gq][(pat.z >> (4 * gq)) & 15u];
                    a3 += sh_tab[gq][(pat.w >> (4 * gq)) & 15u];
                }
            }
        } else {
            double* sh_s = &sh_tab[0][0];
            if (threadIdx.x < nc) sh_s[threadIdx.x] = (double)b.scales_cur[(size_t)(i0 + threadIdx.x) * t.M + blk];
            __syncthreads();
            const int wsel = threadIdx.x >> 3, nsh = (threadIdx.x & 7) * 4;  // this thread's word and its nibble in it
#pragma unroll 4
            for (int c = 0; c < nc; ++c) {
                const double sc = sh_s[c];
                const uint32_t nib = sh_bits[c][wsel] >> nsh;
                all += sc;
                if (nib & 1u) a0 += sc;
                if (nib & 2u) a1 += sc;
                if (nib & 4u) a2 += sc;
                if (nib & 8u) a3 += sc;
            }
        }
    }
    a0 = all - (a0 + a0);
    a1 = all - (a1 + a1);
    a2 = all - (a2 + a2);
    a3 = all - (a3 + a3);
    if (r >= len) return;
    const float gb[4] = {mean_from_acc(a0, hp), mean_from_acc(a1, hp), mean_from_acc(a2, hp),
                         mean_from_acc(a3, hp)};
    if (full) {
        amsgrad_update(gb[0], mm.x, vv.x, hh.x, tt.x, hp);
        amsgrad_update(gb[1], mm.y, vv.y, hh.y, tt.y, hp);
        amsgrad_update(gb[2], mm.z, vv.z, hh.z, tt.z, hp);
        amsgrad_update(gb[3], mm.w, vv.w, hh.w, tt.w, hp);
        if constexpr (RECORD) store4(gbar + r, cls, make_float4(gb[0], gb[1], gb[2], gb[3]));
        store4(m + r, cls, mm);
        store4(v + r, cls, vv);
        store4(vh + r, cls, hh);
        store4(th + r, cls, tt);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (r + k < len) {
                float m1 = m[r + k], v1 = v[r + k], h1 = vh[r + k], t1 = th[r + k];
                amsgrad_update(gb[k], m1, v1, h1, t1, hp);
                if constexpr (RECORD) gbar[r + k] = gb[k];
                m[r + k] = m1;
                v[r + k] = v1;
                vh[r + k] = h1;
                th[r + k] = t1;
            }
        }
    }
}

// The worker-side kernels see this handle's own rows of the message buffers (sign words, scales);
// the server kernel sees the rows of all n_total workers.
static BsBuffers own_rows(const compams_context* c) {
    BsBuffers b = c->bs;
    const size_t r0 = (size_t)c->row0;
    b.bits = c->bs.bits + r0 * (size_t)c->W;
    b.scales_prev = c->scales[c->scales_cur ^ 1] + r0 * (size_t)c->M;
    b.scales_cur = c->scales[c->scales_cur] + r0 * (size_t)c->M;
    return b;
}

template <typename GT>
static cudaError_t launch_sweep_typed(compams_context* c, void (*kernel)(Tables, BsBuffers, const GT*, int, const SegParams), const GT* grads) {
    const dim3 grid((unsigned)c->tab.ntiles, (unsigned)c->n);
    const int deferred = c->e_is_x ? 1 : 0;
    if (c->chain)  // n d <= kChainMaxElems: the launch overlaps the tail of whatever kernel precedes it on the stream
        return counted(c, launch_after(kernel, grid, dim3(kThreads), c->stream, c->tab, own_rows(c), grads, deferred, c->segp));
    kernel<<<grid, kThreads, 0, c->stream>>>(c->tab, own_rows(c), grads, deferred, c->segp);
    return counted(c, cudaGetLastError());
}

// The build that asks ahead takes over where the sweep is many waves long. What it gives depends on the GPU it runs on: us per step without /
// with, on the boxes where most was gained and where least: ResNet-18 shapes, n = 16 395.0 / 389.8, 405.7 / 409.0; 8 of 32 workers, ResNet-50
// shapes 578.3 / 575.2, 597.2 / 597.0; n = 16, d = 2^23 293.6 / 291.8, 300.1 / 302.0; n = 2, d = 90 M 762.1 / 760.0, 769.7 / 770.3; n = 6,
// d = 30 M 479 / 478, 492 / 495. Below it loses everywhere: n = 16, d = 4 M 150 / 152, n = 9, d = 2.9 M 74 / 78, n = 8, d = 2^20 27.5 / 29.8. In
// steps too long to be chained it loses with one block, or a few, more than it gives - n = 32, d = 2^24 1057 / 1064, 1082 / 1109, d = 2^25 2098 /
// 2117, 2141 / 2194, n = 20, d = 40 M 1650 / 1669, 1689 / 1724, n = 16, d = 40 M in two blocks 1378 / 1387 - and gains with many: n = 32, d =
// 25 M in 161 1646 / 1610, 1685 / 1693, n = 13, d = 21.6 M in 134 681 / 672, n = 8, d = 100 M in 21 2049 / 2032, n = 12, d = 50 M in 31 1439 / 1423,
// ten blocks in d = 2^24, n = 32 1117 / 1114.
constexpr int64_t kAheadElems = (int64_t)1 << 26;
static bool sweep_asks_ahead(const compams_context* c) {
    return (int64_t)c->n * c->d >= kAheadElems && (c->chain || c->M > 8);
}

// Where most of the tiles lies outside the blocks (many small ones) the sweep is bound by the instructions of warps that have nothing, or
// little, to do, and the build that lets them stop takes over; one that does not test for it starts 0.5 us earlier, which is what
// counts where the CTAs are few. us per step without / with: 152 blocks in d = 75,215 (17 times as much in tiles), n = 32 72 / 37, n = 4
// 17.5 / 13.5, but n = 1 12.5 / 12.7; 150 in d = 750,007 (2.6 times), n = 8 35.8 / 29.0, bfloat16 39.4 / 37.2, but n = 1 16.3 / 16.9; one block,
// n = 4, d = 100,003 9.2 / 9.8; 80 in d = 3 M (1.2 times), n = 8 75.9 / 76.5.
static bool sweep_is_cut(const compams_context* c) {
    return (int64_t)c->tab.ntiles * kTile >= 2 * c->d && (int64_t)c->n * c->tab.ntiles > 2 * c->num_sms;
}

cudaError_t launch_bs_sweep(compams_context* c, const void* grads) {
    const bool cut = sweep_is_cut(c);
    if (c->grad_bf16)
        return launch_sweep_typed(c, cut ? bs_sweep_kernel<bf16_bits, false, true> : bs_sweep_kernel<bf16_bits, false, false>, (const bf16_bits*)grads);
    const bool ahead = sweep_asks_ahead(c);
    return launch_sweep_typed(c, cut     ? bs_sweep_kernel<float, false, true>
                                 : ahead ? bs_sweep_kernel<float, true, false>
                                         : bs_sweep_kernel<float, false, false>, (const float*)grads);
}

// Whether the server kernel is bs_apply_short: few tiles for the number of workers. us per step (whole vector, bs_apply with the tile
// sums its own business or with bs_scales, whichever is faster, against bs_scales and bs_apply_short): n = 32, d = 65,536 (9 tiles)
// 17.6 / 12.7, n = 16, d = 162,400 (20) 15.3 / 13.3, n = 16, d = 370,001 (46) 18.6 / 18.3, n = 24, d = 524,288 (65) 35.2 / 33.9; beyond the
// line n = 16, d = 750,007 (92) 32.1 / 33.9, n = 32, d = 2^20 (129) 79.7 / 81.8. With few workers and very few tiles the
// launch that is saved is worth more: n = 8, d = 100,003 (13) 10.8 / 11.5, but d = 162,400 (20) 12.3 / 11.9.
static bool bs_apply_is_short(const compams_context* c) {
    return c->tab.ntiles < std::min(4 * c->n_total, 96) && (c->n_total > 8 || c->tab.ntiles >= 16);
}

// Whether bs_apply adds up the tile sums itself, and bs_scales is not launched. Not between compams_compress and compams_apply (the
// messages have to be complete), and not where every CTA would read more sums than its share of the rest, one worker after the other
// by its eight warps. us per step without / with bs_scales: n = 8, d = 2^20 + 1 (129 tiles) 20.6 / 22.3, d = 1.5 M (184) 38.9 / 40.4, d = 2^21
// + 3 (257) 50.9 / 50.9; n = 16, d = 2^20 44.1 / 45.2, d = 1.5 M 66.4 / 65.5; more workers gain only where all blocks are small: n = 32,
// d = 750,007 in 150 blocks (6 tiles at most) 94.2 / 98.5, n = 17 in 40 blocks (21) 42.1 / 42.8, d = 1.5 M in 40 or 150 (34) 77.0 / 75.8
// and 88.0 / 87.9.
bool bs_apply_adds_up(const compams_context* c) {
    if (!c->whole_step || bs_apply_is_short(c)) return false;
    if (c->n <= 8) return c->bs_max_tiles <= kWarpTiles;
    if (c->n <= 2 * kWarps) return c->bs_max_tiles <= 160;
    return (int64_t)c->bs_max_tiles * c->n <= 512;
}

cudaError_t launch_bs_scales(compams_context* c) {
    dim3 grid((unsigned)c->M, (unsigned)c->n);
    if (c->tab.ntiles > 256 * (int64_t)c->M)  // on average more than 256 tiles to a block
        return counted(c, launch_after(bs_scales_kernel<1024>, grid, dim3(1024), c->stream, c->tab, own_rows(c)));
    return counted(c, launch_after(bs_scales_kernel<kThreads>, grid, dim3(kThreads), c->stream, c->tab, own_rows(c)));
}

cudaError_t launch_bs_apply(compams_context* c, float* theta) {
    BsBuffers b = c->bs;
    b.scales_cur = c->scales[c->scales_cur];
    Tables t = c->tab;
    t.n = c->n_total;  // the average runs over every worker's message
    const bool own = bs_apply_adds_up(c), is_short = bs_apply_is_short(c);
    const dim3 grid((unsigned)(c->tab.ntiles * (is_short ? kWarps : kTile / kApplySpan)));
    // (gbar stored or not is a template parameter: a run-time branch around the store slowed the kernel by a tenth)
    void (*kernel)(const Tables, const BsBuffers, float*, const HyperParams, const SegParams) =
        own ? (b.gbar ? bs_apply_kernel<true, true, false> : bs_apply_kernel<false, true, false>)
            : (b.gbar ? bs_apply_kernel<true, false, false> : bs_apply_kernel<false, false, false>);
    // more than 16 workers: one round for up to 32, and lookups without bank conflicts (9 to 16 workers: n = 16, ResNet-18 shapes
    // 406.5 without, 405.5 with, n = 12, d = 9 M 260.2 / 260.4)
    if (c->n_total > kApplyEights)
        kernel = own ? (b.gbar ? bs_apply_kernel<true, true, true> : bs_apply_kernel<false, true, true>)
                     : (b.gbar ? bs_apply_kernel<true, false, true> : bs_apply_kernel<false, false, true>);
    if (is_short)  // tables from 20 workers up: n = 16, d = 162,400 13.6 us with, 13.3 without, n = 32, d = 524,288 43.9 with, 45.8 without
        kernel = c->n_total >= 20 ? (b.gbar ? bs_apply_short_kernel<true, true> : bs_apply_short_kernel<true, false>)
                                  : (b.gbar ? bs_apply_short_kernel<false, true> : bs_apply_short_kernel<false, false>);
    if (c->whole_step) return counted(c, launch_after(kernel, grid, dim3(kThreads), c->stream, t, b, theta, c->hp, c->segp));
    // between compams_compress and compams_apply the caller may have put work on the stream that writes the messages, theta
    // or both, and the kernel reads theta ahead of its wait: a plain launch comes after that work
    kernel<<<grid, dim3(kThreads), 0, c->stream>>>(t, b, theta, c->hp, c->segp);
    return counted(c, cudaGetLastError());
}

cudaError_t launch_bs_materialize(compams_context* c) {
    dim3 grid((unsigned)c->tab.ntiles, (unsigned)c->n);
    bs_materialize_kernel<<<grid, kThreads, 0, c->stream>>>(c->tab, c->E, c->scales[c->scales_cur] + (size_t)c->row0 * (size_t)c->M);
    return counted(c, cudaGetLastError());
}

}  // namespace compams
