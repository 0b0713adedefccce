// Top-k path (Definition 1) of the COMP-AMS step: exact selection of the k_b largest magnitudes
// of every (worker, block), ties at the threshold going to the lower index.
//
// Keys are the fp32 bit patterns of x = g + e with the sign cleared (31 bits); selection is a
// most-significant-digit radix select over them.
//
//   Small problems: topk_fused - sweep and selection of one (worker, block) by one cluster, or one CTA.
//
//   Otherwise blocks of at most kSmallMax coordinates: topk_small - one CTA holds the block in shared
//   memory and does every radix pass there; E is written once. It runs beside the selection of the larger blocks.
//
//   Larger blocks, cut into tiles of kTile coordinates.
//   Candidate path (one pass over [n, d]), for blocks that keep at most 1/9 of their coordinates:
//     topk_sweep    x = g + e written over E (Algorithm 2, the corrected-gradient step); every key >= tau_hat, a threshold
//                   predicted from the previous step, is appended to the segment's candidate list
//     topk_select   if the list holds at least k_b and at most its capacity, the exact Top-k is inside it.
//                   A histogram of the key offsets above tau_hat (bins sized from the last step) finds
//                   the threshold bin; winners above it are emitted, the bin's few candidates are
//                   ordered by (key, lower index first), the best kept, and the next tau_hat predicted. One CTA or one
//                   thread-block cluster per list (select.cuh).
//     topk_emit     writes out the winners of lists so long that their clusters would take many rounds
//   A list that cannot decide: its cluster goes through the block itself (select.cuh), or the segment is marked for the
//   dense passes (exact for any input, e.g. all-equal values), one
//   cooperative kernel topk_dense whose stages are separated by grid-wide barriers:
//     hist<1..3> / find<1..3>  three histogram passes over x, 11 + 10 + 10 key bits
//     collect       keys above the threshold are emitted; threshold ties too unless only some fit,
//                   in which case they are counted per tile
//     ties          takes the lowest-index threshold ties, tile by tile in index order
//   In a whole step whoever emits an (index, value) pair also appends it to the bucket of its coordinate range for the server
//   kernel (the server's average); topk_scatter does that from the messages in compams_apply and after always dense selections.
//   The residual update at a kept coordinate (e = x - x = 0) is deferred: E keeps x there, and every selection
//   leaves one magnitude per segment such that the kept elements are exactly those with |x| at or above it;
//   whoever reads E next - the next sweep, or topk_materialize - treats them as 0. Where a selection cuts through
//   a group of equal magnitudes (some kept, some not), it zeroes the few kept ones in E itself and leaves the
//   next larger magnitude.
#include "context.h"
#include "predict.cuh"
#include "scatter.cuh"
#include "select.cuh"

namespace compams {

// ------------------------------------------------------------------------------------------
// tile addressing shared by the large-block kernels

// First of the 4 consecutive coordinates (relative to the block) that lane `lane` of warp `warp`
// handles at iteration `it` of a tile starting at r0.
__device__ __forceinline__ int lane_r(int r0, int warp, int it, int lane) {
    return r0 + warp * kWarpSpan + it * 128 + lane * 4;
}

// Loads the 32 values of this thread's share of a tile of x (already stored in E).
// Coordinates past the block end read as +0 (callers mask them).
__device__ __forceinline__ void load_x_tile(const float* __restrict__ e, int len, int r0, int warp, int lane,
                                            float4 (&xv)[kIters]) {
    const int ce = align_class(e);
    if (r0 + kTile <= len) {
#pragma unroll
        for (int it = 0; it < kIters; ++it) xv[it] = load4(e + lane_r(r0, warp, it, lane), ce);
    } else {
#pragma unroll
        for (int it = 0; it < kIters; ++it) {
            const int r = lane_r(r0, warp, it, lane);
            if (r + 3 < len) {
                xv[it] = load4(e + r, ce);
            } else {
                float tmp[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) tmp[k] = (r + k < len) ? e[r + k] : 0.0f;
                xv[it] = make_float4(tmp[0], tmp[1], tmp[2], tmp[3]);
            }
        }
    }
}

// ------------------------------------------------------------------------------------------
// sweep: x = g + e -> E; keys >= tau_hat go to the candidate list

// "Nothing kept": as a float this pattern is a NaN, which no magnitude reaches.
constexpr uint32_t kNothingKept = 0xffffffffu;

// A warp's candidates on their way to the list. MANY: of blocks that keep so many entries that most of a warp's
// elements would meet in the shared counter, so the slots come from ballots and the count stays in a register.
template <bool MANY>
struct Stage {
    static constexpr uint32_t kCap = MANY ? kWarpCandMany : kWarpCand;
    uint2* stage;
    uint32_t* staged;  // !MANY: the warp's counter in shared memory
    uint32_t* g_cnt;
    uint2* g_out;
    uint32_t cap, count;
    __device__ __forceinline__ void put(uint32_t slot, uint32_t coord, float x) {
        const uint2 cv = make_uint2(coord, __float_as_uint(x));
        if (slot < kCap) {
            stage[slot] = cv;
        } else {  // a stretch dense with candidates: the staging buffer is full, append directly
            const uint32_t p = atomicAdd(g_cnt, 1u);
            if (p < cap) g_out[p] = cv;
        }
    }
    // Called by the whole warp.
    __device__ __forceinline__ void add(bool is, uint32_t coord, float x) {
        if constexpr (MANY) {
            const unsigned m = __ballot_sync(0xffffffffu, is);
            if (is) put(count + (uint32_t)__popc(m & ((1u << (threadIdx.x & 31)) - 1u)), coord, x);
            count += (uint32_t)__popc(m);
        } else {
            if (is) put(atomicAdd(staged, 1u), coord, x);
        }
    }
};

// One tile of the sweep. The tile starts at r0 (relative to the block), which is the block's tile
// boundary shifted down to a 128-byte line of G and E: r0 may be negative and the tile may reach
// past the block; such coordinates are skipped.
// `kept_from`: elements of E whose magnitude is at or above it were kept by the last step's selection and still
// hold x; their e is 0 (one float comparison: the key order is the order of |x|).
template <bool FULL, typename GT, bool MANY>
__device__ __forceinline__ void topk_sweep_tile(const GT* __restrict__ g, float* __restrict__ e, int len, int r0,
                                                int warp, int lane, uint32_t tau_hat, uint32_t coord0,
                                                Stage<MANY>& stage, float kept_from) {
    const int cg_ = align_class(g + r0), ce = align_class(e + r0);
    constexpr int NB = 2;  // iterations whose loads are in flight together
#pragma unroll
    for (int bt = 0; bt < kIters / NB; ++bt) {
        float4 gv[NB], ev[NB];
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            const int r = lane_r(r0, warp, bt * NB + u, lane);
            if (FULL || (r >= 0 && r + 3 < len)) {
                gv[u] = load4_stream(g + r, cg_);
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
#pragma unroll
        for (int u = 0; u < NB; ++u) {
            const int r = lane_r(r0, warp, bt * NB + u, lane);
            float xs[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                // coordinates kept in the last step still hold x in E: their e is 0 (Algorithm 2, the residual update)
                const float eo = lane_elem(ev[u], k);
                const float ek = fabsf(eo) >= kept_from ? 0.0f : eo;
                xs[k] = __fadd_rn(lane_elem(gv[u], k), ek);  // the corrected-gradient step: x = g + e
                stage.add((FULL || (unsigned)(r + k) < (unsigned)len) && mag_key(xs[k]) >= tau_hat, coord0 + (uint32_t)(r + k), xs[k]);
            }
            if (FULL || (r >= 0 && r + 3 < len)) {
                store4(e + r, ce, make_float4(xs[0], xs[1], xs[2], xs[3]));
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if ((unsigned)(r + k) < (unsigned)len) e[r + k] = xs[k];
            }
        }
    }
}

// The same for bfloat16 gradients on a whole tile whose rows of G and E are 16-byte aligned: 8 coordinates per
// lane and iteration, so that the gradient load is 128 bits wide like the loads and stores of E (with 4
// coordinates per lane the 64-bit gradient loads leave too few bytes in flight). A warp's 1024 coordinates are
// 4 chunks of 256; the next chunk's loads are in flight while one is worked on.
template <bool MANY>
__device__ __forceinline__ void topk_sweep_tile_bf16x8(const bf16_bits* __restrict__ g, float* __restrict__ e, int r0,
                                                       int warp, int lane, uint32_t tau_hat, uint32_t coord0,
                                                       Stage<MANY>& stage, float kept_from) {
    constexpr int NC = kWarpSpan / 256;
    const int rw = r0 + warp * kWarpSpan;
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
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float xs[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t word = gw[h * 2 + (k >> 1)];
                const float gk = __uint_as_float((k & 1) ? (word & 0xffff0000u) : (word << 16));  // exact widening
                // coordinates kept in the last step still hold x in E: their e is 0 (Algorithm 2, the residual update)
                const float eo = lane_elem(ev[h], k);
                const float ek = fabsf(eo) >= kept_from ? 0.0f : eo;
                xs[k] = __fadd_rn(gk, ek);  // the corrected-gradient step: x = g + e
                stage.add(mag_key(xs[k]) >= tau_hat, coord0 + (uint32_t)(r + h * 4 + k), xs[k]);
            }
            *reinterpret_cast<float4*>(e + r + h * 4) = make_float4(xs[0], xs[1], xs[2], xs[3]);
        }
    }
}

// Tiles are shifted down by (i d + o) mod 32, the position of the block's first element within a
// 128-byte line of G and E, so that every warp access covers whole lines (with rows that start
// mid-line a warp's 512 bytes straddle five lines instead of four: measured 7 % slower).
template <typename GT, bool MANY>
__global__ void __launch_bounds__(kThreads, sizeof(GT) == 2 ? 5 : 4) topk_sweep_kernel(Tables t, TopkBuffers b, const GT* __restrict__ G,
                                                                 const __grid_constant__ SegParams sp_) {
    dependency_wait();   // launched as a programmatic dependent while n d <= kChainMaxElems: the kernel before must be done
    allow_dependents();  // ... and the next one may move in behind this one's last wave
    // every warp stages the candidates of its 1024 coordinates by itself: in the list they then lie together, and the
    // selection's warps meet few server buckets at a time
    __shared__ uint2 sh_stage[kWarps][Stage<MANY>::kCap];
    __shared__ uint32_t sh_staged[kWarps], sh_base;
    const TileInfo ti = sp_.nseg ? find_tile(sp_, blockIdx.x) : load_tile(t.tiles, blockIdx.x);
    const int i = blockIdx.y;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t sg = (size_t)i * t.nseg + ti.seg;
    SegState* st = b.seg + sg;
    const uint32_t tau_hat = st->tau_hat;
    const SegInfo* si = t.segs + ti.seg;
    const uint32_t cap = si->cap;
    uint2* out = b.cand + (size_t)i * (size_t)b.cand_total + (size_t)si->cand_off;
    Stage<MANY> stage{sh_stage[warp], &sh_staged[warp], &st->cand_count, out, cap, 0u};
    if (lane == 0) sh_staged[warp] = 0u;
    __syncwarp();
    const int64_t row0 = (int64_t)i * t.d + ti.o;
    const GT* g = G + row0;
    float* e = b.E + row0;
    const int r0s = ti.r0 - (int)(row0 & 31);
    const float kept_from = __uint_as_float(b.use_thr ? b.thr[sg] : kNothingKept);
    const bool whole = r0s >= 0 && r0s + kTile <= ti.len;
    // The tile's lines are asked into the L2 first: four CTAs per SM with registers to spare then do better than six that
    // spill (ResNet-18 shapes whole, n = 16, 0.1 %: step 395.9 -> 388.5 us; the prefetch with six CTAs 401.5, three 389.1;
    // with bfloat16 gradients 386 -> 392, so not there).
    if (sizeof(GT) == 4 && whole) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(e + r0s + warp * kWarpSpan + lane * 32));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(g + r0s + warp * kWarpSpan + lane * 32));
    }
    bool wide = false;
    if constexpr (sizeof(GT) == 2)
        wide = whole && ((reinterpret_cast<uintptr_t>(g + r0s) | reinterpret_cast<uintptr_t>(e + r0s)) & 15u) == 0;
    if (wide) {
        if constexpr (sizeof(GT) == 2)
            topk_sweep_tile_bf16x8(g, e, r0s, warp, lane, tau_hat, (uint32_t)ti.o, stage, kept_from);
    } else if (whole)
        topk_sweep_tile<true>(g, e, ti.len, r0s, warp, lane, tau_hat, (uint32_t)ti.o, stage, kept_from);
    else
        topk_sweep_tile<false>(g, e, ti.len, r0s, warp, lane, tau_hat, (uint32_t)ti.o, stage, kept_from);
    if (MANY && lane == 0) sh_staged[warp] = stage.count;
    __syncthreads();
    uint32_t before = 0, total = 0, mine = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        const uint32_t k = sh_staged[w] < Stage<MANY>::kCap ? sh_staged[w] : Stage<MANY>::kCap;
        if (w < warp) before += k;
        if (w == warp) mine = k;
        total += k;
    }
    if (total == 0u) return;
    if (threadIdx.x == 0) sh_base = atomicAdd(&st->cand_count, total);
    __syncthreads();
    const uint32_t base = sh_base + before;
    for (uint32_t k = lane; k < mine; k += 32)
        if (base + k < cap) out[base + k] = sh_stage[warp][k];
}

// ------------------------------------------------------------------------------------------
// select: exact Top-k inside the candidate list

// One cluster per (worker, block) decides the selection inside the candidate list (see select.cuh) and closes the
// segment. A list that cannot decide: the cluster goes through the block itself, or, where the block is too long for
// its few CTAs, leaves it to the dense passes of the whole GPU. Lists come longest first, every worker's copy of one
// block side by side: the clusters that take longest start first and the last wave holds the shortest.
// Two CTAs of 512 threads per SM, 64 registers: CTAs of 1024 threads were slower for many lists (ResNet-50 shapes layer-wise,
// n = 32: step 1760 -> 1800 us; n = 8, d = 2^20: 42 -> 54; a few that are only counted take them, see fit_topk_cluster), three CTAs
// of 512 at 40 registers faster layer-wise (1744) and slower for single lists (n = 4, d = 65,536: 17.5 -> 19.1).
constexpr int kSelThreads = 512;

template <int NT>
__device__ __forceinline__ void start_select(SelectShared<NT>& sh) {
    clear_hist<NT>(sh);
    if (threadIdx.x == 0) {
        sh.winners = 0u;
        sh.slots = 0u;
        sh.nsurv = 0u;
        sh.listed = 0u;
        sh.undecided = 0u;
    }
    __syncthreads();
}

// What a selection starts from, requested in one go.
struct SelectState {
    uint32_t c, tau_hat, boost;
    int S;
};
__device__ __forceinline__ SelectState load_state(const SegState* st) {
    SelectState s;
    s.c = st->cand_count;
    s.tau_hat = st->tau_hat;
    s.S = (int)st->sel_shift;
    s.boost = st->boost;
    return s;
}

__device__ __forceinline__ SelectJob select_job(const Tables& t, const TopkBuffers& b, const SegInfo& si, int i, bool deliver) {
    SelectJob job;
    job.idx = b.idx + (size_t)i * (size_t)b.K + (size_t)si.slot0;
    job.val = b.val + (size_t)i * (size_t)b.K + (size_t)si.slot0;
    job.erow = b.E + (size_t)i * (size_t)t.d;
    job.kb = si.kb;
    job.cap = si.cap;
    job.deliver = deliver;
    job.defer = false;
    return job;
}

// A block whose list of c candidates has not decided, for the reason `why`: by its group, or left to the dense passes. The
// block's description and state are fetched again, so that a list that decides need not keep them in registers. (As a function
// that is not inlined, around one that is not, it left the inner one too few registers: ResNet-18 shapes whole, n = 16, 1 %, the
// first step 2100 -> 2450 us.)
template <int NT>
__device__ __forceinline__ void select_without_list(Group grp, SelectShared<NT>& sh, const Tables& t, const TopkBuffers& b, int i, int seg,
                                                 uint32_t c, int why, bool deliver) {
    const SegInfo si = t.segs[seg];
    const size_t sg = (size_t)i * t.nseg + seg;
    SegState* st = b.seg + sg;
    const bool first = grp.rank == 0 && threadIdx.x == 0;
    const bool predicted = st->tau_hat != kNoPrediction;
    const uint32_t boost = st->boost;
    if (first && predicted && si.cap) atomicAdd(b.status + why, 1u);
    if ((int64_t)si.len <= (int64_t)b.cluster_max * grp.size) {
        grp.sync();  // the state has been read by all
        if (first && predicted && c < si.kb) margin_came_up_short(st);
        const SelectJob job = select_job(t, b, si, i, deliver);
        select_from_block<NT>(grp, b, job, sh, st, b.thr + sg, job.erow + si.o, (uint32_t)si.len, (uint32_t)si.o, si.cap != 0u, boost);
        if (grp.size > 1) cg::this_cluster().sync();
        return;
    }
    if (first) {
        st->fallback = 1u;
        atomicAdd(b.dense_count, 1u);
        if (predicted && c < si.kb) margin_came_up_short(st);
    }
}

// Called by all threads of the group. `state_read`: a barrier of the group lies between its CTAs' reads of `s` and this call.
template <int NT>
__device__ __forceinline__ void select_segment(Group grp, SelectShared<NT>& sh, const Tables& t, const TopkBuffers& b,
                                               const SegInfo& si, int i, int seg, const SelectState& s, bool state_read, bool deliver,
                                               bool defer) {
    const size_t sg = (size_t)i * t.nseg + seg;
    // the same decision in every CTA of the group: nobody writes these words before all have read them
    int why = s.c < si.kb ? 3 : 4;
    if (s.tau_hat != kNoPrediction && s.c >= si.kb && s.c <= si.cap) {
        // a short list: barriers of the cluster would cost more than the other CTAs save, the first takes it alone. They
        // wait for its verdict: a list that cannot decide needs all of them for the block.
        const bool by_first = grp.size > 1 && s.c <= (uint32_t)(ListSlice::kU * NT);
        // the first will leave the next step's state in the words that they decide by: all must have read them
        if (by_first && !state_read) grp.sync();
        bool decided = false;
        if (!by_first || grp.rank == 0) {
            SelectJob job = select_job(t, b, si, i, deliver);
            job.defer = defer && !by_first;
            const uint2* list = b.cand + (size_t)i * (size_t)b.cand_total + (size_t)si.cand_off;
            decided = select_from_list<NT>(by_first ? Group{1u, 0u} : grp, b, job, sh, b.seg + sg, b.thr + sg, list, s.c, s.tau_hat, s.S,
                                           s.boost, &why);
            if (by_first && !decided && threadIdx.x < grp.size) *grp.of(&sh.undecided, threadIdx.x) = 1u;
        }
        // the first CTA's shared memory stays until all have read from it
        if (grp.size > 1 && (by_first || decided)) cg::this_cluster().sync();
        if (by_first ? sh.undecided == 0u : decided) return;
    }
    select_without_list<NT>(grp, sh, t, b, i, seg, s.c, why, deliver);
}

// seg_list: `nlong` blocks that a cluster selects from, then `nshort` that one CTA does; a cluster's CTAs take as many
// of the latter as they are. `defer`: the long lists' entries are emitted by topk_emit. `early`: the next kernel is topk_small.
template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) topk_select_kernel(const __grid_constant__ Tables t,
                                                                   const __grid_constant__ TopkBuffers b,
                                                                   const int32_t* __restrict__ seg_list, int nlong, int nshort,
                                                                   int deliver, int defer, int early) {
    __shared__ SelectShared<NT> sh;
    Group grp{cg::this_cluster().num_blocks(), cg::this_cluster().block_rank()};
    unsigned item = blockIdx.x / grp.size;
    const unsigned longs = (unsigned)(t.n * nlong);
    const int32_t* segs = seg_list;
    const bool alone = item >= longs;
    if (alone) {
        item = (item - longs) * grp.size + grp.rank;
        segs += nlong;
        grp = Group{1u, 0u};
    }
    const int i = (int)(item % (unsigned)t.n);
    const unsigned q = item / (unsigned)t.n;
    const bool idle = alone && q >= (unsigned)nshort;
    const int seg = segs[idle ? 0u : q];  // the block tables are never written by a kernel
    const SegInfo si = t.segs[seg];
    start_select<NT>(sh);
    if (early) allow_dependents();  // topk_small needs nothing of the sweep's either (which has waited for everything before it)
    dependency_wait();   // launched as a programmatic dependent while n d <= kChainMaxElems: the kernel before must be done
    if (!early) allow_dependents();  // ... and the next one may move in behind this one's last wave
    if (idle) return;
    const SelectState s = load_state(b.seg + (size_t)i * t.nseg + seg);
    select_segment<NT>(grp, sh, t, b, si, i, seg, s, false, deliver != 0, defer != 0 && !alone);
}

// Sweep and selection in one kernel, for problems so small that launches and latency are what a step costs: a cluster, or one CTA, takes one (worker, block), forms x = g + e, lists the candidates and selects
// among them; blocks without a list are selected from directly. A warp takes 512 coordinates at a time, all loads of such
// a stretch in flight together, and its candidates get their places with one atomic.
constexpr int kSpan = 512;

template <bool FULL, typename GT>
__device__ __forceinline__ void fused_span(const GT* __restrict__ g, float* __restrict__ e, int len, int r0, int lane, uint32_t tau_hat,
                                           float kept_from, uint32_t coord0, uint32_t* listed, uint2* out, uint32_t cap) {
    constexpr int NI = kSpan / 128;
    const int cg_ = align_class(g + r0), ce = align_class(e + r0);
    float4 gv[NI], x[NI];
#pragma unroll
    for (int u = 0; u < NI; ++u) {
        const int r = r0 + u * 128 + lane * 4;
        if (FULL || (r >= 0 && r + 3 < len)) {
            gv[u] = load4_stream(g + r, cg_);
            x[u] = load4(e + r, ce);
        } else {
            float gt[4], et[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const bool live = (unsigned)(r + k) < (unsigned)len;
                gt[k] = live ? load1_stream(g + r + k) : 0.0f;
                et[k] = live ? e[r + k] : 0.0f;
            }
            gv[u] = make_float4(gt[0], gt[1], gt[2], gt[3]);
            x[u] = make_float4(et[0], et[1], et[2], et[3]);
        }
    }
    // coordinates kept in the last step still hold x in E: their e is 0 (Algorithm 2, the residual update)
    auto corrected = [&](float gk, float eo) { return __fadd_rn(gk, fabsf(eo) >= kept_from ? 0.0f : eo); };
    auto is = [&](int u, int k) {
        const int r = r0 + u * 128 + lane * 4 + k;
        return (FULL || (unsigned)r < (unsigned)len) && mag_key(lane_elem(x[u], k)) >= tau_hat;
    };
    uint32_t total = 0;
#pragma unroll
    for (int u = 0; u < NI; ++u) {
        const int r = r0 + u * 128 + lane * 4;
        x[u] = make_float4(corrected(gv[u].x, x[u].x), corrected(gv[u].y, x[u].y), corrected(gv[u].z, x[u].z),
                           corrected(gv[u].w, x[u].w));  // the corrected-gradient step: x = g + e
        if (FULL || (r >= 0 && r + 3 < len)) {
            store4(e + r, ce, x[u]);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if ((unsigned)(r + k) < (unsigned)len) e[r + k] = lane_elem(x[u], k);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) total += (uint32_t)__popc(__ballot_sync(0xffffffffu, is(u, k)));
    }
    if (total == 0u) return;
    uint32_t base = 0;
    if (lane == 0) base = atomicAdd(listed, total);
    base = __shfl_sync(0xffffffffu, base, 0);
#pragma unroll
    for (int u = 0; u < NI; ++u) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const bool c = is(u, k);
            const unsigned m = __ballot_sync(0xffffffffu, c);
            const uint32_t p = base + (uint32_t)__popc(m & ((1u << lane) - 1u));
            if (c && p < cap) out[p] = make_uint2(coord0 + (uint32_t)(r0 + u * 128 + lane * 4 + k), __float_as_uint(lane_elem(x[u], k)));
            base += (uint32_t)__popc(m);
        }
    }
}

template <typename GT>
__global__ void __launch_bounds__(kSelThreads, 2) topk_fused_kernel(const __grid_constant__ Tables t,
                                                                           const __grid_constant__ TopkBuffers b,
                                                                           const GT* __restrict__ G,
                                                                           const int32_t* __restrict__ seg_list, int nlong, int nshort,
                                                                           int deliver) {
    constexpr int NT = kSelThreads;
    __shared__ SelectShared<NT> sh;
    Group grp{cg::this_cluster().num_blocks(), cg::this_cluster().block_rank()};
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned item = blockIdx.x / grp.size;
    const unsigned longs = (unsigned)(t.n * nlong);
    const int32_t* segs = seg_list;
    const bool alone = item >= longs;
    if (alone) {
        item = (item - longs) * grp.size + grp.rank;
        segs += nlong;
        grp = Group{1u, 0u};
    }
    const int i = (int)(item % (unsigned)t.n);
    const unsigned q = item / (unsigned)t.n;
    const bool idle = alone && q >= (unsigned)nshort;
    const int seg = segs[idle ? 0u : q];  // the block tables are never written by a kernel
    const SegInfo si = t.segs[seg];
    const size_t sg = (size_t)i * t.nseg + seg;
    start_select<NT>(sh);
    dependency_wait();
    allow_dependents();
    if (idle) return;
    SelectState s = load_state(b.seg + sg);
    const float kept_from = __uint_as_float(b.use_thr ? b.thr[sg] : kNothingKept);
    const int64_t row0 = (int64_t)i * t.d + si.o;
    const GT* g = G + row0;
    float* e = b.E + row0;
    uint2* out = b.cand + (size_t)i * (size_t)b.cand_total + (size_t)si.cand_off;
    grp.sync();  // the first CTA's counter is clear
    uint32_t* listed = grp.of(&sh.listed, 0);
    const int shift = (int)(row0 & 31);  // stretches start on 128-byte lines of G and E, as the sweep's tiles do
    const int spans = (si.len + shift + kSpan - 1) / kSpan;
    for (int u = warp * (int)grp.size + (int)grp.rank; u < spans; u += (int)grp.size * (NT / 32)) {
        const int r0 = u * kSpan - shift;
        if (r0 >= 0 && r0 + kSpan <= si.len)
            fused_span<true>(g, e, si.len, r0, lane, s.tau_hat, kept_from, (uint32_t)si.o, listed, out, si.cap);
        else
            fused_span<false>(g, e, si.len, r0, lane, s.tau_hat, kept_from, (uint32_t)si.o, listed, out, si.cap);
    }
    grp.sync();  // the list and x are complete
    s.c = *listed;
    select_segment<NT>(grp, sh, t, b, si, i, seg, s, true, deliver != 0, false);
}

// Emission of long lists that topk_select has found the threshold of: `parts` CTAs stream through each list, a round's winners
// take their message slots with one atomic, the threshold bin's entries are collected, and the CTA that comes last ranks them
// and closes the segment. A CTA is bound by its chain of dependent accesses - list, slots, stores - and a list by the few CTAs an
// SM holds: the first round's entries do not wait for the list's length, bucket slots and message slots are asked for together,
// and the counter that hands out the message slots counts the parts, too, so that no fence stands behind the stores (n = 8, d =
// 4.2 M, 10 %: this kernel 59.8 -> 50.0 us; n = 32, d = 2^27, 1 % 432 -> 409).
__global__ void __launch_bounds__(kThreads, 4) topk_emit_kernel(const __grid_constant__ Tables t, const __grid_constant__ TopkBuffers b,
                                                             const int32_t* __restrict__ seg_list, int nlong, int parts,
                                                             int deliver) {
    __shared__ uint2 surv[kSurvCap], few[kSurvCap];
    __shared__ uint32_t hist[kThreads], scratch[kWarps], sh_bin[2], sh_above, sh_in;
    __shared__ uint32_t sh_wins[kWarps], sh_first;
    __shared__ int is_last;
    // all lists' first parts first: the workers' entries of one coordinate range then reach its bucket close in time
    const unsigned lists = (unsigned)(t.n * nlong), item = blockIdx.x % lists, part = blockIdx.x / lists;
    const int i = (int)(item % (unsigned)t.n);
    const int seg = seg_list[item / (unsigned)t.n];
    const SegInfo si = t.segs[seg];
    const SelectJob job = select_job(t, b, si, i, deliver != 0);
    dependency_wait();
    allow_dependents();
    const size_t sg = (size_t)i * t.nseg + seg;
    SegState* st = b.seg + sg;
    constexpr int U = ListSlice::kU;
    ListSlice sl;
    sl.list = b.cand + (size_t)i * (size_t)b.cand_total + (size_t)si.cand_off;
    sl.lo = 0u;
    // The first round's loads do not wait for the count. Parts are as many as the longest list has: those of a shorter list read past
    // its end, within its room, which costs nothing that shows (us per step without any early load / so / up to the expected length:
    // n = 8, 10 % of 6 M and 12 x 250,000 320.5 / 310.2 / 310.2; n = 4, 5 % of 20 M and 12 x 1.2 M 545 / 535 / 535; n = 2, 3 % of 16, 8, 4, 2, 1
    // and 0.5 M 366 / 358 / 362).
    sl.hi = si.cap;
    uint2 cv[U];
    uint32_t p0 = part * (U * kThreads);
    sl.load<kThreads>(p0, cv);
    const uint32_t c = st->emit_n;
    if (c == 0u) return;  // decided otherwise (the same word for every part: it changes when the last one is done)
    const uint32_t win_from = st->emit_from, bin_from = st->prefix;
    uint2* gsurv = b.sel_surv + (size_t)item * kSurvCap;
    uint32_t* nsurv = b.sel_ticket + 4 * item;
    unsigned long long* ticket = reinterpret_cast<unsigned long long*>(nsurv + 2);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    sl.hi = c;
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (p0 + u * kThreads + threadIdx.x >= c) cv[u] = make_uint2(0u, kNoCandidate);
    for (;;) {
        const uint32_t next = p0 + (uint32_t)parts * (U * kThreads);
        const bool more = p0 < c && next < c;
        unsigned wins[U];
        uint32_t warp_wins = 0;
        bool any = false;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const bool valid = cv[u].y != kNoCandidate;
            const uint32_t key = cv[u].y & 0x7fffffffu;
            wins[u] = __ballot_sync(0xffffffffu, valid && key >= win_from);
            warp_wins += (uint32_t)__popc(wins[u]);
            any = any || (valid && key >= bin_from && key < win_from);
        }
        if (__any_sync(0xffffffffu, any)) {
            put_survivors<U>(cv, gsurv, nsurv, win_from, bin_from);
            __threadfence();  // there before this CTA's ticket
        }
        // bucket slots and message slots (a round's with one atomic on the list's counter; one per warp: n = 3, d = 117 M, 3.95 %
        // 1573 us against 1496; n = 8, d = 4.2 M, 10 % 163.9 against 162.5) are asked for together
        RunSlots<U> slots;
        if (job.deliver && warp_wins) slots.ask(b, wins, cv);
        if (lane == 0) sh_wins[warp] = warp_wins;
        __syncthreads();
        if (threadIdx.x == 0) {
            uint32_t total = 0;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) total += sh_wins[w];
            // one word: message slots taken, and parts whose last round this is (their entries of the threshold bin are there)
            const unsigned long long old = atomicAdd(ticket, (more ? 0ull : 1ull << 32) + total);
            sh_first = (uint32_t)old;
            is_last = !more && (uint32_t)(old >> 32) == (uint32_t)(parts - 1);
            if (is_last) sh_above = (uint32_t)old + total;  // all slots
        }
        __syncthreads();
        uint32_t slot = sh_first;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) slot += w < warp ? sh_wins[w] : 0u;
        if (warp_wins) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if ((wins[u] >> lane) & 1u) put_pair(b, job, slot + (uint32_t)__popc(wins[u] & ((1u << lane) - 1u)), cv[u].x, cv[u].y);
                slot += (uint32_t)__popc(wins[u]);
            }
            if (job.deliver) slots.put(b, wins, cv);
        }
        if (!more) break;
        p0 = next;
        sl.load<kThreads>(p0, cv);
        __syncthreads();  // the counts have been read
    }
    if (!is_last) return;
    __threadfence();
    // put_survivors counts past kSurvCap but stores no more (topk_select defers no list with more in its threshold bin)
    const uint32_t in_bin = __ldcg(nsurv);
    uint32_t k_rem = st->k_rem, count = k_rem ? (in_bin < (uint32_t)kSurvCap ? in_bin : (uint32_t)kSurvCap) : 0u;
    if (in_bin > (uint32_t)kSurvCap && threadIdx.x == 0) atomicOr(b.status, 1u);
    const uint32_t wins = job.kb - k_rem, taken = sh_above;
    __syncthreads();
    for (uint32_t q = threadIdx.x; q < count; q += kThreads) surv[q] = __ldcg(gsurv + q);
    if (threadIdx.x == 0) sh_bin[0] = sh_bin[1] = sh_above = sh_in = 0u;
    hist[threadIdx.x] = 0u;
    __syncthreads();
    const uint2* last = surv;
    if (count > 64u) {
        // too many for one CTA to rank one against the other: a histogram of 256 bins leaves the few that share a bin
        static_assert(kThreads == 256, "one histogram bin per thread");
        const uint32_t width = win_from - bin_from;
        const int s = width > 256u ? 24 - __clz(width - 1u) : 0;
        for (uint32_t q = threadIdx.x; q < count; q += kThreads) atomicAdd(&hist[((surv[q].y & 0x7fffffffu) - bin_from) >> s], 1u);
        __syncthreads();
        const uint32_t in = hist[255 - threadIdx.x];  // from the top bin down
        uint32_t total;
        const uint32_t incl = block_inclusive_scan(in, scratch, &total);
        if (incl - in < k_rem && k_rem <= incl) {
            sh_bin[0] = 255u - threadIdx.x;
            sh_bin[1] = incl - in;
        }
        __syncthreads();
        for (uint32_t q = threadIdx.x; q < count; q += kThreads) {
            const uint2 cv = surv[q];
            const uint32_t dg = ((cv.y & 0x7fffffffu) - bin_from) >> s;
            if (dg > sh_bin[0]) {
                put_pair(b, job, wins + atomicAdd(&sh_above, 1u), cv.x, cv.y);
                if (job.deliver) scatter_one(b, (int32_t)cv.x, cv.y);
                job.erow[cv.x] = 0.0f;  // the residual of a kept coordinate: e = x - x
            } else if (dg == sh_bin[0]) {
                few[atomicAdd(&sh_in, 1u)] = cv;
            }
        }
        __syncthreads();
        k_rem -= sh_bin[1];
        count = sh_in;
        last = few;
    }
    uint32_t tau = bin_from;
    bool closer = threadIdx.x == 0 && wins == job.kb;
    if (wins != job.kb) closer = rank_survivors(b, job, last, count, k_rem, threadIdx.x >> 5, kWarps, &tau);
    if (closer) {
        if (taken != wins) atomicOr(b.status, 1u);
        st->emit_n = 0u;
        nsurv[0] = 0u;
        *ticket = 0ull;
        close_list(b, job, st, b.thr + sg, wins != job.kb ? tau + 1u : win_from, tau, st->edge, c, st->tau_hat);
    }
}

// ------------------------------------------------------------------------------------------
// dense passes, only for segments marked `fallback`

template <int PASS>
__device__ __forceinline__ void dense_hist(const Tables& t, const TopkBuffers& b, uint32_t* sh) {
    constexpr int NB = (PASS == 1) ? kBins1 : kBins23;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t total = (int64_t)t.n * t.ntiles;
    for (int64_t w = blockIdx.x; w < total; w += gridDim.x) {
        const int i = (int)(w / t.ntiles);
        const TileInfo ti = load_tile(t.tiles, (int)(w % t.ntiles));
        const size_t sg = (size_t)i * t.nseg + ti.seg;
        if (b.seg[sg].fallback == 0u) continue;
        const uint32_t prefix = b.seg[sg].prefix;
        for (int k = threadIdx.x; k < NB; k += kThreads) sh[k] = 0u;
        __syncthreads();
        const float* e = b.E + (size_t)i * (size_t)t.d + (size_t)ti.o;
        float4 xv[kIters];
        load_x_tile(e, ti.len, ti.r0, warp, lane, xv);
        int any = 0;
#pragma unroll
        for (int it = 0; it < kIters; ++it) {
            const int r = lane_r(ti.r0, warp, it, lane);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t key = mag_key(lane_elem(xv[it], k));
                const bool match = (PASS == 1) ? true : (PASS == 2) ? ((key >> 20) == prefix) : ((key >> 10) == prefix);
                if (match && r + k < ti.len) {
                    atomicAdd(&sh[(PASS == 1) ? (key >> 20) : (PASS == 2) ? ((key >> 10) & 1023u) : (key & 1023u)], 1u);
                    any = 1;
                }
            }
        }
        if (__syncthreads_or(any)) {
            uint32_t* h = b.hist + sg * kBins1;
            for (int k = threadIdx.x; k < NB; k += kThreads) {
                const uint32_t v = sh[k];
                if (v) atomicAdd(h + k, v);
            }
        }
        __syncthreads();
    }
}

constexpr int kLowBins = 64;  // fine bins at the bottom of the threshold's pass-1 bin that give the density there

template <int NBINS, int BITS, int PASS>
__device__ __forceinline__ void dense_find(const Tables& t, const TopkBuffers& b, size_t sg, uint32_t* scratch) {
    constexpr int PER = NBINS / kThreads;
    SegState* st = b.seg + sg;
    if (st->fallback == 0u) return;
    const SegInfo* si = t.segs + (sg % (size_t)t.nseg);
    uint32_t* h = b.hist + sg * kBins1;
    const uint32_t kb = si->kb;
    const uint32_t k_rem = (PASS == 1) ? kb : st->k_rem;
    const uint32_t prefix = (PASS == 1) ? 0u : st->prefix;
    // thread t owns the PER bins NBINS-1-t*PER ... downwards, so a scan over threads runs from the top bin down
    uint32_t cnt[PER];
    uint32_t sum = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int bin = NBINS - 1 - ((int)threadIdx.x * PER + j);
        cnt[j] = h[bin];
        h[bin] = 0u;  // leave the histogram clean for the next pass / next step
        sum += cnt[j];
    }
    uint32_t total;
    const uint32_t incl = block_inclusive_scan(sum, scratch, &total);
    const uint32_t excl = incl - sum;
    if (excl < k_rem && k_rem <= incl) {
        uint32_t running = excl;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            if (running < k_rem && k_rem <= running + cnt[j]) {
                const uint32_t bin = (uint32_t)(NBINS - 1 - ((int)threadIdx.x * PER + j));
                const uint32_t np = (prefix << BITS) | bin;
                const uint32_t nk = k_rem - running;
                st->prefix = np;
                st->k_rem = nk;
                if (PASS == 3) {
                    // every key above np is kept, and the ties at np too unless only some fit: then the walk over
                    // the ties zeroes in E the ones it takes and everything from the next key up counts as kept
                    b.thr[sg] = (nk < cnt[j]) ? np + 1u : np;
                    st->tau = np;
                    st->ties_take = nk;
                    st->need_order = (nk < cnt[j]) ? 1u : 0u;
                    // prediction for the next step's sweep (blocks without a candidate buffer never predict)
                    predict_next(st, np, st->edge, si->cap != 0u);
                }
            }
            running += cnt[j];
        }
    }
    if (PASS == 1) {
        // the highest pass-1 bin edge at or above which at least the wanted number of candidates lie (0 if there
        // are fewer); a candidate path that gave up may have handed out message slots: start over
        const uint32_t want = want_candidates(kb, st->boost, si->cap);
        if (threadIdx.x == 0) {
            st->emit_count = 0u;
            if (total < want) st->edge = 0u;
        }
        if (excl < want && want <= incl) {
            uint32_t running = excl;
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                if (running < want && want <= running + cnt[j])
                    st->edge = (uint32_t)(NBINS - 1 - ((int)threadIdx.x * PER + j)) << 20;
                running += cnt[j];
            }
        }
    }
    if constexpr (PASS == 2) {
        // Pass 1 places that edge on a grid of an eighth of a binade. Under error feedback the magnitudes pile up
        // just below the threshold (a coordinate grows until it is kept), so a bin edge a few per cent below the
        // threshold can let through many times the wanted number, more than the list holds, and the segment came
        // back to the dense passes step after step. When the wanted number is reached inside the threshold's own
        // pass-1 bin, this pass places the edge 1024 times finer; when that bin and the bins above hold fewer than
        // wanted, the edge is extrapolated below the bin's lower edge (see there).
        const uint32_t want = want_candidates(kb, st->boost, si->cap);
        const uint32_t above = kb - k_rem;     // keys in the pass-1 bins above the threshold's
        const uint32_t want2 = want - above;   // want > kb > above
        if (excl < want2 && want2 <= incl) {
            uint32_t running = excl;
#pragma unroll
            for (int j = 0; j < PER; ++j) {
                if (running < want2 && want2 <= running + cnt[j])
                    st->edge = (prefix << 20) | ((uint32_t)(NBINS - 1 - ((int)threadIdx.x * PER + j)) << 10);
                running += cnt[j];
            }
        } else if (total < want2 && threadIdx.x == kThreads - 1 - kLowBins / PER) {
            // The wanted count is reached below the threshold's pass-1 bin (the threshold sits just above a bin
            // boundary): the edge goes below the boundary by as far as the missing candidates need at the density
            // of the bin's lowest kLowBins fine bins. Further down the density only grows, so at least the wanted
            // number comes through, and far fewer than down to the next boundary. This thread's bins end where
            // those fine bins begin: `incl` counts everything above them.
            const uint32_t low = total - incl;
            if (low) {
                const unsigned long long ext = (unsigned long long)(want2 - total) * ((unsigned long long)kLowBins << 10) / low;
                const uint32_t top = prefix << 20;
                const uint32_t fine = ext < (unsigned long long)top ? top - (uint32_t)ext : 0u;
                if (fine > st->edge) st->edge = fine;  // never below the pass-1 edge, which is known to suffice
            }
        }
    }
    if (threadIdx.x == 0 && total < k_rem) atomicOr(b.status, 2u);
}

__device__ __forceinline__ void dense_collect(const Tables& t, const TopkBuffers& b, uint32_t* scratch,
                                              uint32_t* sh_base_p, bool deliver) {
    uint32_t& sh_base = *sh_base_p;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t total = (int64_t)t.n * t.ntiles;
    for (int64_t w = blockIdx.x; w < total; w += gridDim.x) {
        const int i = (int)(w / t.ntiles);
        const int tile = (int)(w % t.ntiles);
        const TileInfo ti = load_tile(t.tiles, tile);
        const size_t sg = (size_t)i * t.nseg + ti.seg;
        SegState* st = b.seg + sg;
        if (st->fallback == 0u) continue;
        const uint32_t tau = st->tau;
        const bool need_order = st->need_order != 0u;
        const float* e = b.E + (size_t)i * (size_t)t.d + (size_t)ti.o;
        float4 xv[kIters];
        load_x_tile(e, ti.len, ti.r0, warp, lane, xv);
        uint32_t n_emit = 0, n_tie = 0;
#pragma unroll
        for (int it = 0; it < kIters; ++it) {
            const int r = lane_r(ti.r0, warp, it, lane);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t key = mag_key(lane_elem(xv[it], k));
                const bool live = r + k < ti.len;
                n_emit += (live && key > tau) ? 1u : 0u;
                n_tie += (live && key == tau) ? 1u : 0u;
            }
        }
        if (!need_order) n_emit += n_tie;
        uint32_t tot, tie_tot = 0;
        const uint32_t incl = block_inclusive_scan(n_emit, scratch, &tot);
        if (need_order) {
            block_inclusive_scan(n_tie, scratch, &tie_tot);
            if (threadIdx.x == 0) b.tile_ties[(size_t)i * t.ntiles + tile] = tie_tot;
        }
        if (tot) {
            if (threadIdx.x == 0) sh_base = atomicAdd(&st->emit_count, tot);
            __syncthreads();
            const SegInfo* si = t.segs + ti.seg;
            const uint32_t kb = si->kb;
            const size_t slot0 = (size_t)i * (size_t)b.K + (size_t)si->slot0;
            uint32_t pos = sh_base + (incl - n_emit);
#pragma unroll
            for (int it = 0; it < kIters; ++it) {
                const int r = lane_r(ti.r0, warp, it, lane);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float x = lane_elem(xv[it], k);
                    const uint32_t key = mag_key(x);
                    const bool live = r + k < ti.len;
                    if (live && (key > tau || (!need_order && key == tau))) {
                        if (pos < kb) {
                            b.idx[slot0 + pos] = (int32_t)(ti.o + r + k);
                            b.val[slot0 + pos] = x;
                            if (deliver) scatter_one(b, (int32_t)(ti.o + r + k), __float_as_uint(x));
                        } else {
                            atomicOr(b.status, 1u);
                        }
                        ++pos;
                    }
                }
            }
        }
        __syncthreads();  // sh_base and scratch are reused by the next tile
    }
}

// When the dense passes left threshold ties to order, takes those with the lowest index, tile by
// tile. The ties land in the message slots after the `emit_count` winners; the count itself is
// checked (with the ties added) when the step is closed.
__device__ __forceinline__ void dense_ties(const Tables& t, const TopkBuffers& b, size_t sg, uint32_t* scratch,
                                           uint32_t* sh_c, uint32_t* sh_excl, bool deliver) {
    const int i = (int)(sg / (size_t)t.nseg);
    const SegInfo* si = t.segs + (sg % (size_t)t.nseg);
    const SegState* st = b.seg + sg;
    if (st->fallback == 0u || st->need_order == 0u) return;
    const uint32_t kb = si->kb;
    const uint32_t emitted = st->emit_count;
    const uint32_t tau = st->tau;
    const uint32_t want = st->ties_take;
    if (emitted + want != kb) return;  // inconsistent: reported when the step is closed
    const int tile0 = si->tile0, tile_end = si->tile0 + si->ntile_b;
    const int64_t o = si->o;
    const int len = si->len;
    float* e = b.E + (size_t)i * (size_t)t.d + (size_t)o;
    const size_t slot0 = (size_t)i * (size_t)b.K + (size_t)si->slot0;
    uint32_t taken = 0;  // ties already assigned to earlier tiles (uniform across the CTA)
    for (int tb = tile0; tb < tile_end && taken < want; tb += kThreads) {
        const int tt = tb + (int)threadIdx.x;
        const uint32_t c = (tt < tile_end) ? b.tile_ties[(size_t)i * t.ntiles + tt] : 0u;
        uint32_t batch_total;
        const uint32_t incl = block_inclusive_scan(c, scratch, &batch_total);
        sh_c[threadIdx.x] = c;
        sh_excl[threadIdx.x] = incl - c;
        __syncthreads();
        const int nb = (tile_end - tb < kThreads) ? tile_end - tb : kThreads;
        for (int q = 0; q < nb; ++q) {
            const uint32_t cq = sh_c[q];
            if (cq == 0u) continue;
            const uint32_t before = taken + sh_excl[q];
            if (before >= want) break;
            const uint32_t take = (cq < want - before) ? cq : want - before;
            // tile tb+q in index order: thread j owns the 32 consecutive coordinates r0 + 32 j ...
            const int rs = (tb + q - tile0) * kTile + (int)threadIdx.x * 32;
            uint32_t mine = 0;
            for (int k = 0; k < 32; ++k) {
                const int r = rs + k;
                if (r < len && mag_key(e[r]) == tau) mine |= 1u << k;
            }
            uint32_t tile_tot;
            uint32_t rank = block_inclusive_scan((uint32_t)__popc(mine), scratch, &tile_tot) - __popc(mine);
            while (mine && rank < take) {
                const int k = __ffs(mine) - 1;
                mine &= mine - 1;
                const int r = rs + k;
                const uint32_t pos = emitted + before + rank;
                if (pos < kb) {
                    b.idx[slot0 + pos] = (int32_t)(o + r);
                    b.val[slot0 + pos] = e[r];
                    if (deliver) scatter_one(b, (int32_t)(o + r), __float_as_uint(e[r]));
                }
                e[r] = 0.0f;  // the residual of a kept coordinate: e = x - x (this thread alone reads and writes e[r])
                ++rank;
            }
            __syncthreads();
        }
        taken += batch_total;
        __syncthreads();
    }
    if (threadIdx.x == 0 && taken < want) atomicOr(b.status, 1u);
}

// Closes the step for a segment that the dense passes decided: exactly k_b entries must have been emitted; the
// counters go back to their resting values.
__device__ __forceinline__ void close_segment(const TopkBuffers& b, const SegInfo* si, SegState* st) {
    const uint32_t ties = st->need_order ? st->ties_take : 0u;
    if (st->emit_count + ties != si->kb) atomicOr(b.status, 1u);
    atomicAdd(b.status + 1, 1u);                // selections decided by passes over the block
    if (si->cap) atomicSub(b.dense_count, 1u);  // back to the number of blocks that are always selected here
    st->emit_count = 0u;
    st->cand_count = 0u;
    st->fallback = si->cap ? 0u : 1u;  // a block without a list that came here always does
    st->need_order = 0u;
}

// All dense passes in one cooperative launch: the grid is resident as a whole and the passes are
// separated by grid-wide barriers. When no segment is marked every CTA returns at once, so in the
// steady state the dense path costs one empty launch per step, where it is launched at all.
__global__ void __launch_bounds__(kThreads) topk_dense_kernel(Tables t, TopkBuffers b, int deliver) {
    __shared__ uint32_t sh[kBins1];
    __shared__ uint32_t scratch[kWarps];
    __shared__ uint32_t sh_c[kThreads], sh_excl[kThreads];
    __shared__ uint32_t sh_base;
    // the same word for every CTA; it only changes after the last barrier
    if (*b.dense_count == 0u) return;
    cg::grid_group grid = cg::this_grid();
    const size_t nsg = (size_t)t.n * (size_t)t.nseg;
    dense_hist<1>(t, b, sh);
    grid.sync();
    for (size_t sg = blockIdx.x; sg < nsg; sg += gridDim.x) {
        dense_find<kBins1, 11, 1>(t, b, sg, scratch);
        __syncthreads();
    }
    grid.sync();
    dense_hist<2>(t, b, sh);
    grid.sync();
    for (size_t sg = blockIdx.x; sg < nsg; sg += gridDim.x) {
        dense_find<kBins23, 10, 2>(t, b, sg, scratch);
        __syncthreads();
    }
    grid.sync();
    dense_hist<3>(t, b, sh);
    grid.sync();
    for (size_t sg = blockIdx.x; sg < nsg; sg += gridDim.x) {
        dense_find<kBins23, 10, 3>(t, b, sg, scratch);
        __syncthreads();
    }
    grid.sync();
    dense_collect(t, b, scratch, &sh_base, deliver != 0);
    grid.sync();
    for (size_t sg = blockIdx.x; sg < nsg; sg += gridDim.x) {
        dense_ties(t, b, sg, scratch, sh_c, sh_excl, deliver != 0);
        __syncthreads();
        if (threadIdx.x == 0 && b.seg[sg].fallback) close_segment(b, t.segs + (sg % (size_t)t.nseg), b.seg + sg);
    }
}

// ------------------------------------------------------------------------------------------
// small blocks: the whole selection inside one CTA's shared memory

template <typename GT>
__global__ void __launch_bounds__(kThreads) topk_small_kernel(Tables t, TopkBuffers b, const GT* __restrict__ G, int deliver,
                                                              int after_sweep) {
    __shared__ uint32_t xs[kSmallMax];
    __shared__ uint32_t hist[256];
    __shared__ uint32_t scratch[kWarps];
    __shared__ uint32_t sh_prefix, sh_krem, sh_cnt, sh_rlast, sh_taken;
    // Shares no block with the sweep and the selection: its CTAs move in behind the last wave of the kernel before it, which comes
    // after a sweep that has ordered itself after everything earlier on the stream, and wait for that kernel only at their end, for
    // the sake of the kernel after.
    if (!after_sweep) dependency_wait();
    allow_dependents();
    const int blk = b.small_blk[blockIdx.x];
    const int i = blockIdx.y, lane = threadIdx.x & 31;
    const int64_t o = t.off[blk];
    const int len = (int)(t.off[blk + 1] - o);
    const uint32_t kb = (uint32_t)(b.seg_off[blk + 1] - b.seg_off[blk]);
    const GT* g = G + (size_t)i * (size_t)t.d + (size_t)o;
    float* e = b.E + (size_t)i * (size_t)t.d + (size_t)o;
    for (int r = threadIdx.x; r < len; r += kThreads) xs[r] = __float_as_uint(__fadd_rn(load1_l2(g + r), __ldcg(e + r)));

    // radix select over the 31-bit key: digits of 8, 8, 8 and 7 bits from the top
    uint32_t prefix = 0, k_rem = kb;
    int shift = 31;         // bits below `shift` are still undecided
    bool take_all = false;  // every key in the chosen bin is kept: no tie to break
#pragma unroll 1
    for (int pass = 0; pass < 4 && !take_all; ++pass) {
        const int width = (pass == 3) ? 7 : 8;
        const int nshift = shift - width;
        hist[threadIdx.x] = 0u;
        __syncthreads();
        for (int r = threadIdx.x; r < len; r += kThreads) {
            const uint32_t key = xs[r] & 0x7fffffffu;
            if (pass == 0 || (key >> shift) == prefix) atomicAdd(&hist[(key >> nshift) & ((1u << width) - 1u)], 1u);
        }
        __syncthreads();
        const uint32_t c = hist[255 - threadIdx.x];  // scan from the top bin down
        uint32_t total;
        const uint32_t incl = block_inclusive_scan(c, scratch, &total);
        const uint32_t excl = incl - c;
        if (excl < k_rem && k_rem <= incl) {
            sh_prefix = (prefix << width) | (uint32_t)(255 - threadIdx.x);
            sh_krem = k_rem - excl;
            sh_cnt = c;
        }
        __syncthreads();
        prefix = sh_prefix;
        k_rem = sh_krem;
        take_all = (sh_cnt == k_rem);
        shift = nshift;
        __syncthreads();
    }
    // kept: key >> shift > prefix, or == prefix and (take_all, or among the first k_rem such keys by index)
    const int chunk = (len + kThreads - 1) / kThreads;
    const int lo = (int)threadIdx.x * chunk;
    const int hi = (lo + chunk < len) ? lo + chunk : len;
    if (threadIdx.x == 0) {
        sh_rlast = take_all ? 0x7fffffffu : 0u;
        sh_taken = 0u;
    }
    __syncthreads();
    if (!take_all) {
        uint32_t mine = 0;
        for (int r = lo; r < hi; ++r) mine += ((xs[r] & 0x7fffffffu) == prefix) ? 1u : 0u;  // shift == 0 here
        uint32_t total;
        uint32_t rank = block_inclusive_scan(mine, scratch, &total) - mine;
        for (int r = lo; r < hi; ++r) {
            if ((xs[r] & 0x7fffffffu) == prefix) {
                if (rank == k_rem - 1) sh_rlast = (uint32_t)r;
                ++rank;
            }
        }
        __syncthreads();
    }
    const uint32_t rlast = sh_rlast;
    auto kept = [&](int r) -> bool {
        const uint32_t top = (xs[r] & 0x7fffffffu) >> shift;
        return top > prefix || (top == prefix && (uint32_t)r <= rlast);
    };
    // Emission and residual in one pass, a warp taking 32 consecutive coordinates at a time: its kept entries share an atomic
    // for their message slots and one per server bucket they meet, and e = x - g~ is 0 where kept, x elsewhere (Algorithm 2,
    // the residual update). (With a stretch of coordinates and one atomic per kept entry per thread, n = 32, d = 65,536 in 70
    // blocks took 27 us at 0.1 % and 90 at 10 %.)
    const size_t slot0 = (size_t)i * (size_t)b.K + (size_t)b.seg_off[blk];
    constexpr int U = 4;
    for (int r0 = 0; r0 < len; r0 += U * kThreads) {
        unsigned take[U];
        uint2 cv[U];
        uint32_t rel[U], wins = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int r = r0 + u * kThreads + (int)threadIdx.x;
            const bool live = r < len;
            const bool mine = live && kept(r);
            cv[u] = make_uint2((uint32_t)(o + (live ? r : len - 1)), live ? xs[r] : 0u);
            if (live) e[r] = mine ? 0.0f : __uint_as_float(xs[r]);
            take[u] = __ballot_sync(0xffffffffu, mine);
            rel[u] = wins + (uint32_t)__popc(take[u] & ((1u << lane) - 1u));
            wins += (uint32_t)__popc(take[u]);
        }
        if (wins == 0u) continue;
        uint32_t pos = 0;
        if (lane == 0) pos = atomicAdd(&sh_taken, wins);
        pos = __shfl_sync(0xffffffffu, pos, 0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (((take[u] >> lane) & 1u) && pos + rel[u] < kb) {
                b.idx[slot0 + pos + rel[u]] = (int32_t)cv[u].x;
                b.val[slot0 + pos + rel[u]] = __uint_as_float(cv[u].y);
            }
        }
        if (deliver) scatter_runs<U>(b, take, cv);
    }
    __syncthreads();
    if (threadIdx.x == 0 && sh_taken != kb) atomicOr(b.status, 1u);
    if (after_sweep) dependency_wait();
}

// ------------------------------------------------------------------------------------------
// scatter: the kept (index, value) pairs of the messages are handed to the server grouped by coordinate range.

// All messages at once: `count` pairs of every worker the server averages over. For the messages that the selection did
// not deliver itself: those that compams_apply finds, and of handles whose blocks keep so many entries that the dense passes
// select them (their CTAs append entry by entry; here the lanes of a warp that meet in a bucket share one atomic).
__global__ void __launch_bounds__(kThreads) topk_scatter_kernel(TopkBuffers b, int64_t count) {
    dependency_wait();
    allow_dependents();
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool valid = p < count;
    int32_t j = 0;
    uint32_t xbits = 0;
    if (valid) {
        j = __ldg(b.idx + p);
        xbits = __float_as_uint(__ldg(b.val + p));
    }
    scatter_warp(b, valid, j, xbits);
}

// E holds x at the coordinates kept in the last step: zero them (Algorithm 2, the residual update). One CTA per
// (tile, worker); the kept elements of a segment are those whose magnitude reaches what its selection left.
__global__ void __launch_bounds__(kThreads) topk_materialize_kernel(Tables t, TopkBuffers b) {
    const int i = blockIdx.y;
    const TileInfo ti = load_tile(t.tiles, blockIdx.x);
    const float kept_from = __uint_as_float(b.thr[(size_t)i * t.nseg + ti.seg]);
    float* e = b.E + (size_t)i * (size_t)t.d + (size_t)ti.o;
    const int end = (ti.r0 + kTile < ti.len) ? ti.r0 + kTile : ti.len;
    for (int r = ti.r0 + (int)threadIdx.x; r < end; r += kThreads)
        if (fabsf(e[r]) >= kept_from) e[r] = 0.0f;
}

// ------------------------------------------------------------------------------------------

// The selection kernels see this handle's own rows of the message buffers; the server-side
// kernels see the rows of all n_total workers.
static TopkBuffers own_rows(const compams_context* c) {
    TopkBuffers b = c->tk;
    b.idx = c->tk.idx + (size_t)c->row0 * (size_t)c->K;
    b.val = c->tk.val + (size_t)c->row0 * (size_t)c->K;
    return b;
}

template <typename GT>
static cudaError_t launch_small_typed(compams_context* c, const GT* grads) {
    const dim3 grid((unsigned)c->tk.nsmall, (unsigned)c->n);
    return counted(c, launch_after(topk_small_kernel<GT>, grid, dim3(kThreads), c->stream, c->tab, own_rows(c), grads,
                                   delivers(c) ? 1 : 0, c->tab.ntiles > 0 ? 1 : 0));
}

cudaError_t launch_topk_small(compams_context* c, const void* grads) {
    return c->grad_bf16 ? launch_small_typed(c, (const bf16_bits*)grads) : launch_small_typed(c, (const float*)grads);
}

template <typename GT>
static cudaError_t launch_sweep_typed(compams_context* c, const GT* grads) {
    const dim3 grid((unsigned)c->tab.ntiles, (unsigned)c->n);
    void (*kernel)(Tables, TopkBuffers, const GT*, const SegParams) =
        c->many_candidates ? topk_sweep_kernel<GT, true> : topk_sweep_kernel<GT, false>;
    if (c->chain) return counted(c, launch_after(kernel, grid, dim3(kThreads), c->stream, c->tab, own_rows(c), grads, c->segp));
    kernel<<<grid, kThreads, 0, c->stream>>>(c->tab, own_rows(c), grads, c->segp);
    return counted(c, cudaGetLastError());
}

cudaError_t launch_topk_sweep(compams_context* c, const void* grads) {
    return c->grad_bf16 ? launch_sweep_typed(c, (const bf16_bits*)grads) : launch_sweep_typed(c, (const float*)grads);
}

// While n d <= kChainMaxElems the kernels of a step are launched as programmatic dependents of one another (each waits for its
// predecessor before it touches anything that a kernel of this step, or of the one before, may still write; topk_small, which
// shares no block with topk_sweep and topk_select, starts beside them and waits at its end, which is safe because the sweep's CTAs let
// the next kernel in only behind their own wait): the launch latency and the prologue of a
// kernel then overlap the tail of the one before, which is most of what such a step costs.

typedef void (*SelectKernel)(const Tables, const TopkBuffers, const int32_t*, int, int, int, int, int);

// Whether the device can hold a cluster of `cluster` CTAs of a kernel (more than 8 have to be asked for, once per kernel and
// device).
template <typename... KArgs>
static cudaError_t cluster_fits(void (*kernel)(KArgs...), int threads, int cluster, bool* fits) {
    if (cluster > 8) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cluster);
    cfg.blockDim = dim3((unsigned)threads);
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    *fits = cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters > 0;
    if (!*fits) cudaGetLastError();
    return cudaSuccess;
}

// The clusters were planned without a device, for 148 SMs in GPCs of at least 16. Where SMs are shared out (another process, a
// partition) and none of that size can be resident, smaller ones take over, each CTA with a larger share of the same blocks.
cudaError_t fit_topk_cluster(compams_context* c) {
    // As many long lists as there are GPCs for them, less one, that are only counted by topk_select: twice the threads per CTA
    // (512 / 1024 threads, us per step: d = 2^22, 10 %, n = 1 70.3 / 68.0, n = 5 122.5 / 119.7, n = 7 147.1 / 144.7, n = 8 160.7 / 168.7;
    // d = 9 M, 2 %, n = 1 100.0 / 98.7, n = 7 200.8 / 200.5, n = 8 217.3 / 225.1)
    c->sel_wide = c->sel_parts && c->sel_cluster == 16 && (int64_t)c->n * c->sel_long <= 7;
    const int planned = c->sel_cluster;
    bool fits = planned == 1;
    for (; !fits && c->sel_cluster > 1; c->sel_cluster /= fits ? 1 : 2) {
        cudaError_t e;
        if (c->fused) {
            bool bf16 = false;
            e = cluster_fits(topk_fused_kernel<float>, kSelThreads, c->sel_cluster, &fits);
            if (e == cudaSuccess) e = cluster_fits(topk_fused_kernel<bf16_bits>, kSelThreads, c->sel_cluster, &bf16);
            fits = fits && bf16;
        } else {
            e = cluster_fits(topk_select_kernel<kSelThreads>, kSelThreads, c->sel_cluster, &fits);
        }
        if (e != cudaSuccess) return e;
    }
    if (c->sel_wide && c->sel_cluster == planned) {
        const cudaError_t e = cluster_fits(topk_select_kernel<2 * kSelThreads>, 2 * kSelThreads, c->sel_cluster, &fits);
        if (e != cudaSuccess) return e;
        c->sel_wide = fits;
    } else {
        c->sel_wide = false;
    }
    for (int32_t* most : {&c->cluster_max, &c->cluster_max_first}) {
        const int64_t m = (int64_t)*most * (planned / c->sel_cluster);
        *most = m < INT32_MAX ? (int32_t)m : INT32_MAX;
    }
    return cudaSuccess;
}

cudaError_t launch_topk_select(compams_context* c) {
    const int64_t clusters = (int64_t)c->n * c->sel_long + ((int64_t)c->n * c->sel_short + c->sel_cluster - 1) / c->sel_cluster;
    const SelectKernel kernel = c->sel_wide ? topk_select_kernel<2 * kSelThreads> : topk_select_kernel<kSelThreads>;
    const cudaError_t e = counted(c, launch_cluster(kernel, dim3((unsigned)(clusters * c->sel_cluster)),
                                                    dim3(c->sel_wide ? 2 * kSelThreads : kSelThreads), c->sel_cluster, c->chain, c->stream,
                                                    c->tab, own_rows(c), (const int32_t*)c->sel_segs, c->sel_long, c->sel_short,
                                                    delivers(c) ? 1 : 0, c->sel_parts ? 1 : 0, c->small_last ? 1 : 0));
    if (e != cudaSuccess || !c->sel_parts) return e;
    const dim3 grid((unsigned)((int64_t)c->n * c->sel_long * c->sel_parts));
    if (c->chain)
        return counted(c, launch_after(topk_emit_kernel, grid, dim3(kThreads), c->stream, c->tab, own_rows(c),
                                       (const int32_t*)c->sel_segs, c->sel_long, c->sel_parts, delivers(c) ? 1 : 0));
    topk_emit_kernel<<<grid, kThreads, 0, c->stream>>>(c->tab, own_rows(c), c->sel_segs, c->sel_long, c->sel_parts, delivers(c) ? 1 : 0);
    return counted(c, cudaGetLastError());
}

template <typename GT>
static cudaError_t launch_fused_typed(compams_context* c, const GT* grads) {
    const int64_t clusters = (int64_t)c->n * c->sel_long + ((int64_t)c->n * c->sel_short + c->sel_cluster - 1) / c->sel_cluster;
    return counted(c, launch_cluster(topk_fused_kernel<GT>, dim3((unsigned)(clusters * c->sel_cluster)), dim3(kSelThreads), c->sel_cluster,
                                     true, c->stream, c->tab, own_rows(c), grads, (const int32_t*)c->sel_segs, c->sel_long, c->sel_short,
                                     delivers(c) ? 1 : 0));
}

cudaError_t launch_topk_fused(compams_context* c, const void* grads) {
    return c->grad_bf16 ? launch_fused_typed(c, (const bf16_bits*)grads) : launch_fused_typed(c, (const float*)grads);
}

cudaError_t launch_topk_dense(compams_context* c) {
    if (c->dense_grid == 0) {
        int per_sm = 0;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, topk_dense_kernel, kThreads, 0);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) return cudaErrorLaunchOutOfResources;
        c->dense_grid = per_sm * c->num_sms;  // every CTA resident at once, as a cooperative launch requires
    }
    TopkBuffers b = own_rows(c);
    int deliver = delivers(c) ? 1 : 0;
    void* args[] = {(void*)&c->tab, (void*)&b, (void*)&deliver};
    return counted(c, cudaLaunchCooperativeKernel((const void*)topk_dense_kernel, dim3((unsigned)c->dense_grid),
                                                  dim3(kThreads), args, 0, c->stream));
}

cudaError_t launch_topk_materialize(compams_context* c) {
    dim3 grid((unsigned)c->tab.ntiles, (unsigned)c->n);
    topk_materialize_kernel<<<grid, kThreads, 0, c->stream>>>(c->tab, c->tk);
    return counted(c, cudaGetLastError());
}

cudaError_t launch_topk_scatter(compams_context* c) {
    // one thread per message entry of every worker
    const int64_t count = (int64_t)c->n_total * c->K;
    const unsigned grid = (unsigned)((count + kThreads - 1) / kThreads);
    // (a sharded handle's exchange sits in front of this kernel: a plain launch waits for it)
    if (c->chain && c->n == c->n_total)
        return counted(c, launch_after(topk_scatter_kernel, dim3(grid), dim3(kThreads), c->stream, c->tk, count));
    topk_scatter_kernel<<<grid, kThreads, 0, c->stream>>>(c->tk, count);
    return counted(c, cudaGetLastError());
}

}  // namespace compams
