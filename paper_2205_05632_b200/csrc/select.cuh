// Exact Top-k selection by the CTAs of one thread-block cluster.
//
// A cluster selects the k_b largest magnitudes of one (worker, block): from the block's candidate list when the
// prediction of its threshold held, otherwise from the block itself. Every CTA works on one slice. The CTAs meet in
// distributed shared memory: each counts its slice into a histogram of its own, each adds up one range of bins over
// all of them, the owner of the bin that holds the k_b-th largest key tells the others, and every CTA writes its
// winners to the message. A bin with too many entries is counted again in finer bins. The entries inside the last bin
// (a few hundred) go to the first CTA, are copied to all, and are ranked by (key, lower index first), one per warp of
// the cluster; an entry's rank is its message slot.
//
// Bound by latency: two passes over a slice of a few loads per thread (a list's first round stays in registers) and
// five cluster barriers.
#pragma once

#include <cooperative_groups.h>

#include "context.h"
#include "predict.cuh"
#include "scatter.cuh"

namespace compams {

namespace cg = cooperative_groups;

constexpr int kMaxCluster = 16;
constexpr uint32_t kNoCandidate = 0xffffffffu;  // a NaN's bits: no candidate has them
constexpr uint32_t kNoBin = 0xffffffffu;

template <int NT>
struct SelectShared {
    uint32_t hist[kSelBins];      // this CTA's counts
    uint32_t tot[kSelBins / 2];   // the cluster's counts in this CTA's range of bins (clusters of two CTAs and more)
    uint2 surv[kSurvCap];         // entries of the threshold bin; collected in the first CTA, then copied
    uint32_t warp_sum[NT / 32];
    uint32_t range[kMaxCluster];  // entries in every CTA's range of bins, or ties in every CTA's slice
    uint32_t bin[3];              // threshold bin, entries above it, entries in it
    uint32_t edge[2];             // bin of the wanted number of candidates (kNoBin: fewer than that), entries above it
    uint32_t winners, base;       // winners of this CTA: counted, then written so far; its first message slot
    uint32_t slots, nsurv;        // the first CTA's: message slots handed out, entries collected
    uint32_t listed;              // the first CTA's: candidates listed by a sweep of the same kernel
    uint32_t undecided;           // 1: the first CTA has taken the list alone and could not decide
};

// The CTAs that select together: those of the cluster, or the first of them alone.
struct Group {
    unsigned size, rank;
    __device__ __forceinline__ void sync() const {
        if (size == 1) __syncthreads();
        else cg::this_cluster().sync();
    }
    template <typename T>
    __device__ __forceinline__ T* of(T* mine, unsigned q) const {  // the same shared variable of CTA q
        return size == 1 ? mine : cg::this_cluster().map_shared_rank(mine, q);
    }
};

// Adds the `pred` lanes of a warp to a counter (of this CTA, or of another one of the cluster) with one atomic;
// returns this lane's slot.
__device__ __forceinline__ uint32_t warp_slot(bool pred, uint32_t* counter, int lane) {
    const unsigned m = __ballot_sync(0xffffffffu, pred);
    uint32_t base = 0;
    if (m) {
        const int leader = __ffs(m) - 1;
        if (lane == leader) base = atomicAdd(counter, (uint32_t)__popc(m));
        base = __shfl_sync(0xffffffffu, base, leader);
    }
    return base + (uint32_t)__popc(m & ((1u << lane) - 1u));
}

// Inclusive scan over a CTA of NT threads whose last step is a reduction by every warp of the warps' sums.
template <int NT>
__device__ __forceinline__ uint32_t scan_cta(uint32_t x, uint32_t* warp_sum, uint32_t* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t s = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += y;
    }
    __syncthreads();  // warp_sum may still be read from an earlier call
    if (lane == 31) warp_sum[warp] = s;
    __syncthreads();
    const uint32_t w = lane < NT / 32 ? warp_sum[lane] : 0u;
    *total = __reduce_add_sync(0xffffffffu, w);
    return s + __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u);
}

template <int NT>
__device__ __forceinline__ void clear_hist(SelectShared<NT>& sh) {
    for (int k = threadIdx.x; k < kSelBins / 4; k += NT) reinterpret_cast<uint4*>(sh.hist)[k] = make_uint4(0u, 0u, 0u, 0u);
}

// The CTAs have counted: finds the bin of the `target`-th and of the `want`-th largest entry. Afterwards every CTA of
// the group has sh.bin and sh.edge, and this CTA's entries above the bin are added to sh.winners. Called by all
// threads of the group; hist may be cleared again afterwards.
template <int NT>
__device__ __forceinline__ void locate_bins(const Group& grp, SelectShared<NT>& sh, uint32_t target, uint32_t want) {
    const unsigned C = grp.size, rank = grp.rank;
    const int nb = kSelBins / (int)C;                  // bins of this CTA's range
    const int first = (int)(C - 1 - rank) * nb;        // rank 0 has the topmost range
    const uint32_t* tot = sh.hist;
    if (threadIdx.x == 0) sh.edge[0] = kNoBin;
    grp.sync();  // the histograms
    if (C > 1) {
        for (int k = threadIdx.x; k < nb; k += NT) {
            uint32_t s = 0;
#pragma unroll 8
            for (unsigned q = 0; q < C; ++q) s += grp.of(sh.hist, q)[first + k];
            sh.tot[k] = s;
        }
        tot = sh.tot;
        __syncthreads();
    }
    // every thread owns nb / NT consecutive bins (from the top)
    const int per = nb / NT > 0 ? nb / NT : 1;
    const int top = nb - 1 - (int)threadIdx.x * per;
    uint32_t sum = 0;
    for (int j = 0; j < per; ++j)
        if (top - j >= 0) sum += tot[top - j];
    uint32_t mine, above = 0;
    const uint32_t incl = scan_cta<NT>(sum, sh.warp_sum, &mine);
    if (C > 1) {
        if (threadIdx.x < C) grp.of(sh.range, threadIdx.x)[rank] = mine;
        grp.sync();  // the ranges' totals
        for (unsigned q = 0; q < rank; ++q) above += sh.range[q];
    }
    uint32_t running = above + incl - sum;  // entries above this thread's bins
    if ((running < target && target <= running + sum) || (running < want && want <= running + sum)) {
        for (int j = 0; j < per; ++j) {
            const uint32_t c = tot[top - j];
            if (running < target && target <= running + c)
                for (unsigned q = 0; q < C; ++q) {
                    uint32_t* out = grp.of(sh.bin, q);
                    out[0] = (uint32_t)(first + top - j);
                    out[1] = running;
                    out[2] = c;
                }
            if (running < want && want <= running + c)
                for (unsigned q = 0; q < C; ++q) {
                    uint32_t* out = grp.of(sh.edge, q);
                    out[0] = (uint32_t)(first + top - j);
                    out[1] = running;
                }
            running += c;
        }
    }
    grp.sync();  // the answers
    uint32_t wins = 0;
    for (int k = (int)sh.bin[0] + 1 + (int)threadIdx.x; k < kSelBins; k += NT) wins += sh.hist[k];
    wins = __reduce_add_sync(0xffffffffu, wins);
    if (wins && (threadIdx.x & 31) == 0) atomicAdd(&sh.winners, wins);
    __syncthreads();
}

// Where the kept entries of one (worker, block) go.
struct SelectJob {
    int32_t* idx;  // the segment's message slots
    float* val;
    float* erow;   // the worker's row of E
    uint32_t kb, cap;
    bool deliver;  // kept pairs also go to the server's buckets
    bool defer;    // the entries are emitted by a kernel of their own
};

// One kept pair in message slot `pos`.
__device__ __forceinline__ void put_pair(const TopkBuffers& b, const SelectJob& job, uint32_t pos, uint32_t j, uint32_t xbits) {
    if (pos < job.kb) {
        job.idx[pos] = (int32_t)j;
        job.val[pos] = __uint_as_float(xbits);
    } else {
        atomicOr(b.status, 1u);
    }
}

// The threshold bin's entries among U per thread, a few hundred of a whole list, the whole warp together.
template <int U>
__device__ __forceinline__ void put_survivors(const uint2 (&cv)[U], uint2* surv, uint32_t* nsurv, uint32_t win_from, uint32_t bin_from) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const uint32_t key = cv[u].y & 0x7fffffffu;
        const bool keep = cv[u].y != kNoCandidate && key >= bin_from && key < win_from;
        if (__any_sync(0xffffffffu, keep)) {
            const uint32_t q = warp_slot(keep, nsurv, threadIdx.x & 31);
            if (keep && q < (uint32_t)kSurvCap) surv[q] = cv[u];
        }
    }
}

// Emits U entries per thread, the whole warp together: keys from `win_from` up go to the message, at `base` + slots
// taken from `*taken`; those in [bin_from, win_from) to the survivors.
template <int U>
__device__ __forceinline__ void emit(const TopkBuffers& b, const SelectJob& job, uint32_t base, uint32_t* taken, uint2* surv,
                                     uint32_t* nsurv, const uint2* all, uint32_t win_from, uint32_t bin_from) {
    const int lane = threadIdx.x & 31;
    uint2 cv[U];
    unsigned wins[U];
    uint32_t rel[U], warp_wins = 0;
    bool any = false;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        cv[u] = all[u];
        const bool valid = cv[u].y != kNoCandidate;
        const uint32_t key = cv[u].y & 0x7fffffffu;
        wins[u] = __ballot_sync(0xffffffffu, valid && key >= win_from);
        rel[u] = warp_wins + (uint32_t)__popc(wins[u] & ((1u << lane) - 1u));
        warp_wins += (uint32_t)__popc(wins[u]);
        any = any || (valid && key >= bin_from && key < win_from);
    }
    if (__any_sync(0xffffffffu, any)) put_survivors<U>(cv, surv, nsurv, win_from, bin_from);
    if (warp_wins == 0u) return;
    uint32_t slot = 0;
    if (lane == 0) slot = base + atomicAdd(taken, warp_wins);
    slot = __shfl_sync(0xffffffffu, slot, 0);
#pragma unroll
    for (int u = 0; u < U; ++u)
        if ((wins[u] >> lane) & 1u) put_pair(b, job, slot + rel[u], cv[u].x, cv[u].y);
    if (job.deliver) scatter_runs<U>(b, wins, cv);
}

// The k_rem best of the threshold bin's entries surv[0 .. nsurv), larger key first, then lower index; an entry's rank is
// its slot after the winners. Warp w of W takes the entries w, w + W, ... Returns true in the one thread that holds the
// last one kept, with its key in *tau.
__device__ __forceinline__ bool rank_survivors(const TopkBuffers& b, const SelectJob& job, const uint2* surv, uint32_t nsurv,
                                               uint32_t k_rem, uint32_t w, uint32_t W, uint32_t* tau) {
    const int lane = threadIdx.x & 31;
    auto order = [](const uint2& cv) -> unsigned long long {
        return ((unsigned long long)(cv.y & 0x7fffffffu) << 32) | (unsigned long long)(0xffffffffu - cv.x);
    };
    bool last = false;
    for (uint32_t q = w; q < nsurv; q += W) {
        const uint2 cv = surv[q];
        const unsigned long long mine = order(cv);
        uint32_t beaten = 0;
        for (uint32_t p = lane; p < nsurv; p += 32) beaten += order(surv[p]) > mine ? 1u : 0u;
        beaten = __reduce_add_sync(0xffffffffu, beaten);
        if (lane == 0 && beaten < k_rem) {
            put_pair(b, job, job.kb - k_rem + beaten, cv.x, cv.y);
            if (job.deliver) scatter_one(b, (int32_t)cv.x, cv.y);
            job.erow[cv.x] = 0.0f;  // the residual of a kept coordinate: e = x - x
            if (beaten == k_rem - 1u) {
                last = true;
                *tau = cv.y & 0x7fffffffu;
            }
        }
    }
    return last;
}

// A slice of a candidate list: (coordinate, bits) pairs in any order, but those of one coordinate range mostly together.
// A warp reads 32 consecutive ones at a time, all warps take part in a short list.
struct ListSlice {
    static constexpr int kU = 8;
    static constexpr bool kOrdered = false;
    const uint2* list;
    uint32_t lo, hi;
    template <int NT>
    __device__ __forceinline__ void load(uint32_t p0, uint2 (&cv)[kU]) const {
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const uint32_t p = p0 + u * NT + threadIdx.x;
            cv[u] = p < hi ? __ldcg(list + p) : make_uint2(0u, kNoCandidate);
        }
    }
};

// A stretch of the block itself, in index order. Positions count from the 16-byte boundary at or before the block's first
// element, `skip` elements earlier, so that a thread reads 4 consecutive ones at once; lo is a multiple of 4.
struct BlockSlice {
    static constexpr int kU = 16;
    static constexpr bool kOrdered = true;
    const float* x;
    uint32_t lo, hi, skip, coord0;  // coord0: coordinate of position 0
    __device__ __forceinline__ uint32_t bits(uint32_t r) const {
        return r >= skip && r < hi ? __float_as_uint(__ldcg(x + r)) : kNoCandidate;
    }
    template <int NT>
    __device__ __forceinline__ void load(uint32_t p0, uint2 (&cv)[kU]) const {
#pragma unroll
        for (int u = 0; u < kU; u += 4) {
            const uint32_t r = p0 + u * NT + threadIdx.x * 4;
            float4 v;
            if (r >= skip && r + 3 < hi) {
                v = __ldcg(reinterpret_cast<const float4*>(x + r));
            } else {
                v = make_float4(__uint_as_float(bits(r)), __uint_as_float(bits(r + 1)), __uint_as_float(bits(r + 2)),
                                __uint_as_float(bits(r + 3)));
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) cv[u + k] = make_uint2(coord0 + r + k, __float_as_uint(lane_elem(v, k)));
        }
    }
};

// What a selection leaves: the key from which on everything was kept, the k_b-th largest key (or a lower bound of it,
// when the whole bin was kept), the key that about the wanted number of entries reach (reached = false: fewer do).
struct Selected {
    uint32_t kept_from, tau, edge;
    uint32_t k_rem;  // deferred emission: entries to take from the bin [tau, kept_from), 0: keys from tau = kept_from on
    bool reached;
    bool closer;  // this thread closes the segment's state
    int why;      // not decided: 5 the threshold lies beyond the histogram's range, 6 too many equal keys
};

// Selection of the k_b largest keys from slices whose entries' keys all reach `from`. `open`: the first histogram's
// last bin holds everything beyond its range. False, in all threads of the group and with nothing written: not decided
// (never with an ordered slice). Called by all threads of the group; sh.hist is clear.
template <int NT, typename Slice>
__device__ __forceinline__ bool select_slices(const Group& grp, const TopkBuffers& b, const SelectJob& job, SelectShared<NT>& sh,
                                              const Slice& sl, uint32_t from, int S, bool open, uint32_t want, bool refine_edge,
                                              Selected& out) {
    constexpr int U = Slice::kU;
    constexpr bool kHold = !Slice::kOrdered;  // a slice of one round stays in registers from the count to the emission
    const unsigned C = grp.size, rank = grp.rank;
    const int lane = threadIdx.x & 31;
    uint2 held[U];
    const bool one_round = sl.hi - sl.lo <= (uint32_t)(U * NT);
    if (kHold && one_round) sl.template load<NT>(sl.lo, held);
    auto count = [&](uint32_t base, int s, uint32_t width, bool clip) {  // entries with keys in [base, base + width)
        uint32_t far = 0;
        if (kHold && !one_round) sl.template load<NT>(sl.lo, held);
        for (uint32_t p0 = sl.lo; p0 < sl.hi; p0 += U * NT) {
            uint2 cv[U];
            if constexpr (kHold) {  // the next round is requested before this one is worked on
#pragma unroll
                for (int u = 0; u < U; ++u) cv[u] = held[u];
                if (p0 + U * NT < sl.hi) sl.template load<NT>(p0 + U * NT, held);
            } else {
                sl.template load<NT>(p0, cv);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool valid = cv[u].y != kNoCandidate;
                const uint32_t off = (cv[u].y & 0x7fffffffu) - base;  // wraps beyond every width below `base`
                // the open-ended last bin, most of a list, is counted in registers (by a ballot and one lane's atomic per
                // entry instead, topk_select took 27.7 us of n = 8, d = 4.2 M, 10 %, now 22.6; n = 32, d = 2^27, 1 % 115 -> 93)
                if (clip) {
                    const bool is_far = (off >> s) >= (uint32_t)(kSelBins - 1);
                    far += valid && is_far ? 1u : 0u;
                    if (valid && !is_far) atomicAdd(&sh.hist[off >> s], 1u);
                } else if (valid && off < width) {
                    atomicAdd(&sh.hist[off >> s], 1u);
                }
            }
        }
        if (clip) {
            far = __reduce_add_sync(0xffffffffu, far);
            if (lane == 0 && far) atomicAdd(&sh.hist[kSelBins - 1], far);
        }
    };
    auto again = [&]() {
        __syncthreads();
        clear_hist<NT>(sh);
        __syncthreads();
    };
    uint32_t k_rem = job.kb, edge_need = 0u;
    out.edge = 0u;
    count(from, S, 1u << 31, open);
    locate_bins<NT>(grp, sh, k_rem, want);
    out.reached = sh.edge[0] != kNoBin;
    if (out.reached) {
        out.edge = from + (sh.edge[0] << S);
        edge_need = want - sh.edge[1];
    }
    const int S0 = S;
    bool take_all = false, by_index = false;
    for (bool clipped = open;; clipped = false) {
        const uint32_t c0 = sh.bin[2];
        k_rem -= sh.bin[1];
        take_all = c0 == k_rem;
        if (!take_all && clipped && sh.bin[0] == (uint32_t)(kSelBins - 1)) {
            out.why = 5;
            return false;
        }
        from += sh.bin[0] << S;
        if (take_all || c0 <= (uint32_t)kSurvCap) break;
        if (S == 0) {
            by_index = true;
            break;
        }
        const uint32_t width = 1u << S;
        S = S > 12 ? S - 12 : 0;
        again();
        count(from, S, width, false);
        locate_bins<NT>(grp, sh, k_rem, 0u);
    }
    if (by_index && !Slice::kOrdered) {
        out.why = 6;
        return false;
    }
    const uint32_t c0 = sh.bin[2], my_ties = sh.hist[sh.bin[0]];
    const uint32_t my_wins = sh.winners + (take_all ? my_ties : 0u);
    if (refine_edge && edge_need) {
        // the wanted number of entries is reached inside a wide bin: placed 2^12 times finer, since under error
        // feedback magnitudes pile up just below the threshold
        const int s = S0 > 12 ? S0 - 12 : 0;
        again();
        count(out.edge, s, 1u << S0, false);
        locate_bins<NT>(grp, sh, edge_need, 0u);
        out.edge += sh.bin[0] << s;
    }
    // Keys have 31 bits, the bin holds one of them and S <= 21: the sum fits. Nothing may be cut off at the key of infinity:
    // when the bin lies at or above it (k_b gradients and more that are infinite or NaN) its entries would be emitted as
    // winners, and the ranking would read survivors that nobody has written.
    const uint32_t win_from = take_all ? from : from + (1u << S);
    if (job.defer) {
        out.kept_from = win_from;
        out.tau = from;
        out.k_rem = take_all ? 0u : k_rem;
        out.closer = rank == 0 && threadIdx.x == 0;
        return true;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        sh.base = my_wins ? atomicAdd(grp.of(&sh.slots, 0), my_wins) : 0u;
        sh.winners = 0u;
    }
    __syncthreads();
    uint2* surv = grp.of(sh.surv, 0);
    uint32_t* nsurv = grp.of(&sh.nsurv, 0);
    for (uint32_t p0 = sl.lo; p0 < sl.hi; p0 += U * NT) {
        if (!kHold || !one_round) sl.template load<NT>(p0, held);
#pragma unroll
        for (int h = 0; h < U; h += 4) emit<4>(b, job, sh.base, &sh.winners, surv, nsurv, held + h, win_from, by_index ? win_from : from);
    }
    if (by_index && threadIdx.x < C) grp.of(sh.range, threadIdx.x)[rank] = my_ties;
    grp.sync();  // all winners have their slots, the first CTA has all survivors, everyone the counts of ties
    const uint32_t slots = sh.slots;
    out.tau = from;
    out.closer = rank == 0 && threadIdx.x == 0 && (take_all || by_index);
    if constexpr (Slice::kOrdered) {
        if (by_index) {  // one key: this CTA's share of the k_rem lowest indices
            uint32_t before = 0;
            for (unsigned q = 0; q < rank; ++q) before += sh.range[q];
            for (uint32_t r0 = sl.lo; r0 < sl.hi && before < k_rem; r0 += NT) {
                const uint32_t r = r0 + threadIdx.x;
                const uint32_t xb = sl.bits(r);
                const bool tie = xb != kNoCandidate && (xb & 0x7fffffffu) == from;
                uint32_t total;
                const uint32_t pos = before + scan_cta<NT>(tie ? 1u : 0u, sh.warp_sum, &total) - 1u;
                if (tie && pos < k_rem) {
                    put_pair(b, job, job.kb - k_rem + pos, sl.coord0 + r, xb);
                    if (job.deliver) scatter_one(b, (int32_t)(sl.coord0 + r), xb);
                    job.erow[sl.coord0 + r] = 0.0f;  // the residual of a kept coordinate: e = x - x
                }
                before += total;
            }
        }
    }
    if (!take_all && !by_index) {
        // As many as the histogram has counted, which the arrays have room for; no more than have been collected are ranked. The two
        // counts agree on every path: a slice of one round is the same registers in both passes, and nothing writes a list or a block
        // in between. Should they not, the status word says so and no entry that nobody wrote reaches a message.
        const uint32_t got = *grp.of(&sh.nsurv, 0);  // travels with the entries
        if (rank) {
            const uint2* src = grp.of(sh.surv, 0);
            for (uint32_t q = threadIdx.x; q < c0; q += NT) sh.surv[q] = src[q];
            __syncthreads();
        }
        const uint32_t count = got < c0 ? got : c0;
        if (got != c0 && rank == 0 && threadIdx.x == 0) atomicOr(b.status, 1u);
        out.closer = rank_survivors(b, job, sh.surv, count, k_rem, (threadIdx.x >> 5) * C + rank, C * (NT / 32), &out.tau);
    }
    // with the whole bin kept, everything from its lower edge on; otherwise the kept entries of the bin have been zeroed
    // in E and the next key above the k-th largest is left
    out.kept_from = take_all ? from : out.tau + 1u;
    if (rank == 0 && threadIdx.x == 0 && slots + (take_all ? 0u : k_rem) != job.kb) atomicOr(b.status, 1u);
    return true;
}

// A list of c candidates above tau_hat has decided: leaves what the next step needs. `edge`: see Selected (kNoBin: not
// reached).
__device__ __forceinline__ void close_list(const TopkBuffers& b, const SelectJob& job, SegState* st, uint32_t* thr,
                                           uint32_t kept_from, uint32_t tau, uint32_t edge, uint32_t c, uint32_t tau_hat) {
    *thr = kept_from;
    if (edge == kNoBin) {
        // fewer candidates than wanted: reach further down next time, by half the distance to the threshold
        const uint32_t gap = ((tau - tau_hat) >> 1) + (1u << 16);
        edge = tau_hat > gap ? tau_hat - gap : 0u;
    }
    predict_next(st, tau, edge, true);
    margin_after_selection(st, job.kb, c, job.cap);
    st->cand_count = 0u;
    atomicAdd(b.status + 2, 1u);  // selections decided inside their candidate list
}

// From a candidate list of c entries (k_b <= c) whose keys all reach tau_hat.
template <int NT>
__device__ __forceinline__ bool select_from_list(const Group& grp, const TopkBuffers& b, const SelectJob& job, SelectShared<NT>& sh,
                                                 SegState* st, uint32_t* thr, const uint2* list, uint32_t c, uint32_t tau_hat, int S,
                                                 uint32_t boost, int* why) {
    const uint32_t per = (c + grp.size - 1) / grp.size;
    ListSlice sl;
    sl.list = list;
    sl.lo = grp.rank * per < c ? grp.rank * per : c;
    sl.hi = sl.lo + per < c ? sl.lo + per : c;
    Selected s;
    if (!select_slices<NT>(grp, b, job, sh, sl, tau_hat, S, true, want_candidates(job.kb, boost, job.cap), false, s)) {
        *why = s.why;
        return false;
    }
    if (s.closer) {
        const uint32_t edge = s.reached ? s.edge : kNoBin;
        if (job.defer) {
            st->emit_n = c;
            st->emit_from = s.kept_from;
            st->prefix = s.tau;  // (the dense passes' fields are free while the list decides)
            st->k_rem = s.k_rem;
            st->edge = edge;
            st->cand_count = 0u;
        } else {
            close_list(b, job, st, thr, s.kept_from, s.tau, edge, c, tau_hat);
        }
    }
    return true;
}

// From the block itself, exact for any input: histograms of 2^12 bins narrow the range of keys (31 -> 19 -> 7 -> 0
// open bits) until the bin of the k_b-th largest key is small enough to rank, or holds one key only. `predicts`: the
// block has a candidate list for the next step.
template <int NT>
__device__ __noinline__ void select_from_block(Group grp, const TopkBuffers& b, SelectJob job, SelectShared<NT>& sh, SegState* st,
                                               uint32_t* thr, const float* x, uint32_t len, uint32_t coord0, bool predicts,
                                               uint32_t boost) {
    BlockSlice sl;
    sl.skip = (uint32_t)align_class(x);
    sl.x = x - sl.skip;
    sl.coord0 = coord0 - sl.skip;
    len += sl.skip;
    const uint32_t per = ((len + grp.size - 1) / grp.size + 3u) & ~3u;
    sl.lo = grp.rank * per < len ? grp.rank * per : len;
    sl.hi = sl.lo + per < len ? sl.lo + per : len;
    if (threadIdx.x == 0) sh.winners = 0u;
    clear_hist<NT>(sh);
    __syncthreads();
    Selected s;
    select_slices<NT>(grp, b, job, sh, sl, 0u, 19, false, want_candidates(job.kb, boost, job.cap), predicts, s);
    if (s.closer) {
        *thr = s.kept_from;
        predict_next(st, s.tau, s.edge, predicts);
        st->cand_count = 0u;
        atomicAdd(b.status + 1, 1u);  // selections decided by passes over the block
    }
}

}  // namespace compams
