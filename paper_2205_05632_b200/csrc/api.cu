// C ABI of the COMP-AMS library (see include/compams.h): argument checks, state allocation,
// the per-step launch sequence and the inspection calls.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>

#include "context.h"

using namespace compams;

namespace {

thread_local std::string g_last_cuda_error;

int cuda_fail(cudaError_t e, const char* what) {
    g_last_cuda_error = std::string(what) + ": " + cudaGetErrorString(e);
    return COMPAMS_ERR_CUDA;
}

#define CU(call)                                          \
    do {                                                  \
        cudaError_t _e = (call);                          \
        if (_e != cudaSuccess) return cuda_fail(_e, #call); \
    } while (0)

template <typename T>
int dev_alloc(compams_context* c, T** out, size_t count, bool zero = true) {
    *out = nullptr;
    if (count == 0) count = 1;
    if (c->plan_only || c->ws) {
        // buffers are cut from one region, each on a 256-byte boundary
        const size_t off = (c->ws_used + 255) & ~(size_t)255;
        c->ws_used = off + count * sizeof(T);
        if (c->plan_only) return COMPAMS_OK;
        if (c->ws_used > c->ws_bytes) return COMPAMS_ERR_INVALID_ARG;  // the caller's region is too small
        if (zero) CU(cudaMemsetAsync(c->ws + off, 0, count * sizeof(T), c->stream));
        *out = (T*)(c->ws + off);
        return COMPAMS_OK;
    }
    void* p = nullptr;
    cudaError_t e = cudaMalloc(&p, count * sizeof(T));
    if (e != cudaSuccess) {
        g_last_cuda_error = std::string("cudaMalloc: ") + cudaGetErrorString(e);
        cudaGetLastError();
        return COMPAMS_ERR_ALLOC;
    }
    c->owned.push_back(p);
    if (zero) CU(cudaMemsetAsync(p, 0, count * sizeof(T), c->stream));
    *out = (T*)p;
    return COMPAMS_OK;
}

template <typename T>
int dev_upload(compams_context* c, T** out, const std::vector<T>& host) {
    int rc = dev_alloc(c, out, host.size(), false);
    if (rc) return rc;
    if (!host.empty() && !c->plan_only) CU(cudaMemcpy(*out, host.data(), host.size() * sizeof(T), cudaMemcpyHostToDevice));
    return COMPAMS_OK;
}

#define RC(call)              \
    do {                      \
        int _rc = (call);     \
        if (_rc) return _rc;  \
    } while (0)

// Every enqueueing call must run with the handle's device current: its buffers live there, and on the
// default stream a launch goes to whatever device is current.
int on_handle_device(const compams_context* c) {
    int dev = -1;
    CU(cudaGetDevice(&dev));
    return dev == c->device ? COMPAMS_OK : COMPAMS_ERR_INVALID_ARG;
}

int64_t kept_per_block(double k_ratio, int64_t d_b) {
    int64_t k = (int64_t)std::floor(k_ratio * (double)d_b);
    if (k < 1) k = 1;
    if (k > d_b) k = d_b;
    return k;
}

constexpr int64_t kPlanSms = 148;              // SMs that the choices below count on (a plan is made without a device)
constexpr int64_t kFusedRound = 8192;          // coordinates one CTA of the fused sweep and selection has in flight
constexpr int64_t kListlessFused = 2048;       // blocks up to this size are always selected from directly there (from 0 to 8192 no
                                               // difference in time: n = 3, d = 111,947 in 78 blocks 20.7 us; it saves the lists)
constexpr int64_t kListlessFusedMax = 3 << 18; // n d up to which longer ones are, too
// Coordinates per CTA up to which a cluster goes through a block itself when the list cannot decide: about 0.75 ns each for
// all its passes. Beyond, the dense passes of the whole GPU are launched every step to stand by: about 4 us when they have
// nothing to do, which only matters to short steps.
constexpr int64_t kClusterMax = (int64_t)1 << 21, kClusterMaxLongStep = (int64_t)1 << 17;
// The first steps of a handle, and those after its accumulators have been replaced, are the ones whose lists do fail (none has a
// prediction in the first; later ones fail when the gradient scale drops, or under a cycle of few batches). In these the dense passes
// stand by wherever the clusters would take more than about twice their time, which is 5 ps per worker-element and 30 us
// (first step / later ones, us: n = 1, d = 28.5 M, 1 % 451 / 232, by clusters alone 1329; n = 1, d = 4.2 M 104 / 58, 305; n = 4,
// ResNet-18 shapes whole 498 / 172, 899).
constexpr int kFirstSteps = 32;
// ... of a block that never has a list, where its cluster goes through it on every step. Five passes by a few CTAs: the dense passes of
// the whole GPU are faster from about there on (us per step, clusters / dense passes, 20 % kept: n = 4, d = 162,400 39 / 43, d = 262,144
// 45 / 47, n = 8, d = 262,144 57 / 52 but 64 / 72 with 50 %, n = 1, d = 524,288 59 / 41, d = 2^21 + 3 177 / 56; 70 blocks, n = 8,
// d = 65,536 49 / 57, d = 262,144 72 / 67).
constexpr int64_t kListless = 1 << 14;

// The candidate path pays off for sparse selections only: at most 1/9 of the block kept.
bool has_list(int64_t kb, int64_t len) { return kb * 9 <= len; }

// CTAs per long block when sweep and selection are one kernel, 0 when they are not. It pays where no CTA needs more than
// one round of loads for its share and no two share an SM: n = 4, d = 65,536 15.9 -> 15.3 us, n = 3, d = 111,947 in 78
// blocks 24.2 -> 18.4; but n = 1, d = 2^20 (16 CTAs, eight rounds) 25.7 -> 38.7, n = 32, d = 65,536 (256 CTAs) 17.8 -> 21.3. Blocks
// without a list take five passes by their clusters, which lose to the dense passes of the whole GPU from some problem size on (20 % kept:
// n = 8, d = 65,536 43 against 45 us, n = 4, d = 162,400 in 70 blocks 36 against 62, n = 16, d = 65,536 67 against 55).
int fused_cluster(const compams_context* c) {
    int64_t longest = 0, longs = 0, shorts = 0;
    bool listless = false;
    for (int32_t b = 0; b < c->M; ++b) {
        const int64_t len = c->off[(size_t)b + 1] - c->off[(size_t)b];
        longest = std::max(longest, len);
        (len > kFusedRound ? longs : shorts) += c->n;
        listless = listless || (len > kFusedRound && !has_list(c->seg_off[(size_t)b + 1] - c->seg_off[(size_t)b], len));
    }
    int64_t cluster = 1;
    while (cluster * kFusedRound < longest) cluster *= 2;
    if (listless && c->n * c->d > kListlessFusedMax) return 0;
    return cluster <= 16 && longs * cluster <= kPlanSms && shorts <= 2 * kPlanSms ? (int)cluster : 0;
}

// Decides which kernels select from which blocks, and with how many CTAs.
int group_segments(compams_context* c, const std::vector<SegInfo>& segs) {
    const int64_t elems = (int64_t)c->n * c->d;
    const int64_t cluster_max = elems <= kChainMaxElems ? kClusterMax : kClusterMaxLongStep;
    c->cluster_max = (int32_t)cluster_max;
    c->cluster_max_first = (int32_t)std::min(cluster_max, 80000 + elems / 75);
    c->sel_long = c->sel_short = c->sel_parts = 0;
    c->sel_cluster = 1;
    c->dense_kernel = c->dense_first = false;
    c->seg_always_dense.assign(segs.size(), false);
    if (c->randk) return COMPAMS_OK;
    if (c->fused) {
        std::vector<int32_t> one, several;
        for (size_t s = 0; s < segs.size(); ++s) (segs[s].len <= kFusedRound ? one : several).push_back((int32_t)s);
        c->sel_cluster = fused_cluster(c);
        std::stable_sort(several.begin(), several.end(), [&](int32_t a, int32_t b) { return segs[(size_t)a].len > segs[(size_t)b].len; });
        c->cluster_max = c->cluster_max_first = INT32_MAX;  // the dense passes are never launched
        c->sel_long = (int)several.size();
        c->sel_short = (int)one.size();
        several.insert(several.end(), one.begin(), one.end());
        return dev_upload(c, &c->sel_segs, several);
    }
    // Long candidate lists get a cluster of CTAs each, the others one CTA. Which are long, and how many CTAs they get, is
    // what makes the estimate of the kernel's time least: the longest CTA, or all CTAs over 1.5 per SM. In entries, a CTA
    // costs its share and about a round of 4096 for its fixed latencies, half a round more for the cluster's barriers.
    // More than one cluster of 16 per 16 SMs does not fit the GPCs at once (ResNet-18 shapes whole, n = 16, 1 %, bfloat16:
    // 394 us with 16 CTAs per list, 377 with 8), more than two CTAs per SM wait for others. The choice is within 1.5 % of the best of all
    // cluster sizes and four values of `from` for n = 1 to 32, d = 2^20 and 2^22 whole, ResNet-18 and ResNet-50 shapes by layers (n = 4: 168.4 us
    // against 167.7, with one CTA per list 178.6) and blocks of 1.2 to 2.6 M coordinates.
    auto expected = [&](const SegInfo& si) { return (int64_t)si.kb + si.kb / 4; };
    int cluster = 1;
    int64_t from = INT64_MAX;  // lists are long from here on
    double best = 1e300;
    for (int c16 = 1; c16 <= 16; c16 *= 2) {
        for (int64_t th = 4096; th <= ((int64_t)1 << 20); th *= 2) {
            double longest = 0.0, total = 0.0;
            int64_t longs = 0;
            for (const SegInfo& si : segs) {
                const bool is_long = c16 > 1 && expected(si) >= th;
                const double cost = is_long ? (double)expected(si) / c16 + 6144.0 : (double)expected(si) + 4096.0;
                longest = std::max(longest, cost);
                total += cost * (is_long ? c16 : 1) * c->n;
                longs += is_long ? c->n : 0;
            }
            if (longs * c16 > (c16 == 16 ? 1 : 2) * kPlanSms) continue;
            const double cost = std::max(longest, total / (1.5 * kPlanSms));
            if (cost < 0.98 * best) {
                best = cost;
                cluster = longs ? c16 : 1;
                from = longs ? th : INT64_MAX;
            }
        }
    }
    // A block too long for one CTA to go through gets a cluster however short its list (the first CTA takes that alone), where
    // all CTAs of the kernel are at work at once: the dense passes need not stand by (n = 4, d = 2^21 + 3, 0.1 %: 51.0 -> 46.2 us).
    int64_t lists = 0, by_length = 0, longest = 0;
    for (const SegInfo& si : segs) {
        lists += expected(si) >= from;
        by_length += elems <= kChainMaxElems && expected(si) < from && si.cap && si.len > cluster_max;
        longest = std::max<int64_t>(longest, si.len);
    }
    int lift = 0;
    for (int c16 = cluster > 1 ? cluster : 16; by_length && !lift && c16 > 1; c16 = cluster > 1 ? 1 : c16 / 2) {
        const int64_t ctas = c->n * ((lists + by_length) * c16 + (int64_t)segs.size() - lists - by_length);
        if (ctas <= (c16 == 16 ? 1 : 2) * kPlanSms && longest <= cluster_max * c16) lift = c16;
    }
    if (lift) cluster = lift;
    std::vector<int32_t> few, many;  // blocks for one CTA, for a cluster of them
    for (size_t s = 0; s < segs.size(); ++s) {
        const bool is_many = expected(segs[s]) >= from || (lift && segs[s].cap && segs[s].len > cluster_max);
        (is_many ? many : few).push_back((int32_t)s);
    }
    int64_t entries = 0;
    // blocks without a list go to their clusters where those are short and all at work at once, one per GPC (n = 16, d = 65,536, 16
    // clusters of 8, 20 % kept: 67 us, by the dense passes 55)
    bool walk = (int64_t)many.size() * c->n <= 8 && ((int64_t)many.size() * cluster + (int64_t)few.size()) * c->n <= kPlanSms;
    for (const std::vector<int32_t>* l : {&few, &many})
        for (int32_t s : *l) walk = walk && (segs[(size_t)s].cap || segs[(size_t)s].len <= kListless * (l == &few ? 1 : cluster));
    for (std::vector<int32_t>* l : {&few, &many}) {
        const int64_t ctas = l == &few ? 1 : cluster;
        std::vector<int32_t> listed;
        for (int32_t s : *l) {
            if (segs[(size_t)s].len > cluster_max * ctas) c->dense_kernel = true;
            if (segs[(size_t)s].len > c->cluster_max_first * ctas) c->dense_first = true;
            if (segs[(size_t)s].cap || walk) {
                listed.push_back(s);
                if (l == &many && segs[(size_t)s].cap) entries = std::max(entries, expected(segs[(size_t)s]));
            } else {  // always the dense passes
                c->seg_always_dense[(size_t)s] = true;
                c->dense_kernel = true;
            }
        }
        // longest first (their CTAs differ in length by the lists' lengths)
        std::stable_sort(listed.begin(), listed.end(), [&](int32_t a, int32_t b) { return segs[(size_t)a].cap > segs[(size_t)b].cap; });
        *l = listed;
    }
    c->sel_long = (int)many.size();
    c->sel_short = (int)few.size();
    c->sel_cluster = cluster;
    // Lists that their clusters would have to go through in many rounds are emitted by a kernel of its own: from three
    // rounds on where the clusters leave SMs idle (by the cluster / by topk_emit, us per step: d = 2^22, n = 1, 1.6 rounds 58.2 / 59.7, 3.2
    // 74.1 / 66.2, 8 91.6 / 67.9; n = 8, 2.4 rounds 117 / 122, 4 131.9 / 130.7, 8 170 / 160), from eight where they do not (d = 9 M, n = 16,
    // 3.4 rounds 333 / 334, 6.9 364 / 360, 13.7 429 / 409; d = 4 M, n = 32, 6.1 rounds 329 / 344, 12.2 404 / 423)
    if (c->sel_long && entries >= (cluster == 16 ? 3 : 8) * (int64_t)cluster * 4096) {
        const int64_t lists = (int64_t)c->n * c->sel_long;
        c->sel_parts = (int)((entries + 2047) / 2048);
        RC(dev_alloc(c, &c->tk.sel_ticket, (size_t)lists * 4));
        RC(dev_alloc(c, &c->tk.sel_surv, (size_t)lists * kSurvCap, false));
    }
    many.insert(many.end(), few.begin(), few.end());
    return dev_upload(c, &c->sel_segs, many);
}

// Whether topk_small, whose longest block is `longest`, comes behind topk_select and runs beside it: nothing of either is the other's.
// In front, where it stays with an emission kernel behind the selection, it runs beside the tail of the sweep and delays the selection by
// what sticks out; behind, it starts when all of the selection's CTAs have and costs the step a microsecond or two of its own. us per
// step in front / behind, of 290 layouts of n = 1 to 32, which the conditions divide with no loss above 1.5 % and give up 3 % at most:
// - Blocks of 2500 to 4096 coordinates stick out of any sweep: n = 1, 3 x 600,000 with three of 2500 41.1 / 38.0, n = 8, 8 x 50,000 with
//   eight 36.7 / 26.0, n = 2, d = 2 M in 100 blocks 47.4 / 40.2.
// - Shorter ones only of a sweep of about one wave that has CTAs on all SMs: n = 4, 20 x 20,000 (240 tiles) with 20 of 30 26.6 / 24.0; but
//   n = 4, 3 x 600,000 (888) 45.4 / 47.1, n = 2, d = 200,535 in 15 (58) 19.2 / 21.4; nor where more is kept or the server kernel has more CTAs
//   than fit at once: n = 16, 3 x 50,000, 6 % 30.0 / 32.0, n = 1, 3 x 600,000 (222) 36.2 / 37.9.
// - There is no room beside CTAs of the selection on every SM (n = 32, 8 x 50,000 with eight of 2500 58.8 / 61.9, n = 4, d = 1.7 M in 99
//   50.4 / 51.4), and nothing to gain where both are more than a wave (n = 10, d = 855,151 in 108, bfloat16 62.5 / 66.6) or the small blocks
//   are most of the step (n = 11, d = 135,392 in 128, 6.8 % 40.9 / 42.6, bfloat16 45.4 / 48.9).
bool small_beside_select(const compams_context* c, int64_t longest) {
    const int64_t n = c->n, tiles = n * c->tab.ntiles, small = n * c->tk.nsmall;
    const int64_t ctas = n * ((int64_t)c->sel_long * c->sel_cluster + c->sel_short);
    if (!small || !ctas || c->sel_parts) return false;
    if (c->sel_cluster == 1 && ctas > kPlanSms && ctas <= 2 * kPlanSms) return false;
    if (ctas > 2 * kPlanSms && small > 3 * kPlanSms) return false;
    if (small > 7 * kPlanSms && tiles <= 2 * kPlanSms) return false;
    if (longest >= (tiles > 4 * kPlanSms ? 700 : 1024)) return true;
    return tiles > kPlanSms && tiles <= 4 * kPlanSms && !c->many_candidates &&
           (tiles > 2 * kPlanSms || c->d <= 5 * kPlanSms * kBucketSpan);
}

// Cuts the listed blocks into tiles of kTile coordinates and uploads the tile and segment tables.
// For Top-k (`topk` true) every listed block also gets its message slots and candidate capacity.
int build_tiles(compams_context* c, const std::vector<int32_t>& blocks, bool topk) {
    std::vector<TileInfo> tiles;
    std::vector<SegInfo> segs;
    int64_t cand_total = 0;
    c->bs_max_tiles = 0;
    for (size_t s = 0; s < blocks.size(); ++s) {
        const int32_t b = blocks[s];
        const int64_t len = c->off[b + 1] - c->off[b];
        // The sweeps shift a worker's tiles down by the phase of the block's first element within a
        // 128-byte line, (i d + o) mod 32, so that every warp access covers whole lines; the block
        // needs enough tiles for the largest shift among the workers.
        int64_t smax = 0;
        for (int32_t i = 0; i < c->n && smax < 31; ++i) smax = std::max<int64_t>(smax, ((int64_t)i * c->d + c->off[b]) & 31);
        const int64_t nt = (len + smax + kTile - 1) / kTile;
        if ((int64_t)tiles.size() + nt > (int64_t)0x7fffffff) return COMPAMS_ERR_INVALID_ARG;
        SegInfo si{};
        si.o = c->off[b];
        si.len = (int32_t)len;
        si.blk = b;
        si.tile0 = (int32_t)tiles.size();
        si.ntile_b = (int32_t)nt;
        c->bs_max_tiles = std::max(c->bs_max_tiles, (int)si.ntile_b);
        if (topk) {
            const int64_t kb = c->seg_off[(size_t)b + 1] - c->seg_off[(size_t)b];
            si.slot0 = c->seg_off[(size_t)b];
            si.kb = (uint32_t)kb;
            int64_t cap = !c->randk && has_list(kb, len) ? 8 * kb + 1024 : 0;
            if (c->fused && len <= kListlessFused) cap = 0;
            if (cap) cap = std::min(cap, len <= 65536 ? len : len / 4 + kb);
            cap = (cap + 15) & ~(int64_t)15;  // lists start on 128-byte lines
            si.cap = (uint32_t)cap;
            si.cand_off = cand_total;
            cand_total += cap;
        }
        for (int64_t r0 = 0; r0 < nt * kTile; r0 += kTile) {
            TileInfo ti{};
            ti.o = c->off[b];
            ti.len = (int32_t)len;
            ti.r0 = (int32_t)r0;
            ti.blk = b;
            ti.seg = (int32_t)s;
            ti.tile0 = si.tile0;
            ti.ntile_b = si.ntile_b;
            tiles.push_back(ti);
        }
        segs.push_back(si);
    }
    TileInfo* d_tiles;
    SegInfo* d_segs;
    RC(dev_upload(c, &d_tiles, tiles));
    RC(dev_upload(c, &d_segs, segs));
    c->tab.ntiles = (int32_t)tiles.size();
    c->tab.tiles = d_tiles;
    c->tab.nseg = (int32_t)blocks.size();
    c->tab.segs = d_segs;
    c->segp = SegParams{};
    if (segs.size() <= (size_t)kParamSegs) {
        c->segp.nseg = (int32_t)segs.size();
        for (size_t s = 0; s < segs.size(); ++s) {
            c->segp.tile0[s] = segs[s].tile0;
            c->segp.len[s] = segs[s].len;
            c->segp.blk[s] = segs[s].blk;
            c->segp.o[s] = segs[s].o;
        }
        c->segp.tile0[segs.size()] = (int32_t)tiles.size();
    }
    c->tk.cand_total = cand_total;
    c->many_candidates = 4 * cand_total > c->d;  // more than d / 32 kept (a list has room for 8 k_b)
    if (topk) {
        RC(group_segments(c, segs));
    }
    return COMPAMS_OK;
}

int init_context(compams_context* c, const int64_t* block_offsets) {
    if (!c->plan_only) {
        CU(cudaGetDevice(&c->device));
        CU(cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, c->device));
    }
    const int32_t n = c->n, M = c->M;
    const int64_t d = c->d;
    c->off.assign(block_offsets, block_offsets + M + 1);
    c->tab.n = n;
    c->tab.d = d;
    c->tab.M = M;
    RC(dev_upload(c, &c->d_off, c->off));
    c->tab.off = c->d_off;

    RC(dev_alloc(c, &c->m, (size_t)d));
    RC(dev_alloc(c, &c->v, (size_t)d));
    RC(dev_alloc(c, &c->vhat, (size_t)d));
    RC(dev_alloc(c, &c->gbar, (size_t)d));
    RC(dev_alloc(c, &c->status, 8));

    if (c->sparse()) {
        c->seg_off.assign((size_t)M + 1, 0);
        bool identity = true;
        for (int32_t b = 0; b < M; ++b) {
            const int64_t db = c->off[b + 1] - c->off[b];
            const int64_t kb = kept_per_block(c->k_ratio, db);
            identity = identity && (kb == db);
            c->seg_off[(size_t)b + 1] = c->seg_off[(size_t)b] + kb;
        }
        c->identity = identity;
        c->K = identity ? 0 : c->seg_off[(size_t)M];
    }

    if (c->sparse() && c->identity) {
        // full-precision distributed AMSGrad: e is identically zero and not stored
    } else if (c->sparse()) {
        RC(dev_alloc(c, &c->E, (size_t)n * (size_t)d));
        RC(dev_upload(c, &c->d_seg_off, c->seg_off));
        c->fused = !c->randk && fused_cluster(c) > 0;
        std::vector<int32_t> small, large;
        // (Random-k has no selection: every block is tiled for the sweep, none goes to the shared-memory select)
        for (int32_t b = 0; b < M; ++b)
            ((!c->randk && !c->fused && c->off[b + 1] - c->off[b] <= kSmallMax) ? small : large).push_back(b);
        RC(build_tiles(c, large, true));
        if (!c->plan_only) CU(fit_topk_cluster(c));
        TopkBuffers& t = c->tk;
        t.E = c->E;
        t.K = c->K;
        t.seg_off = c->d_seg_off;
        int32_t* d_small;
        RC(dev_upload(c, &d_small, small));
        t.small_blk = d_small;
        t.nsmall = (int32_t)small.size();
        int64_t longest = 0;
        for (int32_t b : small) longest = std::max(longest, c->off[b + 1] - c->off[b]);
        c->small_last = small_beside_select(c, longest);
        // the messages of all n_total workers: this handle's selection fills its own rows, the other
        // rows are filled by the caller's exchange before compams_apply
        RC(dev_alloc(c, &t.idx, (size_t)c->n_total * (size_t)c->K));
        RC(dev_alloc(c, &t.val, (size_t)c->n_total * (size_t)c->K));
        RC(dev_alloc(c, &t.hist, c->randk ? 1 : (size_t)n * (size_t)c->tab.nseg * kBins1));
        {
            SegState init{};
            init.tau_hat = kNoPrediction;
            init.tau_prev = kNoPrediction;
            std::vector<SegState> seg0((size_t)n * (size_t)c->tab.nseg, init);
            uint32_t never = 0;
            for (size_t k = 0; k < seg0.size(); ++k) {
                seg0[k].fallback = c->seg_always_dense[k % (size_t)c->tab.nseg] ? 1u : 0u;
                never += seg0[k].fallback;
            }
            RC(dev_upload(c, &t.seg, seg0));
            c->seg_init_host = seg0;
            c->dense_count_init = never;
            c->deliver = n == c->n_total && never == 0;
            std::vector<uint32_t> dc(1, never);
            RC(dev_upload(c, &t.dense_count, dc));
        }
        RC(dev_alloc(c, &t.tile_ties, c->randk ? 1 : (size_t)n * (size_t)c->tab.ntiles));
        RC(dev_alloc(c, &t.cand, (size_t)n * (size_t)t.cand_total, false));
        RC(dev_alloc(c, &t.acc, (size_t)d));
        if (c->randk) {
            // workers whose map fits 64 MB of the L2 together, at least one
            constexpr int64_t kMapBits = (int64_t)64 * 8 * 1024 * 1024;
            c->randk_group = (int32_t)std::min<int64_t>(n, std::max<int64_t>(1, kMapBits / d));
            c->randk_words = ((int64_t)c->randk_group * d + 31) / 32 + 1;
            RC(dev_alloc(c, &t.map, (size_t)c->randk_words));
            RC(dev_alloc(c, &t.slots, (size_t)n * (size_t)c->tab.nseg));
        }
        {
            std::vector<uint32_t> none((size_t)n * (size_t)std::max(c->tab.nseg, 1), 0xffffffffu);
            RC(dev_upload(c, &t.thr, none));
        }
        {
            // kept entries are handed to the server grouped by coordinate range: room for four times the
            // average load of a bucket, the rare excess goes through the binary64 accumulator
            t.nbucket = (int32_t)((d + kBucketSpan - 1) / kBucketSpan);
            const int64_t avg = ((int64_t)c->n_total * c->K + t.nbucket - 1) / t.nbucket;
            int64_t cap = 4 * avg + 64;
            if (cap > (int64_t)c->n_total * kBucketSpan) cap = (int64_t)c->n_total * kBucketSpan;
            t.bucket_cap = (int32_t)((cap + 31) / 32 * 32);
            RC(dev_alloc(c, &t.bucket, (size_t)t.nbucket * (size_t)t.bucket_cap, false));
            RC(dev_alloc(c, &t.bcount, (size_t)t.nbucket));
            RC(dev_alloc(c, &t.bdirty, (size_t)t.nbucket));
        }
        t.status = c->status;
        t.gbar = nullptr;  // set by compams_record_average
        t.m = c->m;
        t.v = c->v;
        t.vhat = c->vhat;
    } else {
        RC(dev_alloc(c, &c->E, (size_t)n * (size_t)d));
        std::vector<int32_t> all((size_t)M);
        for (int32_t b = 0; b < M; ++b) all[(size_t)b] = b;
        RC(build_tiles(c, all, false));
        std::vector<int64_t> word_off((size_t)M + 1, 0);
        for (int32_t b = 0; b < M; ++b)
            word_off[(size_t)b + 1] = word_off[(size_t)b] + (c->off[b + 1] - c->off[b] + 31) / 32;
        c->W = word_off[(size_t)M];
        RC(dev_upload(c, &c->d_word_off, word_off));
        if (c->W > (int64_t)INT32_MAX) c->segp.nseg = 0;  // word offsets would not fit the kernel-argument copy
        for (int32_t sg = 0; sg < c->segp.nseg; ++sg) c->segp.wofs[sg] = (int32_t)word_off[(size_t)c->segp.blk[sg]];
        BsBuffers& s = c->bs;
        s.E = c->E;
        s.word_off = c->d_word_off;
        s.W = c->W;
        // sign words and scales of all n_total workers (see the Top-k messages above)
        RC(dev_alloc(c, &s.bits, (size_t)c->n_total * (size_t)c->W));
        RC(dev_alloc(c, &c->scales[0], (size_t)c->n_total * (size_t)M));
        RC(dev_alloc(c, &c->scales[1], (size_t)c->n_total * (size_t)M));
        RC(dev_alloc(c, &s.tile_sum, (size_t)n * (size_t)c->tab.ntiles));
        RC(dev_alloc(c, &s.edge, (size_t)n * (size_t)c->tab.ntiles));
        s.gbar = nullptr;  // set by compams_record_average
        s.status = c->status;
        s.m = c->m;
        s.v = c->v;
        s.vhat = c->vhat;
    }
    if (!c->plan_only) CU(cudaDeviceSynchronize());
    return COMPAMS_OK;
}

void free_context(compams_context* c) {
    for (void* p : c->owned) cudaFree(p);
    c->owned.clear();
    if (c->stage_grads) cudaFree(c->stage_grads);
    if (c->stage_theta) cudaFree(c->stage_theta);
    for (cudaEvent_t e : c->ev_start) cudaEventDestroy(e);
    for (cudaEvent_t e : c->ev_stop) cudaEventDestroy(e);
    delete c;
}

// Runs one launcher, optionally bracketed by an event pair for per-kernel timing.
template <typename F>
int run_kernel(compams_context* c, int kernel, F&& launch) {
    const bool timed = (c->prof_mask >> kernel) & 1u;
    int slot = -1;
    if (timed && c->prof_used < kMaxTimed) {
        slot = c->prof_used++;
        if ((size_t)slot >= c->ev_start.size()) {
            cudaEvent_t a, b;
            CU(cudaEventCreate(&a));
            CU(cudaEventCreate(&b));
            c->ev_start.push_back(a);
            c->ev_stop.push_back(b);
            c->ev_kernel.push_back(kernel);
        }
        c->ev_kernel[(size_t)slot] = kernel;
        CU(cudaEventRecord(c->ev_start[(size_t)slot], c->stream));
    }
    cudaError_t e = launch();  // the launchers count the kernels they enqueue in c->launches
    if (e != cudaSuccess) return cuda_fail(e, compams_kernel_name(kernel));
    if (slot >= 0) CU(cudaEventRecord(c->ev_stop[(size_t)slot], c->stream));
    return COMPAMS_OK;
}

// Worker side of one iteration (Algorithm 2, the workers' loop) for this handle's workers: x = g + e, the
// compression, the residual; the compressed gradients land in this handle's rows of the message buffers.
int compress_device(compams_context* c, const void* grads) {
    ++c->steps_done;
    ++c->iter;
    if (c->compressor == COMPAMS_BLOCKSIGN) {
        c->scales_cur ^= 1;
        RC(run_kernel(c, COMPAMS_K_BS_SWEEP, [&] { return launch_bs_sweep(c, grads); }));
        c->e_is_x = true;
        if (!bs_apply_adds_up(c)) RC(run_kernel(c, COMPAMS_K_BS_SCALES, [&] { return launch_bs_scales(c); }));
        return COMPAMS_OK;
    }
    // a selection leaves x in E at the coordinates it keeps, and the pair that delimits them; their e is zeroed
    // when E is next read (by the next sweep, or by topk_materialize when the caller asks for E)
    c->tk.use_thr = c->e_mask_pending ? 1 : 0;
    if (c->randk) {
        // no selection: the drawn coordinates are marked, and the sweep takes them
        RC(run_kernel(c, COMPAMS_K_RANDK_EMIT, [&] { return launch_randk(c, grads); }));
        return COMPAMS_OK;
    }
    if (c->fused) {
        c->tk.cluster_max = c->cluster_max;
        RC(run_kernel(c, COMPAMS_K_TOPK_SELECT, [&] { return launch_topk_fused(c, grads); }));
        c->e_mask_pending = true;
        return COMPAMS_OK;
    }
    const bool first = c->first_steps > 0;
    if (first) --c->first_steps;
    c->tk.cluster_max = first ? c->cluster_max_first : c->cluster_max;
    if (c->tab.ntiles > 0) RC(run_kernel(c, COMPAMS_K_TOPK_SWEEP, [&] { return launch_topk_sweep(c, grads); }));
    if (c->tk.nsmall > 0 && !c->small_last) RC(run_kernel(c, COMPAMS_K_TOPK_SMALL, [&] { return launch_topk_small(c, grads); }));
    if (c->tab.ntiles > 0) {
        if (c->sel_long + c->sel_short > 0) RC(run_kernel(c, COMPAMS_K_TOPK_SELECT, [&] { return launch_topk_select(c); }));
        if (c->small_last) RC(run_kernel(c, COMPAMS_K_TOPK_SMALL, [&] { return launch_topk_small(c, grads); }));
        if (c->dense_kernel || (first && c->dense_first)) RC(run_kernel(c, COMPAMS_K_TOPK_DENSE, [&] { return launch_topk_dense(c); }));
        c->e_mask_pending = true;
    }
    return COMPAMS_OK;
}

// Server side (Algorithm 2, the server's part): average of the n_total compressed gradients and AMSGrad.
int apply_device(compams_context* c, float* theta) {
    if (c->compressor == COMPAMS_BLOCKSIGN) {
        return run_kernel(c, COMPAMS_K_BS_APPLY, [&] { return launch_bs_apply(c, theta); });
    }
    // (in a whole step Random-k and most selections have delivered their messages already)
    if (!delivers(c)) RC(run_kernel(c, COMPAMS_K_TOPK_SCATTER, [&] { return launch_topk_scatter(c); }));
    RC(run_kernel(c, COMPAMS_K_AMSGRAD, [&] { return launch_amsgrad(c, theta); }));
    return COMPAMS_OK;
}

int step_device(compams_context* c, const void* grads, float* theta) {
    if (c->sparse() && c->identity) {
        ++c->steps_done;
        ++c->iter;
        return run_kernel(c, COMPAMS_K_DENSE_MEAN_AMSGRAD, [&] { return launch_dense_mean_amsgrad(c, grads, theta); });
    }
    c->whole_step = true;
    RC(compress_device(c, grads));
    return apply_device(c, theta);
}

// `ws` null: every buffer is the library's own allocation. `ws` non-null: the buffers are cut from the caller's
// region of `ws_bytes` bytes. `plan` non-null: nothing is created; *plan receives the bytes such a region needs.
int create_handle(compams_handle* out, int32_t n, int32_t n_total, int32_t row0, int64_t d, const int64_t* block_offsets,
                  int32_t num_blocks, int32_t compressor, double k_ratio, float lr, float beta1, float beta2, float eps,
                  void* ws = nullptr, size_t ws_bytes = 0, size_t* plan = nullptr) {
    if ((!out && !plan) || !block_offsets) return COMPAMS_ERR_INVALID_ARG;
    // the tiled kernels address a block with 32-bit coordinates that may run up to two tiles past its end
    if (n < 1 || n_total > 65535 || row0 < 0 || (int64_t)row0 + n > n_total || d < 1 || d > kMaxD ||
        num_blocks < 1 || (int64_t)num_blocks > d)
        return COMPAMS_ERR_INVALID_ARG;
    if (compressor != COMPAMS_TOPK && compressor != COMPAMS_BLOCKSIGN && compressor != COMPAMS_RANDK)
        return COMPAMS_ERR_INVALID_ARG;
    if (compressor != COMPAMS_BLOCKSIGN && !(k_ratio > 0.0 && k_ratio <= 1.0)) return COMPAMS_ERR_INVALID_ARG;
    if (!(lr == lr) || !(beta1 == beta1) || !(beta2 == beta2) || !(eps == eps)) return COMPAMS_ERR_INVALID_ARG;
    if (block_offsets[0] != 0 || block_offsets[num_blocks] != d) return COMPAMS_ERR_INVALID_ARG;
    for (int32_t b = 0; b < num_blocks; ++b)
        if (block_offsets[b + 1] <= block_offsets[b]) return COMPAMS_ERR_INVALID_ARG;

    compams_context* c = new (std::nothrow) compams_context();
    if (!c) return COMPAMS_ERR_ALLOC;
    c->n = n;
    c->n_total = n_total;
    c->row0 = row0;
    c->d = d;
    c->M = num_blocks;
    c->compressor = compressor;
    c->k_ratio = (compressor != COMPAMS_BLOCKSIGN) ? k_ratio : 1.0;
    c->randk = compressor == COMPAMS_RANDK;
    c->hp.lr = lr;
    c->hp.beta1 = beta1;
    c->hp.beta2 = beta2;
    c->hp.omb1 = 1.0f - beta1;
    c->hp.omb2 = 1.0f - beta2;
    c->hp.eps = eps;
    c->chain = (int64_t)n * d <= kChainMaxElems;
    c->first_steps = kFirstSteps;
    c->hp.nf = (float)n_total;
    c->hp.inv_nf = ((n_total & (n_total - 1)) == 0) ? 1.0f / (float)n_total : 0.0f;
    c->plan_only = plan != nullptr;
    c->ws = (unsigned char*)ws;
    c->ws_bytes = ws_bytes;
    int rc;
    try {
        rc = init_context(c, block_offsets);
    } catch (const std::bad_alloc&) {
        rc = COMPAMS_ERR_ALLOC;
    }
    // sharded workers exchange compressed gradients; the uncompressed mode (k = d) has none to exchange
    if (!rc && n != n_total && c->identity) rc = COMPAMS_ERR_INVALID_ARG;
    if (rc || plan) {
        if (!rc) *plan = (c->ws_used + 255) & ~(size_t)255;
        free_context(c);
        return rc;
    }
    *out = c;
    return COMPAMS_OK;
}

}  // namespace

extern "C" {

int compams_create(compams_handle* out, int32_t n, int64_t d, const int64_t* block_offsets, int32_t num_blocks,
                   int32_t compressor, double k_ratio, float lr, float beta1, float beta2, float eps) {
    return create_handle(out, n, n, 0, d, block_offsets, num_blocks, compressor, k_ratio, lr, beta1, beta2, eps);
}

int compams_create_sharded(compams_handle* out, int32_t n_local, int32_t n_total, int32_t first_worker, int64_t d,
                           const int64_t* block_offsets, int32_t num_blocks, int32_t compressor, double k_ratio, float lr,
                           float beta1, float beta2, float eps) {
    return create_handle(out, n_local, n_total, first_worker, d, block_offsets, num_blocks, compressor, k_ratio, lr, beta1,
                         beta2, eps);
}

int compams_workspace_bytes(size_t* bytes, int32_t n_local, int32_t n_total, int64_t d, const int64_t* block_offsets,
                            int32_t num_blocks, int32_t compressor, double k_ratio) {
    if (!bytes) return COMPAMS_ERR_INVALID_ARG;
    return create_handle(nullptr, n_local, n_total, 0, d, block_offsets, num_blocks, compressor, k_ratio, 0.0f, 0.0f, 0.0f,
                         0.0f, nullptr, 0, bytes);
}

int compams_create_in_workspace(compams_handle* out, void* workspace, size_t workspace_bytes, int32_t n_local,
                                int32_t n_total, int32_t first_worker, int64_t d, const int64_t* block_offsets,
                                int32_t num_blocks, int32_t compressor, double k_ratio, float lr, float beta1, float beta2,
                                float eps) {
    if (!workspace || (reinterpret_cast<uintptr_t>(workspace) & 255u)) return COMPAMS_ERR_INVALID_ARG;
    return create_handle(out, n_local, n_total, first_worker, d, block_offsets, num_blocks, compressor, k_ratio, lr, beta1,
                         beta2, eps, workspace, workspace_bytes);
}

static int compress_any(compams_handle c, const void* grads, bool bf16) {
    if (!c || !grads || (reinterpret_cast<uintptr_t>(grads) & (bf16 ? 1u : 3u))) return COMPAMS_ERR_INVALID_ARG;
    if (c->sparse() && c->identity) return COMPAMS_ERR_INVALID_ARG;  // k = d: nothing is compressed
    if (c->compressed) return COMPAMS_ERR_INVALID_ARG;  // the previous compress has not been applied yet
    RC(on_handle_device(c));
    c->grad_bf16 = bf16;
    c->whole_step = false;
    int rc;
    try {
        rc = compress_device(c, grads);
    } catch (const std::bad_alloc&) {
        rc = COMPAMS_ERR_ALLOC;
    }
    if (!rc) c->compressed = true;
    return rc;
}

int compams_compress(compams_handle c, const float* grads) { return compress_any(c, grads, false); }
int compams_compress_bf16(compams_handle c, const void* grads_bf16) { return compress_any(c, grads_bf16, true); }

int compams_apply(compams_handle c, float* theta) {
    if (!c || !theta || (reinterpret_cast<uintptr_t>(theta) & 15u)) return COMPAMS_ERR_INVALID_ARG;
    if (c->sparse() && c->identity) return COMPAMS_ERR_INVALID_ARG;
    if (!c->compressed) return COMPAMS_ERR_INVALID_ARG;  // nothing to apply: compams_compress comes first
    RC(on_handle_device(c));
    c->compressed = false;
    try {
        return apply_device(c, theta);
    } catch (const std::bad_alloc&) {
        return COMPAMS_ERR_ALLOC;
    }
}

static int step_any(compams_handle c, const void* grads, float* theta, bool bf16) {
    if (!c || !grads || !theta) return COMPAMS_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(grads) & (bf16 ? 1u : 3u)) || (reinterpret_cast<uintptr_t>(theta) & 15u))
        return COMPAMS_ERR_INVALID_ARG;
    if (c->n != c->n_total) return COMPAMS_ERR_INVALID_ARG;  // the other workers' messages have to be exchanged first
    if (c->compressed) return COMPAMS_ERR_INVALID_ARG;       // a compams_compress is waiting for its compams_apply
    RC(on_handle_device(c));
    c->grad_bf16 = bf16;
    try {
        return step_device(c, grads, theta);
    } catch (const std::bad_alloc&) {
        return COMPAMS_ERR_ALLOC;
    }
}

int compams_step(compams_handle c, const float* grads, float* theta) { return step_any(c, grads, theta, false); }
int compams_step_bf16(compams_handle c, const void* grads_bf16, float* theta) { return step_any(c, grads_bf16, theta, true); }

int compams_step_host(compams_handle c, const float* grads_host, float* theta_host) {
    if (!c || !grads_host || !theta_host || c->n != c->n_total || c->compressed) return COMPAMS_ERR_INVALID_ARG;
    RC(on_handle_device(c));
    const size_t gbytes = (size_t)c->n * (size_t)c->d * sizeof(float);
    const size_t tbytes = (size_t)c->d * sizeof(float);
    if (!c->stage_grads) {
        cudaError_t e = cudaMalloc((void**)&c->stage_grads, gbytes);
        if (e != cudaSuccess) {
            c->stage_grads = nullptr;
            cudaGetLastError();
            return COMPAMS_ERR_ALLOC;
        }
        e = cudaMalloc((void**)&c->stage_theta, tbytes);
        if (e != cudaSuccess) {
            c->stage_theta = nullptr;
            cudaGetLastError();
            return COMPAMS_ERR_ALLOC;
        }
    }
    CU(cudaMemcpyAsync(c->stage_grads, grads_host, gbytes, cudaMemcpyHostToDevice, c->stream));
    CU(cudaMemcpyAsync(c->stage_theta, theta_host, tbytes, cudaMemcpyHostToDevice, c->stream));
    int rc;
    c->grad_bf16 = false;
    try {
        rc = step_device(c, c->stage_grads, c->stage_theta);
    } catch (const std::bad_alloc&) {
        rc = COMPAMS_ERR_ALLOC;
    }
    if (rc) return rc;
    CU(cudaMemcpyAsync(theta_host, c->stage_theta, tbytes, cudaMemcpyDeviceToHost, c->stream));
    CU(cudaStreamSynchronize(c->stream));
    return COMPAMS_OK;
}

int compams_destroy(compams_handle c) {
    if (!c) return COMPAMS_OK;
    cudaStreamSynchronize(c->stream);
    free_context(c);
    return COMPAMS_OK;
}

int compams_set_stream(compams_handle c, void* cuda_stream) {
    if (!c) return COMPAMS_ERR_INVALID_ARG;
    c->stream = (cudaStream_t)cuda_stream;
    return COMPAMS_OK;
}

int compams_set_seed(compams_handle c, uint64_t seed, uint64_t iterations_done) {
    if (!c || c->compressed) return COMPAMS_ERR_INVALID_ARG;
    c->seed = seed;
    c->iter = iterations_done;
    return COMPAMS_OK;
}

int compams_record_average(compams_handle c, int on) {
    if (!c) return COMPAMS_ERR_INVALID_ARG;
    c->record_gbar = on != 0;
    c->tk.gbar = c->record_gbar ? c->gbar : nullptr;
    c->bs.gbar = c->record_gbar ? c->gbar : nullptr;
    return COMPAMS_OK;
}

int compams_set_lr(compams_handle c, float lr) {
    if (!c || !(lr == lr)) return COMPAMS_ERR_INVALID_ARG;
    c->hp.lr = lr;
    return COMPAMS_OK;
}

// Finishes the residual update where it has been deferred, so that E holds e.
static int finish_residual(compams_context* c) {
    if (c->sparse() && !c->identity && c->e_mask_pending) {
        RC(run_kernel(c, COMPAMS_K_TOPK_MATERIALIZE, [&] { return launch_topk_materialize(c); }));
        c->e_mask_pending = false;
    }
    if (c->compressor == COMPAMS_BLOCKSIGN && c->e_is_x) {
        RC(run_kernel(c, COMPAMS_K_BS_MATERIALIZE, [&] { return launch_bs_materialize(c); }));
        c->e_is_x = false;
    }
    return COMPAMS_OK;
}

int compams_get_state(compams_handle c, float* e, float* m, float* v, float* vhat) {
    if (!c || c->compressed) return COMPAMS_ERR_INVALID_ARG;  // between compress and apply the step is half done
    RC(on_handle_device(c));
    const size_t nd = (size_t)c->n * (size_t)c->d * sizeof(float), db = (size_t)c->d * sizeof(float);
    if (e) {
        if (c->E) {
            RC(finish_residual(c));
            CU(cudaMemcpyAsync(e, c->E, nd, cudaMemcpyDeviceToDevice, c->stream));
        } else {
            CU(cudaMemsetAsync(e, 0, nd, c->stream));
        }
    }
    if (m) CU(cudaMemcpyAsync(m, c->m, db, cudaMemcpyDeviceToDevice, c->stream));
    if (v) CU(cudaMemcpyAsync(v, c->v, db, cudaMemcpyDeviceToDevice, c->stream));
    if (vhat) CU(cudaMemcpyAsync(vhat, c->vhat, db, cudaMemcpyDeviceToDevice, c->stream));
    return COMPAMS_OK;
}

int compams_set_state(compams_handle c, const float* e, const float* m, const float* v, const float* vhat) {
    if (!c || c->compressed) return COMPAMS_ERR_INVALID_ARG;
    RC(on_handle_device(c));
    const size_t nd = (size_t)c->n * (size_t)c->d * sizeof(float), db = (size_t)c->d * sizeof(float);
    if (e && c->E) {
        CU(cudaMemcpyAsync(c->E, e, nd, cudaMemcpyDeviceToDevice, c->stream));
        // E now holds e itself; predictions made from the replaced accumulators are dropped
        c->e_is_x = false;
        c->e_mask_pending = false;
        c->first_steps = kFirstSteps;
        if (c->tk.seg && !c->seg_init_host.empty()) {
            CU(cudaMemcpyAsync(c->tk.seg, c->seg_init_host.data(), c->seg_init_host.size() * sizeof(SegState),
                               cudaMemcpyHostToDevice, c->stream));
            CU(cudaMemcpyAsync(c->tk.dense_count, &c->dense_count_init, sizeof(uint32_t), cudaMemcpyHostToDevice,
                               c->stream));
        }
    }
    if (m) CU(cudaMemcpyAsync(c->m, m, db, cudaMemcpyDeviceToDevice, c->stream));
    if (v) CU(cudaMemcpyAsync(c->v, v, db, cudaMemcpyDeviceToDevice, c->stream));
    if (vhat) CU(cudaMemcpyAsync(c->vhat, vhat, db, cudaMemcpyDeviceToDevice, c->stream));
    return COMPAMS_OK;
}

int compams_bits_transmitted(compams_handle c, uint64_t* out) {
    if (!c || !out) return COMPAMS_ERR_INVALID_ARG;
    const uint64_t full = 32ull * (uint64_t)c->n * (uint64_t)c->d;
    uint64_t payload = full, index = 0;
    if (c->compressor == COMPAMS_BLOCKSIGN) {
        payload = (uint64_t)c->n * ((uint64_t)c->d + 32ull * (uint64_t)c->M);
    } else if (!c->identity) {
        payload = 32ull * (uint64_t)c->n * (uint64_t)c->K;
        index = payload;
    }
    out[0] = full * c->steps_done;
    out[1] = payload * c->steps_done;
    out[2] = index * c->steps_done;
    return COMPAMS_OK;
}

int compams_get_buffer(compams_handle c, int32_t which, void** dev_ptr, int64_t* count) {
    if (!c || !dev_ptr || !count) return COMPAMS_ERR_INVALID_ARG;
    void* p = nullptr;
    int64_t cnt = 0;
    const bool topk = c->sparse() && !c->identity;
    const bool sign = c->compressor == COMPAMS_BLOCKSIGN;
    switch (which) {
        case COMPAMS_BUF_E:
            if (c->compressed) return COMPAMS_ERR_INVALID_ARG;  // the residual is closed by compams_apply
            if (!c->E) break;  // every k_b = d_b: e is identically zero and not stored
            RC(on_handle_device(c));
            RC(finish_residual(c));
            p = c->E;
            cnt = (int64_t)c->n * c->d;
            break;
        case COMPAMS_BUF_M: p = c->m; cnt = c->d; break;
        case COMPAMS_BUF_V: p = c->v; cnt = c->d; break;
        case COMPAMS_BUF_VHAT: p = c->vhat; cnt = c->d; break;
        case COMPAMS_BUF_GBAR:
            if (!c->record_gbar) return COMPAMS_ERR_INVALID_ARG;  // not being written
            p = c->gbar; cnt = c->d; break;
        case COMPAMS_BUF_TOPK_IDX: if (topk) { p = c->tk.idx; cnt = (int64_t)c->n_total * c->K; } break;
        case COMPAMS_BUF_TOPK_VAL: if (topk) { p = c->tk.val; cnt = (int64_t)c->n_total * c->K; } break;
        case COMPAMS_BUF_TOPK_SEG_OFFSETS: if (topk) { p = c->d_seg_off; cnt = c->M + 1; } break;
        case COMPAMS_BUF_SIGN_BITS: if (sign) { p = c->bs.bits; cnt = (int64_t)c->n_total * c->W; } break;
        case COMPAMS_BUF_SIGN_WORD_OFFSETS: if (sign) { p = c->d_word_off; cnt = c->M + 1; } break;
        case COMPAMS_BUF_SCALES: if (sign) { p = c->scales[c->scales_cur]; cnt = (int64_t)c->n_total * c->M; } break;
        case COMPAMS_BUF_STATUS: p = c->status; cnt = 8; break;
        default: return COMPAMS_ERR_INVALID_ARG;
    }
    *dev_ptr = p;
    *count = cnt;
    return COMPAMS_OK;
}

int compams_check_status(compams_handle c, uint32_t* status_word) {
    if (!c) return COMPAMS_ERR_INVALID_ARG;
    CU(cudaStreamSynchronize(c->stream));
    uint32_t w = 0;
    CU(cudaMemcpy(&w, c->status, sizeof w, cudaMemcpyDeviceToHost));
    if (status_word) *status_word = w;
    return w ? COMPAMS_ERR_DEVICE_STATUS : COMPAMS_OK;
}

int compams_set_profiling(compams_handle c, uint32_t kernel_mask) {
    if (!c) return COMPAMS_ERR_INVALID_ARG;
    CU(cudaStreamSynchronize(c->stream));
    c->prof_mask = kernel_mask;
    c->prof_used = 0;
    return COMPAMS_OK;
}

int compams_get_kernel_time(compams_handle c, int32_t kernel, double* total_ms, int64_t* launches) {
    if (!c || !total_ms || !launches || kernel < 0 || kernel >= COMPAMS_K_COUNT) return COMPAMS_ERR_INVALID_ARG;
    CU(cudaStreamSynchronize(c->stream));
    double ms = 0.0;
    int64_t cnt = 0;
    for (int s = 0; s < c->prof_used; ++s) {
        if (c->ev_kernel[(size_t)s] != kernel) continue;
        float t = 0.0f;
        CU(cudaEventElapsedTime(&t, c->ev_start[(size_t)s], c->ev_stop[(size_t)s]));
        ms += (double)t;
        ++cnt;
    }
    *total_ms = ms;
    *launches = cnt;
    return COMPAMS_OK;
}

int64_t compams_launch_count(compams_handle c) { return c ? c->launches : 0; }

const char* compams_error_string(int status) {
    switch (status) {
        case COMPAMS_OK: return "ok";
        case COMPAMS_ERR_INVALID_ARG: return "invalid argument";
        case COMPAMS_ERR_ALLOC: return "allocation failed";
        case COMPAMS_ERR_CUDA: return "CUDA runtime error";
        case COMPAMS_ERR_DEVICE_STATUS: return "device status word is set";
        case COMPAMS_ERR_TOO_LARGE: return "problem size exceeds the fixed scratch capacity";
        default: return "unknown status";
    }
}

const char* compams_kernel_name(int32_t kernel) {
    static const char* names[COMPAMS_K_COUNT] = {
        "dense_mean_amsgrad", "bs_sweep", "bs_apply", "bs_materialize", "topk_sweep", "topk_dense",
        "topk_materialize", "randk_emit", "reserved", "topk_scatter", "amsgrad", "topk_small", "topk_select", "bs_scales"};
    return (kernel >= 0 && kernel < COMPAMS_K_COUNT) ? names[kernel] : "unknown";
}

const char* compams_last_cuda_error(void) { return g_last_cuda_error.c_str(); }

}  // extern "C"
