// Prediction of a segment's next selection threshold and of how many candidates it should let through.
#pragma once

#include "context.h"

namespace compams {

// Prediction for the next step's sweep, from this step's threshold key `tau` and the bin edge
// `edge` at or above which about the wanted number of candidates (want_candidates) lay: the threshold keeps rising while the error
// accumulators fill, so tau_hat follows half of the last rise. `sel_shift` sizes the bins of the
// next select so that the expected threshold lands near the middle of its 4096 bins.
__device__ __forceinline__ void predict_next(SegState* st, uint32_t tau, uint32_t edge, bool enabled) {
    const uint32_t prev = st->tau_prev;
    uint32_t rise = 0;
    if (prev != kNoPrediction && tau > prev) rise = (tau - prev) >> 1;
    if (edge > tau) edge = tau;
    uint32_t next = edge + rise;
    if (next >= 0x7f800000u) next = edge;
    const uint32_t tau_pred = tau + rise;
    uint32_t span = tau_pred > next ? tau_pred - next : 1u;
    // ... but never so fine that the bins end close above the prediction: they cover at least a quarter of a
    // binade (values up to about 19 % above tau_hat), so a threshold that lands higher than predicted - gradients
    // that alternate between two levels do that - is still found inside the list
    if (span < (1u << 19)) span = 1u << 19;
    st->sel_shift = 32u - (uint32_t)__clz(span >> 11);  // smallest S with span >> S < 2048
    st->tau_hat = enabled ? next : kNoPrediction;
    st->tau_prev = tau;
}

// How many candidates the next step's predicted threshold should let through for a segment that keeps kb: the
// count of keys above a fixed threshold moves by about sqrt(kb) from one step to the next (eight of those are
// allowed for), plus a quarter of kb for drift of the gradient scale. A segment whose list came up short gets
// its margin doubled (`boost` times, at most three); the doubling is taken back one step at a time after enough
// selections in a row were decided inside the list (margin_held). Long lists thus carry about 1.26 kb entries, short ones
// (kb = 50: 170) proportionally more.
__device__ __forceinline__ uint32_t want_candidates(uint32_t kb, uint32_t boost, uint32_t cap) {
    const uint32_t margin = ((kb >> 2) + (uint32_t)(8.0f * sqrtf((float)kb)) + 32u) << (boost < 3u ? boost : 3u);
    uint32_t most = 4u * kb + 512u;
    if (most > cap - cap / 4u) most = cap - cap / 4u;  // room for a threshold that lets more through
    if (most < kb) return kb;                          // (cap = 0: the block has no list)
    return kb + (margin < most - kb ? margin : most - kb);
}
// Taking a doubling back is a probe: if the smaller margin comes up short (a dense-pass step, which costs several
// ordinary steps), the margin was needed, and the next probe waits twice as long (32, 64, ... 32768 selections). A
// probe that holds for a whole waiting time halves the wait again. Gradients that alternate between two levels
// need the first doubling for good: with a fixed wait of 32 every 33rd step ran the dense passes (n = 32,
// d = 2^27: 9.1 -> 9.6 ms per step on average).
constexpr uint32_t kHoldMax = 10u;
__device__ __forceinline__ void margin_came_up_short(SegState* st) {
    if (st->boost < 3u) ++st->boost;
    if (st->probing && st->hold < kHoldMax) ++st->hold;
    st->probing = 0u;
    st->streak = 0u;
}
__device__ __forceinline__ void margin_held(SegState* st) {
    if (++st->streak >= (32u << st->hold)) {
        st->streak = 0u;
        if (st->probing && st->hold) --st->hold;
        st->probing = 0u;
        if (st->boost) {
            --st->boost;
            st->probing = 1u;
        }
    }
}

// After a selection decided inside its list of c candidates: a list that held by less than a quarter of its margin
// was a near miss and is treated like a list that came up short, only without the dense passes (thresholds that
// swing from step to step announce themselves this way: d = 2^24, n = 8, two alternating batches: 1.01 k_b
// candidates a dozen steps before 0.94 k_b).
__device__ __forceinline__ void margin_after_selection(SegState* st, uint32_t kb, uint32_t c, uint32_t cap) {
    if (c - kb < (want_candidates(kb, st->boost, cap) - kb) >> 2) margin_came_up_short(st);
    else margin_held(st);
}

}  // namespace compams
