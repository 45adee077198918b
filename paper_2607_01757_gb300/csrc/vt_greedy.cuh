// The greedy min-distance selection for candidates that crowd together, shared
// by the detector's selection and the track bookkeeping.
//
// Both resolve the selection in rounds: a candidate is decided once every
// closer one of higher priority is.  A round walks lists of neighbours, so
// where hundreds of candidates lie within min_dist of each other it takes tens
// of microseconds, and where each depends on the one before it there are as
// many rounds as candidates.  Both leave such sets to greedy_in_order: the next
// 32 undecided candidates are decided by one warp among themselves, the rest of
// the CTA drops what is closer than min_dist to those of them that are kept,
// and so on.  That is at most a step of about 1 us per 32 candidates, and far
// fewer where they crowd, since each kept one takes many others with it.
#pragma once

#include <stdint.h>

namespace vt {

enum : uint8_t { GR_UNDECIDED = 0, GR_KEPT = 1, GR_DROPPED = 2 };

struct GreedySmem {
    int cand[32], kept[32];
    int front, n_kept;
};

// Decides the candidates of 0 .. n - 1 (by priority) that are undecided in
// `state`; closer(a, b): whether a and b lie closer than min_dist.  Every thread
// of the CTA calls it, after a barrier; the states are final when it returns.
template <typename Closer>
__device__ __forceinline__ void greedy_in_order(volatile uint8_t *state, int n, GreedySmem &S, Closer &&closer) {
    const int t = threadIdx.x, lane = t & 31;
    const unsigned full = 0xffffffffu;
    for (int front = 0; front < n;) {
        if (t < 32) {
            // the next 32 undecided ones
            int f = front, cnt = 0;
            while (cnt < 32 && f < n) {
                const bool u = f + lane < n && state[f + lane] == GR_UNDECIDED;
                const unsigned m = __ballot_sync(full, u);
                const int at = cnt + __popc(m & ((1u << lane) - 1u));
                if (u && at < 32) S.cand[at] = f + lane;
                const unsigned last = __ballot_sync(full, u && at == 31);
                cnt = min(32, cnt + __popc(m));
                f += last ? __ffs(last) : 32;
            }
            __syncwarp();
            const int c = lane < cnt ? S.cand[lane] : -1;
            unsigned before = 0;  // those of them that come first and are closer
            for (int j = 0; j < cnt; ++j)
                if (j < lane && c >= 0 && closer(c, S.cand[j])) before |= 1u << j;
            unsigned kept = 0, open = cnt < 32 ? (1u << cnt) - 1u : full;
            while (open) {  // (the first open one is decided each time)
                const bool decided = ((open >> lane) & 1u) && !(before & open);
                kept |= __ballot_sync(full, decided && !(before & kept));
                open &= ~__ballot_sync(full, decided);
            }
            if (c >= 0) {
                const bool k = (kept >> lane) & 1u;
                state[c] = k ? GR_KEPT : GR_DROPPED;
                if (k) S.kept[__popc(kept & ((1u << lane) - 1u))] = c;
            }
            if (lane == 0) S.front = f, S.n_kept = __popc(kept);
        }
        __syncthreads();
        front = S.front;
        const int nk = S.n_kept;
        for (int q = t; q < n; q += blockDim.x) {
            if (q < front || state[q] != GR_UNDECIDED) continue;
            for (int k = 0; k < nk; ++k)
                if (closer(q, S.kept[k])) {
                    state[q] = GR_DROPPED;
                    break;
                }
        }
        __syncthreads();
    }
}

}  // namespace vt
