// Track bookkeeping (K8) for many camera streams at once: identity
// carry-over with age-priority thinning, and spawning of new tracks from
// detections up to each stream's cap.  One CTA per stream; every stream's
// pool stays on the device, counts included, so a step needs no host round
// trip.
//
//   k_tracks_carry  survivors of the temporal step (status 1) in index order,
//                   ages + 1, sorted by (age desc, index asc) in shared
//                   memory (a pool these kernels wrote is in that order and
//                   only checked); the greedy min-distance thinning in that
//                   order finds each survivor's closer higher-priority ones
//                   over a cell grid in shared memory and resolves them in
//                   parallel rounds (a survivor is kept when no kept
//                   higher-priority survivor lies closer than min_dist,
//                   dropped when one does), or one by one where they crowd
//                   (greedy_in_order); kept survivors rewrite the pool in priority order
//                   and, optionally, a detector mask padded with NaN.
//   k_tracks_spawn  accepted detections, in their priority order, appended
//                   until the pool holds `cap` features, with identities
//                   next_id, next_id + 1, ... and age 1.
// Distances are single precision, dx*dx + dy*dy rounded operation by
// operation, as in the oracle, so the result is exact.
#include <cmath>
#include <cstdint>

#include "vt_greedy.cuh"
#include "vt_internal.cuh"

namespace vt {

constexpr int TK_THREADS = 1024;    // threads of the largest CTA
constexpr int TK_MAX_CELLS = 8192;  // the grid's cells: at most TK_CELLS_PER a
constexpr int TK_MIN_CELLS = 4096;  // survivor, within these limits
constexpr int TK_CELLS_PER = 8;
constexpr int kMaxPoolJobs = 192;
// Pools left to greedy_in_order: where a survivor would have to look at more than
// TK_WALK others (TK_WALK_LARGE in pools of more than TK_THREADS, where it costs
// up to 128 steps of 7 us), or TK_ROUNDS rounds have not settled the pool.
constexpr int TK_WALK = 32, TK_WALK_LARGE = 128, TK_ROUNDS = 8;
enum : uint8_t { TK_UNDECIDED = GR_UNDECIDED, TK_KEPT = GR_KEPT, TK_DROPPED = GR_DROPPED };

struct CarryJobs {
    int n;
    float min_dist;
    vt_carry_job j[kMaxPoolJobs];
};

struct SpawnJobs {
    int n;
    vt_spawn_job j[kMaxPoolJobs];
};

// Exclusive block-wide scan of one int per thread; the total through *total.
__device__ __forceinline__ int block_scan(int v, int *warp_sums, int *total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[wid] = x;
    __syncthreads();
    int s = lane < (int)(blockDim.x >> 5) ? warp_sums[lane] : 0;  // every warp sums the warps for itself
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += y;
    }
    *total = __shfl_sync(0xffffffffu, s, 31);
    const int before = __shfl_sync(0xffffffffu, s, wid > 0 ? wid - 1 : 0);
    __syncthreads();  // warp_sums may be written again
    return x - v + (wid > 0 ? before : 0);
}

__device__ __forceinline__ float dist2(float2 a, float2 b) {
    const float dx = __fsub_rn(a.x, b.x), dy = __fsub_rn(a.y, b.y);
    return __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
}

struct CarrySmem {
    float2 pos[VT_POOL_MAX];               // survivor positions by survivor rank
    float2 sorted[VT_POOL_MAX];            // and by priority, where that is another order
    int32_t id[VT_POOL_MAX];
    int32_t age[VT_POOL_MAX];              // already + 1
    union {
        unsigned long long key[VT_POOL_MAX];  // (age << 32) | ~rank, sorted descending
        short4 closer[VT_POOL_MAX];           // by priority: the first closer higher-priority survivors (see k_tracks_carry)
    };
    int16_t rank[VT_POOL_MAX];             // of the survivor at a priority position
    int16_t next[VT_POOL_MAX];             // a cell's survivors, linked from its head
    int head[TK_MAX_CELLS];
    uint8_t state[VT_POOL_MAX];
    int warp_sums[32];
    float red[4][32];
    GreedySmem greedy;
};

// Calls f(o) for the survivors o of higher priority than q that lie closer to
// it than min_dist, until f returns false; false when more than `left`
// survivors would have to be looked at.
template <typename F>
__device__ __forceinline__ bool each_closer(const CarrySmem &S, const float2 *pos, int q, int ix, int iy, int cx, int cy,
                                            float md2, int left, F &&f) {
    const float2 p = pos[q];
    for (int yy = max(0, iy - 1); yy <= min(cy - 1, iy + 1); ++yy)
        for (int xx = max(0, ix - 1); xx <= min(cx - 1, ix + 1); ++xx)
            for (int o = S.head[yy * cx + xx]; o >= 0; o = S.next[o]) {
                if (left-- == 0) return false;
                if (o < q && dist2(p, pos[o]) < md2 && !f(o)) return true;
            }
    return true;
}

// Bound by latency: one CTA per pool, dependent reads and barriers.  A pool as
// the last carry-over and spawning left it needs no sort (66 passes over the
// keys of 2,000 survivors), and the grid is walked once: a survivor's first
// three closer ones of higher priority are kept in `closer`, so a round reads
// three states.  Cold caches, launch included: 8 pools of 250 25 -> 12.5 us,
// 32 of 1,000 41 -> 18, 32 of 2,000 67 -> 22; out of order, 32 of 1,000
// 39 -> 29.  Most of what is left is the launch and three dependent reads from
// memory (count, status, positions).  Crowded pools are left to greedy_in_order
// (one pool, launches of its set-up included): 60 / 1,000 / 4,096 survivors in one
// place 25 / 31 / 59 us (in rounds 235 / 449 / 43,000), a line of 4,096 each in
// conflict with the two before it 738 (2,170), 4,096 spread over 10 min_dist
// squared 89 (1,640).
__global__ void __launch_bounds__(TK_THREADS, 1) k_tracks_carry(const __grid_constant__ CarryJobs J) {
    extern __shared__ __align__(16) uint8_t tk_smem[];
    CarrySmem &S = *reinterpret_cast<CarrySmem *>(tk_smem);
    const vt_carry_job &jb = J.j[blockIdx.x];
    const vt_track_pool &P = jb.pool;
    const float2 *tracked = reinterpret_cast<const float2 *>(jb.tracked);
    const int t = threadIdx.x, T = blockDim.x;
    pdl_wait();  // the tracked positions may be the previous kernel's output
    const int n = min(*P.count, P.cap);
    // 1. survivors in index order (`per` consecutive entries per thread)
    const int per = (n + T - 1) / T;
    int mine = 0;
    for (int k = 0; k < per; ++k) {
        const int i = t * per + k;
        mine += (i < n && jb.status[i] != 0) ? 1 : 0;
    }
    int m;
    int r = block_scan(mine, S.warp_sums, &m);
    for (int k = 0; k < per; ++k) {
        const int i = t * per + k;
        if (i < n && jb.status[i] != 0) {
            S.pos[r] = tracked[i];
            S.id[r] = P.ids[i];
            S.age[r] = P.ages[i] + 1;
            ++r;
        }
    }
    __syncthreads();
    // 2. priority order: age descending, then survivor rank ascending
    int unsorted = 0;
    for (int i = t; i + 1 < m; i += T) unsorted |= (uint32_t)S.age[i] < (uint32_t)S.age[i + 1];
    const float2 *pos = S.pos;  // by priority
    if (__syncthreads_or(unsorted)) {
        int N = 1;
        while (N < m) N <<= 1;
        for (int i = t; i < N; i += T)
            S.key[i] = i < m ? ((unsigned long long)(uint32_t)S.age[i] << 32) | (0xffffffffu - (unsigned)i) : 0ull;
        __syncthreads();
        for (int k = 2; k <= N; k <<= 1)  // bitonic, descending keys
            for (int j = k >> 1; j > 0; j >>= 1) {
                for (int i = t; i < N; i += T) {
                    const int p = i ^ j;
                    if (p > i) {
                        const unsigned long long a = S.key[i], b = S.key[p];
                        if (((i & k) == 0) ? (a < b) : (a > b)) {
                            S.key[i] = b;
                            S.key[p] = a;
                        }
                    }
                }
                __syncthreads();
            }
        for (int q = t; q < m; q += T) {
            const int s = 0xffffffffu - (unsigned)(S.key[q] & 0xffffffffu);
            S.rank[q] = (int16_t)s;
            S.sorted[q] = S.pos[s];
        }
        pos = S.sorted;
    } else {
        for (int q = t; q < m; q += T) S.rank[q] = (int16_t)q;
    }
    // 3. cell grid over the survivors' bounding box: cells wider than
    //    min_dist (by 0.1 %, so rounding cannot separate a close pair by two
    //    cells); a cell holds less than a survivor of a spread-out pool
    float lo_x = INFINITY, lo_y = INFINITY, hi_x = -INFINITY, hi_y = -INFINITY;
    for (int i = t; i < m; i += T) {
        const float2 p = S.pos[i];
        if (!isfinite(p.x) || !isfinite(p.y)) continue;  // non-finite points share cell 0
        lo_x = fminf(lo_x, p.x);
        lo_y = fminf(lo_y, p.y);
        hi_x = fmaxf(hi_x, p.x);
        hi_y = fmaxf(hi_y, p.y);
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        lo_x = fminf(lo_x, __shfl_xor_sync(0xffffffffu, lo_x, o));
        lo_y = fminf(lo_y, __shfl_xor_sync(0xffffffffu, lo_y, o));
        hi_x = fmaxf(hi_x, __shfl_xor_sync(0xffffffffu, hi_x, o));
        hi_y = fmaxf(hi_y, __shfl_xor_sync(0xffffffffu, hi_y, o));
    }
    if ((t & 31) == 0) {
        S.red[0][t >> 5] = lo_x;
        S.red[1][t >> 5] = lo_y;
        S.red[2][t >> 5] = hi_x;
        S.red[3][t >> 5] = hi_y;
    }
    __syncthreads();
    {  // (every warp reduces the warps' boxes for itself)
        const int w = min(t & 31, (T >> 5) - 1);
        lo_x = S.red[0][w], lo_y = S.red[1][w], hi_x = S.red[2][w], hi_y = S.red[3][w];
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        lo_x = fminf(lo_x, __shfl_xor_sync(0xffffffffu, lo_x, o));
        lo_y = fminf(lo_y, __shfl_xor_sync(0xffffffffu, lo_y, o));
        hi_x = fmaxf(hi_x, __shfl_xor_sync(0xffffffffu, hi_x, o));
        hi_y = fmaxf(hi_y, __shfl_xor_sync(0xffffffffu, hi_y, o));
    }
    const float md = J.min_dist, md2 = __fmul_rn(md, md);
    float cs = md * 1.001f;
    int cx = 1, cy = 1;
    if (lo_x <= hi_x && lo_y <= hi_y) {  // some finite survivor
        const float most = (float)min(TK_MAX_CELLS, max(TK_MIN_CELLS, TK_CELLS_PER * m));
        int tries = 0;
        for (;; ++tries) {
            const float fx = floorf((hi_x - lo_x) / cs) + 1.f, fy = floorf((hi_y - lo_y) / cs) + 1.f;
            if (fx * fy <= most) {
                cx = (int)fx;
                cy = (int)fy;
                break;
            }
            if (tries == 64) break;  // one cell for everything: still exact, only slower
            cs *= 1.5f;
        }
    } else {
        lo_x = lo_y = 0.f;
    }
    for (int c = t; c < cx * cy; c += T) S.head[c] = -1;
    __syncthreads();
    auto cell = [&](float2 p, int &ix, int &iy) {
        ix = clampi((int)floorf((p.x - lo_x) / cs), 0, cx - 1);
        iy = clampi((int)floorf((p.y - lo_y) / cs), 0, cy - 1);
    };
    for (int q = t; q < m; q += T) {  // q: priority position
        int ix, iy;
        cell(pos[q], ix, iy);
        S.next[q] = (int16_t)atomicExch(&S.head[iy * cx + ix], q);
    }
    __syncthreads();
    // 4. greedy thinning.  Each survivor's closer ones of higher priority: the
    //    first three, and w = -2 if there are more; with none it is kept.
    const int walk = m <= TK_THREADS ? TK_WALK : TK_WALK_LARGE;
    int crowded = 0;
    for (int q = t; q < m; q += T) {
        int ix, iy, found = 0;
        cell(pos[q], ix, iy);
        short4 c = make_short4(-1, -1, -1, -1);
        const bool all = each_closer(S, pos, q, ix, iy, cx, cy, md2, walk, [&](int o) {
            if (found == 0) c.x = (short)o;
            else if (found == 1) c.y = (short)o;
            else if (found == 2) c.z = (short)o;
            else c.w = -2;
            return ++found < 4;
        });
        crowded |= !all;
        S.closer[q] = c;
        S.state[q] = found ? TK_UNDECIDED : TK_KEPT;
    }
    crowded = __syncthreads_or(crowded);
    //    Rounds: the undecided survivor of highest priority is decided in each.
    for (int round = 0; !crowded; ++round) {
        int undecided = 0;
        for (int q = t; q < m; q += T) {
            volatile uint8_t *state = S.state;
            if (state[q] != TK_UNDECIDED) continue;
            const short4 c = S.closer[q];
            const uint8_t sx = state[c.x], sy = c.y >= 0 ? state[c.y] : (uint8_t)TK_DROPPED,
                          sz = c.z >= 0 ? state[c.z] : (uint8_t)TK_DROPPED;
            bool dropped = sx == TK_KEPT || sy == TK_KEPT || sz == TK_KEPT;
            bool blocked = sx == TK_UNDECIDED || sy == TK_UNDECIDED || sz == TK_UNDECIDED;
            if (c.w == -2 && !dropped && !blocked) {  // the three are dropped: all of them
                int ix, iy;
                cell(pos[q], ix, iy);
                const bool all = each_closer(S, pos, q, ix, iy, cx, cy, md2, walk, [&](int o) {
                    const uint8_t so = state[o];
                    dropped = so == TK_KEPT;
                    blocked |= so == TK_UNDECIDED;
                    return !dropped;
                });
                blocked |= !all;
            }
            if (dropped) state[q] = TK_DROPPED;
            else if (!blocked) state[q] = TK_KEPT;
            else undecided = 1;
        }
        if (!__syncthreads_or(undecided)) break;
        crowded = round + 1 == TK_ROUNDS;
    }
    if (crowded) {  // the same decisions one by one
        for (int q = t; q < m; q += T) S.state[q] = TK_UNDECIDED;
        __syncthreads();
        greedy_in_order(S.state, m, S.greedy, [&](int a, int b) { return dist2(pos[a], pos[b]) < md2; });
    }
    // 5. the kept survivors, in priority order, rewrite the pool
    const int perm = (m + T - 1) / T;
    int kept_mine = 0;
    for (int k = 0; k < perm; ++k) {
        const int q = t * perm + k;
        kept_mine += (q < m && S.state[q] == TK_KEPT) ? 1 : 0;
    }
    int kept;
    int w = block_scan(kept_mine, S.warp_sums, &kept);
    float2 *pts = reinterpret_cast<float2 *>(P.pts);
    float2 *mask = reinterpret_cast<float2 *>(jb.mask);
    for (int k = 0; k < perm; ++k) {
        const int q = t * perm + k;
        if (q < m && S.state[q] == TK_KEPT) {
            const int s = S.rank[q];
            pts[w] = S.pos[s];
            P.ids[w] = S.id[s];
            P.ages[w] = S.age[s];
            if (mask) mask[w] = S.pos[s];
            ++w;
        }
    }
    if (mask)
        for (int i = kept + t; i < P.cap; i += T) mask[i] = make_float2(NAN, NAN);
    if (t == 0) *P.count = kept;
}

__global__ void __launch_bounds__(TK_THREADS) k_tracks_spawn(const __grid_constant__ SpawnJobs J) {
    __shared__ int warp_sums[32];
    const vt_spawn_job &jb = J.j[blockIdx.x];
    const vt_track_pool &P = jb.pool;
    const int T = blockDim.x;
    pdl_wait();  // the detections may be the previous kernel's output
    const int c0 = min(*P.count, P.cap), nc = *jb.n_corners;
    const int room = P.cap - c0, id0 = *P.next_id;
    const float2 *corners = reinterpret_cast<const float2 *>(jb.corners);
    float2 *pts = reinterpret_cast<float2 *>(P.pts);
    int base = 0;
    for (int b0 = 0; b0 < nc && base < room; b0 += T) {  // chunks of T detections, in order
        const int i = b0 + threadIdx.x;
        const int a = (i < nc && (!jb.accept || jb.accept[i] != 0)) ? 1 : 0;
        int total;
        const int r = base + block_scan(a, warp_sums, &total);
        if (a && r < room) {
            pts[c0 + r] = corners[i];
            P.ids[c0 + r] = id0 + r;
            P.ages[c0 + r] = 1;
        }
        base += total;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int added = min(base, room);
        *P.count = c0 + added;
        *P.next_id = id0 + added;
    }
}

// Threads of a call's CTAs: an entry of the largest pool each, where that fits
// (8 pools of 250: 12.3 us with 256 threads, 12.9 with 512, 15.0 with 1,024).
template <typename Job>
static int pool_threads(const Job *jobs, int njobs) {
    int cap = 128;
    for (int i = 0; i < njobs; ++i)
        if (jobs[i].pool.cap > cap) cap = jobs[i].pool.cap;
    return cap >= TK_THREADS ? TK_THREADS : (cap + 31) / 32 * 32;
}

static bool pool_ok(const vt_track_pool &p) {
    return p.pts && p.ids && p.ages && p.count && p.next_id && p.cap >= 1 && p.cap <= VT_POOL_MAX;
}

}  // namespace vt

using namespace vt;

extern "C" {

vt_status vt_tracks_carry(const vt_carry_job *jobs, int njobs, float min_dist, void *cuda_stream) {
    if (njobs < 0 || njobs > kMaxPoolJobs || (njobs > 0 && !jobs) || !(min_dist > 0.f) || !std::isfinite(min_dist))
        return VT_ERR_ARG;
    for (int i = 0; i < njobs; ++i)
        if (!pool_ok(jobs[i].pool) || !jobs[i].tracked || !jobs[i].status) return VT_ERR_ARG;
    if (njobs == 0) return VT_OK;
    CarryJobs J;  // copied into the launch's parameters
    J.n = njobs;
    J.min_dist = min_dist;
    for (int i = 0; i < njobs; ++i) J.j[i] = jobs[i];
    if (!smem_opt_in<k_tracks_carry>(sizeof(CarrySmem))) return VT_ERR_CUDA;
    const cudaError_t e = launch_pdl(k_tracks_carry, njobs, pool_threads(jobs, njobs), sizeof(CarrySmem),
                                     (cudaStream_t)cuda_stream, true, J);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? VT_OK : VT_ERR_CUDA;
}

vt_status vt_tracks_spawn(const vt_spawn_job *jobs, int njobs, void *cuda_stream) {
    if (njobs < 0 || njobs > kMaxPoolJobs || (njobs > 0 && !jobs)) return VT_ERR_ARG;
    for (int i = 0; i < njobs; ++i)
        if (!pool_ok(jobs[i].pool) || !jobs[i].corners || !jobs[i].n_corners) return VT_ERR_ARG;
    if (njobs == 0) return VT_OK;
    SpawnJobs J;
    J.n = njobs;
    for (int i = 0; i < njobs; ++i) J.j[i] = jobs[i];
    const cudaError_t e =
        launch_pdl(k_tracks_spawn, njobs, pool_threads(jobs, njobs), 0, (cudaStream_t)cuda_stream, true, J);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? VT_OK : VT_ERR_CUDA;
}

}  // extern "C"
