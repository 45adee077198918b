// Warp-per-feature pyramidal Lucas-Kanade (K3), shared by the single-pair
// kernels (vt_klt.cu) and the batched persistent kernel (vt_batch.cu) so that
// a point gives bit-identical results alone or in a batch.
//
// The method (textbook coarse-to-fine LK, the tracker the paper uses in
// Sec. IV / Table I; cross-camera check of Sec. V-A):
//   per level l = L-1 .. 0, u_l = u / 2^l:
//     T(x), grad T(x): bilinear samples of I_l and its Scharr planes at u_l + x
//     G = sum grad T grad T^T, reject if lambda_min / (win^2 255^2) < min_eig
//     iterate: q = u_l + g_l + nu (bound test), r = T - J_l(q + x),
//              b = sum r grad T, eta = G^-1 b, nu += eta, stop |eta|^2 < eps^2
//     g_{l-1} = 2 (g_l + nu)
//   result v = u + g_0 + nu (bound test), error = mean |T - J_0(v + x)|.
//
// Mapping to the warp: the window is cut into short runs of rows of one
// column, a lane owning one or two runs (KRuns), so all 32 lanes work on the
// win^2 samples.  Every window sample of one Newton
// iteration shares the same fractional bilinear weights (bx, by), so
// b = sum (T - J(q + x)) grad T expands exactly into bx, by and eight moments
// of the integer footprint of J under the window (cell_moments).  A sweep
// over the footprint is needed only when the integer part of q changes;
// iterations that stay in the same cell reuse the moments.  The template and
// its gradients stay in registers (three floats per owned sample); the image and
// gradient window it is sampled from, and each footprint, are staged in
// per-warp shared memory by cp.async, a level's template while the level
// before it iterates and its first footprint while its template is sampled.  Sums over the window are per-lane FP32
// sums over rows followed by a warp reduction that leaves bit-identical
// totals in every lane (an XOR butterfly, or a reduce-scatter and broadcast),
// so control flow stays warp-uniform.
#pragma once

#include <climits>
#include <cstddef>

#include "vt_internal.cuh"

namespace vt {

// (aligned for the 16-byte loads of track_point_dir, as a kernel parameter too)
struct __align__(16) KPyr {
    Level lv[VT_MAX_LEVELS];
};

struct KOut {
    float x, y;     // level-0 result (last estimate when lost)
    float err;      // mean |T - J| (0 when lost)
    float lmin;     // normalised lambda_min at the last level examined
    int status;     // 1 tracked
    int reason;     // VT_TRACKED / VT_LOST_*
    int iters;      // Newton iterations over all levels (and both passes)
    int tmpl;       // template extractions (window sweeps of 27 FLOP per sample)
    int errp;       // error passes (window sweeps of 9 FLOP per sample)
    int sweeps;     // footprint sweeps the Newton iterations actually needed
};

// Algorithmic FLOPs of a tracked point: per window sample 27 for a template
// sweep (bilinear I, Ix, Iy: 3 x 7; G: 3 FMA), 12 for a Newton sweep
// (bilinear J: 7; residual: 1; b: 2 FMA) and 9 for the error sweep.
__device__ __forceinline__ int klt_flops(int win, const KOut &o) {
    return win * win * (27 * o.tmpl + 12 * o.iters + 9 * o.errp);
}

constexpr unsigned kFull = 0xffffffffu;

// Resident CTAs per SM the tracking kernels are register-budgeted for
// (4-warp CTAs): 4 for windows up to 21 (128 registers per thread).
template <int WIN>
struct KltOcc {
    static constexpr int min_blocks = WIN <= 21 ? 4 : 3;
};

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) v += __shfl_xor_sync(kFull, v, m);
    return v;
}

// Warp totals of eight per-lane values, delivered to every lane: the three
// top butterfly levels are a reduce-scatter (each halves the set a lane
// carries), the last two reduce the lane's single value, and the eight totals
// are broadcast from lanes 0, 4, .., 28.  17 shuffles instead of 5 x 8.
__device__ __forceinline__ void warp_sum8(const float (&a)[8], int lane, float (&m)[8]) {
    const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
    float b[4], c[2];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float send = h16 ? a[k] : a[k + 4], keep = h16 ? a[k + 4] : a[k];
        b[k] = keep + __shfl_xor_sync(kFull, send, 16);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float send = h8 ? b[k] : b[k + 2], keep = h8 ? b[k + 2] : b[k];
        c[k] = keep + __shfl_xor_sync(kFull, send, 8);
    }
    const float send = h4 ? c[0] : c[1], keep = h4 ? c[1] : c[0];
    float d = keep + __shfl_xor_sync(kFull, send, 4);
    d += __shfl_xor_sync(kFull, d, 2);
    d += __shfl_xor_sync(kFull, d, 1);
#pragma unroll
    for (int k = 0; k < 8; ++k) m[k] = __shfl_sync(kFull, d, 4 * k);  // lane 4k holds total k
}

// Warp totals of three per-lane values the same way (the set padded to four
// with a zero; totals broadcast from lanes 0, 8, 16): 9 shuffles instead of
// 5 x 3.
__device__ __forceinline__ void warp_sum3(float x, float y, float z, int lane, float &sx, float &sy, float &sz) {
    const bool h16 = lane & 16, h8 = lane & 8;
    const float s0 = h16 ? x : z, k0 = h16 ? z : x;
    const float s1 = h16 ? y : 0.f, k1 = h16 ? 0.f : y;
    const float b0 = k0 + __shfl_xor_sync(kFull, s0, 16);
    const float b1 = k1 + __shfl_xor_sync(kFull, s1, 16);
    const float sd = h8 ? b0 : b1, kd = h8 ? b1 : b0;
    float d = kd + __shfl_xor_sync(kFull, sd, 8);
    d += __shfl_xor_sync(kFull, d, 4);
    d += __shfl_xor_sync(kFull, d, 2);
    d += __shfl_xor_sync(kFull, d, 1);
    sx = __shfl_sync(kFull, d, 0);
    sy = __shfl_sync(kFull, d, 8);
    sz = __shfl_sync(kFull, d, 16);
}

// Image values in the FP32 sweeps are kept times 2^-22: a byte's bit pattern
// read as a float is the denormal byte * 2^-149, so one FP32 multiplication by
// 2^127 (exact, full rate) converts it, and one FMA converts and subtracts.
// The integer pipe, the busiest one, is left out (a conversion instruction
// per byte kept it 7 % busier and cost an instruction more per pair of
// neighbours).  A power of two changes no rounding: every result is the
// unscaled one's, scaled, until kImgUnscale takes it back.
constexpr float kImgUnscale = 4194304.f;  // 2^22
__device__ __forceinline__ float px_scale() { return __int_as_float(0x7f000000); }  // 2^127
__device__ __forceinline__ float px(uint32_t v) { return __uint_as_float(v) * px_scale(); }
// px(v) - a (a the px of another byte: the difference is exact)
__device__ __forceinline__ float px_minus(uint32_t v, float a) { return fmaf(__uint_as_float(v), px_scale(), -a); }

// Packed FP32 pairs: this GPU issues one instruction for two FMAs, each
// rounded as the scalar one.  y - x as x * (-1) + y: the product is exact, so
// the result is the subtraction's.
__device__ __forceinline__ float2 pair(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 sub2(float2 y, float2 x) { return __ffma2_rn(x, pair(-1.f), y); }

template <int GT>
__device__ __forceinline__ void unpack_grad(uint32_t v, float &gx, float &gy) {
    if (GT == VT_GRAD_S16) {
        gx = (float)(int)(int16_t)(v & 0xffffu);
        gy = (float)((int)v >> 16);
    } else {
        const __half2 h = *reinterpret_cast<const __half2 *>(&v);
        const float2 f = __half22float2(h);
        gx = f.x;
        gy = f.y;
    }
}

// Scale from the stored gradient unit to grey levels per pixel (gradients
// computed on the fly, VT_GRAD_NONE, are raw Scharr like VT_GRAD_S16).
template <int GT>
__device__ __forceinline__ constexpr float grad_unit() { return GT == VT_GRAD_F16 ? 1.0f : 0.03125f; }

// a b - c d by Kahan's FMA scheme: w = c d rounded, its rounding error
// c d - w is exact (one FMA), and the result is round(a b - w) minus that
// error.  Relative error at most 2 ulp and the sign exact (Jeannerod, Louvet
// & Muller, Math. Comp. 82, 2013) -- as good as FP64 products rounded to FP32,
// but on the FP32 pipes: this GPU's FP64 pipe retires about 2 lanes per clock
// per SM, and an FP64 determinant and divides per template kept it 42 % busy.
__device__ __forceinline__ float kdiff(float a, float b, float c, float d) {
    const float w = c * d;
    return fmaf(a, b, -w) - fmaf(c, d, -w);
}

// x^2 + y^2, rounded the same wherever it decides something: left to the
// compiler, which of the products is fused is each kernel's own, and a point's
// result would depend on the kernel that tracked it.
__device__ __forceinline__ float norm2(float x, float y) { return fmaf(x, x, __fmul_rn(y, y)); }

// 2^-l exactly.
__device__ __forceinline__ float pow2neg(int l) { return __int_as_float((127 - l) << 23); }

// Per-warp shared scratch: the staged (win + 1)^2 windows -- the footprint of J
// for one sweep, and the template's image and gradient windows of this level
// and of the next one (levels alternate between the two buffers, so the next
// level's template is copied in while this level iterates) -- in win + 1 rows
// of NC (image) or NG (gradients) 16-byte chunks.
template <int WIN>
struct __align__(16) KSmem {
    static constexpr int NC = (WIN + 31) / 16;  // 16-byte chunks per staged row: cover 15 + win + 1 bytes
    static constexpr int JS = NC * 16;          // staged row stride in bytes
    static_assert(JS >= 15 + WIN + 1, "a staged row covers the footprint row");
    static constexpr int NG = (4 * (3 + WIN + 1) + 15) / 16;  // 16-byte chunks per staged gradient row
    static constexpr int GS = NG * 4;                         // staged gradient row stride in words
    static_assert(GS >= 3 + WIN + 1, "a staged gradient row covers the window row");
    Level lv[2][VT_MAX_LEVELS];  // the point's two pyramids
    // moments of the level's footprint cells that the position left, by the
    // parity of the cell: neighbouring cells never share an entry, so a point
    // that hovers at a cell's edge or corner comes back to kept moments
    float2 cell_m[4][4];
    int2 cell_at[4];
    uint8_t j[(WIN + 1) * JS];
    uint32_t g[2][(WIN + 1) * GS];
    uint8_t t[2][(WIN + 1) * JS];
    // Pyramids without gradient planes: the image windows of this level and the
    // next, one pixel wider on every side, over g[1] and t; the gradients
    // computed from them in g[0].
    static constexpr int RS = (15 + WIN + 3 + 15) / 16 * 16, RAW = (WIN + 3) * RS;
    __device__ __forceinline__ uint8_t *raw(int k) { return reinterpret_cast<uint8_t *>(g[1]) + k * RAW; }
};
template <int WIN>
constexpr bool raw_fits() {
    return 2 * KSmem<WIN>::RAW <= (int)(sizeof(KSmem<WIN>::g) / 2 + sizeof(KSmem<WIN>::t)) &&
           offsetof(KSmem<WIN>, t) == offsetof(KSmem<WIN>, g) + sizeof(KSmem<WIN>::g);
}
static_assert(raw_fits<9>() && raw_fits<15>() && raw_fits<21>() && raw_fits<31>(), "two wider windows over g[1] and t");

// Where a level's staged template is: its image window, rows `stride` bytes
// apart, staged from column sx, of a level w wide; its gradient window
// likewise (gx0: the window's leftmost column in those terms).
struct TWin {
    const uint8_t *st;
    const uint32_t *sg;
    int x0, w, sx;
    int gx0, gw, gsx;
};
template <int WIN, int GT>
__device__ __forceinline__ constexpr int twin_stride() {
    return GT == VT_GRAD_NONE ? KSmem<WIN>::RS : KSmem<WIN>::JS;
}

// Shared scratch of a CTA: its warps' windows, and zeros that a lane's run
// outside the window reads instead of the staged windows (its template
// samples and error terms are then exactly zero without a select per sample):
// a run's rows of two bytes / words at the staged strides.
template <int WIN>
struct KCta {
    static constexpr int RLZ = WIN / (WIN == 31 ? 1 : 3);
    uint8_t zj[RLZ * KSmem<WIN>::RS + 16];
    uint32_t zg[RLZ * KSmem<WIN>::GS + 4];
    KSmem<WIN> warp[1];  // one per warp of the CTA

    static constexpr size_t bytes(int warps) { return sizeof(KCta) + (warps - 1) * sizeof(KSmem<WIN>); }
};

// Clear the zero rows (every thread of the CTA, once per kernel).
template <int WIN>
__device__ __forceinline__ KCta<WIN> &kcta_init(uint8_t *smem) {
    KCta<WIN> &C = *reinterpret_cast<KCta<WIN> *>(smem);
    for (int k = threadIdx.x; k < (int)sizeof(C.zj); k += blockDim.x) C.zj[k] = 0;
    for (int k = threadIdx.x; k < (int)(sizeof(C.zg) / 4); k += blockDim.x) C.zg[k] = 0;
    __syncthreads();
    return C;
}

// Which window samples a lane owns.  The win x win window is cut into runs
// of RL consecutive rows of one column (D bands of RL rows, win * D runs in
// all, numbered band by band so that lanes reading at the same time touch at
// most two staged rows: fewer shared-memory bank conflicts); lane l owns
// runs l, l + 32, ... (at most RPL).  A lane walks each of
// its runs down the column, reading footprint rows r0 .. r0 + RL and the
// neighbouring column from shared memory, so every lane works (with one
// column per lane, 32 - win lanes would idle) and the right neighbour needs
// no shuffle.  The per-sample arithmetic does not depend on the layout; only
// the grouping of the per-lane partial sums does.
template <int WIN>
struct KRuns {
    static constexpr int D = WIN == 31 ? 1 : 3;
    static_assert(WIN % D == 0, "runs tile a column");
    static constexpr int RL = WIN / D;          // samples per run
    static constexpr int NR = WIN * D;          // runs in the window
    static constexpr int RPL = (NR + 31) / 32;  // runs per lane
    static constexpr int NS = RPL * RL;         // samples a lane holds
};

// Run i of a lane: column c, first row r0, and whether it lies in the window
// (a lane's last run may not: it then reads run 0's addresses and its
// samples weigh zero).
template <int WIN>
__device__ __forceinline__ void run_of(int lane, int i, int &c, int &r0, bool &valid) {
    constexpr int RL = KRuns<WIN>::RL;
    const int k = lane + 32 * i;
    valid = k < KRuns<WIN>::NR;
    const int kk = valid ? k : 0;
    const int band = kk / WIN;
    c = kk - band * WIN;
    r0 = band * RL;
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// All but the newest N groups of this thread have arrived.
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Start copying ROWS rows of NCH 16-byte chunks (row pitch `pitch` bytes,
// rows from y0 on, clamped to 0 .. hm1) from `base` to `dst`, the chunks
// below `chunks` of each row.  32 / NCH rows go per step, a lane keeping one
// chunk of a row: its addresses advance by a constant per step, two
// instructions per copied chunk (an index split into row and chunk per copy
// took about 18).  Rows that cross the level's first or last one are clamped
// step by step, unrolled too: half of the windows of the coarse levels do.
template <int ROWS, int NCH>
__device__ __forceinline__ void copy_rows(uint32_t dst, const uint8_t *base, int pitch, int y0, int hm1, int chunks,
                                          int lane) {
    constexpr int RS = 32 / NCH, STEPS = (ROWS + RS - 1) / RS;  // rows per step, steps
    const int r = lane / NCH, c = lane - r * NCH;
    const uint32_t d = dst + 16 * lane;
    const int rows = r < RS && c < chunks ? ROWS - r : 0;  // the lane copies rows r + k RS, k RS < rows
    if (y0 >= 0 && y0 + ROWS - 1 <= hm1) {
        const uint8_t *src = base + (size_t)(y0 + r) * pitch + 16 * c;
#pragma unroll
        for (int k = 0; k < STEPS; ++k) {
            if (k * RS < rows) cp_async16(d + k * RS * NCH * 16, src);
            src += RS * pitch;
        }
    } else {
#pragma unroll
        for (int k = 0; k < STEPS; ++k)
            if (k * RS < rows)
                cp_async16(d + k * RS * NCH * 16, base + (size_t)clampi(y0 + r + k * RS, 0, hm1) * pitch + 16 * c);
    }
}

// First staged column of a window whose leftmost column is x0: the aligned
// column (16 image bytes, 4 gradient words) at or before the first one inside
// the level.
__device__ __forceinline__ int staged_x(int x0, int align) { return max(x0, 0) & ~(align - 1); }

// Start staging the (win + 1)^2 image window with top-left (x0, y0) at `st`
// (and, with GRAD, the gradient window at `sg`): each row, clamped into the
// level, in whole aligned 16-byte chunks from staged_x on, by cp.async (no
// register round trip; the caller commits and waits).  Chunks that begin
// past the level's last column are left out; the last one may read up to 15
// bytes past it, inside the row's pitch.  Columns outside the level are not
// staged: the readers clamp theirs (run_columns).
template <int WIN, bool GRAD>
__device__ __forceinline__ void stage_window(const Level &L, int x0, int y0, int lane, uint8_t *st, uint32_t *sg) {
    const int hm1 = L.h - 1, wx = staged_x(x0, 16);
    __syncwarp();  // every lane is done with what the buffers held
    copy_rows<WIN + 1, KSmem<WIN>::NC>((uint32_t)__cvta_generic_to_shared(st), L.img + wx, L.pitch, y0, hm1,
                                   (L.w - wx + 15) >> 4, lane);
    if constexpr (GRAD) {
        const int gw = staged_x(x0, 4);
        copy_rows<WIN + 1, KSmem<WIN>::NG>((uint32_t)__cvta_generic_to_shared(sg),
                                       reinterpret_cast<const uint8_t *>(L.grad + gw), L.gpitch * 4, y0, hm1,
                                       (L.w - gw + 3) >> 2, lane);
    }
}

// Start staging the image window with top-left (x0, y0) and a border of one
// pixel on every side (pyramids without gradient planes).
template <int WIN>
__device__ __forceinline__ void stage_raw(const Level &L, int x0, int y0, int lane, uint8_t *raw) {
    const int sx = staged_x(x0 - 1, 16);
    __syncwarp();
    copy_rows<WIN + 3, KSmem<WIN>::RS / 16>((uint32_t)__cvta_generic_to_shared(raw), L.img + sx, L.pitch, y0 - 1, L.h - 1,
                                            (L.w - sx + 15) >> 4, lane);
}

// Gradient window of a level without stored gradients, from its staged raw
// window: lane c (c <= win) computes the raw Scharr responses of window
// column c -- the integers the pyramid kernels would have stored for the
// replicate-clamped pixel (reflect-101 neighbours, all inside the raw window)
// -- and stores them as int16 pairs, so the template is then sampled exactly
// as from stored int16 gradients.
//
// Per image row y the lane forms d(y) = I(y, x+1) - I(y, x-1) and
// s(y) = 3 I(y, x-1) + 10 I(y, x) + 3 I(y, x+1); the gradient of row y is
// dx = 3 d(y-1) + 10 d(y) + 3 d(y+1), dy = s(y+1) - s(y-1).  Raw row k holds
// image row clamp(y0 - 1 + k); the rows are read once each (a rolling
// window): for an interior row its neighbours are the raw rows above and
// below; a row at the image's first or last line takes its reflected
// neighbour (row 1 or h-2) on both sides instead.
template <int WIN>
__device__ __forceinline__ void gradients_from_raw(const uint8_t *raw, int w, int h, int x0, int y0, int lane,
                                                   uint32_t *sg) {
    constexpr int RS = KSmem<WIN>::RS, GS = KSmem<WIN>::GS;
    if (lane <= WIN) {
        const int sx = staged_x(x0 - 1, 16), hm1 = h - 1;
        const int q = clampi(x0 + lane, 0, w - 1);
        const uint8_t *pm = raw + refl101(q - 1, w) - sx, *p0 = raw + q - sx, *pp = raw + refl101(q + 1, w) - sx;
        auto terms = [&](int k, int &d, int &s) {  // of raw row k
            const int a = pm[k * RS], b = p0[k * RS], e = pp[k * RS];
            d = e - a;
            s = 3 * (a + e) + 10 * b;
        };
        // reflected neighbours of the first and last image rows (used only when
        // the window reaches them)
        int dt = 0, st = 0, db = 0, sb = 0;
        if (y0 <= 0 || hm1 == 0) terms(refl101(-1, h) - y0 + 1, dt, st);
        if (y0 + WIN >= hm1) terms(refl101(h, h) - y0 + 1, db, sb);
        int dm, sm, d0, s0;
        terms(0, dm, sm);
        terms(1, d0, s0);
#pragma unroll
        for (int r = 0; r <= WIN; ++r) {
            const int yc = clampi(y0 + r, 0, hm1);
            int dp, sp;
            terms(r + 2, dp, sp);
            const bool top = yc == 0, bot = yc == hm1;
            const int du = top ? dt : (bot ? db : dm), su = top ? st : (bot ? sb : sm);
            const int dd = top ? dt : (bot ? db : dp), sd = top ? st : (bot ? sb : sp);
            const int gx = 3 * (du + dd) + 10 * d0, gy = sd - su;
            sg[r * GS + lane] = (uint32_t)(uint16_t)(int16_t)gx | ((uint32_t)(uint16_t)(int16_t)gy << 16);
            dm = d0;
            sm = s0;
            d0 = dp;
            s0 = sp;
        }
    }
    __syncwarp();
}

// Stage the footprint of J with top-left (x0, y0) and wait for it (and for
// every copy under way).
template <int WIN>
__device__ __forceinline__ void stage_footprint(const Level &L, int x0, int y0, int lane, KSmem<WIN> &sm) {
    stage_window<WIN, false>(L, x0, y0, lane, sm.j, nullptr);
    cp_async_commit();
    cp_async_wait<0>();
    __syncwarp();
}

// Where a run's column c and its right neighbour lie in a staged row
// (replicate-clamped into 0 .. w - 1): offsets from the first staged column.
template <int WIN>
__device__ __forceinline__ void run_columns(int x0, int w, int sx, int c, int &o0, int &o1) {
    o0 = x0 + c - sx;
    o1 = o0 + 1;
    if (x0 < 0 || x0 + WIN >= w) {
        o0 = clampi(x0 + c, 0, w - 1) - sx;
        o1 = clampi(x0 + c + 1, 0, w - 1) - sx;
    }
}

// The template at the lane's window samples (KRuns): N = -T (times 2^-22, see
// px) and its gradients,
// sampled at fractional offset (ax, ay) from the staged windows, zero for
// samples outside the window.
template <int WIN, int GT>
__device__ __forceinline__ void sample_template(const KCta<WIN> &C, const TWin &W, float ax, float ay, int lane,
                                                float (&N)[KRuns<WIN>::NS], float2 (&G)[KRuns<WIN>::NS]) {
    constexpr int TS = twin_stride<WIN, GT>(), GS = KSmem<WIN>::GS, RL = KRuns<WIN>::RL, RPL = KRuns<WIN>::RPL;
    // staged gradient words are int16 pairs when computed in place
    constexpr int GTS = GT == VT_GRAD_NONE ? VT_GRAD_S16 : GT;
    const uint8_t *j0[RPL], *j1[RPL];
    const uint32_t *g0[RPL], *g1[RPL];
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
        int c, r0;
        bool valid;
        run_of<WIN>(lane, i, c, r0, valid);
        int o0, o1;
        run_columns<WIN>(W.x0, W.w, W.sx, c, o0, o1);
        j0[i] = valid ? W.st + r0 * TS + o0 : C.zj, j1[i] = valid ? W.st + r0 * TS + o1 : C.zj;
        run_columns<WIN>(W.gx0, W.gw, W.gsx, c, o0, o1);
        g0[i] = valid ? W.sg + r0 * GS + o0 : C.zg, g1[i] = valid ? W.sg + r0 * GS + o1 : C.zg;
    }
    // the image, a lane's two runs as a pair (a lone run's second half is idle)
    float2 pt = pair(0.f);
#pragma unroll
    for (int r = 0; r <= RL; ++r) {
        const float2 l = make_float2(__uint_as_float(j0[0][r * TS]), __uint_as_float(j0[RPL - 1][r * TS]));
        const float2 n = make_float2(__uint_as_float(j1[0][r * TS]), __uint_as_float(j1[RPL - 1][r * TS]));
        float2 nh;  // minus the horizontal lerp
        if constexpr (RPL == 2) {
            const float2 nl = __fmul2_rn(l, pair(-px_scale()));
            nh = __ffma2_rn(pair(-ax), __ffma2_rn(n, pair(px_scale()), nl), nl);
            if (r > 0) {
                const float2 t = __ffma2_rn(pair(ay), sub2(nh, pt), pt);
                N[r - 1] = t.x, N[RL + r - 1] = t.y;  // zero for a run outside the window
            }
        } else {
            const float nl = l.x * -px_scale();
            nh.x = fmaf(-ax, fmaf(n.x, px_scale(), nl), nl);
            nh.y = 0.f;
            if (r > 0) N[r - 1] = fmaf(ay, nh.x - pt.x, pt.x);
        }
        pt = nh;
    }
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
        float2 pg = pair(0.f);
#pragma unroll
        for (int r = 0; r <= RL; ++r) {
            float2 gl, gr;
            unpack_grad<GTS>(g0[i][r * GS], gl.x, gl.y);
            unpack_grad<GTS>(g1[i][r * GS], gr.x, gr.y);
            const float2 hg = __ffma2_rn(pair(ax), sub2(gr, gl), gl);
            if (r > 0) G[i * RL + r - 1] = __ffma2_rn(pair(ay), sub2(hg, pg), pg);
            pg = hg;
        }
    }
}

// Moments of one integer footprint F (top-left (x0, y0)) against the template.
// With F00 = F(y, x), F01 = F(y, x+1), F10 = F(y+1, x), F11 = F(y+1, x+1) for
// window sample (y, x), the bilinear sample at fractional offset (bx, by) is
//   F00 + bx (F01 - F00) + by (F10 - F00) + bx by (F11 - F10 - F01 + F00),
// so for every q with floor(q) = (x0, y0) + (h, h):
//   sum r grad T = R - bx Sx - by Sy - bx by Sxy,
//   R = sum (T - F00) grad T, Sx = sum (F01 - F00) grad T,
//   Sy = sum (F10 - F00) grad T, Sxy = sum (F11 - F10 - F01 + F00) grad T.
// The footprint differences are exact (integers); m: -R, Sx, Sy, Sxy as (x
// part, y part) -- with R negated, -b is a sum without a sign change, and the
// negated 1 / det of the step takes it back.  The footprint is staged in sm.j;
// w: the level's width.
template <int WIN>
__device__ __forceinline__ void cell_moments(int x0, int w, int lane, const float (&N)[KRuns<WIN>::NS],
                                             const float2 (&G)[KRuns<WIN>::NS], const KSmem<WIN> &sm,
                                             float2 (&m)[4]) {
    constexpr int JS = KSmem<WIN>::JS, RL = KRuns<WIN>::RL, RPL = KRuns<WIN>::RPL;
    float2 a[4];  // (x part, y part) of each moment
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] = pair(0.f);
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
        int c, r0;
        bool valid;
        run_of<WIN>(lane, i, c, r0, valid);  // samples of a run outside the window weigh zero
        int o0, o1;
        run_columns<WIN>(x0, w, staged_x(x0, 16), c, o0, o1);
        const uint8_t *j0 = &sm.j[r0 * JS + o0], *j1 = &sm.j[r0 * JS + o1];
        float2 p = pair(0.f);  // F and F(c + 1) - F(c) of the row above
#pragma unroll
        for (int r = 0; r <= RL; ++r) {
            float2 q;
            q.x = px(j0[r * JS]);
            q.y = px_minus(j1[r * JS], q.x);
            if (r > 0) {
                const int s = i * RL + r - 1;
                const float e0 = N[s] + p.x;  // -(T - F00)
                const float2 d = sub2(q, p);  // F10 - F00, F11 - F10 - F01 + F00
                a[0] = __ffma2_rn(pair(e0), G[s], a[0]);
                a[1] = __ffma2_rn(pair(p.y), G[s], a[1]);
                a[2] = __ffma2_rn(pair(d.x), G[s], a[2]);
                a[3] = __ffma2_rn(pair(d.y), G[s], a[3]);
            }
            p = q;
        }
    }
    const float v[8] = {a[0].x, a[1].x, a[2].x, a[3].x, a[0].y, a[1].y, a[2].y, a[3].y};
    float t[8];
    warp_sum8(v, lane, t);
#pragma unroll
    for (int k = 0; k < 4; ++k) m[k] = make_float2(t[k], t[k + 4]);
}

// Error sweep over the staged footprint at fractional offset (bx, by): sum
// |T - J(q + x)| over the window.
template <int WIN>
__device__ __forceinline__ float abs_residual(const KCta<WIN> &C, int x0, int w, float bx, float by, int lane,
                                              const float (&N)[KRuns<WIN>::NS], const KSmem<WIN> &sm) {
    constexpr int JS = KSmem<WIN>::JS, RL = KRuns<WIN>::RL, RPL = KRuns<WIN>::RPL;
    const uint8_t *j0[RPL], *j1[RPL];
#pragma unroll
    for (int i = 0; i < RPL; ++i) {
        int c, r0;
        bool valid;
        run_of<WIN>(lane, i, c, r0, valid);
        int o0, o1;
        run_columns<WIN>(x0, w, staged_x(x0, 16), c, o0, o1);
        j0[i] = valid ? &sm.j[r0 * JS + o0] : C.zj, j1[i] = valid ? &sm.j[r0 * JS + o1] : C.zj;
    }
    float sa = 0.f, sb = 0.f, later[RL];
    float2 ph = pair(0.f);
#pragma unroll
    for (int r = 0; r <= RL; ++r) {
        const float2 l = make_float2(__uint_as_float(j0[0][r * JS]), __uint_as_float(j0[RPL - 1][r * JS]));
        const float2 n = make_float2(__uint_as_float(j1[0][r * JS]), __uint_as_float(j1[RPL - 1][r * JS]));
        const float2 nl = __fmul2_rn(l, pair(-px_scale()));
        const float2 nh = __ffma2_rn(pair(-bx), __ffma2_rn(n, pair(px_scale()), nl), nl);  // minus the horizontal lerp
        if (r > 0) {
            const float2 nj = __ffma2_rn(pair(by), sub2(nh, ph), ph);
            const float e = fabsf(N[r - 1] - nj.x);  // 0 - 0 for a run outside the window
            if (r & 1)
                sa += e;
            else
                sb += e;
            if constexpr (RPL == 2) later[r - 1] = fabsf(N[RL + r - 1] - nj.y);
        }
        ph = nh;
    }
    if constexpr (RPL == 2) {
#pragma unroll
        for (int r = 1; r <= RL; ++r)
            if (r & 1)
                sa += later[r - 1];
            else
                sb += later[r - 1];
    }
    return warp_sum(sa + sb);
}

// ---------------------------------------------------------------------------
// FP64 levels.  Where the gradient matrix of a level's template is
// ill-conditioned (lambda_max / lambda_min above kFp64Cond), the FP32 sums of
// G and b lose the weak direction: their rounding, divided by lambda_min,
// moves the Newton steps along it by more than the flow tolerance.  Such a
// level is tracked in FP64: the template and its gradients are sampled in
// FP64 from the level's staged windows at every sweep, G, the
// footprint moments, the 2x2 solve and the position update are FP64.  The
// branch is warp-uniform; with the default eigenvalue threshold (1e-4) an
// accepted template cannot exceed a condition number of 5e3 (fp64_needed),
// so it is taken only when a caller lowers the threshold.

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) v += __shfl_xor_sync(kFull, v, m);
    return v;
}

// The lane's run c, r0 of a staged template in FP64: horizontal lerps of its
// row r of the image and gradient windows.
template <int WIN, int GT>
struct Run64 {
    const uint8_t *t0, *t1;
    const uint32_t *g0, *g1;

    __device__ __forceinline__ Run64(const TWin &W, int c, int r0) {
        int o0, o1;
        run_columns<WIN>(W.x0, W.w, W.sx, c, o0, o1);
        t0 = W.st + r0 * twin_stride<WIN, GT>() + o0;
        t1 = W.st + r0 * twin_stride<WIN, GT>() + o1;
        run_columns<WIN>(W.gx0, W.gw, W.gsx, c, o0, o1);
        g0 = W.sg + r0 * KSmem<WIN>::GS + o0;
        g1 = W.sg + r0 * KSmem<WIN>::GS + o1;
    }
    __device__ __forceinline__ void row(int r, double ax, double unit, double &hT, double &hGX, double &hGY) const {
        constexpr int TS = twin_stride<WIN, GT>(), GS = KSmem<WIN>::GS;
        constexpr int GTS = GT == VT_GRAD_NONE ? VT_GRAD_S16 : GT;
        const double a = (double)t0[r * TS], b = (double)t1[r * TS];
        float gx0, gy0, gx1, gy1;
        unpack_grad<GTS>(g0[r * GS], gx0, gy0);
        unpack_grad<GTS>(g1[r * GS], gx1, gy1);
        const double x0 = (double)gx0 * unit, x1 = (double)gx1 * unit, y0 = (double)gy0 * unit, y1 = (double)gy1 * unit;
        hT = fma(ax, b - a, a);
        hGX = fma(ax, x1 - x0, x0);
        hGY = fma(ax, y1 - y0, y0);
    }
};

// G of the level's template in FP64 (grey levels per pixel), every lane
// holding the totals.
template <int WIN, int GT>
__device__ __forceinline__ void template_G64(double ax, double ay, const TWin &W, int lane, double &g11, double &g12,
                                             double &g22) {
    constexpr int RL = KRuns<WIN>::RL, RPL = KRuns<WIN>::RPL;
    constexpr double unit = (double)grad_unit<GT>();
    double a11 = 0.0, a12 = 0.0, a22 = 0.0;
#pragma unroll 1
    for (int i = 0; i < RPL; ++i) {
        int c, r0;
        bool valid;
        run_of<WIN>(lane, i, c, r0, valid);
        if (!valid) continue;
        const Run64<WIN, GT> run(W, c, r0);
        double pT, pX, pY;
        run.row(0, ax, unit, pT, pX, pY);
#pragma unroll 1
        for (int r = 1; r <= RL; ++r) {
            double hT, hX, hY;
            run.row(r, ax, unit, hT, hX, hY);
            const double gx = fma(ay, hX - pX, pX), gy = fma(ay, hY - pY, pY);
            a11 = fma(gx, gx, a11);
            a12 = fma(gx, gy, a12);
            a22 = fma(gy, gy, a22);
            pT = hT;
            pX = hX;
            pY = hY;
        }
    }
    g11 = warp_sum_d(a11);
    g12 = warp_sum_d(a12);
    g22 = warp_sum_d(a22);
}

// The eight footprint moments of cell_moments in FP64, the template sampled
// in FP64 from its staged windows (grey levels per pixel).
template <int WIN, int GT>
__device__ __forceinline__ void cell_moments64(const Level &L, int x0, int y0, double ax, double ay, const TWin &W,
                                               int lane, KSmem<WIN> &sm, double (&m)[8]) {
    constexpr int JS = KSmem<WIN>::JS, RL = KRuns<WIN>::RL, RPL = KRuns<WIN>::RPL;
    constexpr double unit = (double)grad_unit<GT>();
    stage_footprint<WIN>(L, x0, y0, lane, sm);
    double a[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) a[k] = 0.0;
#pragma unroll 1
    for (int i = 0; i < RPL; ++i) {
        int c, r0;
        bool valid;
        run_of<WIN>(lane, i, c, r0, valid);
        if (!valid) continue;
        const Run64<WIN, GT> run(W, c, r0);
        int o0, o1;
        run_columns<WIN>(x0, L.w, staged_x(x0, 16), c, o0, o1);
        const uint8_t *j0 = &sm.j[r0 * JS + o0], *j1 = &sm.j[r0 * JS + o1];
        double pT, pX, pY;
        run.row(0, ax, unit, pT, pX, pY);
        double pmv = (double)j0[0];
        double pdx = (double)j1[0] - pmv;
#pragma unroll 1
        for (int r = 1; r <= RL; ++r) {
            double hT, hX, hY;
            run.row(r, ax, unit, hT, hX, hY);
            const double T = fma(ay, hT - pT, pT), gx = fma(ay, hX - pX, pX), gy = fma(ay, hY - pY, pY);
            const double mv = (double)j0[r * JS];
            const double dx = (double)j1[r * JS] - mv;
            const double e0 = T - pmv, sy = mv - pmv, sxy = dx - pdx;
            a[0] = fma(e0, gx, a[0]);
            a[1] = fma(pdx, gx, a[1]);
            a[2] = fma(sy, gx, a[2]);
            a[3] = fma(sxy, gx, a[3]);
            a[4] = fma(e0, gy, a[4]);
            a[5] = fma(pdx, gy, a[5]);
            a[6] = fma(sy, gy, a[6]);
            a[7] = fma(sxy, gy, a[7]);
            pT = hT;
            pX = hX;
            pY = hY;
            pmv = mv;
            pdx = dx;
        }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) m[k] = warp_sum_d(a[k]);
}

// Result of one FP64 level.
struct Level64 {
    double nx, ny;  // step sum from the level's guess
    float lmin;     // normalised lambda_min (FP64, rounded)
    int reason;     // VT_TRACKED, VT_LOST_EIG or VT_LOST_OOB
    int iters, sweeps;
};

// One level in FP64 (see kFp64Cond): the eigenvalue test and the Newton
// iterations from the level's guess (gx, gy).
template <int WIN, int GT>
__device__ __forceinline__ Level64 track_level64(const Level Jl, const int max_iters, const float eps2,
                                              const float min_eig, float ux, float uy, float gx, float gy,
                                              const TWin &W, int lane, KSmem<WIN> *smp) {
    constexpr int HW = WIN / 2;
    constexpr double N = (double)(WIN * WIN);
    KSmem<WIN> &sm = *smp;
    Level64 o;
    o.reason = VT_TRACKED;
    o.iters = 0;
    o.sweeps = 0;
    o.nx = o.ny = 0.0;
    const double ax = (double)(ux - floorf(ux)), ay = (double)(uy - floorf(uy));
    double G11, G12, G22;
    template_G64<WIN, GT>(ax, ay, W, lane, G11, G12, G22);
    const double det64 = G11 * G22 - G12 * G12;
    const double lmax64 = 0.5 * (G11 + G22 + sqrt((G11 - G22) * (G11 - G22) + 4.0 * G12 * G12));
    const double lmin64 = det64 / lmax64 / (N * 65025.0);
    o.lmin = (float)lmin64;
    if (!(lmin64 >= (double)min_eig) || !(det64 > 0.0)) {
        o.reason = VT_LOST_EIG;
        return o;
    }
    int cx = INT_MIN, cy = INT_MIN;
    double m[8];
    const double uxd = (double)ux + (double)gx, uyd = (double)uy + (double)gy;
    for (int k = 0; k < max_iters; ++k) {
        const double qx = uxd + o.nx, qy = uyd + o.ny;
        const double dist = fmin(fmin(qx + (double)HW, (double)(Jl.w - 1 + HW) - qx),
                                 fmin(qy + (double)HW, (double)(Jl.h - 1 + HW) - qy));
        if (!(dist >= 0.0)) {
            o.reason = VT_LOST_OOB;
            return o;
        }
        const double fx = floor(qx), fy = floor(qy);
        const int ix = (int)fx - HW, iy = (int)fy - HW;
        if (ix != cx || iy != cy) {
            cell_moments64<WIN, GT>(Jl, ix, iy, ax, ay, W, lane, sm, m);
            cx = ix;
            cy = iy;
            ++o.sweeps;
        }
        const double bx = qx - fx, by = qy - fy, bxy = bx * by;
        const double b1 = m[0] - bx * m[1] - by * m[2] - bxy * m[3];
        const double b2 = m[4] - bx * m[5] - by * m[6] - bxy * m[7];
        const double ex = (G22 * b1 - G12 * b2) / det64;
        const double ey = (G11 * b2 - G12 * b1) / det64;
        o.nx += ex;
        o.ny += ey;
        ++o.iters;
        if (ex * ex + ey * ey < (double)eps2) break;
    }
    return o;
}

// Internal reason of a point the FP32 tracker leaves to the FP64-capable one
// (its status is written as kStatusPending until that second launch).
constexpr int kReasonPending = 255;
constexpr uint8_t kStatusPending = 2;

// Track one point u = (ux0, uy0) from pyramid I to pyramid J.  The FP32
// tracker (F64 = false) stops at a level whose template is ill-conditioned
// (kFp64Cond) and marks the point pending (kReasonPending); the kernels then
// leave it to a second, FP64-capable launch (F64 = true) that tracks it again
// from the start with such levels in FP64.  Levels are deterministic, so its
// coarser levels give the same results the second time.  Keeping the FP64
// code out of the FP32 kernels keeps their registers free of it.
template <int WIN, int GT, bool F64>
__device__ __forceinline__ void track_point(const Level *I, const Level *J, const KParams &P, float ux0, float uy0,
                                            bool has_guess, float gux, float guy, int lane, const KCta<WIN> &C,
                                            KSmem<WIN> &sm, KOut &o, bool want_err) {
    constexpr int HW = WIN / 2;
    constexpr float N = (float)(WIN * WIN);
    constexpr float unit = grad_unit<GT>();
    // lambda_min normalisation: stored units^2 -> (grey/px)^2, / (N 255^2)
    const float inv_norm = unit * unit / (N * 65025.0f);
    constexpr int NS = KRuns<WIN>::NS;
    float T[NS];
    float2 G[NS];
    const int L = P.levels;
    float gx = 0.f, gy = 0.f, nux = 0.f, nuy = 0.f;
    double nx64 = 0.0, ny64 = 0.0;  // the step sum of an FP64 level
    bool level64 = false;           // the last level examined ran in FP64
    int lost_level = 0;
    o.status = 1;
    o.reason = VT_TRACKED;
    o.iters = 0;
    o.tmpl = 0;
    o.errp = 0;
    o.sweeps = 0;
    o.err = 0.f;
    o.lmin = __int_as_float(0x7fc00000);
    if (!(ux0 >= 0.f && ux0 <= (float)(I[0].w - 1) && uy0 >= 0.f && uy0 <= (float)(I[0].h - 1))) {
        o.status = 0;
        o.reason = VT_LOST_INPUT;
        o.x = ux0;
        o.y = uy0;
        return;
    }
    if (has_guess) {
        const float s = pow2neg(L - 1);
        gx = (gux - ux0) * s;
        gy = (guy - uy0) * s;
    }
    // integer part of the current footprint cell (unknown: NaN)
    constexpr float kNone = __builtin_nanf("");
    float cfx = kNone, cfy = kNone;
    bool staged = true;  // whether sm.j holds that cell's footprint
    // the template started by the previous iteration: position, its floor, the level's width
    float ux = 0.f, uy = 0.f, ufx = 0.f, ufy = 0.f;
    int tw = 0;
    float s = pow2neg(L);
    // Level l's iteration starts its own first footprint (its position is known
    // now) and the next level's template (known from the start) before it
    // samples its own template, which the previous iteration started: the
    // copies arrive while the warp computes.  l = L only starts the first
    // template.  Two commit groups per level, so the waits below count them.
    for (int l = L; l >= 0; --l) {
        const float ax = ux - ufx, ay = uy - ufy;
        const int tx0 = (int)ufx - HW, ty0 = (int)ufy - HW, w_I = tw;  // the template's window
        const float qx0 = ux + gx, qy0 = uy + gy;  // the level's first footprint position
        float limx = 0.f, limy = 0.f;              // footprint positions lie in [-HW, limx] x [-HW, limy]
        bool inside = false;
        Level Jl;
        cfx = kNone;
        if (l < L) {
            Jl = J[l];  // by value: the fields stay in registers across the copies
            limx = (float)(Jl.w - 1 + HW);
            limy = (float)(Jl.h - 1 + HW);
            inside = qx0 >= -(float)HW && qx0 <= limx && qy0 >= -(float)HW && qy0 <= limy;
            if (inside) {
                cfx = floorf(qx0);
                cfy = floorf(qy0);
                staged = true;
                stage_window<WIN, false>(Jl, (int)cfx - HW, (int)cfy - HW, lane, sm.j, nullptr);
            }
            cp_async_commit();
        }
        if (l > 0) {
            const Level In = I[l - 1];
            s += s;
            ux = ux0 * s, uy = uy0 * s;
            ufx = floorf(ux), ufy = floorf(uy);
            tw = In.w;
            if constexpr (GT == VT_GRAD_NONE)
                stage_raw<WIN>(In, (int)ufx - HW, (int)ufy - HW, lane, sm.raw((l - 1) & 1));
            else
                stage_window<WIN, true>(In, (int)ufx - HW, (int)ufy - HW, lane, sm.t[(l - 1) & 1], sm.g[(l - 1) & 1]);
        }
        cp_async_commit();
        if (l == L) continue;
        TWin W;
        W.x0 = tx0, W.w = w_I;
        cp_async_wait<2>();
        __syncwarp();
        if constexpr (GT == VT_GRAD_NONE) {
            gradients_from_raw<WIN>(sm.raw(l & 1), w_I, I[l].h, tx0, ty0, lane, sm.g[0]);
            W.st = sm.raw(l & 1) + KSmem<WIN>::RS;
            W.sg = sm.g[0];
            W.sx = staged_x(tx0 - 1, 16);
            W.gx0 = 0, W.gw = WIN + 1, W.gsx = 0;  // window columns, clamped already
        } else {
            W.st = sm.t[l & 1];
            W.sg = sm.g[l & 1];
            W.sx = staged_x(tx0, 16);
            W.gx0 = tx0, W.gw = w_I, W.gsx = staged_x(tx0, 4);
        }
        sample_template<WIN, GT>(C, W, ax, ay, lane, T, G);
        ++o.tmpl;
        float2 aii = pair(0.f);
        float a12 = 0.f;
#pragma unroll
        for (int r = 0; r < NS; ++r) {
            aii = __ffma2_rn(G[r], G[r], aii);
            a12 = fmaf(G[r].x, G[r].y, a12);
        }
        float g11, g12, g22;
        warp_sum3(aii.x, a12, aii.y, lane, g11, g12, g22);
        const float tr = g11 + g22, df = g11 - g22;
        const float det = kdiff(g11, g22, g12, g12);  // sign exact, 2 ulp
        nux = nuy = 0.f;
        // lambda_min = det / lambda_max >= det / tr: a template that passes with
        // that bound by more than the rounding of all this (1e-5 against a few
        // 1e-7) passes, and the square root and the division are left out
        // unless the caller wants lambda_min (or a level may need FP64)
        const bool passes = det * inv_norm > 1.00001f * P.min_eig * tr;
        if (F64 || P.fp64 || P.want_lmin || !passes) {
            // det / lambda_max avoids the cancellation of (tr - disc) / 2
            const float lmax = 0.5f * (tr + sqrtf(fmaf(df, df, 4.f * g12 * g12)));
            const float lmin = det / lmax;
            o.lmin = lmin * inv_norm;
            // ill-conditioned (or det <= 0): decided and tracked in FP64
            level64 = P.fp64 && !(lmin * kFp64Cond >= lmax);
        }
        if (level64) {
            if constexpr (!F64) {
                cp_async_wait<0>();  // nothing may land after the buffers are used again
                o.status = 0;
                o.reason = kReasonPending;
                return;
            } else {
                cp_async_wait<0>();  // the first footprint started above: sm.j is staged anew
                const Level64 r = track_level64<WIN, GT>(Jl, P.max_iters, P.eps2, P.min_eig, ux0 * pow2neg(l),
                                                         uy0 * pow2neg(l), gx, gy, W, lane, &sm);
                cfx = kNone;
                o.lmin = r.lmin;
                o.iters += r.iters;
                o.sweeps += r.sweeps;
                nx64 = r.nx;
                ny64 = r.ny;
                if (r.reason != VT_TRACKED) {
                    o.status = 0;
                    o.reason = r.reason;
                    lost_level = l;
                    break;
                }
                if (l > 0) {
                    gx = (float)(2.0 * ((double)gx + nx64));
                    gy = (float)(2.0 * ((double)gy + ny64));
                    level64 = false;
                }
                continue;
            }
        }
        if (!passes && (!(o.lmin >= P.min_eig) || !(det > 0.f))) {
            o.status = 0;
            o.reason = VT_LOST_EIG;
            lost_level = l;
            break;
        }
        // eta = G^-1 b in grey/px units: G = unit^2 G_s, b = unit b_s => eta = adj(G_s) b_s / (unit det_s)
        // (unit is a power of two, so det * unit is exact; the adjugate
        // products cancel for ill-conditioned G, hence kdiff)
        const float inv_det = -1.0f / (det * unit) * kImgUnscale;  // of -b, which carries the image scale
        if (!inside) {
            o.status = 0;
            o.reason = VT_LOST_OOB;
            lost_level = l;
            break;
        }
        // the moments of a footprint cell serve every position in it; the
        // first cell's copy was started above
        float2 m[4];
        cp_async_wait<1>();
        __syncwarp();
        cell_moments<WIN>((int)cfx - HW, Jl.w, lane, T, G, sm, m);
        ++o.sweeps;
        float bx = qx0 - cfx, by = qy0 - cfy;
        // A position is in the cell when both offsets lie in [0, 1): as bit
        // patterns, below that of 1 (negative numbers and NaN are above).  A
        // cell that begins at the bound holds positions outside: there every
        // step takes the full test (0).
        constexpr unsigned kOne = 0x3f800000u;
        unsigned cell_end = cfx >= limx || cfy >= limy ? 0u : kOne;
        bool left_cell = false;  // whether sm.cell_* hold this level's entries
        for (int k = 1;; ++k) {
            const float bxy = bx * by;
            float2 b = __ffma2_rn(pair(bx), m[1], m[0]);  // -b
            b = __ffma2_rn(pair(by), m[2], b);
            b = __ffma2_rn(pair(bxy), m[3], b);
            const float ex = kdiff(g22, b.x, g12, b.y) * inv_det;
            const float ey = kdiff(g11, b.y, g12, b.x) * inv_det;
            nux += ex;
            nuy += ey;
            ++o.iters;
            if (norm2(ex, ey) < P.eps2 || k >= P.max_iters) break;
            const float qx = qx0 + nux, qy = qy0 + nuy;
            bx = qx - cfx, by = qy - cfy;
            if (max(__float_as_uint(bx), __float_as_uint(by)) >= cell_end) {
                if (!(qx >= -(float)HW && qx <= limx && qy >= -(float)HW && qy <= limy)) {
                    o.status = 0;
                    o.reason = VT_LOST_OOB;
                    break;
                }
                const float fx = floorf(qx), fy = floorf(qy);
                if (fx != cfx || fy != cfy) {
                    // every lane stores and reads back the same values
                    const int ix = (int)fx, iy = (int)fy, px = (int)cfx, py = (int)cfy;
                    const int slot = (ix & 1) | (iy & 1) << 1, old = (px & 1) | (py & 1) << 1;
                    if (!left_cell) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) sm.cell_at[q] = make_int2(INT_MIN, INT_MIN);
                        left_cell = true;
                    }
#pragma unroll
                    for (int q = 0; q < 4; ++q) sm.cell_m[old][q] = m[q];
                    sm.cell_at[old] = make_int2(px, py);
                    cfx = fx, cfy = fy;
                    const int2 at = sm.cell_at[slot];
                    if (at.x == ix && at.y == iy) {
#pragma unroll
                        for (int q = 0; q < 4; ++q) m[q] = sm.cell_m[slot][q];
                        staged = false;
                    } else {
                        stage_footprint<WIN>(Jl, ix - HW, iy - HW, lane, sm);
                        cell_moments<WIN>(ix - HW, Jl.w, lane, T, G, sm, m);
                        ++o.sweeps;
                        staged = true;
                    }
                    bx = qx - fx, by = qy - fy;
                    cell_end = fx >= limx || fy >= limy ? 0u : kOne;
                }
            }
        }
        if (!o.status) {
            lost_level = l;
            break;
        }
        if (l > 0) {
            gx = 2.f * (gx + nux);
            gy = 2.f * (gy + nuy);
        }
    }
    cp_async_wait<0>();  // a point lost early leaves copies under way; nothing may land after this
    {
        const float sc = (float)(1 << lost_level);
        const float si = pow2neg(lost_level);
        if (F64 && level64) {
            o.x = (float)(((double)(ux0 * si) + (double)gx + nx64) * (double)sc);
            o.y = (float)(((double)(uy0 * si) + (double)gy + ny64) * (double)sc);
        } else {
            o.x = (ux0 * si + gx + nux) * sc;
            o.y = (uy0 * si + gy + nuy) * sc;
        }
    }
    if (o.status) {
        const float dist = fminf(fminf(o.x, (float)(I[0].w - 1) - o.x), fminf(o.y, (float)(I[0].h - 1) - o.y));
        if (!(dist >= 0.f)) {
            o.status = 0;
            o.reason = VT_LOST_OOB;
        } else {
            // T still holds level 0's template, and sm.j its last footprint
            if (want_err) {
                const float fx = floorf(o.x), fy = floorf(o.y);
                const int ix = (int)fx - HW, iy = (int)fy - HW;
                if (fx != cfx || fy != cfy || !staged) stage_footprint<WIN>(J[0], ix, iy, lane, sm);
                o.err = abs_residual<WIN>(C, ix, J[0].w, o.x - fx, o.y - fy, lane, T, sm) * kImgUnscale / N;
                ++o.errp;
            }
        }
    }
}

// Forward I->J (pass 0) and, with fb, backward J->I from the forward result
// (pass 1) followed by the FB test.  One inlined copy of track_point serves
// both passes, and every kernel (single-pair or batched) calls this function,
// so a point's result does not depend on which kernel tracked it.
template <int WIN, int GT, bool F64>
__device__ __forceinline__ void track_point_dir(const Level *I, const Level *J, const KParams &P, float ux0,
                                                float uy0, bool fb, bool has_guess, float gux, float guy, int lane,
                                                const KCta<WIN> &C, KSmem<WIN> &sm, KOut &o) {
    // the two level tables next to the warp: a level's fields are one shared
    // load away, not a chain of global ones
    static_assert(sizeof(Level) * VT_MAX_LEVELS == 16 * 16, "16 lanes copy a table");
    static_assert(offsetof(KSmem<WIN>, lv) % 16 == 0 && alignof(KSmem<WIN>) >= 16, "16-byte stores");
    __syncwarp();
    reinterpret_cast<uint4 *>(sm.lv)[lane] = reinterpret_cast<const uint4 *>(lane < 16 ? I : J)[lane & 15];
    __syncwarp();
    const Level *A = sm.lv[0], *B = sm.lv[1];
    float x = ux0, y = uy0;
    const int npass = fb ? 2 : 1;
#pragma unroll 1
    for (int pass = 0; pass < npass; ++pass) {
        KOut r;
        // the backward pass only decides the status: its error is not an output
        track_point<WIN, GT, F64>(A, B, P, x, y, pass == 0 && has_guess, gux, guy, lane, C, sm, r, pass == 0);
        if (pass == 0) {
            o = r;
            if (!r.status) return;
            x = r.x;
            y = r.y;
            A = sm.lv[1];
            B = sm.lv[0];
        } else {
            o.iters += r.iters;
            o.tmpl += r.tmpl;
            o.errp += r.errp;
            o.sweeps += r.sweeps;
            if (!r.status) {
                o.status = 0;
                o.reason = r.reason;
                return;
            }
            const float dx = ux0 - r.x, dy = uy0 - r.y;
            if (!(norm2(dx, dy) <= P.fb_thr2)) {
                o.status = 0;
                o.reason = VT_LOST_FB;
            }
        }
    }
}

}  // namespace vt
