// Gaussian pyramid (K1) and Scharr gradients (K2) for the LK tracker.
//
// K1: level l+1 = 5x5 separable [1 4 6 4 1]^2 / 256 sum centred at (2x, 2y)
//     of level l, reflect-101 borders, (s + 128) >> 8.  Integer arithmetic,
//     no rounding between the vertical and horizontal passes: bit-exact.
// K2: Scharr dx = [-3 0 3; -10 0 10; -3 0 3] * I, dy = transpose, reflect-101,
//     stored as (dx, dy) int16 pairs or (dx/32, dy/32) half pairs.
// The paper names the pyramidal LK tracker without its filters (Sec. IV,
// Table I); these are the readings implemented.
//
// Layout: a CTA stages its input tile (plus halo) in shared memory with
// 16-byte loads, the reflected columns of edge tiles filled in afterwards.
// The same staged tile serves the pyramid step and, in the fused variant, the
// gradients of the source level and the copy of a caller's frame.  A frame's
// small levels are built together from shared memory (tail_build).
#include <cuda.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "vt_internal.cuh"

namespace vt {

constexpr int PD_TW = 64;              // output tile width (level l+1)
constexpr int PD_TH = 16;              // output tile height
constexpr int PD_IW = 2 * PD_TW + 32;  // staged bytes per row (16-byte chunks)
constexpr int PD_IH = 2 * PD_TH + 3;   // staged rows
constexpr int PD_VW = 2 * PD_TW + 8;   // vertical-pass columns (staged columns 12 .. 12 + PD_VW)
constexpr int PD_THREADS = 256;

constexpr int SC_TW = 64;
constexpr int SC_TH = 16;
constexpr int SC_IW = SC_TW + 32;
constexpr int SC_IH = SC_TH + 2;
constexpr int SC_THREADS = 256;

template <int GT>
__device__ __forceinline__ uint32_t pack_grad(int dx, int dy) {
    if (GT == VT_GRAD_S16) {
        return (uint32_t)(uint16_t)(int16_t)dx | ((uint32_t)(uint16_t)(int16_t)dy << 16);
    } else {
        // raw / 32 is exact in FP32; the conversion to half rounds to nearest even
        __half2 h = __floats2half2_rn((float)dx * 0.03125f, (float)dy * 0.03125f);
        return *reinterpret_cast<uint32_t *>(&h);
    }
}

// Scharr of the staged tile at staged (row sr, column sc).
template <int IW>
__device__ __forceinline__ void scharr_at(const uint8_t (*s)[IW], int sr, int sc, int &dx, int &dy) {
    const int a00 = s[sr - 1][sc - 1], a01 = s[sr - 1][sc], a02 = s[sr - 1][sc + 1];
    const int a10 = s[sr][sc - 1], a12 = s[sr][sc + 1];
    const int a20 = s[sr + 1][sc - 1], a21 = s[sr + 1][sc], a22 = s[sr + 1][sc + 1];
    dx = 3 * (a02 - a00) + 10 * (a12 - a10) + 3 * (a22 - a20);
    dy = 3 * (a20 - a00) + 10 * (a21 - a01) + 3 * (a22 - a02);
}

// `n` bytes (1 .. 16) at any address, by the aligned words that hold them (each
// holds at least one of the bytes, so none lies outside the caller's allocation).
__device__ __forceinline__ uint4 load16_any(const uint8_t *p, unsigned n) {
    const unsigned a = (unsigned)(uintptr_t)p & 3u;
    const uint32_t *q = reinterpret_cast<const uint32_t *>(p - a);
    uint32_t v[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) v[k] = 4 * k < a + n ? q[k] : 0u;
    return make_uint4(__funnelshift_r(v[0], v[1], 8 * a), __funnelshift_r(v[1], v[2], 8 * a),
                      __funnelshift_r(v[2], v[3], 8 * a), __funnelshift_r(v[3], v[4], 8 * a));
}

// Stage rows [iy0, iy0 + IH) and columns [ix0, ix0 + IW) of an image (ix0 a
// multiple of 16), rows and columns reflected into it; ends with a barrier.
// The 16-byte chunks inside the image are copied whole (one load where the
// rows are 16-byte aligned, vec_ok, else word by word), of the chunk that holds
// the last column only the words that reach into the row (a caller's last row
// may end there); the columns -2, -1, w and w + 1 are then filled
// from the staged ones (the reflected columns lie in the same tile for w >= 4;
// the readers use no others outside the image).  A tile at the image's edge
// so costs about what an inner one does: mapping every byte of it through the
// reflection took most of a small level's launch (all of its tiles are at an
// edge): 11.7 -> 4.5 us at 752 x 480, and level 0 of 32 frames 144 -> 89 us.
//
// Pixels are read by ordinary loads, here and in tail_build: the launch before
// may still be writing them when this one starts (programmatic dependent
// launch), and a read-only load (__ldg) wants data that nothing writes while
// the kernel runs; it need not stay behind pdl_wait() either.  A thread's
// chunks are all loaded before the first is stored, which the compiler does not
// do for ordinary loads by itself (752 x 480 build 13.44 us without, 12.38 so;
// 12.94 with read-only loads; 1919 x 1199 half planes 21.0, 17.8 and 20.7).
template <int IH, int IW>
__device__ __forceinline__ void stage_tile(uint8_t (*s)[IW], const uint8_t *src, int w, int h, int pitch, int ix0,
                                           int iy0, bool vec_ok) {
    constexpr int C16 = IW / 16;
    if (w >= 4) {
        const bool inner = ix0 >= 0 && ix0 + IW <= w && iy0 >= 0 && iy0 + IH <= h;
        constexpr int N = (IH * C16 + PD_THREADS - 1) / PD_THREADS;  // chunks a thread (of at least PD_THREADS)
        uint4 v[N];
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const int i = threadIdx.x + k * blockDim.x, r = i / C16, x = ix0 + 16 * (i - r * C16);
            if (i < IH * C16 && (inner || (x >= 0 && x < w))) {
                const uint8_t *p = src + (size_t)(inner ? iy0 + r : refl101(iy0 + r, h)) * pitch + x;
                v[k] = vec_ok && x + 16 <= w ? *reinterpret_cast<const uint4 *>(p) : load16_any(p, min(16, w - x));
            }
        }
#pragma unroll
        for (int k = 0; k < N; ++k) {
            const int i = threadIdx.x + k * blockDim.x, r = i / C16, c = i - r * C16, x = ix0 + 16 * c;
            if (i < IH * C16 && (inner || (x >= 0 && x < w))) *reinterpret_cast<uint4 *>(&s[r][c * 16]) = v[k];
        }
        if (!inner) {
            __syncthreads();
            static_assert(IH <= 64, "one row per thread of two warps");
            if (threadIdx.x < IH) {
                const int r = threadIdx.x, e = w - ix0;
                if (ix0 < 0) {
                    s[r][-2 - ix0] = s[r][2 - ix0];
                    s[r][-1 - ix0] = s[r][1 - ix0];
                }
                if (e < IW) s[r][e] = s[r][e - 2];
                if (e + 1 < IW) s[r][e + 1] = s[r][e - 3];
            }
            __syncwarp();
        }
    } else {
        for (int i = threadIdx.x; i < IH * IW; i += blockDim.x) {
            const int r = i / IW, c = i - r * IW;
            const int sy = refl101(iy0 + r, h), sx = refl101(ix0 + c, w);
            s[r][c] = src[(size_t)sy * pitch + sx];
        }
    }
    __syncthreads();
}

// Copy the staged rows [r0, r0 + nr) x staged columns [c0, c0 + 128) to
// dst rows y0.. / columns x0.. (x0 a multiple of 128, dst rows 16-byte aligned).
template <int IW>
__device__ __forceinline__ void copy_out(const uint8_t (*s)[IW], int r0, int c0, int nr, uint8_t *dst, int dpitch,
                                         int x0, int y0, int w, int h) {
    for (int i = threadIdx.x; i < nr * 8; i += blockDim.x) {
        const int r = i >> 3, c = (i & 7) * 16;
        const int y = y0 + r, x = x0 + c;
        if (y >= h || x >= w) continue;
        uint8_t *d = dst + (size_t)y * dpitch + x;
        if (x + 16 <= w) {
            *reinterpret_cast<uint4 *>(d) = *reinterpret_cast<const uint4 *>(&s[r0 + r][c0 + c]);
        } else {
            for (int q = 0; q < 16 && x + q < w; ++q) d[q] = s[r0 + r][c0 + c + q];
        }
    }
}

// Four columns x .. x+3 of a staged row as the packed Scharr pass holds them:
// two columns two apart in the 16-bit lanes of a word, (x, x+2), (x+1, x+3),
// and the edge columns (x-1, x+4).
struct Row4 {
    uint32_t c13, c24, ce;
};
// From the words that hold columns x-4 .. x-1, x .. x+3 and x+4 .. x+7.
__device__ __forceinline__ Row4 row4(uint32_t a, uint32_t b, uint32_t c) {
    return {b & 0x00FF00FFu, (b >> 8) & 0x00FF00FFu, (a >> 24) | ((c << 16) & 0x00FF0000u)};
}

// Scharr (int16 output) of 4 consecutive columns of the row between `t` and
// `u` (m: the row itself), two pixels per 32-bit operation.  Per lane, the
// vertical smoothing V = 3 top + 10 mid + 3 bottom is at most 4080 and the
// biased difference D = bottom - top + 2048 lies in [1793, 2303], so
//   dx + 32768 = V(x+1) - V(x-1) + 32768,
//   dy + 32768 = 3 D(x-1) + 10 D(x) + 3 D(x+1)      (bias 16 * 2048)
// both lie in [28688, 36848]: no lane ever borrows from or carries into its
// neighbour, and flipping bit 15 of a lane turns the biased value into the
// int16 two's complement of dx or dy.  Same results as the scalar form.
__device__ __forceinline__ uint4 scharr4_s16(const Row4 &t, const Row4 &m, const Row4 &u) {
    const uint32_t v13 = 3u * (t.c13 + u.c13) + 10u * m.c13;
    const uint32_t v24 = 3u * (t.c24 + u.c24) + 10u * m.c24;
    const uint32_t ve = 3u * (t.ce + u.ce) + 10u * m.ce;
    const uint32_t d13 = u.c13 + 0x08000800u - t.c13;
    const uint32_t d24 = u.c24 + 0x08000800u - t.c24;
    const uint32_t de = u.ce + 0x08000800u - t.ce;
    const uint32_t vm = __byte_perm(ve, v24, 0x5410), vp = __byte_perm(v13, ve, 0x7632);  // (x-1, x+1), (x+2, x+4)
    const uint32_t dm = __byte_perm(de, d24, 0x5410), dp = __byte_perm(d13, de, 0x7632);
    const uint32_t dx13 = (v24 + 0x80008000u - vm) ^ 0x80008000u;  // columns (x, x+2)
    const uint32_t dx24 = (vp + 0x80008000u - v13) ^ 0x80008000u;  // columns (x+1, x+3)
    const uint32_t dy13 = (3u * (dm + d24) + 10u * d13) ^ 0x80008000u;
    const uint32_t dy24 = (3u * (d13 + dp) + 10u * d24) ^ 0x80008000u;
    return make_uint4(__byte_perm(dx13, dy13, 0x5410), __byte_perm(dx24, dy24, 0x5410),
                      __byte_perm(dx13, dy13, 0x7632), __byte_perm(dx24, dy24, 0x7632));
}

// The gradient words of columns x .. x+3 to a row of w columns.
__device__ __forceinline__ void store_grad4(uint32_t *row, int x, int w, const uint4 &g) {
    if (x + 3 < w) {
        *reinterpret_cast<uint4 *>(row + x) = g;
    } else {
        const uint32_t gq[4] = {g.x, g.y, g.z, g.w};
        for (int q = 0; q < 4 && x + q < w; ++q) row[x + q] = gq[q];
    }
}

// Scharr (int16 output) of 4 consecutive columns x .. x+3 and 4 rows y0 ..
// y0+3 of the staged tile.  `sr0` is the staged row above y0; `xr` the staged
// column offset of x.
__device__ __forceinline__ void scharr_4x4_s16(const uint8_t (*s)[PD_IW], int sr0, int xr, int x, int y0, int w,
                                               int h, uint32_t *grad, int gpitch) {
    auto load_row = [&](int sr) {
        const uint32_t *wp = reinterpret_cast<const uint32_t *>(&s[sr][12 + xr]);
        return row4(wp[0], wp[1], wp[2]);  // columns x-4 .. x+7
    };
    Row4 r0 = load_row(sr0), r1 = load_row(sr0 + 1);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const Row4 r2 = load_row(sr0 + 2 + i);
        const int y = y0 + i;
        if (y < h && x < w) store_grad4(grad + (size_t)y * gpitch, x, w, scharr4_s16(r0, r1, r2));
        r0 = r1;
        r1 = r2;
    }
}

// Vertical [1 4 6 4 1] sums of a word's columns over five rows: (columns 0, 2)
// and (1, 3) in 16-bit lanes (at most 16 * 255, no carry between lanes).
__device__ __forceinline__ void vsum4(const uint32_t (&v)[5], uint32_t &sl, uint32_t &sh) {
    uint32_t lo[5], hi[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
        lo[k] = v[k] & 0x00FF00FFu;
        hi[k] = (v[k] >> 8) & 0x00FF00FFu;
    }
    sl = lo[0] + lo[4] + 4u * (lo[1] + lo[3]) + 6u * lo[2];
    sh = hi[0] + hi[4] + 4u * (hi[1] + hi[3]) + 6u * hi[2];
}

// Four consecutive pyramid outputs from the vertical sums of their columns,
// two outputs per 32-bit operation: p[k] holds columns (2k - 2, 2k - 1)
// relative to the first output's centre, and output q needs columns 2q - 2 ..
// 2q + 2, so lane pairs (c, c+2) are gathered by byte permutes; a lane's sum
// is at most 16 * 4080 + 128 and never carries into its neighbour.
__device__ __forceinline__ uint32_t hsum4(const uint32_t (&p)[6]) {
    auto lo2 = [](uint32_t a, uint32_t b) { return __byte_perm(a, b, 0x5410); };
    auto hi2 = [](uint32_t a, uint32_t b) { return __byte_perm(a, b, 0x7632); };
    auto down2 = [](uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, uint32_t w4) {
        const uint32_t sum = w0 + w4 + 0x00800080u + 4u * (w1 + w3) + 6u * w2;
        return (sum >> 8) & 0x00FF00FFu;
    };
    const uint32_t w4 = lo2(p[2], p[3]);
    const uint32_t ra = down2(lo2(p[0], p[1]), hi2(p[0], p[1]), lo2(p[1], p[2]), hi2(p[1], p[2]), w4);
    const uint32_t rb = down2(w4, hi2(p[2], p[3]), lo2(p[3], p[4]), hi2(p[3], p[4]), lo2(p[4], p[5]));
    return __byte_perm(ra, rb, 0x6420);  // bytes o0, o1, o2, o3
}

// Four outputs x .. x+3 to a row of w columns.
__device__ __forceinline__ void store_px4(uint8_t *row, int x, int w, uint32_t packed) {
    if (x + 3 < w) {
        *reinterpret_cast<uint32_t *>(row + x) = packed;
    } else {
        for (int q = 0; q < 4 && x + q < w; ++q) row[x + q] = (uint8_t)(packed >> (8 * q));
    }
}

// One output tile (tx, ty) of the pyramid step src -> dst; with GRAD also the
// Scharr planes of src over the matching 2*TW x 2*TH region, and with `copy`
// a copy of that src region (level 0 of a pyramid built from a caller image).
// Needs blockDim.x == PD_THREADS.
//
// The staged tile holds image columns ix0 .. ix0 + PD_IW with ix0 = 2*ox0 - 16
// and rows iy0 .. iy0 + PD_IH with iy0 = 2*oy0 - 2.
//  * vertical [1 4 6 4 1] pass on 32-bit words: the even and odd bytes of a
//    word are summed as two packed 16-bit lanes (at most 16 * 255 = 4080, no
//    carry between lanes), 4 columns per operation;
//  * horizontal pass: 4 outputs per thread from 6 packed column pairs, two
//    outputs per 32-bit operation;
//  * Scharr: each thread owns 4 columns x 4 rows and slides a 3-row window of
//    6 bytes per row (3 aligned word loads per row), with the separable form
//    dx = s(x+1) - s(x-1), s = 3 top + 10 mid + 3 bottom, and
//    dy = 3 d(x-1) + 10 d(x) + 3 d(x+1), d = bottom - top; int16 planes two
//    pixels per 32-bit operation (scharr_4x4_s16), half planes per pixel.
template <bool GRAD, int GT>
__device__ __forceinline__ void pyr_tile_compute(int w, int h, uint8_t *dst, int dpitch, uint32_t *grad, int gpitch,
                                                 uint8_t *copy, int cpitch, int tx, int ty,
                                                 uint8_t (*s_in)[PD_IW], uint16_t (*s_v)[PD_VW]);

template <bool GRAD, int GT>
__device__ __forceinline__ void pyr_tile(const uint8_t *src, int w, int h, int spitch, bool vec_ok, uint8_t *dst,
                                         int dpitch, uint32_t *grad, int gpitch, uint8_t *copy, int cpitch, int tx,
                                         int ty, uint8_t (*s_in)[PD_IW], uint16_t (*s_v)[PD_VW]) {
    stage_tile<PD_IH, PD_IW>(s_in, src, w, h, spitch, 2 * tx * PD_TW - 16, 2 * ty * PD_TH - 2, vec_ok);
    pyr_tile_compute<GRAD, GT>(w, h, dst, dpitch, grad, gpitch, copy, cpitch, tx, ty, s_in, s_v);
}

// The computing part of pyr_tile on an already staged tile.
template <bool GRAD, int GT>
__device__ __forceinline__ void pyr_tile_compute(int w, int h, uint8_t *dst, int dpitch, uint32_t *grad, int gpitch,
                                                 uint8_t *copy, int cpitch, int tx, int ty,
                                                 uint8_t (*s_in)[PD_IW], uint16_t (*s_v)[PD_VW]) {
    const int W = (w + 1) >> 1, H = (h + 1) >> 1;
    const int ox0 = tx * PD_TW, oy0 = ty * PD_TH;

    // vertical pass: s_v[r][c] = sum_k [1 4 6 4 1]_k staged(2r + k, 12 + c)
    for (int i = threadIdx.x; i < PD_TH * (PD_VW / 4); i += PD_THREADS) {
        const int r = i / (PD_VW / 4), j = i - r * (PD_VW / 4);
        uint32_t v[5], sl, sh;
#pragma unroll
        for (int k = 0; k < 5; ++k) v[k] = *reinterpret_cast<const uint32_t *>(&s_in[2 * r + k][12 + 4 * j]);
        vsum4(v, sl, sh);
        uint32_t *out = reinterpret_cast<uint32_t *>(&s_v[r][0]) + 2 * j;
        *reinterpret_cast<uint2 *>(out) = make_uint2(__byte_perm(sl, sh, 0x5410), __byte_perm(sl, sh, 0x7632));
    }
    if constexpr (GRAD && GT == VT_GRAD_S16) {
        const int g = threadIdx.x & 31, rg = threadIdx.x >> 5;
        scharr_4x4_s16(s_in, 4 * rg + 1, 4 * g, 2 * ox0 + 4 * g, 2 * oy0 + 4 * rg, w, h, grad, gpitch);
    } else if constexpr (GRAD) {
        const int g = threadIdx.x & 31, rg = threadIdx.x >> 5;
        const int xr = 4 * g, x = 2 * ox0 + xr;
        int t0[6], t1[6], t2[6];
        auto load_row = [&](int sr, int (&v)[6]) {
            const uint32_t *wp = reinterpret_cast<const uint32_t *>(&s_in[sr][12 + xr]);
            const uint32_t a = wp[0], b = wp[1], c = wp[2];
            v[0] = (int)(a >> 24);
            v[1] = (int)(b & 0xffu);
            v[2] = (int)((b >> 8) & 0xffu);
            v[3] = (int)((b >> 16) & 0xffu);
            v[4] = (int)(b >> 24);
            v[5] = (int)(c & 0xffu);
        };
        load_row(4 * rg + 1, t0);
        load_row(4 * rg + 2, t1);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            load_row(4 * rg + 3 + i, t2);
            const int y = 2 * oy0 + 4 * rg + i;
            if (y < h && x < w) {
                int sm[6], dd[6];
#pragma unroll
                for (int k = 0; k < 6; ++k) {
                    sm[k] = 3 * (t0[k] + t2[k]) + 10 * t1[k];
                    dd[k] = t2[k] - t0[k];
                }
                uint32_t gq[4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    gq[q] = pack_grad<GT>(sm[q + 2] - sm[q], 3 * (dd[q] + dd[q + 2]) + 10 * dd[q + 1]);
                uint32_t *d = grad + (size_t)y * gpitch + x;
                if (x + 3 < w) {
                    *reinterpret_cast<uint4 *>(d) = make_uint4(gq[0], gq[1], gq[2], gq[3]);
                } else {
                    for (int q = 0; q < 4 && x + q < w; ++q) d[q] = gq[q];
                }
            }
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                t0[k] = t1[k];
                t1[k] = t2[k];
            }
        }
    }
    if (copy) copy_out<PD_IW>(s_in, 2, 16, 2 * PD_TH, copy, cpitch, 2 * ox0, 2 * oy0, w, h);
    __syncthreads();
    // horizontal pass: 4 consecutive outputs per thread; output x uses
    // s_v columns 2x + 2 .. 2x + 6
    {
        const int r = threadIdx.x >> 4, x4 = (threadIdx.x & 15) * 4;
        const int oy = oy0 + r, ox = ox0 + x4;
        if (oy < H && ox < W) {
            const uint32_t *pr = reinterpret_cast<const uint32_t *>(&s_v[r][0]) + x4 + 1;
            uint32_t p[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) p[k] = pr[k];
            store_px4(dst + (size_t)oy * dpitch, ox, W, hsum4(p));
        }
    }
}

// One Scharr tile (tx, ty) of a level; with `copy` also a copy of the tile.
template <int GT>
__device__ __forceinline__ void scharr_tile(const uint8_t *src, int w, int h, int spitch, bool vec_ok,
                                            uint32_t *grad, int gpitch, uint8_t *copy, int cpitch, int tx, int ty,
                                            uint8_t (*s_in)[SC_IW]) {
    const int x0 = tx * SC_TW, y0 = ty * SC_TH;
    stage_tile<SC_IH, SC_IW>(s_in, src, w, h, spitch, x0 - 16, y0 - 1, vec_ok);
    for (int i = threadIdx.x; i < SC_TH * (SC_TW / 4); i += blockDim.x) {
        const int r = i / (SC_TW / 4), x4 = (i - r * (SC_TW / 4)) * 4;
        const int y = y0 + r, x = x0 + x4;
        if (y >= h || x >= w) continue;
        uint32_t g[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            int dx, dy;
            scharr_at<SC_IW>(s_in, r + 1, x4 + q + 16, dx, dy);
            g[q] = pack_grad<GT>(dx, dy);
        }
        uint32_t *d = grad + (size_t)y * gpitch + x;
        if (x + 3 < w) {
            *reinterpret_cast<uint4 *>(d) = make_uint4(g[0], g[1], g[2], g[3]);
        } else {
            for (int q = 0; q < 4 && x + q < w; ++q) d[q] = g[q];
        }
    }
    if (copy) {
        // SC_TW = 64 columns: copy with 16-byte stores per 16 columns
        for (int i = threadIdx.x; i < SC_TH * 4; i += blockDim.x) {
            const int r = i >> 2, c = (i & 3) * 16;
            const int y = y0 + r, x = x0 + c;
            if (y >= h || x >= w) continue;
            uint8_t *d = copy + (size_t)y * cpitch + x;
            if (x + 16 <= w) {
                *reinterpret_cast<uint4 *>(d) = *reinterpret_cast<const uint4 *>(&s_in[r + 1][c + 16]);
            } else {
                for (int q = 0; q < 16 && x + q < w; ++q) d[q] = s_in[r + 1][c + 16 + q];
            }
        }
    }
    __syncthreads();
}

// One level of one frame (level 0 may come from the caller's image, with the
// level-0 copy written from the same tile).
template <bool GRAD, int GT>
__global__ void __launch_bounds__(PD_THREADS) k_pyrdown(const __grid_constant__ PyrJob J) {
    __shared__ __align__(16) uint8_t s_in[PD_IH][PD_IW];
    __shared__ uint16_t s_v[PD_TH][PD_VW];
    pdl_wait();  // the level (or the caller's image) is the previous launch's output
    pdl_trigger();
    const int ty = blockIdx.x / J.tiles_x, tx = blockIdx.x - ty * J.tiles_x;
    pyr_tile<GRAD, GT>(J.src, J.w, J.h, J.spitch, J.vec_ok != 0, J.dst, J.dpitch, J.grad, J.gpitch, J.copy, J.cpitch,
                       tx, ty, s_in, s_v);
}

template <int GT>
__global__ void __launch_bounds__(SC_THREADS) k_scharr(const __grid_constant__ GradJobs J) {
    __shared__ __align__(16) uint8_t s_in[SC_IH][SC_IW];
    pdl_wait();
    int k = 0;
    while (k + 1 < J.njobs && (int)blockIdx.x >= J.j[k + 1].tile0) ++k;
    const GradJob &jb = J.j[k];
    const int t = blockIdx.x - jb.tile0;
    const int ty = t / jb.tiles_x, tx = t - ty * jb.tiles_x;
    scharr_tile<GT>(jb.src, jb.w, jb.h, jb.spitch, jb.vec_ok != 0, jb.grad, jb.gpitch, jb.copy, jb.cpitch, tx, ty, s_in);
}

// --------------------------------------------------------- batched (persistent)
// Largest k with tile0[k] <= t over n jobs of stride `stride` ints.
__device__ __forceinline__ int find_job(const BLvlJob *jobs, int n, int t) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (jobs[mid].tile0 <= t) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Launch `l` (< VT_MAX_LEVELS - 1): level l -> l+1 plus the Scharr planes of
// level l for every frame of the batch whose tail starts above l (no Scharr
// planes for GT = VT_GRAD_NONE: the tracker computes gradients itself).  Level 0
// reads the caller's image and writes the pyramid's level-0 copy from the
// same tile (unless the frame is built in place).  The job list is first
// copied to shared memory so the per-tile job search does not chain global
// loads, and each job's source and destination are resolved on the host
// (BTileSrc), one load per tile, fetched a tile ahead.
constexpr int kJobsInSmem = 256;

// Six CTAs per SM (at most 40 registers a thread, no spills with the packed
// Scharr and horizontal passes): more tiles' loads in flight per SM.
template <int GT>
__global__ void __launch_bounds__(PD_THREADS, 6) k_pyr_batch(const uint8_t *tab, int l) {
    __shared__ __align__(16) uint8_t s_in[PD_IH][PD_IW];
    __shared__ uint16_t s_v[PD_TH][PD_VW];
    __shared__ BLvlJob s_jobs[kJobsInSmem];
    const BatchHdr *H = reinterpret_cast<const BatchHdr *>(tab);
    const int njobs = H->njobs[l], tiles = H->ntiles[l];
    if ((int)blockIdx.x >= tiles) return;
    const BLvlJob *gjobs = reinterpret_cast<const BLvlJob *>(tab + H->off_jobs) + (size_t)l * H->cap_frames;
    const bool in_smem = njobs <= kJobsInSmem;
    if (in_smem) {
        for (int i = threadIdx.x; i < njobs; i += blockDim.x) s_jobs[i] = gjobs[i];
        __syncthreads();
    }
    const BLvlJob *jobs = in_smem ? s_jobs : gjobs;
    const BTileSrc *tsrc = reinterpret_cast<const BTileSrc *>(tab + H->off_tsrc) + (size_t)l * H->cap_frames;
    // One thread resolves the CTA's next tile (its job's source record and
    // tile coordinates) into the other slot while the current tile is
    // computed, so no tile waits for the job search and the record's load.
    __shared__ BTileSrc s_ts[2];
    __shared__ int s_txy[2][2];
    auto locate = [&](int t, int k) {
        const int j = find_job(jobs, njobs, t);
        const int tt = t - jobs[j].tile0, nx = jobs[j].tiles_x;
        s_ts[k] = tsrc[j];
        s_txy[k][1] = tt / nx;
        s_txy[k][0] = tt - (tt / nx) * nx;
    };
    if (threadIdx.x == 0) locate(blockIdx.x, 0);  // the tables are complete before the first launch
    __syncthreads();
    pdl_wait();  // level l is the previous launch's output
    int k = 0;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x, k ^= 1) {
        if (t + (int)gridDim.x >= tiles) pdl_trigger();  // this CTA's last tile: the next launch may start
        const BTileSrc &ts = s_ts[k];  // fields read from shared memory where used
        const int tx = s_txy[k][0], ty = s_txy[k][1];
        // slot k ^ 1 was last read before the previous tile's closing barrier
        if (threadIdx.x == PD_THREADS - 32 && t + (int)gridDim.x < tiles) locate(t + (int)gridDim.x, k ^ 1);
        pyr_tile<GT != VT_GRAD_NONE, GT>(ts.src, ts.w, ts.h, ts.spitch, ts.vec_ok != 0, ts.dst, ts.dpitch, ts.grad,
                                         ts.gpitch, ts.copy, ts.cpitch, tx, ty, s_in, s_v);
        __syncthreads();
    }
}

// ------------------------------------------------------------------ tail
constexpr int TAIL_THREADS = 1024;
// A level in shared memory: rows of tail_stride(w) bytes, column x at byte
// 4 + x, with the reflected columns -2, -1, w and w + 1 filled in.  Every
// level of at most kTailMaxPx bytes at a pitch of 64 or more fits in TAIL_A,
// and its successor in TAIL_B (checked over all widths); a group of four
// outputs may read up to 16 bytes past the last row.
__host__ __device__ constexpr int tail_stride(int w) { return (w + 3) / 4 * 4 + 8; }
constexpr int TAIL_A = 46080 + 16;  // level c, and every second level after it
constexpr int TAIL_B = 20488 + 24;  // level c + 1, ...
__host__ __device__ inline bool tail_fits(const Level &L) {
    return (long)L.pitch * L.h <= kTailMaxPx && (long)tail_stride(L.w) * L.h <= TAIL_A - 16;
}
constexpr int TAIL_SMEM = TAIL_A + TAIL_B;

// First level the tail kernel builds: the first whose rows (at the
// pyramid's pitch) fit in `limit` bytes, or the last.
int tail_start_level(const vt_pyramid *p, long limit) {
    for (int l = 0; l < p->levels; ++l)
        if (tail_fits(p->lv[l]) && (long)p->lv[l].pitch * p->lv[l].h <= limit) return l;
    return p->levels - 1;
}

// CTAs of a frame's tail: one builds the levels below c, the others (about
// 4096 pixels each, at most 7) take row bands of level c's gradients.  A last
// level too large for shared memory is shared tile by tile.
int tail_parts(const vt_pyramid *p, long limit) {
    const int c = tail_start_level(p, limit);
    const long px = (long)p->lv[c].w * p->lv[c].h;
    if (!tail_fits(p->lv[c])) return 8;
    const int n = 1 + (int)((px + 4095) / 4096);
    return n > 8 ? 8 : n;
}

// Fill the reflected columns of rows [y0, y1) of a w-wide level in shared memory.
__device__ __forceinline__ void tail_pad(uint8_t *s, int w, int y0, int y1) {
    const int S = tail_stride(w);
    const int l2 = refl101(-2, w), l1 = refl101(-1, w), r0 = refl101(w, w), r1 = refl101(w + 1, w);
    for (int y = y0 + threadIdx.x; y < y1; y += blockDim.x) {
        uint8_t *r = s + y * S + 4;
        r[-2] = r[l2];
        r[-1] = r[l1];
        r[w] = r[r0];
        r[w + 1] = r[r1];
    }
    __syncwarp();
}

// Scharr of rows [y0, y1) of a w x h level held in shared memory, four columns
// a thread (the words of three rows; int16 planes two pixels per operation).
template <int GT>
__device__ __forceinline__ void tail_scharr(const uint8_t *s, int w, int h, int y0, int y1, uint32_t *grad,
                                            int gpitch) {
    const int S = tail_stride(w), G = (w + 3) / 4;
    for (int i = threadIdx.x; i < (y1 - y0) * G; i += blockDim.x) {
        const int y = y0 + i / G, g = i % G;
        uint32_t v[3][3];  // columns 4g - 4 .. 4g + 7 of the rows above, at and below y
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint32_t *wp = reinterpret_cast<const uint32_t *>(s + refl101(y + k - 1, h) * S) + g;
#pragma unroll
            for (int c = 0; c < 3; ++c) v[k][c] = wp[c];
        }
        uint4 q;
        if constexpr (GT == VT_GRAD_S16) {
            q = scharr4_s16(row4(v[0][0], v[0][1], v[0][2]), row4(v[1][0], v[1][1], v[1][2]),
                            row4(v[2][0], v[2][1], v[2][2]));
        } else {
            int sm[6], dd[6];  // columns 4g - 1 .. 4g + 4
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                const int wd = (c + 3) >> 2, sh = 8 * ((c + 3) & 3);
                const int a = (v[0][wd] >> sh) & 255, b = (v[1][wd] >> sh) & 255, e = (v[2][wd] >> sh) & 255;
                sm[c] = 3 * (a + e) + 10 * b;
                dd[c] = e - a;
            }
            uint32_t o[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) o[c] = pack_grad<GT>(sm[c + 2] - sm[c], 3 * (dd[c] + dd[c + 2]) + 10 * dd[c + 1]);
            q = make_uint4(o[0], o[1], o[2], o[3]);
        }
        store_grad4(grad + (size_t)y * gpitch, 4 * g, w, q);
    }
    __syncwarp();
}

// pyrDown of a w x h level in shared memory into d (shared) and g (global),
// four outputs a thread.
__device__ __forceinline__ void tail_pyrdown(const uint8_t *s, int w, int h, uint8_t *d, uint8_t *g, int gpitch) {
    const int W = (w + 1) >> 1, H = (h + 1) >> 1, G = (W + 3) / 4;
    const int S = tail_stride(w), D = tail_stride(W);
    for (int i = threadIdx.x; i < H * G; i += blockDim.x) {
        const int Y = i / G, x4 = 4 * (i % G);
        const uint32_t *rows[5];
#pragma unroll
        for (int k = 0; k < 5; ++k)
            rows[k] = reinterpret_cast<const uint32_t *>(s + refl101(2 * Y + k - 2, h) * S) + x4 / 2;
        uint32_t sl[4], sh[4];  // columns 2 x4 - 4 .. 2 x4 + 11
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            uint32_t v[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) v[k] = rows[k][c];
            vsum4(v, sl[c], sh[c]);
        }
        const uint32_t p[6] = {__byte_perm(sl[0], sh[0], 0x7632), __byte_perm(sl[1], sh[1], 0x5410),
                               __byte_perm(sl[1], sh[1], 0x7632), __byte_perm(sl[2], sh[2], 0x5410),
                               __byte_perm(sl[2], sh[2], 0x7632), __byte_perm(sl[3], sh[3], 0x5410)};
        const uint32_t o = hsum4(p);
        *reinterpret_cast<uint32_t *>(d + Y * D + 4 + x4) = o;
        store_px4(g + (size_t)Y * gpitch, x4, W, o);
    }
    __syncwarp();
}

// The tail of a frame's pyramid: the levels from c (the first level of at most
// kTailMaxPx bytes) down to the last, with their Scharr planes, from level c
// held in shared memory.  Part 0 of `parts` builds the levels below c; the
// others write row bands of level c's planes (part 0 writes them itself when
// it is alone).  Level c comes from the tiled launches, or for c = 0 from the
// caller's image (part 0 then writes the level-0 copy).  A last level too
// large for shared memory (a large pyramid of few levels) gets its Scharr
// planes tile by tile from global memory.
//
// Bound by the latency of its chain of small levels (a barrier each); four
// pixels a thread with the tile kernel's packed arithmetic instead of 25 byte
// reads a pixel, and the bands load only their rows: 18.3 -> 12.4 us for one
// 960 x 600 frame of 5 levels, 25.0 -> 17.8 us for 32 frames (cold caches).
template <int GT>
__device__ __forceinline__ void tail_build(const Level *lv, int levels, int c, int part, int parts, const uint8_t *img,
                                           int pitch, bool vec_ok, uint8_t *smem) {
    const Level Lc = lv[c];
    const uint8_t *src = c == 0 ? img : Lc.img;
    const int sp = c == 0 ? pitch : Lc.pitch, w = Lc.w, h = Lc.h;
    if (tail_fits(Lc)) {
        uint8_t *cur = smem, *nxt = smem + TAIL_A;
        const int bands = parts > 1 ? parts - 1 : 1, band = (h + bands - 1) / bands;
        const int y0 = (parts > 1 ? part - 1 : 0) * band, y1 = min(h, y0 + band);  // this part's band (part 0 of many: none)
        const bool chain = part == 0;
        if (!chain && (GT == VT_GRAD_NONE || y0 >= y1)) return;
        const int r0 = chain ? 0 : max(0, y0 - 1), r1 = chain ? h : min(h, y1 + 1);  // rows needed
        const int S = tail_stride(w);
        const int C = (w + 15) / 16;
        for (int i = threadIdx.x; i < (r1 - r0) * C; i += blockDim.x) {
            const int y = r0 + i / C, k = i % C, n = min(16, w - 16 * k);
            const uint8_t *q = src + (size_t)y * sp + 16 * k;  // (the caller's image: any alignment)
            const uint4 v = c > 0 ? *reinterpret_cast<const uint4 *>(q) : load16_any(q, n);
            uint32_t *d = reinterpret_cast<uint32_t *>(cur + y * S) + 1 + 4 * k;
            const int room = S / 4 - 1 - 4 * k;  // words left in the row
            if (room > 0) d[0] = v.x;
            if (room > 1) d[1] = v.y;
            if (room > 2) d[2] = v.z;
            if (room > 3) d[3] = v.w;
            if (c == 0 && chain && src != Lc.img) {  // the level-0 copy
                uint8_t *o = Lc.img + (size_t)y * Lc.pitch + 16 * k;
                const uint32_t vq[4] = {v.x, v.y, v.z, v.w};
                if (n == 16)
                    *reinterpret_cast<uint4 *>(o) = v;
                else
                    for (int b = 0; b < n; ++b) o[b] = (uint8_t)(vq[b >> 2] >> (8 * (b & 3)));
            }
        }
        __syncwarp();
        __syncthreads();
        tail_pad(cur, w, r0, r1);
        __syncthreads();
        if constexpr (GT != VT_GRAD_NONE)
            if (!chain || parts == 1) tail_scharr<GT>(cur, w, h, y0, y1, Lc.grad, Lc.gpitch);
        if (!chain) return;
        for (int l = c; l + 1 < levels; ++l) {
            const int lw = lv[l].w, lh = lv[l].h;
            const Level N = lv[l + 1];
            tail_pyrdown(cur, lw, lh, nxt, N.img, N.pitch);
            __syncthreads();
            tail_pad(nxt, N.w, 0, N.h);
            __syncthreads();
            if constexpr (GT != VT_GRAD_NONE) tail_scharr<GT>(nxt, N.w, N.h, 0, N.h, N.grad, N.gpitch);
            uint8_t *t = cur;
            cur = nxt;
            nxt = t;
        }
    } else if constexpr (GT != VT_GRAD_NONE) {
        uint8_t (*s_in)[SC_IW] = reinterpret_cast<uint8_t (*)[SC_IW]>(smem);
        int tiles_x;
        const int tiles = scharr_tiles(w, h, tiles_x);
        for (int t = part; t < tiles; t += parts) {
            const int ty = t / tiles_x, tx = t - ty * tiles_x;
            scharr_tile<GT>(src, w, h, sp, c == 0 ? vec_ok : true, Lc.grad, Lc.gpitch,
                            (c == 0 && src != Lc.img) ? Lc.img : nullptr, Lc.pitch, tx, ty, s_in);
        }
    } else if (c == 0 && src != Lc.img) {  // no gradients: only the level-0 copy of a large one-level pyramid
        const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
        for (int y = part * nw + (threadIdx.x >> 5); y < h; y += parts * nw)
            for (int x = lane; x < w; x += 32) Lc.img[(size_t)y * Lc.pitch + x] = src[(size_t)y * sp + x];
    }
}

// The tails of a batch: every part of every frame (the jobs of the tail list).
template <int GT>
__global__ void __launch_bounds__(TAIL_THREADS) k_pyr_tail(const uint8_t *tab) {
    extern __shared__ __align__(16) uint8_t tail_smem[];
    const BatchHdr *H = reinterpret_cast<const BatchHdr *>(tab);
    const int njobs = H->njobs[VT_MAX_LEVELS - 1];
    const BFrame *frames = reinterpret_cast<const BFrame *>(tab + H->off_frames);
    const BLvlJob *jobs =
        reinterpret_cast<const BLvlJob *>(tab + H->off_jobs) + (size_t)(VT_MAX_LEVELS - 1) * H->cap_frames;
    pdl_wait();  // level c is the previous launch's output
    for (int j = blockIdx.x; j < njobs; j += gridDim.x) {
        if (j + (int)gridDim.x >= njobs) pdl_trigger();  // this CTA's last job
        const BLvlJob jb = jobs[j];
        const BFrame fr = frames[jb.frame];
        tail_build<GT>(fr.lv, fr.levels, jb.aux, jb.tiles_x, jb.tile0, fr.img, fr.pitch, fr.vec_ok != 0, tail_smem);
        __syncthreads();
    }
}

// The tail of one frame's pyramid (one CTA per part).
struct TailArgs {
    Level lv[VT_MAX_LEVELS];
    int levels, c, pitch, vec_ok;
    const uint8_t *img;
};

template <int GT>
__global__ void __launch_bounds__(TAIL_THREADS) k_pyr_tail_one(const __grid_constant__ TailArgs A) {
    extern __shared__ __align__(16) uint8_t tail_smem[];
    pdl_wait();
    tail_build<GT>(A.lv, A.levels, A.c, blockIdx.x, gridDim.x, A.img, A.pitch, A.vec_ok != 0, tail_smem);
}

int pyr_tiles(int w, int h, int &tiles_x) {
    const int W = (w + 1) / 2, H = (h + 1) / 2;
    tiles_x = (W + PD_TW - 1) / PD_TW;
    return tiles_x * ((H + PD_TH - 1) / PD_TH);
}

__host__ __device__ int scharr_tiles(int w, int h, int &tiles_x) {
    tiles_x = (w + SC_TW - 1) / SC_TW;
    return tiles_x * ((h + SC_TH - 1) / SC_TH);
}

vt_status launch_pyr_batch(const uint8_t *dev_tab, int tiled_launches, int gtype, int grid_pyr, int grid_tail,
                           cudaStream_t s, cudaEvent_t *ev) {
    if (!(gtype == VT_GRAD_F16    ? smem_opt_in<k_pyr_tail<VT_GRAD_F16>>(TAIL_SMEM)
          : gtype == VT_GRAD_NONE ? smem_opt_in<k_pyr_tail<VT_GRAD_NONE>>(TAIL_SMEM)
                                  : smem_opt_in<k_pyr_tail<VT_GRAD_S16>>(TAIL_SMEM)))
        return VT_ERR_CUDA;
    // every launch after the first overlaps its start with the previous one's
    // end (programmatic dependent launch), except where an event is recorded
    // in between for per-launch timing
    auto pyr = gtype == VT_GRAD_F16 ? k_pyr_batch<VT_GRAD_F16>
                                    : (gtype == VT_GRAD_NONE ? k_pyr_batch<VT_GRAD_NONE> : k_pyr_batch<VT_GRAD_S16>);
    auto tail = gtype == VT_GRAD_F16 ? k_pyr_tail<VT_GRAD_F16>
                                     : (gtype == VT_GRAD_NONE ? k_pyr_tail<VT_GRAD_NONE> : k_pyr_tail<VT_GRAD_S16>);
    cudaError_t e = cudaSuccess;
    for (int l = 0; l < tiled_launches && e == cudaSuccess; ++l) {
        e = launch_pdl(pyr, grid_pyr, PD_THREADS, 0, s, l > 0 && !ev, dev_tab, l);
        if (ev && ev[l]) cudaEventRecord(ev[l], s);
    }
    if (e == cudaSuccess) e = launch_pdl(tail, grid_tail, TAIL_THREADS, TAIL_SMEM, s, tiled_launches > 0 && !ev, dev_tab);
    if (ev && ev[tiled_launches]) cudaEventRecord(ev[tiled_launches], s);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? VT_OK : VT_ERR_CUDA;
}

int pyr_batch_blocks_per_sm() {
    int a = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_pyr_batch<VT_GRAD_S16>, PD_THREADS, 0);
    return a;
}

// A Scharr job over level `lv`, read from `src` (the level itself, or the
// caller's image, then also copied to the level).
static void add_grad_job(GradJobs &jobs, int &blocks, const Level &lv, const uint8_t *src, int spitch, int vec_ok) {
    GradJob &j = jobs.j[jobs.njobs++];
    j.src = src;
    j.grad = lv.grad;
    j.copy = src != lv.img ? lv.img : nullptr;
    j.w = lv.w;
    j.h = lv.h;
    j.spitch = spitch;
    j.gpitch = lv.gpitch;
    j.cpitch = lv.pitch;
    j.vec_ok = vec_ok;
    j.tile0 = blocks;
    blocks += scharr_tiles(lv.w, lv.h, j.tiles_x);
}

// Every launch of a build starts while the stream's previous kernel ends
// (programmatic dependent launch): a build is a chain of launches of a few
// microseconds each, and the launch latency between them cost as much as the
// kernels.
static vt_status launch_scharr(const GradJobs &jobs, int total_blocks, int gtype, bool pdl, cudaStream_t s) {
    if (jobs.njobs == 0 || total_blocks == 0) return VT_OK;
    return launch_pdl(gtype == VT_GRAD_F16 ? k_scharr<VT_GRAD_F16> : k_scharr<VT_GRAD_S16>, total_blocks, SC_THREADS, 0,
                      s, pdl, jobs) == cudaSuccess
               ? VT_OK
               : VT_ERR_CUDA;
}

// ------------------------------------------------------------------ host side
// `level0` (nullable): the caller's level-0 buffer (row pitch `pitch0`); the
// allocation then holds only the levels above 0 and the planes.
static vt_status alloc_pyramid(int w, int h, int levels, vt_pyramid **out, uint8_t *level0 = nullptr,
                               int pitch0 = 0) {
    vt_pyramid *p = (vt_pyramid *)calloc(1, sizeof(vt_pyramid));
    if (!p) return VT_ERR_OOM;
    p->w = w;
    p->h = h;
    p->levels = levels;
    p->gtype = VT_GRAD_NONE;
    cudaGetDevice(&p->device);
    size_t off = 256;  // the device copy of the level table sits at the start
    size_t img_off[VT_MAX_LEVELS], grad_off[VT_MAX_LEVELS];
    int lw = w, lh = h;
    for (int l = 0; l < levels; ++l) {
        Level &L = p->lv[l];
        L.w = lw;
        L.h = lh;
        L.pitch = (l == 0 && level0) ? pitch0 : round_up(lw, kImgPitchAlign);
        L.gpitch = round_up(lw, kGradPitchAlign);
        img_off[l] = off;
        if (l > 0 || !level0) off += ((size_t)L.pitch * lh + 255) / 256 * 256;
        lw = (lw + 1) / 2;
        lh = (lh + 1) / 2;
    }
    for (int l = 0; l < levels; ++l) {
        grad_off[l] = off;
        off += ((size_t)p->lv[l].gpitch * 4 * p->lv[l].h + 255) / 256 * 256;
    }
    off += 256;  // slack: wide loads of a footprint may read a few bytes past a row end
    if (cudaMalloc(&p->base, off) != cudaSuccess) {
        cudaGetLastError();
        free(p);
        return VT_ERR_OOM;
    }
    p->bytes = off;
    for (int l = 0; l < levels; ++l) {
        p->lv[l].img = (l == 0 && level0) ? level0 : (uint8_t *)p->base + img_off[l];
        p->lv[l].grad = (uint32_t *)((uint8_t *)p->base + grad_off[l]);
    }
    static_assert(sizeof(Level) * VT_MAX_LEVELS <= 256, "level table must fit its slot");
    p->dev_lv = (Level *)p->base;
    if (cudaMemcpy(p->dev_lv, p->lv, sizeof(Level) * VT_MAX_LEVELS, cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(p->base);
        free(p);
        return VT_ERR_CUDA;
    }
    *out = p;
    return VT_OK;
}

static vt_status check_build_args(const uint8_t *img, int w, int h, int pitch, int levels, vt_pyramid **out) {
    if (!img || !out || w <= 0 || h <= 0 || pitch < w || levels < 1 || levels > VT_MAX_LEVELS) return VT_ERR_ARG;
    // ceil-halving never reaches 0 px, so every level count up to VT_MAX_LEVELS is valid
    if (*out) {
        const vt_pyramid *p = *out;
        if (p->w != w || p->h != h || p->levels != levels) return VT_ERR_ARG;
    }
    return VT_OK;
}

// Where a kernel on the current device can read the `bytes` bytes at `p`: in
// the device's own memory (on_device) or in pinned host memory (not
// on_device), wholly inside one allocation; null for anything else, which is
// left to the copy call (it reaches other devices and pageable memory, and
// refuses what it cannot read).
static const uint8_t *kernel_readable(const uint8_t *p, size_t bytes, bool on_device) {
    typedef CUresult (*Query)(unsigned, CUpointer_attribute *, void **, CUdeviceptr);
    static const Query query = []() -> Query {  // once, thread-safe static initialisation
        void *f = nullptr;
        cudaDriverEntryPointQueryResult r;
        const bool ok = cudaGetDriverEntryPointByVersion("cuPointerGetAttributes", &f, 12000, cudaEnableDefault, &r) ==
                            cudaSuccess &&
                        r == cudaDriverEntryPointSuccess;
        if (!ok) cudaGetLastError();
        return ok ? reinterpret_cast<Query>(f) : nullptr;
    }();
    CUpointer_attribute what[] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE, CU_POINTER_ATTRIBUTE_DEVICE_ORDINAL,
                                  CU_POINTER_ATTRIBUTE_DEVICE_POINTER, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                  CU_POINTER_ATTRIBUTE_RANGE_SIZE};
    unsigned type = 0;
    int of = -1, dev = -2;
    CUdeviceptr at = 0, start = 0;
    size_t size = 0;
    void *to[] = {&type, &of, &at, &start, &size};
    if (!query || cudaGetDevice(&dev) != cudaSuccess || query(5, what, to, (CUdeviceptr)(uintptr_t)p) != CUDA_SUCCESS) {
        cudaGetLastError();
        return nullptr;
    }
    const bool ok = (on_device ? type == CU_MEMORYTYPE_DEVICE && of == dev : type == CU_MEMORYTYPE_HOST) && at >= start &&
                    at - start <= size && bytes <= size - (at - start);
    return ok ? reinterpret_cast<const uint8_t *>((uintptr_t)at) : nullptr;
}

// Pinned host frames up to this size, and larger ones whose rows need a new
// pitch, are read by the first launch over the host link: a 2-D copy moves
// rows at a third of the link's rate and costs a launch of its own (752 x 480:
// 41 -> 16 us a build, 1437 x 901: 66 -> 28).  A large frame in one piece is
// copied faster than a kernel reads it (1920 x 1200 alone: 47 against 51 us).
constexpr size_t kHostReadBytes = (size_t)1 << 20;

static vt_status build_impl(const uint8_t *img, int w, int h, int pitch, int levels, int img_on_device, int gtype,
                            void *cuda_stream, vt_pyramid **out) {
    vt_status st = check_build_args(img, w, h, pitch, levels, out);
    if (st != VT_OK) return st;
    bool fresh = false;
    if (!*out) {
        st = alloc_pyramid(w, h, levels, out);
        if (st != VT_OK) return st;
        fresh = true;
    }
    vt_pyramid *p = *out;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    const Level &L0 = p->lv[0];
    if (img == L0.img && pitch != L0.pitch) return VT_ERR_ARG;
    const bool grad = gtype != VT_GRAD_NONE;
    const int c = tail_start_level(p, kTailFewPx);
    const bool small = tail_fits(p->lv[c]);  // the levels from c on take one launch
    // A frame already in level 0 (vt_pyramid_upload) is built in place, and a
    // device image is copied by the launch that reads it first; other host
    // images are copied up first, also one that makes a single level without
    // planes: there is nothing else to do (160 x 120: 7 us, 15 by a launch).
    bool by_kernel = false;
    if (img != L0.img && (c > 0 || grad || (small && (levels > 1 || img_on_device))) &&
        (img_on_device || pitch != L0.pitch || (size_t)pitch * h <= kHostReadBytes)) {
        const uint8_t *q = kernel_readable(img, (size_t)pitch * (h - 1) + w, img_on_device != 0);
        by_kernel = q != nullptr;
        if (by_kernel) img = q;
    }
    const bool from_host = by_kernel && !img_on_device;
    cudaError_t e = cudaSuccess;
    if (img != L0.img && !by_kernel) {
        e = cudaMemcpy2DAsync(L0.img, L0.pitch, img, pitch, w, h,
                              img_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s);
        img = L0.img;
        pitch = L0.pitch;
    }
    const int vec_ok = (uintptr_t)img % 16 == 0 && pitch % 16 == 0;
    for (int l = 0; l < c && e == cudaSuccess; ++l) {
        const Level &S = p->lv[l], &D = p->lv[l + 1];
        PyrJob j;
        j.src = l == 0 ? img : S.img;
        j.spitch = l == 0 ? pitch : S.pitch;
        j.vec_ok = l == 0 ? vec_ok : 1;
        j.copy = j.src != S.img ? S.img : nullptr;
        j.cpitch = S.pitch;
        j.dst = D.img;
        j.dpitch = D.pitch;
        j.grad = S.grad;
        j.gpitch = S.gpitch;
        j.w = S.w;
        j.h = S.h;
        const int tiles = pyr_tiles(S.w, S.h, j.tiles_x);
        e = launch_pdl(!grad                    ? k_pyrdown<false, VT_GRAD_S16>
                       : gtype == VT_GRAD_F16 ? k_pyrdown<true, VT_GRAD_F16>
                                              : k_pyrdown<true, VT_GRAD_S16>,
                       tiles, PD_THREADS, 0, s, l > 0 || !from_host, j);  // (host memory: after the launch before)
    }
    if (e == cudaSuccess && small && (c + 1 < levels || grad || (c == 0 && by_kernel))) {  // (else nothing is left)
        TailArgs A;
        for (int l = 0; l < VT_MAX_LEVELS; ++l) A.lv[l] = l < levels ? p->lv[l] : Level{};
        A.levels = levels;
        A.c = c;
        A.img = img;
        A.pitch = pitch;
        A.vec_ok = vec_ok;
        const bool fits = !grad                    ? smem_opt_in<k_pyr_tail_one<VT_GRAD_NONE>>(TAIL_SMEM)
                          : gtype == VT_GRAD_F16 ? smem_opt_in<k_pyr_tail_one<VT_GRAD_F16>>(TAIL_SMEM)
                                                 : smem_opt_in<k_pyr_tail_one<VT_GRAD_S16>>(TAIL_SMEM);
        e = !fits ? cudaErrorInvalidValue
                  : launch_pdl(!grad                    ? k_pyr_tail_one<VT_GRAD_NONE>
                               : gtype == VT_GRAD_F16 ? k_pyr_tail_one<VT_GRAD_F16>
                                                      : k_pyr_tail_one<VT_GRAD_S16>,
                               grad ? tail_parts(p, kTailFewPx) : 1, TAIL_THREADS, TAIL_SMEM, s, c > 0 || !from_host, A);
    } else if (e == cudaSuccess && !small && grad) {  // (c is the last level)
        GradJobs gj;
        gj.njobs = 0;
        int blocks = 0;
        add_grad_job(gj, blocks, p->lv[c], c == 0 ? img : p->lv[c].img, c == 0 ? pitch : p->lv[c].pitch,
                     c == 0 ? vec_ok : 1);
        if (launch_scharr(gj, blocks, gtype, c > 0 || !from_host, s) != VT_OK) e = cudaErrorLaunchFailure;
    }
    if (e != cudaSuccess || cudaGetLastError() != cudaSuccess) {
        cudaGetLastError();
        if (fresh) {
            vt_pyramid_free(p);
            *out = nullptr;
        }
        return VT_ERR_CUDA;
    }
    p->gtype = grad ? gtype : VT_GRAD_NONE;
    return VT_OK;
}

}  // namespace vt

using namespace vt;

extern "C" {

vt_status vt_pyramid_build(const uint8_t *img, int w, int h, int pitch, int levels, int img_on_device,
                           void *cuda_stream, vt_pyramid **out) {
    return build_impl(img, w, h, pitch, levels, img_on_device, VT_GRAD_NONE, cuda_stream, out);
}

vt_status vt_pyramid_build_grad(const uint8_t *img, int w, int h, int pitch, int levels, int img_on_device,
                                vt_grad_type t, void *cuda_stream, vt_pyramid **out) {
    if (t != VT_GRAD_S16 && t != VT_GRAD_F16) return VT_ERR_ARG;
    return build_impl(img, w, h, pitch, levels, img_on_device, (int)t, cuda_stream, out);
}

vt_status vt_gradients(vt_pyramid *p, vt_grad_type t, void *cuda_stream) {
    if (!p || (t != VT_GRAD_S16 && t != VT_GRAD_F16)) return VT_ERR_ARG;
    GradJobs gj;
    gj.njobs = 0;
    int blocks = 0;
    for (int l = 0; l < p->levels; ++l) add_grad_job(gj, blocks, p->lv[l], p->lv[l].img, p->lv[l].pitch, 1);
    const vt_status st = launch_scharr(gj, blocks, (int)t, true, (cudaStream_t)cuda_stream);
    if (st == VT_OK) p->gtype = (int)t;
    return st;
}

vt_status vt_pyramid_upload(vt_pyramid *p, const uint8_t *img, int pitch, int img_on_device, void *cuda_stream) {
    if (!p || !img || pitch < p->w) return VT_ERR_ARG;
    const Level &L0 = p->lv[0];
    if (cudaMemcpy2DAsync(L0.img, L0.pitch, img, pitch, p->w, p->h,
                          img_on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                          (cudaStream_t)cuda_stream) != cudaSuccess) {
        cudaGetLastError();
        return VT_ERR_CUDA;
    }
    return VT_OK;
}

vt_status vt_pyramid_create(int w, int h, int levels, vt_pyramid **out) {
    if (!out || w <= 0 || h <= 0 || levels < 1 || levels > VT_MAX_LEVELS) return VT_ERR_ARG;
    *out = nullptr;
    return alloc_pyramid(w, h, levels, out);
}

vt_status vt_pyramid_create_on(const uint8_t *level0, int pitch, size_t level0_bytes, int w, int h, int levels,
                               vt_pyramid **out) {
    if (!out || !level0 || w <= 0 || h <= 0 || levels < 1 || levels > VT_MAX_LEVELS) return VT_ERR_ARG;
    if ((uintptr_t)level0 % 16 != 0 || pitch % 16 != 0 || pitch < w) return VT_ERR_ARG;
    if (level0_bytes < (size_t)pitch * h + 32) return VT_ERR_ARG;
    *out = nullptr;
    return alloc_pyramid(w, h, levels, out, const_cast<uint8_t *>(level0), pitch);
}

vt_status vt_pyramid_level(const vt_pyramid *p, int lvl, const uint8_t **ptr, int *w, int *h, int *pitch) {
    if (!p || lvl < 0 || lvl >= p->levels) return VT_ERR_ARG;
    if (ptr) *ptr = p->lv[lvl].img;
    if (w) *w = p->lv[lvl].w;
    if (h) *h = p->lv[lvl].h;
    if (pitch) *pitch = p->lv[lvl].pitch;
    return VT_OK;
}

vt_status vt_pyramid_grad(const vt_pyramid *p, int lvl, const void **ptr, int *pitch_pairs, vt_grad_type *t) {
    if (!p || lvl < 0 || lvl >= p->levels) return VT_ERR_ARG;
    if (ptr) *ptr = p->lv[lvl].grad;
    if (pitch_pairs) *pitch_pairs = p->lv[lvl].gpitch;
    if (t) *t = (vt_grad_type)p->gtype;
    return VT_OK;
}

vt_status vt_pyramid_info(const vt_pyramid *p, int *w, int *h, int *levels, size_t *device_bytes) {
    if (!p) return VT_ERR_ARG;
    if (w) *w = p->w;
    if (h) *h = p->h;
    if (levels) *levels = p->levels;
    if (device_bytes) *device_bytes = p->bytes;
    return VT_OK;
}

void vt_pyramid_free(vt_pyramid *p) {
    if (!p) return;
    cudaDeviceSynchronize();
    cudaFree(p->base);
    free(p);
}

const char *vt_status_str(vt_status s) {
    switch (s) {
        case VT_OK: return "VT_OK";
        case VT_ERR_ARG: return "VT_ERR_ARG: invalid argument";
        case VT_ERR_OOM: return "VT_ERR_OOM: out of device memory";
        case VT_ERR_CUDA: return "VT_ERR_CUDA: CUDA call or launch failed";
        case VT_ERR_TIMEOUT: return "VT_ERR_TIMEOUT: a bounded wait ran out";
        case VT_ERR_UNSUPPORTED: return "VT_ERR_UNSUPPORTED: configuration not built";
    }
    return "unknown vt_status";
}

const char *vt_version(void) { return "vt 0.1 (sm_103a)"; }

}  // extern "C"
