// Stereo triangulation gate (K7): the per-point geometric check of stereo
// correspondences (Sec. III-C: negligible-disparity matches are dropped, the
// rest triangulated with the rig's extrinsics and kept only with a positive
// depth inside a valid range and at most 1.5 px of reprojection error in
// both views).  One thread per correspondence; decisions and points are FP64's
// (the eigenvectors are found in FP32 and refined, see gate_fast):
//
//   disparity  |p_R - pi_R(R K_L^-1 p_L)| (image of the left ray's point at
//              infinity in the right view; infinite when it lies behind the
//              right camera), kept when > min_disp;
//   DLT        the homogeneous point is the eigenvector of the smallest
//              eigenvalue of A^T A, A = [x_L P_L^3 - P_L^1; y_L P_L^3 - P_L^2;
//              x_R P_R^3 - P_R^1; y_R P_R^3 - P_R^2] on normalised
//              coordinates, P_L = [I | 0], P_R = [R | t]; cyclic Jacobi
//              rotations on the 4x4 (at most kJacobiSweeps sweeps);
//   depth      X_4 != 0, Z_R > 0, z_min <= Z_L <= z_max;
//   reprojection  both views' pixel errors <= max_reproj.
#include <cmath>
#include <cstdint>

#include "vt_internal.cuh"

namespace vt {

constexpr int kJacobiSweeps = 12;

// Rigs with a shorter translation go to the FP64 route alone: the spectrum's gap
// shrinks with its square (at 0.016 to 5e-5 of the largest eigenvalue, where half
// of the pairs are left to that route anyway).
constexpr double kGateMinT = 0.015625;

struct GateArgs {
    vt_stereo_rig rig;
    vt_gate_params prm;
    GateScale k;
};

// The constants of a rig that the fast route uses.
GateScale gate_scale(const vt_stereo_rig &rig) {
    GateScale k;
    k.ikl[0] = 1.0 / rig.kl[0], k.ikl[1] = 1.0 / rig.kl[1];
    k.ikr[0] = 1.0 / rig.kr[0], k.ikr[1] = 1.0 / rig.kr[1];
    const double t = std::fmax(std::fabs(rig.t[0]), std::fmax(std::fabs(rig.t[1]), std::fabs(rig.t[2])));
    k.unit = t >= 2.0 ? std::ldexp(1.0, std::ilogb(t)) : 1.0;
    k.beta = 1.0 / k.unit / k.unit;
    for (int i = 0; i < 3; ++i) k.t[i] = rig.t[i] / k.unit;
    double r = 1.0, f = 0.0, c = 0.0;
    for (int i = 0; i < 3; ++i)
        r = std::fmax(r, std::fabs(rig.R[3 * i]) + std::fabs(rig.R[3 * i + 1]) + std::fabs(rig.R[3 * i + 2]));
    for (int i = 0; i < 2; ++i) {
        f = std::fmax(f, std::fmax(std::fabs(rig.kl[i]), std::fabs(rig.kr[i])));
        c = std::fmax(c, std::fmax(std::fabs(rig.kl[2 + i]), std::fabs(rig.kr[2 + i])));
    }
    k.rows = (float)r;
    k.px = (float)(f + c);
    k.fast = t >= kGateMinT;
    return k;
}

// One Jacobi rotation in the (P, Q) plane of the symmetric M (upper
// triangle M[i][j], i < j, and the diagonal are kept), accumulating V.
//
// GB300 issues FP64 at a small fraction of its FP32 rate, so the angle is
// found in FP32 (tan t, the smaller root of t^2 + 2 tau t - 1 = 0,
// tau = (M_QQ - M_PP) / 2 M_PQ) and only made exactly orthogonal in FP64:
// c = 1 / sqrt(1 + t^2) by two Newton steps from the FP32 estimate, s = t c,
// so c^2 + s^2 = 1 to FP64 rounding.  An approximate angle leaves a small
// M_PQ behind for the next sweep; the update itself is the full similarity
// J^T M J in FP64, so the eigenvectors keep FP64 accuracy.
template <int P, int Q>
__device__ __forceinline__ void jacobi_rotate(double (&M)[4][4], double (&V)[4][4]) {
    const double apq = M[P][Q];
    if (apq == 0.0) return;
    const float tau = (float)(M[Q][Q] - M[P][P]) / (2.0f * (float)apq);
    const float tf = copysignf(1.0f, tau) / (fabsf(tau) + sqrtf(fmaf(tau, tau, 1.0f)));
    if (tf == 0.0f) return;  // |M_PQ| negligible against |M_QQ - M_PP|
    const double t = tf;
    const double x = fma(t, t, 1.0);
    double c = (double)rsqrtf((float)x);
    c = c * fma(-0.5 * x, c * c, 1.5);
    c = c * fma(-0.5 * x, c * c, 1.5);
    const double s = t * c;
    const double cc = c * c, ss = s * s, cs = c * s;
    const double app = M[P][P], aqq = M[Q][Q];
    M[P][P] = fma(cc, app, fma(-2.0 * cs, apq, ss * aqq));
    M[Q][Q] = fma(ss, app, fma(2.0 * cs, apq, cc * aqq));
    M[P][Q] = fma(cc - ss, apq, cs * (app - aqq));
#pragma unroll
    for (int k = 0; k < 4; ++k) {  // the other rows / columns of J^T M J
        if (k == P || k == Q) continue;
        double &mkp = k < P ? M[k][P] : M[P][k];
        double &mkq = k < Q ? M[k][Q] : M[Q][k];
        const double a = mkp, b = mkq;
        mkp = fma(c, a, -s * b);
        mkq = fma(s, a, c * b);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {  // eigenvectors accumulate as columns of V J
        const double a = V[k][P], b = V[k][Q];
        V[k][P] = fma(c, a, -s * b);
        V[k][Q] = fma(s, a, c * b);
    }
}

// Homogeneous point X (4) minimising |A X| / |X|, from the 4 rows of A.
__device__ __forceinline__ void dlt_null_vector(const double (&A)[4][4], double (&X)[4]) {
    double M[4][4], V[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            double s = 0.0;
            if (j >= i) {  // upper triangle only
#pragma unroll
                for (int r = 0; r < 4; ++r) s += A[r][i] * A[r][j];
            }
            M[i][j] = s;
            V[i][j] = i == j ? 1.0 : 0.0;
        }
    for (int sweep = 0; sweep < kJacobiSweeps; ++sweep) {
        const double off = M[0][1] * M[0][1] + M[0][2] * M[0][2] + M[0][3] * M[0][3] + M[1][2] * M[1][2] +
                           M[1][3] * M[1][3] + M[2][3] * M[2][3];
        const double dia = M[0][0] * M[0][0] + M[1][1] * M[1][1] + M[2][2] * M[2][2] + M[3][3] * M[3][3];
        if (off <= 1e-34 * dia) break;
        jacobi_rotate<0, 1>(M, V);
        jacobi_rotate<0, 2>(M, V);
        jacobi_rotate<0, 3>(M, V);
        jacobi_rotate<1, 2>(M, V);
        jacobi_rotate<1, 3>(M, V);
        jacobi_rotate<2, 3>(M, V);
    }
    // column of the smallest eigenvalue (constant indices only: M and V stay in registers)
    double best = M[0][0];
#pragma unroll
    for (int i = 0; i < 4; ++i) X[i] = V[i][0];
#pragma unroll
    for (int j = 1; j < 4; ++j)
        if (M[j][j] < best) {
            best = M[j][j];
#pragma unroll
            for (int i = 0; i < 4; ++i) X[i] = V[i][j];
        }
}

struct GateOut {
    float x, y, z;
    uint8_t status, reason;
};

__device__ __forceinline__ GateOut gate_point(const GateArgs &g, float2 pl, float2 pr, bool tracked) {
    GateOut o{0.f, 0.f, 0.f, 0, VT_LOST_INPUT};
    if (!tracked || !isfinite(pl.x) || !isfinite(pl.y) || !isfinite(pr.x) || !isfinite(pr.y)) return o;
    const double *KL = g.rig.kl, *KR = g.rig.kr, *R = g.rig.R, *T = g.rig.t;
    const double ul = pl.x, vl = pl.y, ur = pr.x, vr = pr.y;
    const double xl = (ul - KL[2]) / KL[0], yl = (vl - KL[3]) / KL[1];
    const double xr = (ur - KR[2]) / KR[0], yr = (vr - KR[3]) / KR[1];
    // disparity against the right image of the left ray's point at infinity
    const double rx = R[0] * xl + R[1] * yl + R[2];
    const double ry = R[3] * xl + R[4] * yl + R[5];
    const double rz = R[6] * xl + R[7] * yl + R[8];
    if (rz > 0.0) {
        const double dx = ur - (KR[0] * rx / rz + KR[2]);
        const double dy = vr - (KR[1] * ry / rz + KR[3]);
        if (!(sqrt(dx * dx + dy * dy) > g.prm.min_disp)) {
            o.reason = VT_LOST_DISP;
            return o;
        }
    }
    // rows x P^3 - P^1 and y P^3 - P^2 of both views
    const double A[4][4] = {{-1.0, 0.0, xl, 0.0},
                            {0.0, -1.0, yl, 0.0},
                            {xr * R[6] - R[0], xr * R[7] - R[1], xr * R[8] - R[2], xr * T[2] - T[0]},
                            {yr * R[6] - R[3], yr * R[7] - R[4], yr * R[8] - R[5], yr * T[2] - T[1]}};
    double Xh[4];
    dlt_null_vector(A, Xh);
    o.reason = VT_LOST_DEPTH;
    if (Xh[3] == 0.0) return o;
    const double X = Xh[0] / Xh[3], Y = Xh[1] / Xh[3], Z = Xh[2] / Xh[3];
    o.x = (float)X;
    o.y = (float)Y;
    o.z = (float)Z;
    const double XR = R[0] * X + R[1] * Y + R[2] * Z + T[0];
    const double YR = R[3] * X + R[4] * Y + R[5] * Z + T[1];
    const double ZR = R[6] * X + R[7] * Y + R[8] * Z + T[2];
    if (!(ZR > 0.0 && Z >= g.prm.z_min && Z <= g.prm.z_max)) return o;
    const double exl = KL[0] * X / Z + KL[2] - ul, eyl = KL[1] * Y / Z + KL[3] - vl;
    const double exr = KR[0] * XR / ZR + KR[2] - ur, eyr = KR[1] * YR / ZR + KR[3] - vr;
    const double el = sqrt(exl * exl + eyl * eyl), er = sqrt(exr * exr + eyr * eyr);
    if (!(fmax(el, er) <= g.prm.max_reproj)) {
        o.reason = VT_LOST_REPROJ;
        return o;
    }
    o.status = 1;
    o.reason = VT_TRACKED;
    return o;
}

// ----------------------------------------------------------------------------
// The same decisions with a tenth of the FP64 instructions.  GB300 retires two
// FP64 lanes per clock and SM against 128 FP32 lanes, and gate_point's four
// FP64 Jacobi sweeps, 13 divides and three square roots are about 2,000 FP64
// instructions a pair.  Here
//   - the eigenvectors of A^T A are found in FP32 (all Jacobi sweeps), and the
//     null vector x is refined against the FP64 rows: the residual
//     r = A^T (A x) - |A x|^2 x in FP64, the correction
//     sum_k -(v_k . r) / (l_k - l_0) v_k from the FP32 eigenpairs.  A step
//     shrinks the error by the relative error of those (about 1e-6 |A|^2 /
//     (l_1 - l_0)); the steps end when the next one, judged by the last two,
//     is below the rounding (`err` below): usually after two;
//   - one reciprocal serves the divisions by the same number, and distances are
//     compared squared.
// The unit that minimises |A x| is the one in the rig's own unit of length, but it
// is sought in coordinates whose last column is scaled by a power of two to the
// translation's size (y_4 = unit x_4, |x|^2 = y_1^2 + y_2^2 + y_3^2 + y_4^2 /
// unit^2): gap and stop then mean the same for a rig in millimetres.  Without it
// the gap shrank with the square of the translation, and from 250 on every pair
// went through both routes (19,000 pairs at 250: 68 us, 13.0 so; 12.1 at 0.11).
//
// The null vector's error is at most `err` = 2e-15 l_3 / (l_1 - l_0) + 1e-15 for
// the rounding of the residual (an FP64 row of four terms is off by 4 2^-53
// |A_i|, the squares of the |A_i| add up to at most 4 l_3, and the gap carries
// that to the vector) and as much again for the refinement's stop; the point's is
// `rel` (unit + |X|), rel = 4 err / |y_4|, a factor of two to spare.  A pair is
// left to gate_point when the refinement has not converged, when the spectrum has
// no gap, when rel passes 1e-7 (points beyond some 1e4 to 1e7 translations), or
// when a decision lies within that error of its threshold (at least 1e-8,
// relative, for depths).  Not-a-numbers fail these tests and go there, too.
// Measured: 19,000 pairs 78 -> 11.8 us, about 6,000 pairs of a batched run 76 ->
// 14.7 us (one warp a CTA spreads them; cold caches); hardly a pair of either is
// left to gate_point.

// One FP32 Jacobi rotation in the (P, Q) plane (see jacobi_rotate).
template <int P, int Q>
__device__ __forceinline__ void jacobi_rotate32(float (&M)[4][4], float (&V)[4][4]) {
    const float apq = M[P][Q];
    const float tau = __fdividef(M[Q][Q] - M[P][P], 2.0f * apq);
    const float h = fmaf(tau, tau, 1.0f);
    float t = __fdividef(copysignf(1.0f, tau), fabsf(tau) + h * rsqrtf(h));
    if (!(fabsf(tau) < 1e9f)) t = 0.0f;  // nothing to rotate (or no number)
    const float c = rsqrtf(fmaf(t, t, 1.0f)), s = t * c;
    M[P][P] = fmaf(-t, apq, M[P][P]);
    M[Q][Q] = fmaf(t, apq, M[Q][Q]);
    M[P][Q] = 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (k == P || k == Q) continue;
        float &mkp = k < P ? M[k][P] : M[P][k];
        float &mkq = k < Q ? M[k][Q] : M[Q][k];
        const float a = mkp, b = mkq;
        mkp = fmaf(c, a, -s * b);
        mkq = fmaf(s, a, c * b);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float a = V[k][P], b = V[k][Q];
        V[k][P] = fmaf(c, a, -s * b);
        V[k][Q] = fmaf(s, a, c * b);
    }
}

// 1 / v to FP64 accuracy, from the FP32 reciprocal `seed` by two Newton steps.
// Beyond FP32's range both are 0: the callers test the seed (kSeedMin).
constexpr float kSeedMin = 1e-30f;
__device__ __forceinline__ double recip(double v, float &seed) {
    seed = __frcp_rn((float)v);
    double r = (double)seed;
    r = fma(r, fma(-v, r, 1.0), r);
    return fma(r, fma(-v, r, 1.0), r);
}

// The null vector of the rows (-1, 0, xl, 0), (0, -1, yl, 0), a and b: the unit
// x that minimises |A x|, or false (see above).
// x: in scaled coordinates (a[3], b[3] scaled; beta = 1 / unit^2); err: its error.
__device__ __forceinline__ bool null_vector_fast(double xl, double yl, const double (&a)[4], const double (&b)[4],
                                                 double beta, double (&x)[4], float &err) {
    constexpr int kSweeps = 4, kSteps = 8;
    float m[4][4], V[4][4];
    {
        const float u = (float)xl, v = (float)yl;
        float fa[4], fb[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) fa[i] = (float)a[i], fb[i] = (float)b[i];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (j >= i) m[i][j] = fmaf(fa[i], fa[j], fb[i] * fb[j]);
                V[i][j] = i == j ? 1.0f : 0.0f;
            }
        m[0][0] += 1.0f, m[1][1] += 1.0f;
        m[0][2] -= u, m[1][2] -= v;
        m[2][2] += fmaf(u, u, v * v);
    }
#pragma unroll 1
    for (int k = 0; k < kSweeps; ++k) {
        jacobi_rotate32<0, 1>(m, V);
        jacobi_rotate32<0, 2>(m, V);
        jacobi_rotate32<0, 3>(m, V);
        jacobi_rotate32<1, 2>(m, V);
        jacobi_rotate32<1, 3>(m, V);
        jacobi_rotate32<2, 3>(m, V);
    }
    float l[4] = {m[0][0], m[1][1], m[2][2], m[3][3]};
#pragma unroll
    for (int j = 1; j < 4; ++j)  // the smallest first
        if (l[j] < l[0]) {
            float t = l[0];
            l[0] = l[j];
            l[j] = t;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                t = V[i][0];
                V[i][0] = V[i][j];
                V[i][j] = t;
            }
        }
    const float top = fmaxf(fmaxf(l[1], l[2]), l[3]), gap = fminf(fminf(l[1], l[2]), l[3]) - l[0];
    if (!(gap > 2e-5f * top)) return false;
    err = fmaf(2e-15f, top / gap, 1e-15f);
    const float w[3] = {1.0f / (l[0] - l[1]), 1.0f / (l[0] - l[2]), 1.0f / (l[0] - l[3])};
    const float n0 = rsqrtf(fmaf(V[0][0], V[0][0], fmaf(V[1][0], V[1][0], fmaf(V[2][0], V[2][0], V[3][0] * V[3][0]))));
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = V[i][0] * n0;
    float last = 1e-2f;  // the step before (a first step as large is no refinement)
#pragma unroll 1
    for (int k = 0; k < kSteps; ++k) {
        const double e0 = fma(xl, x[2], -x[0]), e1 = fma(yl, x[2], -x[1]);
        const double e2 = fma(a[0], x[0], fma(a[1], x[1], fma(a[2], x[2], a[3] * x[3])));
        const double e3 = fma(b[0], x[0], fma(b[1], x[1], fma(b[2], x[2], b[3] * x[3])));
        // (unscaled, |x| is 1 within 1e-6, and what that leaves of rho x in r is along x)
        double rho = fma(e0, e0, fma(e1, e1, fma(e2, e2, e3 * e3)));
        double rb = rho;
        if (beta != 1.0) {
            float seed;
            rho *= recip(fma(x[0], x[0], fma(x[1], x[1], fma(x[2], x[2], beta * (x[3] * x[3])))), seed);
            rb = rho * beta;
        }
        const float r[4] = {(float)fma(a[0], e2, fma(b[0], e3, fma(-rho, x[0], -e0))),
                            (float)fma(a[1], e2, fma(b[1], e3, fma(-rho, x[1], -e1))),
                            (float)fma(a[2], e2, fma(b[2], e3, fma(xl, e0, fma(yl, e1, -rho * x[2])))),
                            (float)fma(a[3], e2, fma(b[3], e3, -rb * x[3]))};
        float d[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float f = w[j] * fmaf(V[0][j + 1], r[0], fmaf(V[1][j + 1], r[1], fmaf(V[2][j + 1], r[2], V[3][j + 1] * r[3])));
#pragma unroll
            for (int i = 0; i < 4; ++i) d[i] = fmaf(f, V[i][j + 1], d[i]);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] += (double)d[i];
        const float step = fmaxf(fmaxf(fabsf(d[0]), fabsf(d[1])), fmaxf(fabsf(d[2]), fabsf(d[3])));
        if (!(step < 0.1f * last)) return step < err;  // does not shrink (or has reached the rounding)
        if (k > 0 && step * step < err * last) return true;
        last = step;
    }
    return false;
}

// Whether v >= 0 is infinite.
__device__ __forceinline__ bool infinite(double v) { return __double2hiint(v) == 0x7ff00000; }

// gate_point's result, or false when the pair is to be left to it.
__device__ __forceinline__ bool gate_fast(const GateArgs &g, float2 pl, float2 pr, bool tracked, GateOut &o) {
    o = {0.f, 0.f, 0.f, 0, VT_LOST_INPUT};
    if (!tracked || !isfinite(pl.x) || !isfinite(pl.y) || !isfinite(pr.x) || !isfinite(pr.y)) return true;
    const double *KL = g.rig.kl, *KR = g.rig.kr, *R = g.rig.R, *T = g.rig.t, *t = g.k.t;
    const double ul = pl.x, vl = pl.y, ur = pr.x, vr = pr.y;
    const double xl = (ul - KL[2]) * g.k.ikl[0], yl = (vl - KL[3]) * g.k.ikl[1];
    const double xr = (ur - KR[2]) * g.k.ikr[0], yr = (vr - KR[3]) * g.k.ikr[1];
    const double rx = fma(R[0], xl, fma(R[1], yl, R[2]));
    const double ry = fma(R[3], xl, fma(R[4], yl, R[5]));
    const double rz = fma(R[6], xl, fma(R[7], yl, R[8]));
    float seed;
    if (!(fabs(rz) > 1e-6)) return false;
    if (rz > 0.0) {
        const double iz = recip(rz, seed);
        if (!(seed > kSeedMin)) return false;
        const double dx = ur - fma(KR[0], rx * iz, KR[2]), dy = vr - fma(KR[1], ry * iz, KR[3]);
        const double d2 = fma(dx, dx, dy * dy), m2 = g.prm.min_disp * g.prm.min_disp;
        if (!(infinite(m2) ? d2 < m2 : fabs(d2 - m2) > fma(1e-8, d2 + m2, 1e-9))) return false;
        if (d2 < m2) {
            o.reason = VT_LOST_DISP;
            return true;
        }
    }
    const double a[4] = {fma(xr, R[6], -R[0]), fma(xr, R[7], -R[1]), fma(xr, R[8], -R[2]), fma(xr, t[2], -t[0])};
    const double b[4] = {fma(yr, R[6], -R[3]), fma(yr, R[7], -R[4]), fma(yr, R[8], -R[5]), fma(yr, t[2], -t[1])};
    double x[4];
    float err;
    if (!null_vector_fast(xl, yl, a, b, g.k.beta, x, err)) return false;
    double iw = recip(x[3], seed);
    const float rel = 4.0f * err * fabsf(seed);
    if (!(rel < 1e-7f)) return false;  // near infinity
    if (g.k.beta != 1.0) iw *= g.k.unit;
    const double X = x[0] * iw, Y = x[1] * iw, Z = x[2] * iw;
    o.x = (float)X;
    o.y = (float)Y;
    o.z = (float)Z;
    o.reason = VT_LOST_DEPTH;
    const double XR = fma(R[0], X, fma(R[1], Y, fma(R[2], Z, T[0])));
    const double YR = fma(R[3], X, fma(R[4], Y, fma(R[5], Z, T[1])));
    const double ZR = fma(R[6], X, fma(R[7], Y, fma(R[8], Z, T[2])));
    const double size = fabs(X) + fabs(Y) + fabs(Z) + g.k.unit;
    const double band = (double)(fmaxf(1e-8f, rel) * g.k.rows) * size;
    if (!(fabs(ZR) > band) || !(Z < g.prm.z_min - band || Z > g.prm.z_min + band) ||
        !(Z < g.prm.z_max - band || Z > g.prm.z_max + band))
        return false;
    if (!(ZR > 0.0 && Z > g.prm.z_min && Z < g.prm.z_max)) return true;
    if (!(fabs(Z) > band)) return false;
    float sl, sr;
    const double il = recip(Z, sl), ir = recip(ZR, sr);
    sl = fabsf(sl);
    if (!(fminf(sl, sr) > kSeedMin)) return false;
    const double exl = fma(KL[0], X * il, KL[2] - ul), eyl = fma(KL[1], Y * il, KL[3] - vl);
    const double exr = fma(KR[0], XR * ir, KR[2] - ur), eyr = fma(KR[1], YR * ir, KR[3] - vr);
    // An error e is off by at most d = rel size |R| / |Z| times f + f |X / Z|, and
    // f |X / Z| by at most the observation's distance from the principal point
    // and e.  e and the threshold m compare as their squares where those differ by
    // more than d (e + m), which is at most d's factor (px + um + 2) (1 + e^2 + m^2).
    const float um = fmaxf(fmaxf(fabsf(pl.x), fabsf(pl.y)), fmaxf(fabsf(pr.x), fabsf(pr.y)));
    const float de = 2.0f * rel * (float)size * g.k.rows * fmaxf(sl, sr) * (g.k.px + um + 2.0f);
    const double tol = (double)fmaxf(de, 1e-10f);
    const double e2 = fmax(fma(exl, exl, eyl * eyl), fma(exr, exr, eyr * eyr)), m2 = g.prm.max_reproj * g.prm.max_reproj;
    if (!(infinite(m2) ? e2 < m2 : fabs(e2 - m2) > fma(tol, e2 + m2, tol))) return false;
    if (e2 > m2) {
        o.reason = VT_LOST_REPROJ;
        return true;
    }
    o.status = 1;
    o.reason = VT_TRACKED;
    return true;
}

__device__ __forceinline__ GateOut gate(const GateArgs &g, float2 pl, float2 pr, bool tracked) {
    GateOut o;
    if (!g.k.fast || !gate_fast(g, pl, pr, tracked, o)) o = gate_point(g, pl, pr, tracked);
    return o;
}

// One warp a CTA: the few hundred warps of a call spread over all SMs instead
// of filling a third of them.
constexpr int GATE_THREADS = 32;

__global__ void __launch_bounds__(GATE_THREADS) k_stereo_gate(const float2 *pl, const float2 *pr, const uint8_t *st_in, int n,
                                                     const __grid_constant__ GateArgs g, float *xyz, uint8_t *st_out,
                                                              uint8_t *reason) {
    pdl_wait();  // the pairs may be the previous kernel's output
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const GateOut o = gate(g, pl[i], pr[i], st_in ? st_in[i] != 0 : true);
    if (xyz) {
        xyz[3 * i + 0] = o.x;
        xyz[3 * i + 1] = o.y;
        xyz[3 * i + 2] = o.z;
    }
    st_out[i] = o.status;
    if (reason) reason[i] = o.reason;
}

// Batched form: every gate task of a vt_batch table, one thread per pair,
// grid-stride (the grid is fixed so a captured graph replays any batch).
__global__ void __launch_bounds__(GATE_THREADS) k_gate_batch(const uint8_t *tab) {
    const BatchHdr *H = reinterpret_cast<const BatchHdr *>(tab);
    const GTask *gates = reinterpret_cast<const GTask *>(tab + H->off_gates);
    const int *p0s = reinterpret_cast<const int *>(tab + H->off_gprefix);
    const int total = H->gate_points, ng = H->ngates;
    pdl_wait();  // the pairs are the tracking launch's output
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < total; p += gridDim.x * blockDim.x) {
        int lo = 0, hi = ng - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(p0s + mid) <= p) lo = mid;
            else hi = mid - 1;
        }
        const GTask &t = gates[lo];
        const int i = p - t.p0;
        GateArgs g;
        g.rig = t.rig;
        g.prm = H->G;
        g.k = t.k;
        const GateOut o = gate(g, t.pts_l[i], t.pts_r[i], t.status_in ? t.status_in[i] != 0 : true);
        if (t.xyz) {
            t.xyz[3 * i + 0] = o.x;
            t.xyz[3 * i + 1] = o.y;
            t.xyz[3 * i + 2] = o.z;
        }
        t.status_out[i] = o.status;
        if (t.reason) t.reason[i] = o.reason;
    }
}

static bool finite_all(const double *v, int n) {
    for (int i = 0; i < n; ++i)
        if (!std::isfinite(v[i])) return false;
    return true;
}

bool gate_args_ok(const vt_stereo_rig *rig, const vt_gate_params *prm) {
    if (!rig || !prm) return false;
    if (!finite_all(rig->kl, 4) || !finite_all(rig->kr, 4) || !finite_all(rig->R, 9) || !finite_all(rig->t, 3))
        return false;
    if (rig->kl[0] == 0.0 || rig->kl[1] == 0.0 || rig->kr[0] == 0.0 || rig->kr[1] == 0.0) return false;
    return prm->min_disp >= 0.0 && prm->max_reproj >= 0.0 && prm->z_min <= prm->z_max && std::isfinite(prm->z_min);
}

vt_status launch_gate_batch(const uint8_t *dev_tab, int sms, bool pdl, cudaStream_t s) {
    return launch_pdl(k_gate_batch, 16 * sms, GATE_THREADS, 0, s, pdl, dev_tab) == cudaSuccess ? VT_OK : VT_ERR_CUDA;
}

}  // namespace vt

using namespace vt;

extern "C" vt_status vt_stereo_gate(const float *pts_l, const float *pts_r, const uint8_t *status_in, int n,
                                    const vt_stereo_rig *rig, const vt_gate_params *prm, float *xyz_out,
                                    uint8_t *status_out, uint8_t *reason_out, void *cuda_stream) {
    if (n < 0 || !gate_args_ok(rig, prm)) return VT_ERR_ARG;
    if (n > 0 && (!pts_l || !pts_r || !status_out)) return VT_ERR_ARG;
    if (n == 0) return VT_OK;
    GateArgs g;
    g.rig = *rig;
    g.prm = *prm;
    g.k = gate_scale(*rig);
    const cudaError_t e = launch_pdl(k_stereo_gate, (n + GATE_THREADS - 1) / GATE_THREADS, GATE_THREADS, 0,
                                     (cudaStream_t)cuda_stream, true, reinterpret_cast<const float2 *>(pts_l),
                                     reinterpret_cast<const float2 *>(pts_r), status_in, n, g, xyz_out, status_out,
                                     reason_out);
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? VT_OK : VT_ERR_CUDA;
}
