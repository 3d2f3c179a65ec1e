// Device helpers of the descriptors (App. A): the Darboux-frame pair
// features of Eq. A2, the binning of Eq. A3 and the compensated sum used for
// Eq. A5.  Shared by Faster-PFH and the classic FPFH baseline, which differ
// only in which pairs they visit.
#pragma once

#include "kmx_internal.cuh"

namespace kmxp {

constexpr int kH = 11;
constexpr int kD = 3 * kH;  // 33
constexpr int kStride = KMX_DESC_STRIDE;
static_assert(kD == KMX_DESC_DIM, "three sub-histograms of H bins");

__device__ __forceinline__ float dot3(float ax, float ay, float az, float bx, float by, float bz)
{
    return fmaf(az, bz, fmaf(ay, by, ax * bx));
}

// Angular features of the pair (q, k) (Eq. A2): the point whose normal is
// closer to parallel with the connecting line is the source; v and w are unit
// vectors.  Returns false for coincident points or |d x u| < 1e-6.
__device__ __forceinline__ bool pair_features(float4 pq, float4 nq, float4 pk, float4 nk, float* f)
{
    float dx = pk.x - pq.x, dy = pk.y - pq.y, dz = pk.z - pq.z;
    const float dd = dot3(dx, dy, dz, dx, dy, dz);
    if (!(dd > 0.f)) return false;
    const float inv = 1.0f / sqrtf(dd);
    dx *= inv;
    dy *= inv;
    dz *= inv;
    const float cq = fabsf(dot3(nq.x, nq.y, nq.z, dx, dy, dz));
    const float ck = fabsf(dot3(nk.x, nk.y, nk.z, dx, dy, dz));
    float4 u = nq, nb = nk;
    if (!(cq >= ck)) {
        u = nk;
        nb = nq;
        dx = -dx;
        dy = -dy;
        dz = -dz;
    }
    // v = d x u / |d x u|
    float vx = dy * u.z - dz * u.y;
    float vy = dz * u.x - dx * u.z;
    float vz = dx * u.y - dy * u.x;
    const float s = sqrtf(dot3(vx, vy, vz, vx, vy, vz));
    if (s < 1e-6f) return false;
    const float is = 1.0f / s;
    vx *= is;
    vy *= is;
    vz *= is;
    // w = u x v
    const float wx = u.y * vz - u.z * vy;
    const float wy = u.z * vx - u.x * vz;
    const float wz = u.x * vy - u.y * vx;
    f[0] = atan2f(dot3(wx, wy, wz, nb.x, nb.y, nb.z), dot3(u.x, u.y, u.z, nb.x, nb.y, nb.z));
    f[1] = dot3(vx, vy, vz, nb.x, nb.y, nb.z);
    f[2] = dot3(u.x, u.y, u.z, dx, dy, dz);
    return true;
}

// 0-based bin (Eq. A3) with the upper end clamped to H-1.
__device__ __forceinline__ int feature_bin(float f, float lo, float hi)
{
    float t = floorf((float)kH * (f - lo) / (hi - lo));
    t = fminf(fmaxf(t, 0.f), (float)(kH - 1));
    return (int)t;
}

// The bins of the pair (q, k) by the expressions above, packed b0 | b1 << 8 |
// b2 << 16, or ~0 for a degenerate pair.  Out of line: the fast path below
// needs it for about one pair in a thousand.
static __device__ __noinline__ unsigned pair_bins_exact(float4 pq, float4 nq, float4 pk, float4 nk)
{
    const float PI = 3.14159265358979f;
    float f[3];
    if (!pair_features(pq, nq, pk, nk, f)) return ~0u;
    return (unsigned)feature_bin(f[0], -PI, PI) | (unsigned)feature_bin(f[1], -1.f, 1.f) << 8 |
           (unsigned)feature_bin(f[2], -1.f, 1.f) << 16;
}

// The bins of feature values are all that SPFH needs, so they are found from
// cheap approximations wherever those decide them, and by pair_bins_exact
// elsewhere: the same bins for every pair.  What the approximations leave out
// are the IEEE square roots and divisions and atan2f (about two thirds of the
// instructions of a pair).
//
// Differences between the two evaluations, with e = 2^-24, |d| = |u| = |nb| = 1:
// the direction d carries a common factor within 2^-21 of 1 (the approximate
// reciprocal square root) and a few e per component.  The factor cancels in
// v = d x u / |d x u| and in the source test, which leaves v within 10 e / s of
// the exact path's, s = |d x u|.  So, as positions t among the 11 bins,
//   f3 = u . d            t differs by 5.5 (2^-21 + 10 e)   < 6e-6
//   f2 = v . nb           t differs by 5.5 (10 e / s + 6 e) < 6e-6 / s
//   f1 = atan2(y, x)      the angle differs by (10 e / s + 6 e) sqrt(2) / h, h =
//                         |(x, y)|, by the polynomial's 1.7e-6 (odd, degree 11,
//                         least maximum error on [0, 1]) and by rounding: t
//                         differs by less than 4e-6 / (s h) + 6e-6
// and the exact path's own t rounds within 2e-6.  The result stands when every
// t is farther from its nearest bin edge than 6e-5 / s^2 (6e-5 / (s h)^2 for
// f1), several times these bounds as s, h <= 1; the source test when the two
// cosines differ by 2e-6 (they differ by at most 16 e between the paths).
// Inputs outside the assumptions (coincident or huge distances, s < 1e-3,
// normals that are not unit vectors, NaN) fail one of the tests.
// nq_unit: unit_normal(nq).
__device__ __forceinline__ bool unit_normal(float4 n)
{
    return fabsf(dot3(n.x, n.y, n.z, n.x, n.y, n.z) - 1.f) < 1e-3f;
}

__device__ __forceinline__ unsigned pair_bins(float4 pq, float4 nq, bool nq_unit, float4 pk, float4 nk)
{
    constexpr float kMagic = 12582912.f;  // 1.5 2^23: adding it rounds to an integer in the low bits
    const float dx = pk.x - pq.x, dy = pk.y - pq.y, dz = pk.z - pq.z;
    const float dd = dot3(dx, dy, dz, dx, dy, dz);
    const float inv = rsqrtf(dd);
    const float a = dot3(nq.x, nq.y, nq.z, dx, dy, dz) * inv, b = dot3(nk.x, nk.y, nk.z, dx, dy, dz) * inv;
    const bool src = fabsf(a) >= fabsf(b);
    const float ux = src ? nq.x : nk.x, uy = src ? nq.y : nk.y, uz = src ? nq.z : nk.z;
    const float bx = src ? nk.x : nq.x, by = src ? nk.y : nq.y, bz = src ? nk.z : nq.z;
    const float si = src ? inv : -inv;
    const float ex = dx * si, ey = dy * si, ez = dz * si;
    const float vx = ey * uz - ez * uy, vy = ez * ux - ex * uz, vz = ex * uy - ey * ux;
    const float ss = dot3(vx, vy, vz, vx, vy, vz);
    const float is = rsqrtf(ss);
    const float f2 = dot3(vx, vy, vz, bx, by, bz) * is;
    // (u x v) . nb = v . (nb x u)
    const float y = dot3(vx, vy, vz, by * uz - bz * uy, bz * ux - bx * uz, bx * uy - by * ux) * is;
    const float x = dot3(ux, uy, uz, bx, by, bz);
    const float ax = fabsf(x), ay = fabsf(y);
    const float r = __fdividef(fminf(ax, ay), fmaxf(ax, ay)), r2 = r * r;
    // atan(r) in bins (times 11 / 2 pi)
    float t = fmaf(r2, fmaf(r2, fmaf(r2, fmaf(r2, fmaf(r2, -0.020516733f, 0.09216993f), -0.20382833f), 0.33883196f),
                            -0.58232427f), 1.7506645f) * r;
    t = ay > ax ? 2.75f - t : t;
    t = x < 0.f ? 5.5f - t : t;
    // positions less half a bin: the nearest integer is the bin
    const float t1 = copysignf(t, y) + 5.f, t2 = fmaf(f2, 5.5f, 5.f), t3 = fmaf(src ? a : -b, 5.5f, 5.f);
    const float m1 = t1 + kMagic, m2 = t2 + kMagic, m3 = t3 + kMagic;
    // distances to the nearest bin edge
    const float g1 = 0.5f - fabsf(t1 - (m1 - kMagic)), g2 = 0.5f - fabsf(t2 - (m2 - kMagic));
    const float g3 = 0.5f - fabsf(t3 - (m3 - kMagic));
    const float hh = fmaf(x, x, y * y);
    const float g = fminf(fminf(g1 * hh, g2), g3) * ss;
    const bool ok = nq_unit && unit_normal(nk) && g > 6e-5f && ss > 1e-6f && hh > 1e-6f && dd > 0x1p-100f && dd < 0x1p100f &&
                    fabsf(fabsf(a) - fabsf(b)) > 2e-6f;
    if (!ok) return pair_bins_exact(pq, nq, pk, nk);
    return (__float_as_uint(m1) & 15u) | (__float_as_uint(m2) & 15u) << 8 | (__float_as_uint(m3) & 15u) << 16;
}

__device__ __forceinline__ void count_bins(int* hist, unsigned bins)
{
    atomicAdd(&hist[bins & 255u], 1);
    atomicAdd(&hist[kH + ((bins >> 8) & 255u)], 1);
    atomicAdd(&hist[2 * kH + (bins >> 16)], 1);
}

__device__ __forceinline__ void kahan_add(float& sum, float& comp, float term)
{
    const float y = term - comp;
    const float t = sum + y;
    comp = (t - sum) - y;
    sum = t;
}

// Compensated sum of the term a * b, its product fused with the subtraction
// of the compensation (one rounding), so that every kernel that adds the
// same terms in the same order gets the same bits.
__device__ __forceinline__ void kahan_add_prod(float& sum, float& comp, float a, float b)
{
    const float y = fmaf(a, b, -comp);
    const float t = sum + y;
    comp = (t - sum) - y;
    sum = t;
}

// kahan_add_prod on two independent sums at once, in paired FP32
// instructions; ncomp holds the negated compensation.  Each component takes
// exactly kahan_add_prod's roundings: fma(a, b, -c), then s + y, then
// -((t - s) - y) computed as y + (s - t) (round-to-nearest is symmetric under
// negation, and s - t is the fma of t, -1 and s).  The paired form issues half
// the instructions for the same bits.
__device__ __forceinline__ void kahan_add_prod2(float2& sum, float2& ncomp, float2 a, float2 b)
{
    const float2 y = __ffma2_rn(a, b, ncomp);
    const float2 t = __fadd2_rn(sum, y);
    const float2 e = __ffma2_rn(t, make_float2(-1.f, -1.f), sum);
    ncomp = __fadd2_rn(y, e);
    sum = t;
}

}  // namespace kmxp
