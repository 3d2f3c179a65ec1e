// Device helpers of the radius searches: the grid view, the exact radius
// test of Eq. A1, the 27-cell stencil walked by a warp, and the FP64
// eigen-solve and orientation that turn second moments into a normal
// (Sec. III-C).  Shared by the Faster-PFH search (one search, r_FPFH) and the
// classic FPFH baseline (separate searches).
#pragma once

#include "kmx_internal.cuh"
#include "grid_common.cuh"

#include <climits>

namespace kmxs {

constexpr unsigned kFull = 0xffffffffu;

struct GridView {
    const float4* __restrict__ sorted;
    const int2* __restrict__ cells;
    const unsigned long long* __restrict__ keys;
    uint32_t T;
    double inv_cell;
    const int64_t* n_sorted;
    const int32_t* __restrict__ sslot;  // hash slot of each sorted point's cell
};

struct Radii {
    float rf2, rn2;     // FP32 squared radii
    double rf2d, rn2d;  // FP64 squared radii, (double)r * (double)r
    float ef, en;       // half-widths of the bands around them in which FP64 decides (within)
};

inline Radii make_radii(const kmx_params* prm)
{
    Radii R;
    R.rf2 = prm->r_fpfh * prm->r_fpfh;
    R.rn2 = prm->r_normal * prm->r_normal;
    R.rf2d = (double)prm->r_fpfh * (double)prm->r_fpfh;
    R.rn2d = (double)prm->r_normal * (double)prm->r_normal;
    R.ef = 1e-5f * R.rf2;
    R.en = 1e-5f * R.rn2;
    return R;
}

// Is a within radius of q?  FP32 unless the FP32 distance lies within 1e-5
// (relative) of r^2, where the FP64 expression ((dx*dx + dy*dy) + dz*dz) <
// r*r decides; FP32 error is far below that band, so the set is exact.
__device__ __forceinline__ bool within(float4 a, float4 q, float d2, float r2, double r2d)
{
    if (fabsf(d2 - r2) > 1e-5f * r2) return d2 < r2;
    double dx = __dsub_rn((double)a.x, (double)q.x);
    double dy = __dsub_rn((double)a.y, (double)q.y);
    double dz = __dsub_rn((double)a.z, (double)q.z);
    double e = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    return e < r2d;
}

// The packed cell key of the point at sorted position p: the grid build
// computed it (FP64 floor of x / cell) and kept its hash slot.
__device__ __forceinline__ unsigned long long cell_key_at(const GridView& g, int64_t p)
{
    return __ldg(g.keys + __ldg(g.sslot + p));
}

__device__ __forceinline__ void unpack_cell(unsigned long long key, int* cx, int* cy, int* cz)
{
    *cx = (int)((key >> 42) & 0x1FFFFFull) - KMX_KEY_BIAS;
    *cy = (int)((key >> 21) & 0x1FFFFFull) - KMX_KEY_BIAS;
    *cz = (int)(key & 0x1FFFFFull) - KMX_KEY_BIAS;
}

// Lane l < 27 gets (start, count) of cell l of the stencil around cell
// (cx, cy, cz); returns the candidate total and leaves each lane's exclusive
// prefix in *excl.  Every query of one cell has the same stencil.
__device__ __forceinline__ int stencil_at(const GridView& g, int cx, int cy, int cz, int lane, int* start, int* excl)
{
    int st = 0, ct = 0;
    if (lane < 27) {
        int dx = lane % 3 - 1, dy = (lane / 3) % 3 - 1, dz = lane / 9 - 1;
        int slot = kmx_hash_find(g.keys, g.T, kmx_pack_key(cx + dx, cy + dy, cz + dz));
        if (slot >= 0) {
            int2 c = g.cells[slot];
            st = c.x;
            ct = c.y;
        }
    }
    int incl = ct;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    *start = st;
    *excl = incl - ct;
    return __shfl_sync(kFull, incl, 31);
}

// The stencil of the query at sorted position p.
__device__ __forceinline__ int stencil(const GridView& g, int64_t p, int lane, int* start, int* excl)
{
    int cx, cy, cz;
    unpack_cell(cell_key_at(g, p), &cx, &cy, &cz);
    return stencil_at(g, cx, cy, cz, lane, start, excl);
}

// Candidate number t -> position in the sorted point array.
__device__ __forceinline__ int candidate(int t, int start, int excl)
{
    int lo = 0;
#pragma unroll
    for (int step = 16; step >= 1; step >>= 1) {
        int e = __shfl_sync(kFull, excl, lo + step);
        if (e <= t) lo += step;
    }
    int cs = __shfl_sync(kFull, start, lo);
    int ce = __shfl_sync(kFull, excl, lo);
    return cs + (t - ce);
}

// Device point count from which the radius searches (normals, the list-free
// FPFH path) give each query one lane of a warp (LaneQueries); below it one
// warp takes a query, so that a small cloud still fills the GPU.  Every search
// kernel applies the same rule, which keeps the list and list-free paths
// bit-identical.
constexpr int64_t kThreadQueryMin = 65536;

constexpr int kStep = 4;        // 32-candidate words a warp holds in registers at once
constexpr int kKeepWords = 32;  // words of P_normal hits kept per query between the two sweeps
constexpr int kLaneWarps = 4;   // warps per block of the lane-per-query kernels

// Shared memory of one warp of the lane-per-query search.
struct LaneQueries {
    float4 neg[32][2];              // the warp's queries negated, each coordinate twice: (x x y y), (z z - -)
    float4 c[32 * kStep];           // the candidates of the current step
    unsigned keep[kKeepWords][32];  // r_normal hits of query l in word w
};

// Candidates of 32 kStep consecutive stencil positions, one per lane and word,
// the words paired for paired FP32 instructions; lanes past the end hold a
// point at infinity, which is inside no radius.  Lane 31 holds a word's first
// candidate, so that the highest set bit of a ballot is the next in list order
// (one instruction to find).
struct Words {
    float2 x[kStep / 2], y[kStep / 2], z[kStep / 2];
    int idx[kStep];

    __device__ __forceinline__ void load(const GridView& g, int base, int total, int start, int excl, int lane,
                                         float4* stage)
    {
#pragma unroll
        for (int w = 0; w < kStep; ++w) {
            const int t = base + 32 * w + 31 - lane;
            const int pos = candidate(t, start, excl);
            const float4 a = t < total ? __ldg(g.sorted + pos) : make_float4(INFINITY, INFINITY, INFINITY, 0.f);
            if (w & 1) {
                x[w / 2].y = a.x;
                y[w / 2].y = a.y;
                z[w / 2].y = a.z;
            } else {
                x[w / 2].x = a.x;
                y[w / 2].x = a.y;
                z[w / 2].x = a.z;
            }
            idx[w] = __float_as_int(a.w);
            if (stage) stage[32 * w + lane] = a;
        }
    }
};

// The FP64 decision of hit_words for one word: rare, so it is kept out of
// line (the unrolled tests stay small enough for the instruction cache).
// Bits 0 and 1: within r_FPFH, within r_normal.
static __device__ __noinline__ unsigned within_both(float ax, float ay, float az, float qx, float qy, float qz, float d2,
                                             float rf2, float rn2, double rf2d, double rn2d)
{
    const float4 a = make_float4(ax, ay, az, 0.f), q = make_float4(qx, qy, qz, 0.f);
    if (!(ax < INFINITY)) return 0u;  // no candidate in this lane
    const bool f = within(a, q, d2, rf2, rf2d);
    return (f ? 1u : 0u) | (f && within(a, q, d2, rn2, rn2d) ? 2u : 0u);
}

// Hits of query j among the warp's candidate words: bit l of bf[w] (bn[w]) is
// set when the candidate of lane l in word w lies within r_FPFH (r_normal).
// A step in which some distance falls into an FP64 band is decided again.
template <bool kF, bool kN>
__device__ __forceinline__ void hit_words(const Words& c, const float4 (&neg)[2], const Radii& R,
                                          unsigned (&bf)[kStep], unsigned (&bn)[kStep])
{
    const float2 qx = make_float2(neg[0].x, neg[0].y), qy = make_float2(neg[0].z, neg[0].w);
    const float2 qz = make_float2(neg[1].x, neg[1].y);
    bool band = false;
    float2 d2[kStep / 2];
#pragma unroll
    for (int h = 0; h < kStep / 2; ++h) {
        const float2 dx = __fadd2_rn(c.x[h], qx), dy = __fadd2_rn(c.y[h], qy), dz = __fadd2_rn(c.z[h], qz);
        d2[h] = __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
        if (kF) {
            const float2 e = __fadd2_rn(d2[h], make_float2(-R.rf2, -R.rf2));
            band |= !(fabsf(e.x) > R.ef);
            band |= !(fabsf(e.y) > R.ef);
            bf[2 * h] = __ballot_sync(kFull, e.x < 0.f);
            bf[2 * h + 1] = __ballot_sync(kFull, e.y < 0.f);
        }
        if (kN) {
            const float2 e = __fadd2_rn(d2[h], make_float2(-R.rn2, -R.rn2));
            band |= !(fabsf(e.x) > R.en);
            band |= !(fabsf(e.y) > R.en);
            bn[2 * h] = __ballot_sync(kFull, e.x < 0.f);
            bn[2 * h + 1] = __ballot_sync(kFull, e.y < 0.f);
        }
    }
    if (__any_sync(kFull, band)) {
#pragma unroll
        for (int w = 0; w < kStep; ++w) {
            const int h = w / 2;
            const unsigned in = within_both((w & 1) ? c.x[h].y : c.x[h].x, (w & 1) ? c.y[h].y : c.y[h].x,
                                            (w & 1) ? c.z[h].y : c.z[h].x, -qx.x, -qy.x, -qz.x,
                                            (w & 1) ? d2[h].y : d2[h].x, R.rf2, R.rn2, R.rf2d, R.rn2d);
            if (kF) bf[w] = __ballot_sync(kFull, in & 1u);
            if (kN) bn[w] = __ballot_sync(kFull, in & 2u);
        }
    }
}

// The lane-per-query kernels take the queries in batches of up to 32 of one
// cell: positions 0, 32, 64, .. of a cell's run start a batch.  The warp that
// takes a window of 32 sorted positions takes the batches that start in it, at
// most 63 queries.  (Batches cut at the windows, whatever the cells, gave 18.4k
// batches of 16 queries on a 300k-point indoor cloud instead of 14k; whole
// cells per warp left a tail of dense cells, 0.61 -> 1.03 ms.)
// Bit l: a batch starts at sorted position p0 + l; (*slot, *end) are that
// position's cell and the end of its run.
__device__ __forceinline__ unsigned batch_heads(const GridView& g, int64_t p0, int64_t n_sorted, int lane, int* slot,
                                                int* end)
{
    const int64_t p = p0 + lane;
    bool head = false;
    *slot = *end = 0;
    if (p < n_sorted) {
        *slot = __ldg(g.sslot + p);
        const int2 cell = __ldg(g.cells + *slot);
        *end = cell.x + cell.y;
        head = (((int)p - cell.x) & 31) == 0;
    }
    return __ballot_sync(kFull, head);
}

// Leave the queries of a batch negated in shared memory, for the whole warp.
__device__ __forceinline__ void stage_queries(float4 q, int lane, float4 (&neg)[32][2])
{
    __syncwarp();
    neg[lane][0] = make_float4(-q.x, -q.x, -q.y, -q.y);
    neg[lane][1] = make_float4(-q.z, -q.z, 0.f, 0.f);
    __syncwarp();
}

// Calls f(a) for the candidates behind the set bits of the lane's words m, in
// list order, all lanes together.  A lane moves on to its next word when the
// current one is used up, so the lanes stay busy until the fullest one ends.
template <typename F>
__device__ __forceinline__ void for_each_hit(const unsigned (&words)[kStep], const float4* stage, F&& f)
{
    unsigned m[kStep];
    int left = 0;
#pragma unroll
    for (int w = 0; w < kStep; ++w) {
        m[w] = words[w];
        left += max(__popc(m[w]), 1);
    }
    int at = 0;
    for (left = __reduce_max_sync(kFull, left); left > 0; --left) {
        const int bit = 31 - __clz(m[0]);
        if (m[0]) {
            f(stage[at + bit]);
            m[0] ^= 1u << bit;
        }
        if (!m[0]) {
#pragma unroll
            for (int w = 0; w + 1 < kStep; ++w) m[w] = m[w + 1];
            m[kStep - 1] = 0u;
            at += 32;
        }
    }
}

// |I| (r_FPFH), |P_normal| (r_normal) and the centred P_normal moments of the
// nq <= 32 queries of one batch, one per lane: mom = s1 (3), then xx xy xz yy yz
// zz of the offsets centred on their mean.  (start, excl, total) is the
// stencil of their cell (stencil_at).
//
// The distance tests run one candidate per lane and one query per step, with
// the candidates of 4 words held in registers for all queries of the batch; the
// sums run one query per lane over its hit bits, in list order, the candidate
// read from shared memory.
__device__ __forceinline__ void lane_moments(const GridView& g, const Radii& R, int start, int excl, int total, int nq,
                                             int lane, LaneQueries& sm, float4 q, int* nf_out, int* nn_out,
                                             float (&mom)[9])
{
    stage_queries(q, lane, sm.neg);
    int nf = 0, nn = 0;
    float sx = 0.f, sy = 0.f, sz = 0.f;
#pragma unroll
    for (int i = 0; i < 9; ++i) mom[i] = 0.f;
    const bool mine = lane < nq, kept = total <= 32 * kKeepWords;
    for (int base = 0; base < total; base += 32 * kStep) {
        Words c;
        __syncwarp();
        c.load(g, base, total, start, excl, lane, sm.c);
        unsigned mf[kStep], mn[kStep];
#pragma unroll
        for (int w = 0; w < kStep; ++w) mf[w] = mn[w] = 0u;
        for (int j = 0; j < nq; ++j) {
            unsigned bf[kStep], bn[kStep];
            hit_words<true, true>(c, sm.neg[j], R, bf, bn);
            if (lane == j) {
#pragma unroll
                for (int w = 0; w < kStep; ++w) {
                    mf[w] = bf[w];
                    mn[w] = bn[w];
                }
            }
        }
        const int word0 = kept ? base >> 5 : 0;
#pragma unroll
        for (int w = 0; w < kStep; ++w) {
            nf += __popc(mf[w]);
            nn += __popc(mn[w]);
            if (mine) sm.keep[word0 + w][lane] = mn[w];
        }
        __syncwarp();
        for_each_hit(mn, sm.c, [&](float4 e) {
            sx += e.x - q.x;
            sy += e.y - q.y;
            sz += e.z - q.z;
        });
    }
    const float inv = nn > 0 ? 1.0f / (float)nn : 0.0f;
    const float mx = sx * inv, my = sy * inv, mz = sz * inv;
    for (int base = 0; base < total; base += 32 * kStep) {
        const int word0 = kept ? base >> 5 : 0;
        if (total > 32 * kStep) {  // a single step's candidates are still there
            Words c;
            __syncwarp();
            c.load(g, base, total, start, excl, lane, sm.c);
            if (!kept) {
                for (int j = 0; j < nq; ++j) {
                    unsigned bf[kStep], bn[kStep];
                    hit_words<false, true>(c, sm.neg[j], R, bf, bn);
                    if (lane == j) {
#pragma unroll
                        for (int w = 0; w < kStep; ++w) sm.keep[w][lane] = bn[w];
                    }
                }
            }
            __syncwarp();
        }
        unsigned mn[kStep];
#pragma unroll
        for (int w = 0; w < kStep; ++w) mn[w] = mine ? sm.keep[word0 + w][lane] : 0u;
        for_each_hit(mn, sm.c, [&](float4 e) {
            const float dx = e.x - q.x, dy = e.y - q.y, dz = e.z - q.z;
            const float ex = dx - mx, ey = dy - my, ez = dz - mz;
            mom[0] += ex;
            mom[1] += ey;
            mom[2] += ez;
            mom[3] = fmaf(ex, ex, mom[3]);
            mom[4] = fmaf(ex, ey, mom[4]);
            mom[5] = fmaf(ex, ez, mom[5]);
            mom[6] = fmaf(ey, ey, mom[6]);
            mom[7] = fmaf(ey, ez, mom[7]);
            mom[8] = fmaf(ez, ez, mom[8]);
        });
    }
    *nf_out = nf;
    *nn_out = nn;
}

// Every batch of the calling warp's windows: f(q, nq, start, excl, total) with
// the lane's query (lanes past nq repeat the last one) and its cell's stencil,
// looked up once per batch, 27 lookups at once.
template <typename F>
__device__ __forceinline__ void for_each_batch(const GridView& g, int64_t warp0, int64_t warps, int lane, F&& f)
{
    const int64_t n_sorted = *g.n_sorted;
    for (int64_t p0 = 32 * warp0; p0 < n_sorted; p0 += 32 * warps) {
        int slot, end;
        unsigned heads = batch_heads(g, p0, n_sorted, lane, &slot, &end);
        while (heads) {
            const int l = __ffs(heads) - 1;
            heads &= heads - 1u;
            int cx, cy, cz, start, excl;
            unpack_cell(__ldg(g.keys + __shfl_sync(kFull, slot, l)), &cx, &cy, &cz);
            const int total = stencil_at(g, cx, cy, cz, lane, &start, &excl);
            const int first = (int)p0 + l, nq = min(32, __shfl_sync(kFull, end, l) - first);
            f(__ldg(g.sorted + first + min(lane, nq - 1)), nq, start, excl, total);
        }
    }
}

// The candidates of the last query a warp searched, kept while the next
// queries (consecutive in cell order) sit in the same cell: the stencil and its
// first 32 kStep candidates.
struct WarpQuery {
    unsigned long long key = KMX_EMPTY_KEY;
    int start = 0, excl = 0, total = 0;
    Words first;

    __device__ __forceinline__ void set(const GridView& g, int64_t p, int lane)
    {
        const unsigned long long k = cell_key_at(g, p);
        if (k == key) return;
        int x, y, z;
        unpack_cell(k, &x, &y, &z);
        total = stencil_at(g, x, y, z, lane, &start, &excl);
        first.load(g, 0, total, start, excl, lane, nullptr);
        key = k;
    }

    // f(words, base) for every 32 kStep candidates
    template <typename F>
    __device__ __forceinline__ void for_each(const GridView& g, int lane, F&& f) const
    {
        f(first, 0);
        for (int base = 32 * kStep; base < total; base += 32 * kStep) {
            Words c;
            c.load(g, base, total, start, excl, lane, nullptr);
            f(c, base);
        }
    }
};

// Offset of the lane's candidate in word w from the query (-neg).
__device__ __forceinline__ float3 offset_of(const Words& c, int w, const float4 (&neg)[2])
{
    const int h = w / 2;
    return make_float3(((w & 1) ? c.x[h].y : c.x[h].x) + neg[0].x, ((w & 1) ? c.y[h].y : c.y[h].x) + neg[0].z,
                       ((w & 1) ? c.z[h].y : c.z[h].x) + neg[1].x);
}

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

__device__ __forceinline__ void cross3(const double* a, const double* b, double* c)
{
    c[0] = a[1] * b[2] - a[2] * b[1];
    c[1] = a[2] * b[0] - a[0] * b[2];
    c[2] = a[0] * b[1] - a[1] * b[0];
}

// Eigenvalues l1 >= l2 >= l3 of a symmetric 3x3 matrix and a unit eigenvector
// of l3.  Returns false if the matrix is a multiple of the identity.
//
// GB300 issues FP64 at a small fraction of the FP32 rate, and an FP64 divide
// or square root is a long instruction sequence, so the reciprocals and
// reciprocal square roots below start from the FP32 intrinsic and take one
// FP64 Newton-Raphson step (r <- r (2 - x r) for 1/x, r <- r (3 - x r^2) / 2
// for 1/sqrt(x)), which squares the FP32 start's relative error (about 1e-7)
// to about 1e-14: far below the 1e-8 the eigenvalues are accurate to.
// Arguments outside [2^-100, 2^100] take the FP64 operation itself.
__device__ __forceinline__ bool fp32_range(double x) { return x > 0x1p-100 && x < 0x1p100; }

__device__ __forceinline__ double recip64(double x)
{
    if (!fp32_range(x)) return 1.0 / x;
    const double r = (double)__frcp_rn((float)x);
    return r * fma(-x, r, 2.0);
}

__device__ __forceinline__ double rsqrt64(double x)
{
    if (!fp32_range(x)) return 1.0 / sqrt(x);
    const double r = (double)rsqrtf((float)x);
    return r * fma(-0.5 * x, r * r, 1.5);
}

// sqrt(x) = x / sqrt(x) for x > 0, 0 for x <= 0
__device__ __forceinline__ double sqrt64(double x)
{
    if (!(x > 0.0)) return 0.0;
    return fp32_range(x) ? x * rsqrt64(x) : sqrt(x);
}

__device__ __forceinline__ bool eig_sym3(double a00, double a01, double a02, double a11, double a12, double a22,
                                         double* l, double* nv)
{
    const double p1 = a01 * a01 + a02 * a02 + a12 * a12;
    const double q = (a00 + a11 + a22) * (1.0 / 3.0);
    const double b00 = a00 - q, b11 = a11 - q, b22 = a22 - q;
    const double p2 = b00 * b00 + b11 * b11 + b22 * b22 + 2.0 * p1;
    if (!(p2 > 0.0)) {
        l[0] = l[1] = l[2] = q;
        nv[0] = 0.0;
        nv[1] = 0.0;
        nv[2] = 1.0;
        return false;
    }
    // Eigenvalues of the traceless B = A - qI are the roots of
    // g(mu) = mu^3 - (p2 / 2) mu - det(B), i.e. 2p cos(phi + 2 pi k / 3) with
    // p = sqrt(p2 / 6), phi = acos(r) / 3, r = det(B) / (2 p^3).  GB300 issues
    // FP64 slowly and acos / cos in FP64 dominated this solve, so: the
    // trigonometric form in FP32 for a start, two FP64 Newton steps on the
    // extreme root that is well separated (the largest when r >= 0, i.e. when
    // the two smaller roots are the closer pair; else the smallest), and the
    // other two in FP64 from the quadratic mu^2 + m mu + (m^2 - p2 / 2) = 0
    // (sum of the roots 0, sum of their pairwise products -p2 / 2), whose
    // square root resolves a close pair to ~1e-8 p.  Beyond p (below -p) g is
    // increasing and convex (concave), so Newton started there (the start is
    // clamped; pf is within 2^-23 of p) moves monotonically to that extreme
    // root.  Eigenvalues come out to ~1e-8 relative or better, the smallest
    // one to FP64 accuracy where the normal is well posed.
    const double det = b00 * (b11 * b22 - a12 * a12) - a01 * (a01 * b22 - a12 * a02) + a02 * (a01 * a12 - b11 * a02);
    const float pf = sqrtf((float)p2 / 6.0f);
    const float rf = fminf(1.0f, fmaxf(-1.0f, (float)det / (2.0f * pf * pf * pf)));
    const float phi = acosf(rf) / 3.0f;
    const double edge = (double)pf * (1.0 + 0x1p-20);
    const bool top = rf >= 0.0f;
    double mu = top ? fmax((double)(2.0f * pf * cosf(phi)), edge)
                    : fmin((double)(2.0f * pf * cosf(phi + 2.0943951f)), -edge);
    const double h = 0.5 * p2;
#pragma unroll
    for (int it = 0; it < 2; ++it) {
        const double g = mu * (mu * mu - h) - det;
        const double dg = 3.0 * mu * mu - h;
        if (dg > 0.0) mu -= g * recip64(dg);  // dg > 0 beyond +-p
    }
    const double sd = sqrt64(2.0 * p2 - 3.0 * mu * mu);
    if (top) {
        l[0] = q + mu;
        l[1] = q + 0.5 * (-mu + sd);
        l[2] = q + 0.5 * (-mu - sd);
    } else {
        l[0] = q + 0.5 * (-mu + sd);
        l[1] = q + 0.5 * (-mu - sd);
        l[2] = q + mu;
    }
    const double r0[3] = {a00 - l[2], a01, a02};
    const double r1[3] = {a01, a11 - l[2], a12};
    const double r2[3] = {a02, a12, a22 - l[2]};
    double c0[3], c1[3], c2[3];
    cross3(r0, r1, c0);
    cross3(r0, r2, c1);
    cross3(r1, r2, c2);
    const double n0 = c0[0] * c0[0] + c0[1] * c0[1] + c0[2] * c0[2];
    const double n1 = c1[0] * c1[0] + c1[1] * c1[1] + c1[2] * c1[2];
    const double n2 = c2[0] * c2[0] + c2[1] * c2[1] + c2[2] * c2[2];
    double cx = c0[0], cy = c0[1], cz = c0[2], nb = n0;
    if (n1 > nb) {
        cx = c1[0];
        cy = c1[1];
        cz = c1[2];
        nb = n1;
    }
    if (n2 > nb) {
        cx = c2[0];
        cy = c2[1];
        cz = c2[2];
        nb = n2;
    }
    if (!(nb > 0.0)) {
        nv[0] = 0.0;
        nv[1] = 0.0;
        nv[2] = 1.0;
        return true;
    }
    const double inv = rsqrt64(nb);
    nv[0] = cx * inv;
    nv[1] = cy * inv;
    nv[2] = cz * inv;
    return true;
}

// Normal of a query from the moments of its P_normal offsets e = (a - q) - m0
// (m0 the FP32 mean used for centring): mom = (sum e, then the six products
// xx xy xz yy yz zz).  The covariance (1/n normaliser) is formed and solved
// in FP64, the normal oriented toward vp (first non-zero component positive
// when n . (vp - q) = 0) and p_lin = (l1 - l2) / l1 stored in w.  Returns
// false (and a zero normal) when l1 = 0.
__device__ __forceinline__ bool normal_from_moments(const float* mom, int nN, float qx, float qy, float qz,
                                                    const float* vp, float4* nout, double* plin_out)
{
    const double inv = recip64((double)nN);
    const double m0 = (double)mom[0] * inv, m1 = (double)mom[1] * inv, m2 = (double)mom[2] * inv;
    const double c00 = (double)mom[3] * inv - m0 * m0, c01 = (double)mom[4] * inv - m0 * m1;
    const double c02 = (double)mom[5] * inv - m0 * m2, c11 = (double)mom[6] * inv - m1 * m1;
    const double c12 = (double)mom[7] * inv - m1 * m2, c22 = (double)mom[8] * inv - m2 * m2;
    double l[3], nv[3];
    eig_sym3(c00, c01, c02, c11, c12, c22, l, nv);
    *nout = make_float4(0.f, 0.f, 0.f, 0.f);
    *plin_out = 0.0;
    if (!(l[0] > 0.0)) return false;
    const double view = nv[0] * ((double)vp[0] - (double)qx) + nv[1] * ((double)vp[1] - (double)qy) +
                        nv[2] * ((double)vp[2] - (double)qz);
    bool flip = view < 0.0;
    if (view == 0.0) flip = nv[0] != 0.0 ? nv[0] < 0.0 : (nv[1] != 0.0 ? nv[1] < 0.0 : nv[2] < 0.0);
    const double sgn = flip ? -1.0 : 1.0;
    const double plin = (l[0] - l[1]) / l[0];
    *nout = make_float4((float)(sgn * nv[0]), (float)(sgn * nv[1]), (float)(sgn * nv[2]), (float)plin);
    *plin_out = plin;
    return true;
}

}  // namespace kmxs
