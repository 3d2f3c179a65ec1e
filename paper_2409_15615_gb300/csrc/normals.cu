// Algorithm 1, step 1 (Sec. III-C, App. A): one radius search per point with
// r_FPFH (Eq. A1), the r_normal subsample P_normal, PCA normal and linearity,
// and the reliability flag B.
//
// Queries are taken in cell order so that neighbouring lanes or warps walk the
// same cells.  The kernels pick one of two layouts from the device point count,
// the same way in every launch (kThreadQueryMin, search_common.cuh):
//  - large clouds: 32 queries per warp, one per lane (lane_moments).  The
//    distance tests run one candidate per lane, the sums one query per lane in
//    the order of the stored lists.
//  - small clouds (too few queries to fill the GPU that way): one warp per
//    query.  The 27 stencil cells are looked up by 27 lanes at once, their
//    candidate ranges are flattened into one index space, and all 32 lanes
//    test candidates.
// Two passes: the first counts |I|, takes the P_normal mean and the covariance
// centred on it; after a prefix sum of the counts the second tests again and
// writes the CSR lists.  Keeping the first pass's hits would need a bit per
// candidate and query in memory of no fixed size.
//
// Bound by instruction issue (2.4 a cycle of 4).  On a 300k-point indoor cloud
// (166 neighbours of 600 candidates a query): one thread per query, each
// looking up its 27 cells, walking twice and writing its own list, took 636 us
// (count), 792 us (fill) and 103 us (solve) with 17 to 19 of 32 lanes active;
// this form takes 535 us (lane_normals, solve included) and 300 us
// (search_fill).  On a 19k-point LiDAR scan the small-cloud kernels went from
// 23 + 25 + 17 us to 25 + 17 (fill) + 11 us (solve) by holding 128 candidates
// in registers across a cell's queries and both sweeps.
//
// The 3x3 eigen-problem starts from the closed form (Smith 1961:
// trigonometric eigenvalues) in FP32, refines the well-separated extreme
// eigenvalue by FP64 Newton steps on the characteristic polynomial and takes
// the other two from a quadratic in FP64; the normal is the best-conditioned
// cross product of two rows of A - l3 I in FP64 (search_common.cuh).  GB300 issues FP64
// at a small fraction of the FP32 rate and a warp instruction costs the same
// with 1 or 32 active lanes, so a solve always takes 32 queries at once: at the
// end of a warp's 32 queries on a large cloud (where the FP64 pipe works beside
// the other warps' tests), in a pass of its own over the stored moments on a
// small one.
#include "search_common.cuh"

using namespace kmxs;

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kQPerWarp = 4;                    // queries per warp in the warp-per-query mode
constexpr int kQPerBlock = kWarps * kQPerWarp;  // = 32, queries per block per step in that mode

struct NormScratch {
    int32_t* cnt;    // [n+1] |I(q)|
    float4* mom;     // [sorted position][3] small clouds: centred moments s1x s1y s1z sxx | sxy sxz syy syz | szz |P_normal| - -
};

NormScratch carve(void* base, int64_t n, size_t* total)
{
    NormScratch s{};
    kmx_arena a{static_cast<char*>(base), 0};
    s.cnt = (int32_t*)a.take(sizeof(int32_t) * (n + 1));
    s.mom = (float4*)a.take(sizeof(float4) * 3 * ((n < kThreadQueryMin ? n : kThreadQueryMin) + 1));
    *total = kmx_align_up(a.used, 256);
    return s;
}

struct NormOut {
    float4* normal4;
    uint8_t* flags;
    const int64_t* offs;
    int32_t* nbr;
    int64_t nbr_cap;
    int64_t n_cap;
    int64_t* needed;
    int tau_num;
    float tau_lin;
    float vp[3];
};

// The FP64 eigen-solve of one query's moments, orientation toward the
// viewpoint and the linearity test.
__device__ __forceinline__ void solve_one(const NormOut& o, float4 q, int nF, int nN, const float* mom)
{
    const int qi = __float_as_int(q.w);
    uint8_t flag = 0;
    float4 nout = make_float4(0.f, 0.f, 0.f, 0.f);
    if (nF >= o.tau_num && nN >= o.tau_num) {
        double plin;
        flag |= 4;
        if (normal_from_moments(mom, nN, q.x, q.y, q.z, o.vp, &nout, &plin) && plin < (double)o.tau_lin) flag |= 1;
    }
    o.normal4[qi] = nout;
    o.flags[qi] = flag;
}

// Pass 1 of a large cloud: |I(q)|, |P_normal|, the P_normal moments and the
// normal.
__global__ void __launch_bounds__(32 * kLaneWarps, 6) lane_normals(GridView g, Radii R, NormScratch s, NormOut o)
{
    __shared__ LaneQueries sm[kLaneWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n_sorted = *g.n_sorted;
    if (n_sorted < kThreadQueryMin) return;
    for_each_batch(g, (int64_t)blockIdx.x * kLaneWarps + warp, (int64_t)gridDim.x * kLaneWarps, lane,
                   [&](float4 q, int nq, int start, int excl, int total) {
                       int nf, nn;
                       float mom[9];
                       lane_moments(g, R, start, excl, total, nq, lane, sm[warp], q, &nf, &nn, mom);
                       if (lane < nq) {
                           s.cnt[__float_as_int(q.w)] = nf;
                           solve_one(o, q, nf, nn, mom);
                       }
                   });
}

// Pass 1 of a small cloud: |I(q)|, |P_normal| and the P_normal moments.
__global__ void __launch_bounds__(kThreads) search_moments(GridView g, Radii R, NormScratch s)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n_sorted = *g.n_sorted;
    const int64_t warps = (int64_t)gridDim.x * kWarps;
    if (n_sorted >= kThreadQueryMin) return;
    for (int64_t w = (int64_t)blockIdx.x * kWarps + warp; w * kQPerWarp < n_sorted; w += warps) {
        WarpQuery c;  // the warp's queries are consecutive in cell order
        for (int k = 0; k < kQPerWarp && w * kQPerWarp + k < n_sorted; ++k) {
            const int64_t p = w * kQPerWarp + k;
            const float4 q = g.sorted[p];
            c.set(g, p, lane);
            const float4 neg[2] = {make_float4(-q.x, -q.x, -q.y, -q.y), make_float4(-q.z, -q.z, 0.f, 0.f)};
            int nf = 0, nn = 0;
            float sx = 0.f, sy = 0.f, sz = 0.f;
            unsigned first[kStep];  // the first words' P_normal hits, for the second sweep
            c.for_each(g, lane, [&](const Words& a, int base) {
                unsigned bf[kStep], bn[kStep];
                hit_words<true, true>(a, neg, R, bf, bn);
#pragma unroll
                for (int i = 0; i < kStep; ++i) {
                    nf += __popc(bf[i]);
                    nn += __popc(bn[i]);
                    if (base == 0) first[i] = bn[i];
                    if ((bn[i] >> lane) & 1u) {
                        const float3 d = offset_of(a, i, neg);
                        sx += d.x;
                        sy += d.y;
                        sz += d.z;
                    }
                }
            });
            sx = warp_sum(sx);
            sy = warp_sum(sy);
            sz = warp_sum(sz);
            const float inv = nn > 0 ? 1.0f / (float)nn : 0.0f;
            const float mx = sx * inv, my = sy * inv, mz = sz * inv;
            float m[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) m[i] = 0.f;
            c.for_each(g, lane, [&](const Words& a, int base) {
                unsigned bf[kStep], bn[kStep];
                if (base == 0) {
#pragma unroll
                    for (int i = 0; i < kStep; ++i) bn[i] = first[i];
                } else {
                    hit_words<false, true>(a, neg, R, bf, bn);
                }
#pragma unroll
                for (int i = 0; i < kStep; ++i) {
                    if ((bn[i] >> lane) & 1u) {
                        const float3 d = offset_of(a, i, neg);
                        const float ex = d.x - mx, ey = d.y - my, ez = d.z - mz;
                        m[0] += ex;
                        m[1] += ey;
                        m[2] += ez;
                        m[3] = fmaf(ex, ex, m[3]);
                        m[4] = fmaf(ex, ey, m[4]);
                        m[5] = fmaf(ex, ez, m[5]);
                        m[6] = fmaf(ey, ey, m[6]);
                        m[7] = fmaf(ey, ez, m[7]);
                        m[8] = fmaf(ez, ez, m[8]);
                    }
                }
            });
#pragma unroll
            for (int i = 0; i < 9; ++i) m[i] = warp_sum(m[i]);
            if (lane == 0) {
                s.cnt[__float_as_int(q.w)] = nf;
                float4* o = s.mom + 3 * p;
                o[0] = make_float4(m[0], m[1], m[2], m[3]);
                o[1] = make_float4(m[4], m[5], m[6], m[7]);
                o[2] = make_float4(m[8], __int_as_float(nn), 0.f, 0.f);
            }
        }
    }
}

// Small clouds: the solve of the stored moments, one point per thread.  Blocks
// of 64 spread a scan's 20k points over every SM's FP64 pipe.
constexpr int kSolveThreads = 64;
__global__ void __launch_bounds__(kSolveThreads) solve_normals(GridView g, NormScratch s, NormOut o)
{
    const int64_t n_sorted = *g.n_sorted;
    if (n_sorted >= kThreadQueryMin) return;  // lane_normals solved them
    for (int64_t p = (int64_t)blockIdx.x * kSolveThreads + threadIdx.x; p < n_sorted;
         p += (int64_t)gridDim.x * kSolveThreads) {
        const float4 q = g.sorted[p];
        const float4* m = s.mom + 3 * p;
        const float4 m0 = m[0], m1 = m[1], m2 = m[2];
        const float mom[9] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w, m2.x};
        solve_one(o, q, s.cnt[__float_as_int(q.w)], __float_as_int(m2.y), mom);
    }
}

// Pass 2: the CSR lists.  On a large cloud the warp tests 32 candidates at a
// time against each of its 32 queries in turn, as pass 1 does, so that the
// hits of a query are written next to one another (a lane per query would
// write 32 lists at once, a sector per entry).
__global__ void __launch_bounds__(kThreads, 4) search_fill(GridView g, Radii R, NormOut o, unsigned int* err)
{
    __shared__ float4 neg[kWarps][32][2];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t total_list = o.offs[o.n_cap];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *o.needed = total_list;
        if (o.nbr && total_list > o.nbr_cap) kmx_raise(err, KMX_DERR_CAPACITY);
    }
    if (!o.nbr || total_list > o.nbr_cap) return;
    const int64_t n_sorted = *g.n_sorted;
    const int64_t warps = (int64_t)gridDim.x * kWarps;
    const unsigned above = ~((2u << lane) - 1u);  // bits before this lane's in list order
    if (n_sorted >= kThreadQueryMin) {
        for_each_batch(g, (int64_t)blockIdx.x * kWarps + warp, warps, lane,
                       [&](float4 q, int nq, int start, int excl, int total) {
                           stage_queries(q, lane, neg[warp]);
                           int64_t out = o.offs[__float_as_int(q.w)];
                           for (int base = 0; base < total; base += 32 * kStep) {
                               Words c;
                               c.load(g, base, total, start, excl, lane, nullptr);
                               for (int j = 0; j < nq; ++j) {
                                   unsigned bf[kStep], bn[kStep];
                                   hit_words<true, false>(c, neg[warp][j], R, bf, bn);
                                   int32_t* list = o.nbr + __shfl_sync(kFull, out, j);
                                   int at = 0;
#pragma unroll
                                   for (int w = 0; w < kStep; ++w) {
                                       if ((bf[w] >> lane) & 1u) list[at + __popc(bf[w] & above)] = c.idx[w];
                                       at += __popc(bf[w]);
                                   }
                                   if (lane == j) out += at;
                               }
                           }
                       });
        return;
    }
    for (int64_t w = (int64_t)blockIdx.x * kWarps + warp; w * kQPerWarp < n_sorted; w += warps) {  // one warp per query
        WarpQuery c;
        for (int k = 0; k < kQPerWarp && w * kQPerWarp + k < n_sorted; ++k) {
            const int64_t p = w * kQPerWarp + k;
            const float4 q = g.sorted[p];
            c.set(g, p, lane);
            const float4 qn[2] = {make_float4(-q.x, -q.x, -q.y, -q.y), make_float4(-q.z, -q.z, 0.f, 0.f)};
            int32_t* list = o.nbr + o.offs[__float_as_int(q.w)];
            c.for_each(g, lane, [&](const Words& a, int) {
                unsigned bf[kStep], bn[kStep];
                hit_words<true, false>(a, qn, R, bf, bn);
#pragma unroll
                for (int i = 0; i < kStep; ++i) {
                    if ((bf[i] >> lane) & 1u) list[__popc(bf[i] & above)] = a.idx[i];
                    list += __popc(bf[i]);
                }
            });
        }
    }
}

// Zero the counts |I(q)| of the actual points, and the normals and flags of
// the whole capacity: points that a range error kept out of the grid keep
// zeros, the others are written by search_fill.
__global__ void clear_counts(int32_t* cnt, float4* normal4, uint8_t* flags, const int64_t* d_n, int64_t n_cap)
{
    const int64_t n = kmx_count(d_n, n_cap);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_cap; i += (int64_t)gridDim.x * blockDim.x) {
        if (i < n) cnt[i] = 0;
        normal4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        flags[i] = 0;
    }
}

// When the lists did not fit (search_fill wrote none of them), every offset
// becomes 0: a later stage then reads empty lists instead of entries past
// the end of the list buffer.  `needed` (the full length) is left for the
// caller to size the buffer.
__global__ void empty_lists_on_overflow(int64_t* offs, int64_t n_cap, const int64_t* needed, int64_t nbr_cap)
{
    if (*needed <= nbr_cap) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= n_cap; i += (int64_t)gridDim.x * blockDim.x)
        offs[i] = 0;
}

}  // namespace

size_t kmx_normals_scratch_bytes(int64_t n_cap)
{
    size_t total = 0;
    carve(nullptr, n_cap, &total);
    return total;
}

cudaError_t kmx_normals_launch(kmx_ctx* ctx, const kmx_grid* g, const kmx_params* prm, float* normal4,
                               uint8_t* flags, int64_t* offs, int32_t* nbr, int64_t nbr_cap, int64_t* needed,
                               void* scratch)
{
    cudaStream_t st = ctx->stream;
    size_t total = 0;
    NormScratch s = carve(scratch, g->n_cap, &total);
    GridView gv{g->sorted, g->cells, g->keys, g->table_size, g->inv_cell, g->d_n_sorted, g->sslot};
    const Radii R = make_radii(prm);
    const int64_t n = g->n_cap;
    cudaError_t e;
    KMX_COUNT_LAUNCH();
    clear_counts<<<kmx_stride_blocks(n, 256, ctx->sm_count), 256, 0, st>>>(
        s.cnt, reinterpret_cast<float4*>(normal4), flags, g->d_n, n);
    NormOut o{reinterpret_cast<float4*>(normal4), flags, offs, nbr, nbr_cap, n, needed, prm->tau_num,
              prm->tau_lin, {prm->viewpoint[0], prm->viewpoint[1], prm->viewpoint[2]}};
    // enough blocks for one warp step each at the sizes that fill the GPU, so
    // that uneven stencils balance over the SMs as blocks retire
    const unsigned nb = kmx_stride_blocks(n, kQPerBlock, ctx->sm_count, 16);
    if (n >= kThreadQueryMin) {
        KMX_COUNT_LAUNCH();
        lane_normals<<<kmx_stride_blocks(n, 32 * kLaneWarps, ctx->sm_count, 32), 32 * kLaneWarps, 0, st>>>(gv, R, s, o);
    }
    KMX_COUNT_LAUNCH();
    search_moments<<<nb, kThreads, 0, st>>>(gv, R, s);
    KMX_COUNT_LAUNCH();
    solve_normals<<<kmx_stride_blocks(n < kThreadQueryMin ? n : kThreadQueryMin, kSolveThreads, ctx->sm_count),
                    kSolveThreads, 0, st>>>(gv, s, o);
    if ((e = kmx_scan_i32(ctx, s.cnt, n, g->d_n, offs))) return e;
    KMX_COUNT_LAUNCH();
    search_fill<<<nb, kThreads, 0, st>>>(gv, R, o, ctx->d_err);
    if (nbr) {
        KMX_COUNT_LAUNCH();
        empty_lists_on_overflow<<<kmx_stride_blocks(n + 1, 256, ctx->sm_count), 256, 0, st>>>(offs, n, needed,
                                                                                             nbr_cap);
    }
    return cudaGetLastError();
}
