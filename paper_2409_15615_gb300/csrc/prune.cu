// Correspondence pruning of Sec. III-D on the device: the ratio filter (the
// N_tau correspondences with the lowest d1 / d2), the pairwise-invariant
// compatibility graph of Eq. 3, and the maximum k-core.
//
//   ratio_keys        ratio = d1 / d2 in FP64 (1 when d2 = 0), a 4096-bucket
//                     histogram of it.
//   ratio_threshold   one block: the buckets' first places and the first
//                     bucket B at which the cumulative count reaches N_tau.
//   ratio_candidates  the correspondences in buckets <= B, bucket by bucket
//                     (every one of the N_tau lowest is among them; all others
//                     rank higher).
//   ratio_rank        each candidate's exact rank by (ratio, i) among its
//                     bucket's, after the buckets below; ranks < N_tau give
//                     the selection in ascending order, with both end points
//                     gathered.
//   graph_build       32-bit words of the adjacency bit matrix, two per lane and
//                     32 pair tests:
//                     k ~ k' iff | |b_k - b_k'| - |a_k - a_k'| | <= 2 beta.  The
//                     test runs in FP32; within a band around the threshold it
//                     is decided again in FP64 as ((dx dx + dy dy) + dz dz),
//                     sqrt, |db - da| <= 2 beta, so every edge is the FP64
//                     decision.
//   kcore             one cooperative launch: the core numbers as the fixed
//                     point of c(v) <- H({c(u) : u ~ v}) started from the
//                     degrees (H = h-index: the largest h with at least h
//                     values >= h; the values only decrease and stay above the
//                     core numbers, so updates in any order converge to them).
//                     Rounds of kPasses passes over the vertices, separated by
//                     a bounded grid barrier, until a round changes nothing;
//                     then the largest core number and the positions of the
//                     maximum k-core in ascending order.
#include "kmx_internal.cuh"

#include <cooperative_groups.h>

namespace {

constexpr int kBuckets = 4096;
constexpr int kThreads = 256;
constexpr uint32_t kSpinLimit = 1u << 24;
constexpr int kMaxRounds = 1 << 16;
constexpr int kCoreThreads = 1024;
constexpr int kCoreWarps = kCoreThreads / 32;
constexpr int kSyncGen = 64;                // words from the arrivals, which the pollers of the generation leave alone
constexpr int kPasses = 3;                  // passes between two grid barriers
constexpr size_t kCoreSmem = 136 * 1024;    // snapshot, vertex states and neighbour lists of a kcore CTA

struct PruneScratch {
    double* ratio;            // [n_cap]
    int32_t* bucket;          // [n_cap]
    int32_t* hist;            // [kBuckets] counts, then the places left to fill
    int32_t* first;           // [kBuckets + 1] first place of each bucket; from the last candidate bucket on, their number
    int32_t* cand;            // [n_cap]
    unsigned long long* ckey; // [n_cap] candidate ratio bits
    int32_t* ci;              // [n_cap] candidate source index i
    int32_t* thr;             // [1] threshold bucket
    int32_t* odd;             // [1] some ratio's bits do not order like its bucket (NaN or a set sign)
    float4* pa;               // [n_tau] source end point of each selected correspondence
    float4* pb;               // [n_tau] target end point
    uint32_t* adj;            // [n_tau][words]
    uint16_t* core;           // [n_tau, padded to 8] working values
    uint32_t* sync;           // barrier arrivals (changed blocks in the high half); at [kSyncGen] its generation
};

__device__ __forceinline__ int64_t corr_count(const int64_t* d_n, int64_t cap)
{
    if (!d_n) return cap;
    const int64_t n = *d_n;
    return n < 0 ? 0 : (n > cap ? cap : n);
}

__global__ void __launch_bounds__(kThreads) ratio_keys(const kmx_corr* __restrict__ corr, int64_t cap,
                                                      const int64_t* d_n, PruneScratch s)
{
    const int64_t n = corr_count(d_n, cap);
    for (int64_t k = (int64_t)blockIdx.x * kThreads + threadIdx.x; k < n; k += (int64_t)gridDim.x * kThreads) {
        const double d1 = (double)corr[k].d1, d2 = (double)corr[k].d2;
        const double r = d2 > 0.0 ? __ddiv_rn(d1, d2) : 1.0;
        s.ratio[k] = r;
        int b = (int)(r * (double)kBuckets);  // r in [0, 1]; exact scaling by a power of two
        b = b < 0 ? 0 : (b >= kBuckets ? kBuckets - 1 : b);
        s.bucket[k] = b;
        if (!(r >= 0.0) || signbit(r)) *s.odd = 1;
        atomicAdd(&s.hist[b], 1);
    }
}

// exclusive prefix over the CTA's 1024 threads
__device__ __forceinline__ int32_t block_prefix(int32_t x, int32_t* wsum)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    int32_t before = 0;
    if (lane < warp) before = wsum[lane];
    before = __reduce_add_sync(0xffffffffu, before);
    return before + inc - x;
}

__global__ void __launch_bounds__(1024) ratio_threshold(const int64_t* d_n, int64_t cap, int32_t n_tau, PruneScratch s,
                                                        int64_t* __restrict__ n_sel)
{
    __shared__ int32_t wsum[32];
    constexpr int kPer = kBuckets / 1024;
    static_assert(kPer == 4, "one int4 per thread");
    const int4 h = reinterpret_cast<const int4*>(s.hist)[threadIdx.x];
    const int32_t f0 = block_prefix(h.x + h.y + h.z + h.w, wsum);
    const int32_t f1 = f0 + h.x, f2 = f1 + h.y, f3 = f2 + h.z, f4 = f3 + h.w;
    reinterpret_cast<int4*>(s.first)[threadIdx.x] = make_int4(f0, f1, f2, f3);
    if (threadIdx.x == 1023) {
        s.first[kBuckets] = f4;
        if (f4 < n_tau) *s.thr = kBuckets - 1;  // fewer than N_tau in all
        const int64_t n = corr_count(d_n, cap);
        *n_sel = n < n_tau ? n : n_tau;
    }
    if (f0 < n_tau && f4 >= n_tau) *s.thr = threadIdx.x * kPer + (f1 >= n_tau ? 0 : f2 >= n_tau ? 1 : f3 >= n_tau ? 2 : 3);
}

__global__ void __launch_bounds__(kThreads) ratio_candidates(const kmx_corr* __restrict__ corr, int64_t cap,
                                                            const int64_t* d_n, PruneScratch s)
{
    const int64_t n = corr_count(d_n, cap);
    const int32_t thr = *s.thr;
    for (int64_t k = (int64_t)blockIdx.x * kThreads + threadIdx.x; k < n; k += (int64_t)gridDim.x * kThreads) {
        const int b = s.bucket[k];
        if (b > thr) continue;
        const int c = s.first[b] + atomicSub(&s.hist[b], 1) - 1;
        s.cand[c] = (int32_t)k;
        s.ckey[c] = (unsigned long long)__double_as_longlong(s.ratio[k]);
        s.ci[c] = corr[k].i;
    }
}

// (ratio, i) lexicographic: a non-negative double orders like its bits.
__device__ __forceinline__ bool key_less(unsigned long long ra, int32_t ia, unsigned long long rb, int32_t ib)
{
    return ra < rb || (ra == rb && ia < ib);
}

// One warp per candidate: its rank among its bucket's (the lanes stride over
// the compact keys), after the buckets below.
__global__ void __launch_bounds__(kThreads) ratio_rank(const kmx_corr* __restrict__ corr, int32_t n_tau,
                                                      const float4* __restrict__ src4,
                                                      const float4* __restrict__ tgt4, PruneScratch s,
                                                      int32_t* __restrict__ sel)
{
    const int m = s.first[*s.thr + 1];
    const int lane = threadIdx.x & 31;
    const int warps = gridDim.x * (kThreads / 32);
    for (int c = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5); c < m; c += warps) {
        const int32_t k = s.cand[c];
        const unsigned long long rk = s.ckey[c];
        const int32_t ik = s.ci[c];
        const kmx_corr e = corr[k];
        const int b = s.bucket[k];
        const bool odd = *s.odd != 0;
        const int f0 = odd ? 0 : s.first[b], f1 = odd ? m : s.first[b + 1];
        int rank = 0;
        for (int f = f0 + lane; f < f1; f += 32) rank += key_less(s.ckey[f], s.ci[f], rk, ik);
        rank = f0 + __reduce_add_sync(0xffffffffu, rank);
        if (rank < n_tau) {
            if (lane == 0) {
                sel[rank] = k;
                s.pa[rank] = src4[e.i];
            } else if (lane == 1) {
                s.pb[rank] = tgt4[e.j];
            }
        }
    }
}

__device__ __forceinline__ float sqrt_approx(float x)
{
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ bool edge_fp64(float4 a, float4 a2, float4 b, float4 b2, double two_beta)
{
    const double ax = (double)a.x - (double)a2.x, ay = (double)a.y - (double)a2.y, az = (double)a.z - (double)a2.z;
    const double bx = (double)b.x - (double)b2.x, by = (double)b.y - (double)b2.y, bz = (double)b.z - (double)b2.z;
    const double da = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(ax, ax), __dmul_rn(ay, ay)), __dmul_rn(az, az)));
    const double db = __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(bx, bx), __dmul_rn(by, by)), __dmul_rn(bz, bz)));
    return fabs(__dadd_rn(db, -da)) <= two_beta;
}

// One warp per pair of 32-vertex blocks (bv >= bu): lane = vertex of bv, its
// word for the block bu; the ballot over the lanes is the word of each vertex of
// bu for the block bv, so every pair is tested once.  Bound by instruction issue
// and the latency of the warp's uniform loads; 3000 vertices with every word
// from its own 32 tests took 24 us, this form 15 us.
__global__ void __launch_bounds__(kThreads) graph_build(int32_t n_tau, const int64_t* d_n_sel, double two_beta,
                                                       PruneScratch s, int32_t words)
{
    const int nsel = (int)*d_n_sel;
    const int nb = (nsel + 31) / 32;
    const int64_t total = (int64_t)nb * (nb + 1) / 2;
    const float tb = (float)two_beta;
    const int lane = threadIdx.x & 31;
    for (int64_t t = (int64_t)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5); t < total;
         t += (int64_t)gridDim.x * (kThreads / 32)) {
        // t = bv (bv + 1) / 2 + bu
        int bv = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
        while ((int64_t)(bv + 1) * (bv + 2) / 2 <= t) ++bv;
        while ((int64_t)bv * (bv + 1) / 2 > t) --bv;
        const int bu = (int)(t - (int64_t)bv * (bv + 1) / 2);
        const int v = bv * 32 + lane;
        const bool valid = v < nsel;
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 a = valid ? s.pa[v] : zero, b = valid ? s.pb[v] : zero;
        uint32_t bits = 0, back = 0;
        const int last = min(32, nsel - bu * 32);
#pragma unroll 4
        for (int e = 0; e < last; ++e) {
            const int u = bu * 32 + e;
            const float4 a2 = s.pa[u], b2 = s.pb[u];
            const float ax = a.x - a2.x, ay = a.y - a2.y, az = a.z - a2.z;
            const float bx = b.x - b2.x, by = b.y - b2.y, bz = b.z - b2.z;
            const float da = sqrt_approx(fmaf(az, az, fmaf(ay, ay, ax * ax)));
            const float db = sqrt_approx(fmaf(bz, bz, fmaf(by, by, bx * bx)));
            const float gap = fabsf(db - da) - tb;
            // FP32 carries a few ulp of the distances (the approximate root,
            // which halves the instructions of a pair, one more); decide again
            // in FP64 near the threshold
            const float band = 1e-5f * (1.0f + da + db);
            bool on = gap < -band;
            if (!on && !(gap > band)) on = edge_fp64(a, a2, b, b2, two_beta);
            on = on && valid && u != v;
            const unsigned all = __ballot_sync(0xffffffffu, on);
            bits |= (uint32_t)on << e;
            if (lane == e) back = all;
        }
        if (valid) s.adj[(int64_t)v * words + bu] = bits;
        if (bu != bv && lane < last) s.adj[(int64_t)(bu * 32 + lane) * words + bv] = back;
    }
}

__device__ __forceinline__ uint32_t ld_volatile(const uint32_t* p) { return *reinterpret_cast<const volatile uint32_t*>(p); }

// Bounded grid barrier (generation `round` + 1 once every block has arrived);
// `changed` of any block reaches all of them as *any.  False when a spin ran out.
__device__ bool grid_barrier(uint32_t* sync, uint32_t nblocks, uint32_t round, bool changed, bool* any)
{
    __shared__ uint32_t state;
    const int mine = __syncthreads_or(changed);
    if (threadIdx.x == 0) {
        const uint32_t want = round + 1;
        uint32_t seen;
        __threadfence();
        const uint32_t add = mine ? 0x10001u : 1u;
        const uint32_t sum = atomicAdd(sync, add) + add;
        if ((sum & 0xffffu) == nblocks) {
            seen = want | (sum >> 16 ? 0x80000000u : 0u);
            atomicExch(sync, 0u);
            __threadfence();
            atomicExch(sync + kSyncGen, seen);
        } else {
            uint32_t it = 0;
            while (((seen = ld_volatile(sync + kSyncGen)) & 0x7fffffffu) != want) {
                if (++it > kSpinLimit) {
                    seen = 0xffffffffu;
                    break;
                }
            }
        }
        __threadfence();
        state = seen;
    }
    __syncthreads();
    const uint32_t st = state;
    *any = (st >> 31) != 0;
    return st != 0xffffffffu;
}

// values of a snapshot: n_tau rounded up to whole words of the bit rows
__host__ __device__ constexpr int32_t snap_len(int32_t n_tau) { return (n_tau + 31) / 32 * 32; }

struct CoreVertex {
    int32_t c;      // current value
    int32_t deg;
    int32_t start;  // of the neighbour list in the warp's part, -1: the list did not fit
};

// The values of a vertex's neighbours for the counts of one visit: per lane in
// registers up to 32 kHeld neighbours, else read again for every count, from the
// list or by the bit row.
constexpr int kHeld = 16;
struct Neighbours {
    int held[kHeld];
    const uint16_t* list;
    const uint32_t* row;
    const uint16_t* snap;
    int deg, words;

    __device__ __forceinline__ void load()
    {
        const int lane = threadIdx.x & 31;
        if (!list || deg > 32 * kHeld) return;
#pragma unroll
        for (int e = 0; e < kHeld; ++e)
            if (32 * e < deg) held[e] = 32 * e + lane < deg ? snap[list[32 * e + lane]] : -1;
    }

    // number of neighbours with a value >= h > 0 (warp-wide, every lane gets it)
    __device__ __forceinline__ int count_ge(int h) const
    {
        const int lane = threadIdx.x & 31;
        int cnt = 0;
        if (list && deg <= 32 * kHeld) {
#pragma unroll
            for (int e = 0; e < kHeld; ++e)
                if (32 * e < deg) cnt += held[e] >= h;
        } else if (list) {
#pragma unroll 4
            for (int e = lane; e < deg; e += 32) cnt += snap[list[e]] >= h;
        } else {
            for (int w = lane; w < words; w += 32) {
                uint32_t bits = row[w];
                while (bits) {
                    const int e = __ffs(bits) - 1;
                    bits &= bits - 1;
                    cnt += snap[w * 32 + e] >= h;
                }
            }
        }
        return __reduce_add_sync(0xffffffffu, cnt);
    }
};

// One warp per vertex (per_warp of them at most), whose neighbour list it keeps
// in shared memory as 16-bit indices.  A pass reads all values (2 n bytes from
// L2) and lowers the CTA's own; passes of different CTAs are not ordered, and
// only the barrier after kPasses of them decides whether anything still moves
// (a round without a change saw the same values in all its passes).  What
// bounds it: the L2 round trip of a pass and the barrier's.  Before, a pass took
// vertices from a global counter, walked 32-bit rows in L2 and ended in a
// barrier: 3000 vertices of 160 neighbours took 1042 us; with lists and four
// passes to a barrier 263 us, with the values of a visit held in registers and three passes
// 245 us.
__global__ void __launch_bounds__(kCoreThreads, 1) kcore(const int64_t* d_n_sel, int32_t words, int32_t per_warp,
                                                         int32_t list_len, PruneScratch s,
                                                         int32_t* __restrict__ core_out, int32_t* __restrict__ kmax_out,
                                                         int32_t* __restrict__ inlier, int64_t* __restrict__ n_inlier,
                                                         unsigned int* __restrict__ err)
{
    const int n = (int)*d_n_sel;
    const int n_words = (n + 31) / 32;  // of the row's `words` (graph_build writes no others)
    const uint32_t nblocks = gridDim.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // dynamic shared memory: the values at the start of a pass, the warps'
    // vertices, their neighbour lists
    extern __shared__ __align__(16) uint8_t dyn[];
    uint16_t* snap = reinterpret_cast<uint16_t*>(dyn);
    const int n8 = (n + 7) / 8;
    CoreVertex* vert = reinterpret_cast<CoreVertex*>(dyn + sizeof(uint16_t) * snap_len(words * 32));
    uint16_t* list = reinterpret_cast<uint16_t*>(vert + kCoreWarps * per_warp) + (size_t)warp * list_len;
    vert += warp * per_warp;
    // vertex k of the warp
    const int step = kCoreWarps * (int)nblocks, v0 = warp * (int)nblocks + (int)blockIdx.x;
    int used = 0;
    for (int k = 0, v = v0; v < n; ++k, v += step) {
        const uint32_t* row = s.adj + (int64_t)v * words;
        int deg = 0;
        for (int w0 = 0; w0 < n_words; w0 += 32) {
            uint32_t bits = w0 + lane < n_words ? row[w0 + lane] : 0u;
            const int mine = __popc(bits);
            int inc = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += y;
            }
            int at = used + deg + inc - mine;
            while (bits) {
                const int e = __ffs(bits) - 1;
                bits &= bits - 1;
                if (at < list_len) list[at] = (uint16_t)((w0 + lane) * 32 + e);
                ++at;
            }
            deg += __shfl_sync(0xffffffffu, inc, 31);
        }
        const bool fits = used + deg <= list_len;
        if (lane == 0) {
            vert[k] = CoreVertex{deg, deg, fits ? used : -1};
            *reinterpret_cast<volatile uint16_t*>(s.core + v) = (uint16_t)deg;
        }
        if (fits) used += deg;
        __syncwarp();
    }
    bool any = false;
    bool ok = grid_barrier(s.sync, nblocks, 0, false, &any);
    for (uint32_t round = 1; ok && round <= kMaxRounds; ++round) {
        bool changed = false;
        for (int pass = 0; pass < kPasses; ++pass) {
            for (int i = tid; i < n8; i += kCoreThreads) {
                uint4 q;
                asm volatile("ld.relaxed.gpu.global.v4.u32 {%0, %1, %2, %3}, [%4];"
                             : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w)
                             : "l"(reinterpret_cast<const uint4*>(s.core) + i)
                             : "memory");
                reinterpret_cast<uint4*>(snap)[i] = q;
            }
            __syncthreads();
            for (int k = 0, v = v0; v < n; ++k, v += step) {
                const CoreVertex x = vert[k];
                if (x.c == 0) continue;
                Neighbours nb;
                nb.list = x.start >= 0 ? list + x.start : nullptr;
                nb.row = s.adj + (int64_t)v * words;
                nb.snap = snap;
                nb.deg = x.deg;
                nb.words = n_words;
                nb.load();
                // count_ge falls as h grows: with `lo` values >= c, at least
                // `lo` are >= lo
                int lo = nb.count_ge(x.c);
                if (lo >= x.c) continue;
                int hi = x.c - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (nb.count_ge(mid) >= mid)
                        lo = mid;
                    else
                        hi = mid - 1;
                }
                if (lane == 0) {
                    vert[k].c = lo;
                    *reinterpret_cast<volatile uint16_t*>(s.core + v) = (uint16_t)lo;
                }
                __syncwarp();
                changed = true;
            }
            __syncthreads();  // the values are read before the next pass overwrites them
        }
        ok = grid_barrier(s.sync, nblocks, round, changed, &any);
        if (!any) break;
    }
    if (!ok || any) {
        if (tid == 0) kmx_raise(err, KMX_DERR_TIMEOUT);
        return;
    }
    if (blockIdx.x != 0) return;
    // block 0: largest core number, then the maximum k-core in ascending order
    // (the last round changed nothing: snap holds the core numbers)
    __shared__ int32_t wsum[kCoreWarps];
    int32_t mx = 0;
    for (int v = tid; v < n; v += kCoreThreads) {
        const int32_t cv = snap[v];
        core_out[v] = cv;
        mx = max(mx, cv);
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) wsum[warp] = mx;
    __syncthreads();
    const int32_t kmax = __reduce_max_sync(0xffffffffu, wsum[lane]);
    __syncthreads();
    int32_t base = 0;
    for (int b = 0; b < n; b += kCoreThreads) {
        const int v = b + tid;
        const bool in = v < n && snap[v] == kmax;
        const int32_t at = base + block_prefix(in, wsum);
        if (in) inlier[at] = v;
        base += __syncthreads_count(in);
    }
    if (tid == 0) {
        *kmax_out = kmax;
        *n_inlier = base;
    }
}

int32_t words_for(int32_t n_tau) { return (n_tau + 31) / 32; }

size_t zero_bytes() { return sizeof(int32_t) * (kBuckets + 2 + kSyncGen + 1); }

PruneScratch carve(void* base, int64_t cap, int32_t n_tau, size_t* total)
{
    kmx_arena a{static_cast<char*>(base), 0};
    PruneScratch s{};
    s.ratio = static_cast<double*>(a.take(sizeof(double) * (cap + 1)));
    s.bucket = static_cast<int32_t*>(a.take(sizeof(int32_t) * (cap + 1)));
    s.cand = static_cast<int32_t*>(a.take(sizeof(int32_t) * (cap + 1)));
    s.ckey = static_cast<unsigned long long*>(a.take(sizeof(unsigned long long) * (cap + 1)));
    s.ci = static_cast<int32_t*>(a.take(sizeof(int32_t) * (cap + 1)));
    s.pa = static_cast<float4*>(a.take(sizeof(float4) * (n_tau + 1)));
    s.pb = static_cast<float4*>(a.take(sizeof(float4) * (n_tau + 1)));
    s.adj = static_cast<uint32_t*>(a.take(sizeof(uint32_t) * ((size_t)n_tau * words_for(n_tau) + 1)));
    s.first = static_cast<int32_t*>(a.take(sizeof(int32_t) * (kBuckets + 1)));
    s.core = static_cast<uint16_t*>(a.take(sizeof(uint16_t) * (size_t)snap_len(n_tau)));
    // zeroed together: histogram, threshold, odd flag, sync words
    int32_t* z = static_cast<int32_t*>(a.take(zero_bytes()));
    s.hist = z;
    s.thr = z + kBuckets;
    s.odd = z + kBuckets + 1;
    s.sync = reinterpret_cast<uint32_t*>(z + kBuckets + 2);
    *total = kmx_align_up(a.used, 256);
    return s;
}

}  // namespace

size_t kmx_prune_scratch_bytes(int64_t corr_cap, int32_t n_tau)
{
    size_t total = 0;
    carve(nullptr, corr_cap, n_tau, &total);
    return total;
}

cudaError_t kmx_prune_launch(kmx_ctx* ctx, const kmx_corr* corr, int64_t cap, const int64_t* d_n,
                             const float4* src4, const float4* tgt4, int32_t n_tau, double beta, int32_t* sel,
                             int64_t* n_sel, int32_t* core_out, int32_t* kmax, int32_t* inlier, int64_t* n_inlier,
                             void* scratch)
{
    cudaStream_t st = ctx->stream;
    size_t total = 0;
    PruneScratch s = carve(scratch, cap, n_tau, &total);
    cudaError_t e;
    if ((e = cudaMemsetAsync(s.hist, 0, zero_bytes(), st))) return e;
    const unsigned grid = 4u * (unsigned)ctx->sm_count;
    KMX_COUNT_LAUNCH();
    ratio_keys<<<grid, kThreads, 0, st>>>(corr, cap, d_n, s);
    KMX_COUNT_LAUNCH();
    ratio_threshold<<<1, 1024, 0, st>>>(d_n, cap, n_tau, s, n_sel);
    KMX_COUNT_LAUNCH();
    ratio_candidates<<<grid, kThreads, 0, st>>>(corr, cap, d_n, s);
    KMX_COUNT_LAUNCH();
    ratio_rank<<<grid, kThreads, 0, st>>>(corr, n_tau, src4, tgt4, s, sel);
    const int32_t words = words_for(n_tau);
    KMX_COUNT_LAUNCH();
    graph_build<<<2 * grid, kThreads, 0, st>>>(n_tau, n_sel, 2.0 * beta, s, words);
    // one CTA per SM (co-resident under a cooperative launch: the rounds wait
    // on one another through the grid barrier)
    const unsigned kgrid = (unsigned)ctx->sm_count;
    const int per_warp = (n_tau + kCoreWarps * (int)kgrid - 1) / (kCoreWarps * (int)kgrid);
    const size_t fixed = sizeof(uint16_t) * (size_t)snap_len(n_tau) + sizeof(CoreVertex) * kCoreWarps * (size_t)per_warp;
    // 16384 vertices of four a warp take 34 KB of it
    const size_t smem = kCoreSmem > fixed ? kCoreSmem : fixed;
    const int list_len = (int)((smem - fixed) / (sizeof(uint16_t) * kCoreWarps));
    if ((e = kmx_once_per_device(kmx_attr_kcore, [] {
            return cudaFuncSetAttribute(kcore, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024 - 1024);
        })))
        return e;
    const int64_t* n_sel_c = n_sel;
    int32_t words_c = words, per_warp_c = per_warp, list_len_c = list_len;
    unsigned int* err = ctx->d_err;
    void* args[] = {(void*)&n_sel_c, (void*)&words_c, (void*)&per_warp_c, (void*)&list_len_c, (void*)&s, (void*)&core_out,
                    (void*)&kmax, (void*)&inlier, (void*)&n_inlier, (void*)&err};
    KMX_COUNT_LAUNCH();
    return cudaLaunchCooperativeKernel((const void*)kcore, dim3(kgrid), dim3(kCoreThreads), args, smem, st);
}
