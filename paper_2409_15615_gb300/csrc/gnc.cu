// Robust pose from the pruned correspondences (Sec. III-E): graduated
// non-convexity with the truncated-least-squares loss (GNC-TLS, Yang et al.,
// RA-L 2020) around a weighted closed-form rigid alignment (Horn 1987, unit
// quaternions).
//
// One CTA per problem (the maximum k-core holds a few thousand
// correspondences).  The points sit in shared memory, centred on their
// unweighted centroids (taken in FP64), so the FP32 residuals and moments
// carry only the spread of the cloud; the block reductions end in FP64.  The
// GNC schedule is the one of the paper's solver:
// weights w = 1 first; mu = c^2 / (2 r_max^2 - c^2); each iteration sets
// w = 1 for r^2 <= mu/(mu+1) c^2, 0 for r^2 >= (mu+1)/mu c^2 and
// c sqrt(mu (mu+1)) / r - mu between, refits, and multiplies mu by the
// factor; it stops when fewer than 3 weights are positive (keeping the
// previous fit) or when the weighted cost repeats within tol.
//
// What bounds it: one CTA's serial chain.  An FP64 instruction occupies its
// pipe for tens of cycles whatever the number of active lanes, so FP64 work is
// laid across lanes and out of the threads that do not need it: the schedule's
// roots and divisions for 32 iterations at a time (they do not depend on the
// data), the warp sums' tree with a few lanes per total, centroids, covariance
// and rotation with a lane per entry.  One pass over the points per iteration
// forms the residuals, the cost of the last fit, the next weights and their
// moments, with one reduction.  269 points, 22 iterations: 570 -> 203 us.
#include "kmx_internal.cuh"

namespace {

constexpr int kThreads = 512;
constexpr int kMaxPoints = 4096;
constexpr int kWarpsG = kThreads / 32;

struct GncOut {
    double* R;       // [9] row-major
    double* t;       // [3]
    float* w;        // [cap] final weights
    int32_t* stats;  // [4]: iterations, weights > 0.5, points, status (0 ok, 1 fewer than 3 points, 2 too many)
};

constexpr int kSums = 18;  // 16 moments, the weighted cost, the positive weights

struct Shared {
    float part[kWarpsG][kSums + 1];  // warp sums (stride 19: no bank conflicts)
    double tot[kSums];               // block sums
    float4 sched[32];                // lo, hi, c sqrt(mu (mu+1)), mu of 32 iterations
    float R[9];                      // current rotation (FP32, for the residuals)
    float tc[3];                     // translation in the centred frame: b' = R a' + tc
    double Rd[9];                    // current rotation, FP64 copy for the output
    double ca[6];                    // weighted centroids of a and b
    float H[9];                      // weighted cross-covariance
    float q[4];                      // the quaternion
    int32_t count[kWarpsG];
};

// One step of a warp's sum of N values per lane: the lanes with bit O keep the
// upper half of the values, the others the lower half, each added to the other
// side's.  After O = 16, 8, 4, 2, 1 from 16 values lane pairs hold one whole sum
// each, added in the order of a butterfly over every value.
template <int N, int O>
__device__ __forceinline__ void sum_step(float (&v)[16], int lane)
{
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        const bool up = (lane & O) != 0;
        const float keep = up ? v[i + N / 2] : v[i], give = up ? v[i] : v[i + N / 2];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, give, O);
    }
}

// Warp sums of v[0..15], cost and npos into S.part[warp].
__device__ __forceinline__ void warp_sums(float (&v)[16], float cost, float npos, Shared& S)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    sum_step<16, 16>(v, lane);
    sum_step<8, 8>(v, lane);
    sum_step<4, 4>(v, lane);
    sum_step<2, 2>(v, lane);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        cost += __shfl_xor_sync(0xffffffffu, cost, o);
        npos += __shfl_xor_sync(0xffffffffu, npos, o);
    }
    // bit 4 of the lane chose the upper eight values, bit 3 the upper four of those, ...
    const int i = ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 + ((lane >> 1) & 1);
    if (!(lane & 1)) S.part[warp][i] = v[0];
    if (lane == 0) S.part[warp][16] = cost;
    if (lane == 1) S.part[warp][17] = npos;
}

// Block sums in FP64 of the warp sums: warps 0..4 take four sums each, eight
// lanes per sum.  Ends with a barrier; S.tot holds them.
__device__ __forceinline__ void block_sums(Shared& S)
{
    static_assert(kWarpsG == 16, "eight lanes per sum add two warps each");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (warp < (kSums + 3) / 4) {
        const int i = warp * 4 + (lane >> 3), w = lane & 7;
        double y = 0.0;
        if (i < kSums) y = (double)S.part[w][i] + (double)S.part[w + 8][i];
#pragma unroll
        for (int o = 4; o >= 1; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
        if (i < kSums && w == 0) S.tot[i] = y;
    }
    __syncthreads();
}

// Eigenvector of the largest eigenvalue of a symmetric 4 x 4 matrix (cyclic
// Jacobi rotations).
__device__ void jacobi4_max(float (&A)[4][4], float (&q)[4])
{
    float V[4][4] = {{1.f, 0.f, 0.f, 0.f}, {0.f, 1.f, 0.f, 0.f}, {0.f, 0.f, 1.f, 0.f}, {0.f, 0.f, 0.f, 1.f}};
    // every index below is a compile-time constant after unrolling, so the
    // two matrices stay in registers
    for (int sweep = 0; sweep < 12; ++sweep) {
        float off = 0.f, diag = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            diag += A[i][i] * A[i][i];
#pragma unroll
            for (int j = i + 1; j < 4; ++j) off += A[i][j] * A[i][j];
        }
        if (off <= 1e-14f * diag) break;
#pragma unroll
        for (int p = 0; p < 3; ++p) {
#pragma unroll
            for (int r = p + 1; r < 4; ++r) {
                const float apr = A[p][r];
                if (apr == 0.f) continue;
                const float theta = (A[r][r] - A[p][p]) / (2.f * apr);
                const float tt = (theta >= 0.f ? 1.f : -1.f) / (fabsf(theta) + sqrtf(theta * theta + 1.f));
                const float c = 1.f / sqrtf(tt * tt + 1.f), s = tt * c;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float akp = A[k][p], akr = A[k][r];
                    A[k][p] = c * akp - s * akr;
                    A[k][r] = s * akp + c * akr;
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float apk = A[p][k], ark = A[r][k];
                    A[p][k] = c * apk - s * ark;
                    A[r][k] = s * apk + c * ark;
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float vkp = V[k][p], vkr = V[k][r];
                    V[k][p] = c * vkp - s * vkr;
                    V[k][r] = s * vkp + c * vkr;
                }
            }
        }
    }
    float bestv = A[0][0];
    float qv[4] = {V[0][0], V[1][0], V[2][0], V[3][0]};
#pragma unroll
    for (int i = 1; i < 4; ++i) {
        if (A[i][i] > bestv) {
            bestv = A[i][i];
#pragma unroll
            for (int k = 0; k < 4; ++k) qv[k] = V[k][i];
        }
    }
    float nrm = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) nrm += qv[k] * qv[k];
    nrm = 1.f / sqrtf(nrm);
#pragma unroll
    for (int k = 0; k < 4; ++k) q[k] = qv[k] * nrm;
}

// Per-point state in dynamic shared memory (struct of arrays).
struct Pts {
    float* ax;
    float* ay;
    float* az;
    float* bx;
    float* by;
    float* bz;
};

__device__ __forceinline__ void add_moments(float (&v)[16], const Pts& P, int k, float wk)
{
    const float ax = P.ax[k], ay = P.ay[k], az = P.az[k], bx = P.bx[k], by = P.by[k], bz = P.bz[k];
    v[0] += wk;
    v[1] += wk * ax;
    v[2] += wk * ay;
    v[3] += wk * az;
    v[4] += wk * bx;
    v[5] += wk * by;
    v[6] += wk * bz;
    v[7] += wk * ax * bx;
    v[8] += wk * ax * by;
    v[9] += wk * ax * bz;
    v[10] += wk * ay * bx;
    v[11] += wk * ay * by;
    v[12] += wk * ay * bz;
    v[13] += wk * az * bx;
    v[14] += wk * az * by;
    v[15] += wk * az * bz;
}

// Weighted fit in the centred frame from the moments in S.tot: Horn's
// quaternion, rotation and translation.  Warp 0 works, one lane per entry;
// ends with a barrier.
__device__ void fit(Shared& S)
{
    const int lane = threadIdx.x & 31;
    if (threadIdx.x < 32) {
        const double sw = S.tot[0] > 0.0 ? S.tot[0] : 1.0;
        if (lane < 6) S.ca[lane] = S.tot[1 + lane] / sw;
        __syncwarp();
        const int e = lane < 9 ? lane : 8, i = e / 3, j = e - 3 * i;
        // centred cross-covariance S_ij = sum w (a_i - ca_i)(b_j - cb_j)
        const float h = (float)(S.tot[7 + e] - sw * S.ca[i] * S.ca[3 + j]);
        if (lane < 9) S.H[lane] = h;
        __syncwarp();
        if (lane == 0) {
            const float Sxx = S.H[0], Sxy = S.H[1], Sxz = S.H[2];
            const float Syx = S.H[3], Syy = S.H[4], Syz = S.H[5];
            const float Szx = S.H[6], Szy = S.H[7], Szz = S.H[8];
            float N[4][4] = {{Sxx + Syy + Szz, Syz - Szy, Szx - Sxz, Sxy - Syx},
                             {Syz - Szy, Sxx - Syy - Szz, Sxy + Syx, Szx + Sxz},
                             {Szx - Sxz, Sxy + Syx, -Sxx + Syy - Szz, Syz + Szy},
                             {Sxy - Syx, Szx + Sxz, Syz + Szy, -Sxx - Syy + Szz}};
            float q[4];
            jacobi4_max(N, q);
#pragma unroll
            for (int k = 0; k < 4; ++k) S.q[k] = q[k];
        }
        __syncwarp();
        // R = (q0^2 - |v|^2) I + 2 v v^T + 2 q0 [v]x, one entry per lane
        const double q0 = S.q[0], vi = S.q[1 + i], vj = S.q[1 + j];
        double r;
        if (i == j) {
            const double va = S.q[1 + (i + 1) % 3], vb = S.q[1 + (i + 2) % 3];
            r = q0 * q0 + vi * vi - va * va - vb * vb;
        } else {
            const double vk = S.q[1 + 3 - i - j];
            const double turn = q0 * vk;
            r = 2 * (vi * vj + ((j + 3 - i) % 3 == 1 ? -turn : turn));
        }
        if (lane < 9) {
            S.Rd[lane] = r;
            S.R[lane] = (float)r;
        }
        __syncwarp();
        if (lane < 3)
            S.tc[lane] = (float)(S.ca[3 + lane] - (S.Rd[3 * lane] * S.ca[0] + S.Rd[3 * lane + 1] * S.ca[1] +
                                                   S.Rd[3 * lane + 2] * S.ca[2]));
    }
    __syncthreads();
}

__device__ __forceinline__ float resid2(const Shared& S, float ax, float ay, float az, float bx, float by, float bz)
{
    const float rx = bx - (S.R[0] * ax + S.R[1] * ay + S.R[2] * az) - S.tc[0];
    const float ry = by - (S.R[3] * ax + S.R[4] * ay + S.R[5] * az) - S.tc[1];
    const float rz = bz - (S.R[6] * ax + S.R[7] * ay + S.R[8] * az) - S.tc[2];
    return rx * rx + ry * ry + rz * rz;
}

__global__ void __launch_bounds__(kThreads, 1)
    gnc_tls(const kmx_corr* __restrict__ corr, const int32_t* __restrict__ sel, const int32_t* __restrict__ inlier,
            const int64_t* __restrict__ d_n, int64_t cap, const float4* __restrict__ src4,
            const float4* __restrict__ tgt4, double c2, int max_iters, double mu_factor, double tol, GncOut o,
            unsigned int* err)
{
    __shared__ Shared S;
    const int64_t n64 = d_n ? min(*d_n, cap) : cap;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (n64 > (int64_t)kMaxPoints) {  // more points than shared memory holds
        if (tid == 0) {
            kmx_raise(err, KMX_DERR_CAPACITY);
            o.stats[3] = 2;
        }
        return;
    }
    const int n = (int)n64;
    if (n < 3) {
        if (tid == 0) {
            for (int i = 0; i < 9; ++i) o.R[i] = (i % 4 == 0) ? 1.0 : 0.0;
            o.t[0] = o.t[1] = o.t[2] = 0.0;
            o.stats[0] = 0;
            o.stats[1] = 0;
            o.stats[2] = n;
            o.stats[3] = 1;
        }
        for (int k = tid; k < n; k += kThreads) o.w[k] = 0.f;
        return;
    }
    extern __shared__ float dyn[];
    const Pts P{dyn, dyn + kMaxPoints, dyn + 2 * kMaxPoints, dyn + 3 * kMaxPoints, dyn + 4 * kMaxPoints,
                dyn + 5 * kMaxPoints};
    float* w = dyn + 6 * kMaxPoints;       // the weights of the latest fit
    float* w_next = dyn + 7 * kMaxPoints;  // the next ones
    // unweighted centroids in FP64, the reference frame of the FP32 work:
    // offsets from the first point are summed, then it is added back
    const kmx_corr c0 = corr[sel[inlier[0]]];
    const float4 a0 = src4[c0.i], b0 = tgt4[c0.j];
    float v[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = 0.f;
    for (int k = tid; k < n; k += kThreads) {
        const kmx_corr c = corr[sel[inlier[k]]];
        const float4 a = src4[c.i], b = tgt4[c.j];
        P.ax[k] = a.x;  // raw for now, centred below
        P.ay[k] = a.y;
        P.az[k] = a.z;
        P.bx[k] = b.x;
        P.by[k] = b.y;
        P.bz[k] = b.z;
        v[0] += a.x - a0.x;
        v[1] += a.y - a0.y;
        v[2] += a.z - a0.z;
        v[3] += b.x - b0.x;
        v[4] += b.y - b0.y;
        v[5] += b.z - b0.z;
    }
    warp_sums(v, 0.f, 0.f, S);
    block_sums(S);
    double ca0[3], cb0[3];
    {
        const float first[6] = {a0.x, a0.y, a0.z, b0.x, b0.y, b0.z};
        if (tid < 6) S.ca[tid] = (double)first[tid] + S.tot[tid] / n;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            ca0[i] = S.ca[i];
            cb0[i] = S.ca[3 + i];
        }
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = 0.f;
    for (int k = tid; k < n; k += kThreads) {
        P.ax[k] = (float)((double)P.ax[k] - ca0[0]);
        P.ay[k] = (float)((double)P.ay[k] - ca0[1]);
        P.az[k] = (float)((double)P.az[k] - ca0[2]);
        P.bx[k] = (float)((double)P.bx[k] - cb0[0]);
        P.by[k] = (float)((double)P.by[k] - cb0[1]);
        P.bz[k] = (float)((double)P.bz[k] - cb0[2]);
        w[k] = 1.f;
        add_moments(v, P, k, 1.f);
    }
    warp_sums(v, 0.f, 0.f, S);
    block_sums(S);
    fit(S);
    float rmax = 0.f;
    for (int k = tid; k < n; k += kThreads)
        rmax = fmaxf(rmax, resid2(S, P.ax[k], P.ay[k], P.az[k], P.bx[k], P.by[k], P.bz[k]));
    {
        // residuals are >= 0 (or NaN, which fmaxf drops): their bits order like integers
        const unsigned wm = __reduce_max_sync(0xffffffffu, __float_as_uint(rmax));
        if (lane == 0) S.count[warp] = (int32_t)wm;
        __syncthreads();
        rmax = __uint_as_float(__reduce_max_sync(0xffffffffu, (unsigned)S.count[lane % kWarpsG]));
        __syncthreads();
    }
    int iters = 0;
    if ((double)rmax > c2) {
        double mu0 = c2 / fmax(2.0 * (double)rmax - c2, 1e-30);  // of the schedule's first entry
        double prev_cost = INFINITY;
        for (int it = 0; it < max_iters; ++it) {
            if ((it & 31) == 0) {
                // the schedule of 32 iterations, by as many lanes (every warp
                // has passed the last barrier, so the last entries are read)
                if (warp == 0) {
                    double mu = mu0;
                    for (int i = 0; i < lane; ++i) mu *= mu_factor;
                    S.sched[lane] = make_float4((float)(mu / (mu + 1.0) * c2), (float)((mu + 1.0) / mu * c2),
                                                (float)(sqrt(c2) * sqrt(mu * (mu + 1.0))), (float)mu);
                    mu0 = __shfl_sync(0xffffffffu, mu, 31) * mu_factor;
                }
                __syncthreads();
            }
            // residuals of the last fit, its cost, and the next weights with
            // their moments
            const float4 sc = S.sched[it & 31];
            float cost = 0.f, npos = 0.f;
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = 0.f;
            for (int k = tid; k < n; k += kThreads) {
                const float r = resid2(S, P.ax[k], P.ay[k], P.az[k], P.bx[k], P.by[k], P.bz[k]);
                cost += w[k] * r;
                const float wk = r <= sc.x ? 1.f : (r >= sc.y ? 0.f : sc.z / sqrtf(fmaxf(r, 1e-30f)) - sc.w);
                w_next[k] = wk;
                npos += wk > 0.f ? 1.f : 0.f;
                add_moments(v, P, k, wk);
            }
            warp_sums(v, cost, npos, S);
            block_sums(S);
            if (it > 0) {
                if (fabs(S.tot[16] - prev_cost) < tol) break;
                prev_cost = S.tot[16];
            }
            float* const t = w;
            w = w_next;
            w_next = t;
            if (S.tot[17] < 3.0) break;  // the current fit stays; w are the weights that stopped it
            fit(S);
            ++iters;
        }
    }
    // outputs: R, t in the original frame (b = R a + t with t = cb0 + tc - R ca0)
    int good = 0;
    for (int k = tid; k < n; k += kThreads) {
        const float wk = w[k];
        o.w[k] = wk;
        good += wk > 0.5f;
    }
    good = __reduce_add_sync(0xffffffffu, good);
    if (lane == 0) S.count[warp] = good;
    __syncthreads();
    if (tid == 0) {
        for (int i = 0; i < 9; ++i) o.R[i] = S.Rd[i];
        for (int i = 0; i < 3; ++i)
            o.t[i] = cb0[i] + (double)S.tc[i] -
                     (S.Rd[3 * i] * ca0[0] + S.Rd[3 * i + 1] * ca0[1] + S.Rd[3 * i + 2] * ca0[2]);
        o.stats[0] = iters;
        good = 0;
        for (int i = 0; i < kWarpsG; ++i) good += S.count[i];
        o.stats[1] = good;
        o.stats[2] = n;
        o.stats[3] = 0;
    }
}

size_t smem_bytes() { return sizeof(float) * 8 * (size_t)kMaxPoints; }

}  // namespace

int64_t kmx_gnc_max_points() { return kMaxPoints; }

cudaError_t kmx_gnc_launch(kmx_ctx* ctx, const kmx_corr* corr, const int32_t* sel, const int32_t* inlier,
                           const int64_t* d_n, int64_t cap, const float4* src4, const float4* tgt4, double noise_bound,
                           int max_iters, double mu_factor, double tol, double* R, double* t, float* w,
                           int32_t* stats)
{
    cudaError_t e = kmx_once_per_device(kmx_attr_gnc, [] {
        return cudaFuncSetAttribute(gnc_tls, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes());
    });
    if (e) return e;
    KMX_COUNT_LAUNCH();
    gnc_tls<<<1, kThreads, smem_bytes(), ctx->stream>>>(corr, sel, inlier, d_n, cap, src4, tgt4, noise_bound * noise_bound,
                                             max_iters, mu_factor, tol, GncOut{R, t, w, stats}, ctx->d_err);
    return cudaGetLastError();
}
