// Mini bundle adjustment of the initial pose estimation (Sec. 4.1 and App. A.1):
// Levenberg-Marquardt over a shared focal length, the poses of frames 1..F-1
// (frame 0 fixed: the gauge) and P points, each observed in all F frames - the
// fixed-size layout that makes every block of the problem a fixed-size
// computation. One iteration:
//   k_ba_begin      (one cluster) accepts or rejects the previous trial state,
//                   residual norms e of all P F observations, and the lower median
//                   of e and of |e - median| by radix select: median + 4 MAD
//   k_ba_points     each point's Huber-weighted 3x3 block (damped) and its inverse,
//                   gradient, coupling rows K (Nc x 3) and H_pp^-1 K
//   k_ba_normal     per chunk of 32 points: threads owning entries of the reduced
//                   camera system accumulate H_cc - sum_p K H_pp^-1 K^T and its
//                   right-hand side in FP64, in a fixed order (deterministic)
//   k_ba_reduce     fixed-order sum of the chunk partials
//   k_ba_solve      one CTA: Marquardt damping, L D L^T factorisation and the
//                   triangular solves in FP64, the trial cameras
//   k_ba_step       point steps dp = -H_pp^-1 (g_p + K^T dc), the trial points and
//                   the robust cost of the trial state on the same observation set
// and, after the last one, k_ba_sum and k_ba_accept. Problems with more
// observations than k_ba_begin's cluster holds in registers run its three parts as
// kernels of their own. Everything stays on the device, so the iterations can be
// captured into one CUDA graph and replayed without host work.
#include <cooperative_groups.h>
#include <mutex>
#include <type_traits>

#include "common.cuh"

namespace gs {

constexpr int kBaMaxF = 8;
constexpr int kBaMaxNc = 6 * (kBaMaxF - 1) + 1;  // 43 camera parameters

__device__ __forceinline__ int ba_nc(int F) { return 6 * (F - 1) + 1; }
__device__ __forceinline__ int ba_nup(int nc) { return nc * (nc + 1) / 2; }
__device__ __forceinline__ int ba_stride(int nc) { return ba_nup(nc) + 2 * nc; }  // S_up | H diag | rhs

struct BaObs {
    float r[2], e, w;
    float jq[2][3];  // d pixel / d q (camera-space point)
    float q[3];
};

// Residual of point X in frame (R, t) against its observation, with the
// derivative of the projection with respect to the camera-space point.
__device__ __forceinline__ void ba_observe(const float* Rt, float4 X, float fl, float cx, float cy, float2 uv,
                                           BaObs& o) {
    const float x = Rt[0] * X.x + Rt[1] * X.y + Rt[2] * X.z + Rt[9];
    const float y = Rt[3] * X.x + Rt[4] * X.y + Rt[5] * X.z + Rt[10];
    const float z = Rt[6] * X.x + Rt[7] * X.y + Rt[8] * X.z + Rt[11];
    const float iz = 1.f / z;
    o.q[0] = x; o.q[1] = y; o.q[2] = z;
    o.r[0] = fl * x * iz + cx - uv.x;
    o.r[1] = fl * y * iz + cy - uv.y;
    o.e = sqrtf(o.r[0] * o.r[0] + o.r[1] * o.r[1]);
    const float a = fl * iz;
    o.jq[0][0] = a; o.jq[0][1] = 0.f; o.jq[0][2] = -a * x * iz;
    o.jq[1][0] = 0.f; o.jq[1][1] = a; o.jq[1][2] = -a * y * iz;
}

// Huber weight and cost of an observation kept by the median + 4 MAD rule.
__device__ __forceinline__ float ba_weight(float e, bool keep, float delta) {
    return keep ? (e <= delta ? 1.f : delta / e) : 0.f;
}
__device__ __forceinline__ double ba_cost(float e, bool keep, float delta) {
    if (!keep) return 0.0;
    return e <= delta ? 0.5 * (double)e * e : (double)delta * ((double)e - 0.5 * delta);
}

__global__ void k_ba_residual(const float2* __restrict__ obs, const float* __restrict__ poses,
                              const float4* __restrict__ pts, const float* __restrict__ fl, float cx, float cy,
                              int F, int64_t P, float* __restrict__ e_out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P * F) return;
    const int64_t p = i / F;
    const int f = (int)(i % F);
    BaObs o;
    ba_observe(poses + 12 * f, pts[p], *fl, cx, cy, obs[i], o);
    e_out[i] = o.e;
}

// Median + 4 MAD threshold in one CTA: radix select (8 bits per pass, most
// significant first) of the lower median of e, then of |e - median|; the
// values are re-read from global memory (L1-resident) on every pass, so any
// P F fits. Non-negative floats order like their bits. The residual norms share
// a handful of exponents, so the first pass would pile every atomic onto a few
// bins: each lane counts into its own copy of the histogram (row stride 257,
// so equal digits of one warp fall into distinct banks).
constexpr int kBaSelThreads = 1024;
constexpr int64_t kBaMaxObs = int64_t(1) << 26;  // P F bound: 32-bit indexing everywhere
constexpr int kBaHistStride = 257;

template <bool kAbsDev>
__device__ uint32_t select_rank(const float* __restrict__ e, int n, float med, int rank, uint32_t* hist,
                                uint32_t* s_wsum, uint32_t* s_pref) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t* my = hist + lane * kBaHistStride;
    uint32_t prefix = 0, mask = 0;
    int k = rank;
    for (int shift = 24; shift >= 0; shift -= 8) {
        for (int i = tid; i < 32 * kBaHistStride; i += blockDim.x) hist[i] = 0;
        __syncthreads();
        for (int i = tid; i < n; i += blockDim.x) {
            const float x = kAbsDev ? fabsf(e[i] - med) : e[i];
            const uint32_t u = __float_as_uint(x);
            if ((u & mask) == prefix) atomicAdd(&my[(u >> shift) & 255u], 1u);
        }
        __syncthreads();
        uint32_t c = 0, incl = 0;
        if (tid < 256) {  // bin tid over the 32 copies, then a block scan of the 256 bins
            for (int l = 0; l < 32; l++) c += hist[l * kBaHistStride + tid];
            incl = c;
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            if (lane == 31) s_wsum[warp] = incl;
        }
        __syncthreads();
        if (tid < 256) {
            for (int w = 0; w < warp; w++) incl += s_wsum[w];
            const uint32_t excl = incl - c;
            if (excl <= (uint32_t)k && (uint32_t)k < incl) {  // exactly one bin holds rank k
                s_pref[0] = prefix | ((uint32_t)tid << shift);
                s_pref[1] = (uint32_t)k - excl;
            }
        }
        __syncthreads();
        prefix = s_pref[0];
        k = (int)s_pref[1];
        mask |= 255u << shift;
        __syncthreads();
    }
    return prefix;
}

__global__ void __launch_bounds__(kBaSelThreads) k_ba_median_mad(const float* __restrict__ e, int n,
                                                                 float* __restrict__ thr) {
    __shared__ uint32_t hist[32 * kBaHistStride];
    __shared__ uint32_t s_wsum[8];
    __shared__ uint32_t s_pref[2];
    const float med = __uint_as_float(select_rank<false>(e, n, 0.f, (n - 1) / 2, hist, s_wsum, s_pref));
    const float mad = __uint_as_float(select_rank<true>(e, n, med, (n - 1) / 2, hist, s_wsum, s_pref));
    if (threadIdx.x == 0) *thr = med + 4.f * mad;
}

// The same order statistic of values in registers: NV per thread of a cluster of CS
// CTAs of kBaSelThreads threads each (count: how many of the thread's values
// exist). 11, 11 and 10 bits per pass. Each CTA counts its values into a histogram
// of its own; in a cluster each then sums its share of the bins over all of them
// and writes the sums to every CTA (reading all of the cluster's histograms in every
// CTA takes twice as long). The counts are cleared only after the barrier that
// follows their last reading, and so are the sums.
struct SelScratch {
    uint32_t hist[2048];    // this CTA's counts
    uint32_t merged[2048];  // the cluster's
    uint32_t wsum[kBaSelThreads / 32];
    uint32_t pick[2];
};

template <int NV, int CS>
__device__ uint32_t select_in_registers(const uint32_t (&key)[NV], int count, int rank, SelScratch& sc) {
    namespace cg = cooperative_groups;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t prefix = 0, mask = 0;
    uint32_t k = (uint32_t)rank;
#pragma unroll
    for (int pass = 0; pass < 3; pass++) {
        const int shift = pass == 0 ? 21 : pass == 1 ? 10 : 0;
        const uint32_t digits = pass == 2 ? 1023u : 2047u;
        reinterpret_cast<uint2*>(sc.hist)[tid] = make_uint2(0u, 0u);
        __syncthreads();
#pragma unroll
        for (int v = 0; v < NV; v++)
            if (v < count && (key[v] & mask) == prefix) atomicAdd(&sc.hist[(key[v] >> shift) & digits], 1u);
        uint2 c;  // bins 2 tid and 2 tid + 1
        if constexpr (CS > 1) {
            auto cluster = cg::this_cluster();
            constexpr int SHARE = 2048 / CS;
            cluster.sync();
            if (tid < SHARE) {
                const int bin = (int)cluster.block_rank() * SHARE + tid;
                uint32_t t = 0;
#pragma unroll
                for (int r = 0; r < CS; r++) t += *cluster.map_shared_rank(&sc.hist[bin], r);
#pragma unroll
                for (int r = 0; r < CS; r++) *cluster.map_shared_rank(&sc.merged[bin], r) = t;
            }
            cluster.sync();
            c = reinterpret_cast<const uint2*>(sc.merged)[tid];
        } else {
            __syncthreads();
            c = reinterpret_cast<const uint2*>(sc.hist)[tid];
            __syncthreads();
        }
        uint32_t incl = c.x + c.y;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        if (lane == 31) sc.wsum[warp] = incl;
        __syncthreads();
        const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? sc.wsum[lane] : 0u);
        const uint32_t excl = before + incl - c.x - c.y;
        if (excl <= k && k < before + incl) {  // exactly one thread's two bins hold rank k
            const bool second = k >= excl + c.x;
            sc.pick[0] = prefix | ((uint32_t)(2 * tid + (second ? 1 : 0)) << shift);
            sc.pick[1] = k - excl - (second ? c.x : 0u);
        }
        __syncthreads();
        prefix = sc.pick[0];
        k = sc.pick[1];
        mask |= digits << shift;
    }
    return prefix;
}

// Opens an iteration, one cluster of 8 CTAs with NV observations a thread: accepts
// or rejects the trial state of the iteration before (as k_ba_sum and k_ba_accept),
// forms the residual norms at the resulting state and their median + 4 MAD.
// 49,152 observations: 78 us of three kernels, of which 70 the select in one CTA
// with its values read again in every pass -> 21 us.
constexpr int kBaCluster = 8;
constexpr int kBaMaxNV = 8;
constexpr int64_t kBaClusterObs = (int64_t)kBaCluster * kBaSelThreads * kBaMaxNV;  // 65,536

// k_ba_sum's total in every thread of a CTA of kBaSelThreads threads.
__device__ double ba_trial_total(const double* __restrict__ part, int nb, double* s /* [256] */) {
    const int tid = threadIdx.x;
    if (tid < 256) {
        double a = 0.0;
        for (int b = tid; b < nb; b += 256) a += part[b];
        s[tid] = a;
    }
    __syncthreads();
    if (tid < 64) {  // the tree of k_ba_sum: 256 -> 128 -> 64 -> 32, then in a warp
        double a = (s[tid] + s[tid + 128]) + (s[tid + 64] + s[tid + 192]);
        s[tid] = a;
    }
    __syncthreads();
    if (tid < 32) {
        double a = s[tid] + s[tid + 32];
        for (int o = 16; o > 0; o >>= 1) a += __shfl_down_sync(0xffffffffu, a, o);
        if (tid == 0) s[0] = a;
    }
    __syncthreads();
    return s[0];
}

template <int NV>
__global__ void __cluster_dims__(kBaCluster) __launch_bounds__(kBaSelThreads)
    k_ba_begin(const float2* __restrict__ obs, float* __restrict__ poses, float4* __restrict__ pts,
               float* __restrict__ fl, float cx, float cy, int F, int64_t P, bool first,
               const double* __restrict__ trial_partial, int nt, const double* __restrict__ cost_cur,
               const float* __restrict__ poses_t, const float4* __restrict__ pts_t, const float* __restrict__ fl_t,
               float* __restrict__ lam, float nu, float* __restrict__ history, int* __restrict__ iter,
               float* __restrict__ e_out, float* __restrict__ thr) {
    __shared__ SelScratch sc;
    __shared__ double s_sum[256];
    __shared__ float s_pose[12 * kBaMaxF];
    __shared__ float s_fl;
    const int tid = threadIdx.x;
    const int cta = blockIdx.x;  // the grid is one cluster
    bool acc = false;
    if (!first) {
        const double tc = ba_trial_total(trial_partial, nt, s_sum), cur = *cost_cur;
        acc = tc < cur;
        if (cta == 0 && tid == 0) {
            // lam is kept within [1e-12, 1e10]: a converged run rejects every further
            // step, and unbounded growth would reach infinity
            *lam = fminf(1e10f, fmaxf(1e-12f, acc ? *lam / nu : *lam * nu));
            if (history) {
                const int it = *iter;
                history[3 * it] = (float)cur;
                history[3 * it + 1] = (float)tc;
                history[3 * it + 2] = acc ? 1.f : 0.f;
            }
            *iter += 1;
        }
        if (acc) {  // every CTA reads the trial state below; it becomes the state here
            for (int64_t p = (int64_t)cta * kBaSelThreads + tid; p < P; p += kBaCluster * kBaSelThreads) pts[p] = pts_t[p];
            if (cta == 0 && tid < 12 * F) poses[tid] = poses_t[tid];
            if (cta == 0 && tid == 0) *fl = *fl_t;
        }
    }
    const float* from = acc ? poses_t : poses;
    const float4* X = acc ? pts_t : pts;
    if (tid < 12 * F) s_pose[tid] = from[tid];
    if (tid == 0) s_fl = acc ? *fl_t : *fl;
    __syncthreads();
    const int64_t n = P * F;
    uint32_t key[NV];
    int count = 0;
#pragma unroll
    for (int v = 0; v < NV; v++) {
        const int64_t i = ((int64_t)v * kBaCluster + cta) * kBaSelThreads + tid;
        key[v] = 0;
        if (i < n) {
            const int p = (int)i / F, f = (int)i - p * F;
            BaObs o;
            ba_observe(s_pose + 12 * f, X[p], s_fl, cx, cy, obs[i], o);
            e_out[i] = o.e;
            key[v] = __float_as_uint(o.e);
            count = v + 1;  // the values that exist come first
        }
    }
    const int rank = (int)((n - 1) / 2);
    const float med = __uint_as_float(select_in_registers<NV, kBaCluster>(key, count, rank, sc));
#pragma unroll
    for (int v = 0; v < NV; v++) key[v] = __float_as_uint(fabsf(__uint_as_float(key[v]) - med));
    const float mad = __uint_as_float(select_in_registers<NV, kBaCluster>(key, count, rank, sc));
    if (cta == 0 && tid == 0) *thr = med + 4.f * mad;
    cooperative_groups::this_cluster().sync();  // no CTA leaves while its histogram may be read
}

// x in FP64 by integer operations: the FP64 pipe (two lanes a clock and SM) is what
// bounds this file's kernels, and a conversion would take as long as an addition.
__device__ __noinline__ double widen_rare(float x) { return (double)x; }
__device__ __forceinline__ double widen(float x) {
    const uint32_t u = __float_as_uint(x), a = u & 0x7fffffffu;
    if (a - 0x00800000u >= 0x7f000000u && a != 0) return widen_rare(x);  // subnormal, infinite or NaN
    const uint32_t hi = (u & 0x80000000u) | (a ? (a >> 3) + 0x38000000u : 0u);
    return __hiloint2double((int)hi, (int)(u << 29));
}

// One observation's part of its point's system: Huber weight, cost, the terms of
// H_pp (6) and g_p (3) and of the focal length's coupling row (3) before weighting,
// the pose's six coupling rows, and (when asked for) the camera Jacobian rows.
struct BaTerms {
    float w, cost_e;  // cost_e: the residual norm where kept, or -1
    float h[6], g[3], kf[3];
};

__device__ __forceinline__ void ba_terms(const float* Rt, float4 X, float fl, float cx, float cy, float2 uv, float e_cur,
                                         float thr, float delta, bool pose_rows, BaTerms& t,
                                         float (*K)[3] /* the pose's 6 rows */, float (*Jc)[8] /* [2][8] or null */) {
    BaObs o;
    ba_observe(Rt, X, fl, cx, cy, uv, o);
    const bool keep = e_cur <= thr;
    const float w = ba_weight(o.e, keep, delta);
    t.w = w;
    t.cost_e = keep ? o.e : -1.f;
    float Jp[2][3];  // point Jacobian jq R
#pragma unroll
    for (int k = 0; k < 2; k++)
#pragma unroll
        for (int c = 0; c < 3; c++) Jp[k][c] = o.jq[k][0] * Rt[c] + o.jq[k][1] * Rt[3 + c] + o.jq[k][2] * Rt[6 + c];
    t.h[0] = Jp[0][0] * Jp[0][0] + Jp[1][0] * Jp[1][0];
    t.h[1] = Jp[0][0] * Jp[0][1] + Jp[1][0] * Jp[1][1];
    t.h[2] = Jp[0][0] * Jp[0][2] + Jp[1][0] * Jp[1][2];
    t.h[3] = Jp[0][1] * Jp[0][1] + Jp[1][1] * Jp[1][1];
    t.h[4] = Jp[0][1] * Jp[0][2] + Jp[1][1] * Jp[1][2];
    t.h[5] = Jp[0][2] * Jp[0][2] + Jp[1][2] * Jp[1][2];
#pragma unroll
    for (int c = 0; c < 3; c++) t.g[c] = Jp[0][c] * o.r[0] + Jp[1][c] * o.r[1];
    // camera Jacobian rows: pose (rho: jq, phi: jq (-q^)) for f > 0, focal (x/z, y/z)
    float jc[2][7];
    const float qx = o.q[0], qy = o.q[1], qz = o.q[2];
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const float a0 = o.jq[k][0], a1 = o.jq[k][1], a2 = o.jq[k][2];
        jc[k][0] = a0; jc[k][1] = a1; jc[k][2] = a2;
        // row of jq (-q^): -q^ = [[0, qz, -qy], [-qz, 0, qx], [qy, -qx, 0]]
        jc[k][3] = -a1 * qz + a2 * qy;
        jc[k][4] = a0 * qz - a2 * qx;
        jc[k][5] = -a0 * qy + a1 * qx;
        jc[k][6] = (k == 0 ? qx : qy) / qz;
    }
    if (Jc) {
#pragma unroll
        for (int k = 0; k < 2; k++) {
#pragma unroll
            for (int a = 0; a < 6; a++) Jc[k][a] = pose_rows ? jc[k][a] : 0.f;
            Jc[k][6] = jc[k][6];
            Jc[k][7] = w * o.r[k];
        }
    }
    if (pose_rows) {
#pragma unroll
        for (int a = 0; a < 6; a++)
#pragma unroll
            for (int c = 0; c < 3; c++) K[a][c] = w * (jc[0][a] * Jp[0][c] + jc[1][a] * Jp[1][c]);
    }
#pragma unroll
    for (int c = 0; c < 3; c++) t.kf[c] = jc[0][6] * Jp[0][c] + jc[1][6] * Jp[1][c];
}

// A point's damped block and its inverse from its observations' terms (in frame
// order): H_pp with Marquardt damping and the absolute floor, the symmetric 3x3
// inverse in FP64 (00 01 02 11 12 22), the gradient, the focal length's coupling
// row and the robust cost.
__device__ __forceinline__ void ba_point(const BaTerms* t, int F, float delta, float lam, double (&Hinv)[6], float (&g)[3],
                                         float (&kf)[3], double& cost) {
    float H[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    g[0] = g[1] = g[2] = kf[0] = kf[1] = kf[2] = 0.f;
    cost = 0.0;
    for (int f = 0; f < F; f++) {
        const BaTerms& o = t[f];
        const float w = o.w;
        cost += ba_cost(o.cost_e, o.cost_e >= 0.f, delta);
#pragma unroll
        for (int c = 0; c < 6; c++) H[c] += w * o.h[c];
#pragma unroll
        for (int c = 0; c < 3; c++) g[c] += w * o.g[c];
#pragma unroll
        for (int c = 0; c < 3; c++) kf[c] += w * o.kf[c];
    }
    const double a = (double)H[0] * (1.0 + lam) + 1e-9, b = H[1], c = H[2];
    const double d = (double)H[3] * (1.0 + lam) + 1e-9, e = H[4];
    const double ff = (double)H[5] * (1.0 + lam) + 1e-9;
    const double c00 = d * ff - e * e, c01 = c * e - b * ff, c02 = b * e - c * d;
    const double c11 = a * ff - c * c, c12 = b * c - a * e, c22 = a * d - b * b;
    const double idet = 1.0 / (a * c00 + b * c01 + c * c02);
    Hinv[0] = c00 * idet; Hinv[1] = c01 * idet; Hinv[2] = c02 * idet;
    Hinv[3] = c11 * idet; Hinv[4] = c12 * idet; Hinv[5] = c22 * idet;
}

__device__ __forceinline__ void sym3_mul(const double* S, const float* v, double* o) {
    const double x = widen(v[0]), y = widen(v[1]), z = widen(v[2]);
    o[0] = S[0] * x + S[1] * y + S[2] * z;
    o[1] = S[1] * x + S[3] * y + S[4] * z;
    o[2] = S[2] * x + S[4] * y + S[5] * z;
}

// Upper-triangle index e -> (i, j), i <= j, row-major over i.
__device__ __forceinline__ void up_ij(int e, int nc, int& i, int& j) {
    int r = 0, left = e;
    while (left >= nc - r) { left -= nc - r; r++; }
    i = r;
    j = r + left;
}

// What k_ba_points leaves of each point for the kernels after it.
struct BaPoints {
    float* K;        // [P][Nc][3] coupling rows
    float* V;        // [P][Nc][3] H_pp^-1 K
    double* Hinv;    // [P][6]
    double* u;       // [P][3] H_pp^-1 g
    float* g;        // [P][3]
    double* cost;    // [P] robust cost
    float* J;        // [P][F][2][8] camera Jacobian rows and weighted residual
    float* w;        // [P][F] weights
};

constexpr int kBaChunk = 32;  // points per chunk of k_ba_normal

// The point systems: one thread per observation forms its terms, one per point
// sums and inverts its block, one per point and camera parameter forms H_pp^-1 K.
constexpr int kBaPointsPts = 16;
constexpr int kBaPointsThreads = 128;

__global__ void __launch_bounds__(kBaPointsThreads) k_ba_points(const float2* __restrict__ obs,
                                                                const float* __restrict__ poses,
                                                                const float4* __restrict__ pts,
                                                                const float* __restrict__ fl_p, float cx, float cy,
                                                                int F, int64_t P, const float* __restrict__ e_cur,
                                                                const float* __restrict__ thr_p, float delta,
                                                                const float* __restrict__ lam_p, BaPoints out) {
    __shared__ float s_pose[12 * kBaMaxF];
    __shared__ BaTerms s_t[kBaPointsPts][kBaMaxF];
    __shared__ float s_K[kBaPointsPts][kBaMaxNc][3];
    __shared__ double s_Hinv[kBaPointsPts][6];
    const int nc = ba_nc(F), tid = threadIdx.x;
    for (int i = tid; i < 12 * F; i += kBaPointsThreads) s_pose[i] = poses[i];
    __syncthreads();
    const int64_t p0 = (int64_t)blockIdx.x * kBaPointsPts;
    const int np = (int)min((int64_t)kBaPointsPts, P - p0);
    const float thr = *thr_p, fl = *fl_p, lam = *lam_p;
    for (int i = tid; i < np * F; i += kBaPointsThreads) {
        const int pt = i / F, f = i % F;
        const int64_t ob = (p0 + pt) * F + f;
        float Jc[2][8];
        ba_terms(s_pose + 12 * f, pts[p0 + pt], fl, cx, cy, obs[ob], e_cur[ob], thr, delta, f > 0, s_t[pt][f],
                 &s_K[pt][6 * (f > 0 ? f - 1 : 0)], Jc);
        float4* dst = reinterpret_cast<float4*>(out.J + ob * 16);
        dst[0] = make_float4(Jc[0][0], Jc[0][1], Jc[0][2], Jc[0][3]);
        dst[1] = make_float4(Jc[0][4], Jc[0][5], Jc[0][6], Jc[0][7]);
        dst[2] = make_float4(Jc[1][0], Jc[1][1], Jc[1][2], Jc[1][3]);
        dst[3] = make_float4(Jc[1][4], Jc[1][5], Jc[1][6], Jc[1][7]);
        out.w[ob] = s_t[pt][f].w;
    }
    __syncthreads();
    if (tid < np) {
        float g[3], kf[3];
        double Hinv[6], c, u[3];
        ba_point(s_t[tid], F, delta, lam, Hinv, g, kf, c);
        sym3_mul(Hinv, g, u);
        out.cost[p0 + tid] = c;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            s_K[tid][nc - 1][k] = kf[k];
            out.g[(p0 + tid) * 3 + k] = g[k];
            out.u[(p0 + tid) * 3 + k] = u[k];
        }
#pragma unroll
        for (int k = 0; k < 6; k++) {
            s_Hinv[tid][k] = Hinv[k];
            out.Hinv[(p0 + tid) * 6 + k] = Hinv[k];
        }
    }
    __syncthreads();
    for (int i = tid; i < np * nc; i += kBaPointsThreads) {
        const int pt = i / nc, c = i % nc;
        double v[3];
        sym3_mul(s_Hinv[pt], s_K[pt][c], v);
        const int64_t o = (p0 * nc + i) * 3;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            out.K[o + k] = s_K[pt][c][k];
            out.V[o + k] = (float)v[k];
        }
    }
}

// Entries of the reduced camera system per chunk of 32 points: h = the entry of
// H_cc and h - sum_p K_i . H^-1 K_j, the points in order, FP32 products summed in
// FP64. FP64 is what bounds this (a warp instruction takes 16 cycles of an SM), so
// its threads are dealt densely: the 21 (F - 1) + Nc entries that have an h first,
// then the others, 512 entries per CTA (two CTAs per chunk at 8 frames: 384, all
// resident); behind a chunk's last entries two warps take the right-hand side, its
// products formed by all warps before. The focal length's chain of adds is F times as
// long as the others' and would come last, at its share of a busy FP64 pipe: CTAs of
// their own, first in the grid, take it, one thread per chunk. 8 frames x 6144 points:
// 190 us with k_ba_points' work in it and the right-hand side in one warp -> 38 -> 30,
// k_ba_points 16.
constexpr int kBaNormalThreads = 512;
constexpr int kBaFocalChunks = 8;  // chunks per focal CTA

static size_t ba_normal_smem(int F, int nc) {
    return sizeof(float) * (2 * kBaChunk * nc * 3 + kBaChunk * F * 17) + sizeof(double) * kBaChunk * (3 + 2 * (nc - 1));
}

__global__ void __launch_bounds__(kBaNormalThreads) k_ba_normal(BaPoints in, int F, int64_t P,
                                                                double* __restrict__ partial) {
    extern __shared__ __align__(16) double sm[];
    const int nc = ba_nc(F), nup = ba_nup(nc), tid = threadIdx.x;
    const int nb = (int)ceil_div(P, kBaChunk), nfocal = (nb + kBaFocalChunks - 1) / kBaFocalChunks;
    if ((int)blockIdx.x < nfocal) {  // the focal length's right-hand side of these chunks
        const int c0 = blockIdx.x * kBaFocalChunks, nch = min(kBaFocalChunks, nb - c0), per = kBaChunk * F;
        double* s_gf = (double*)sm;                     // [32 F][8] gradient terms
        double* s_kf = s_gf + per * kBaFocalChunks;     // [32][8] K . u
        for (int i = tid; i < nch * per; i += kBaNormalThreads) {
            const int64_t o = (int64_t)c0 * per + i;
            if (o >= P * F) break;
            const float2 a = *reinterpret_cast<const float2*>(in.J + o * 16 + 6);
            const float2 b = *reinterpret_cast<const float2*>(in.J + o * 16 + 14);
            s_gf[i % per * kBaFocalChunks + i / per] = widen(a.x) * widen(a.y) + widen(b.x) * widen(b.y);
        }
        for (int i = tid; i < nch * kBaChunk; i += kBaNormalThreads) {
            const int64_t p = (int64_t)c0 * kBaChunk + i;
            if (p >= P) break;
            const float* K = in.K + (p * nc + nc - 1) * 3;
            const double* u = in.u + p * 3;
            s_kf[i % kBaChunk * kBaFocalChunks + i / kBaChunk] = widen(K[0]) * u[0] + widen(K[1]) * u[1] + widen(K[2]) * u[2];
        }
        __syncthreads();
        if (tid < nch) {
            const int np = (int)min((int64_t)kBaChunk, P - (int64_t)(c0 + tid) * kBaChunk);
            double gc = 0.0, ku = 0.0;
#pragma unroll 8
            for (int i = 0; i < np * F; i++) gc += s_gf[i * kBaFocalChunks + tid];
#pragma unroll 4
            for (int pt = 0; pt < np; pt++) ku += s_kf[pt * kBaFocalChunks + tid];
            partial[(int64_t)(c0 + tid) * ba_stride(nc) + nup + nc + nc - 1] = -gc + ku;
        }
        return;
    }
    const int part = ((int)blockIdx.x - nfocal) / nb, chunk = ((int)blockIdx.x - nfocal) % nb;
    const bool last = (int)blockIdx.x >= (int)gridDim.x - nb;  // this CTA's row has the right-hand side too
    const int64_t p0 = (int64_t)chunk * kBaChunk;
    const int np = (int)min((int64_t)kBaChunk, P - p0);
    double* out = partial + (int64_t)chunk * ba_stride(nc);
    double* s_u = (double*)sm;                       // [32][3]
    double* s_gc = s_u + kBaChunk * 3;               // [32][Nc - 1] gradient terms of the pose parameters
    double* s_ku = s_gc + kBaChunk * (nc - 1);       // [32][Nc - 1] K . u
    float* s_K = (float*)(s_ku + kBaChunk * (nc - 1));  // [32][Nc][3]
    float* s_V = s_K + kBaChunk * nc * 3;            // [32][Nc][3]
    float* s_J = s_V + kBaChunk * nc * 3;            // [32][F][16]
    float* s_w = s_J + kBaChunk * F * 16;            // [32][F]
#pragma unroll 4
    for (int i = tid; i < np * nc * 3; i += kBaNormalThreads) {
        s_K[i] = in.K[p0 * nc * 3 + i];
        s_V[i] = in.V[p0 * nc * 3 + i];
    }
#pragma unroll 4
    for (int i = tid; i < np * F * 16; i += kBaNormalThreads) s_J[i] = in.J[p0 * F * 16 + i];
    for (int i = tid; i < np * F; i += kBaNormalThreads) s_w[i] = in.w[p0 * F + i];
    if (tid < np * 3) s_u[tid] = in.u[p0 * 3 + tid];
    __syncthreads();
    if (last) {  // the products of the right-hand side, spread over all warps
        for (int i = tid; i < np * (nc - 1); i += kBaNormalThreads) {
            const int pt = i / (nc - 1), c = i % (nc - 1), f = c / 6 + 1, a = c % 6;
            const float* K = s_K + (pt * nc + c) * 3;
            const double* u = s_u + pt * 3;
            s_ku[i] = widen(K[0]) * u[0] + widen(K[1]) * u[1] + widen(K[2]) * u[2];
            const float* J = s_J + (pt * F + f) * 16;
            s_gc[i] = widen(J[a]) * widen(J[7]) + widen(J[8 + a]) * widen(J[15]);
        }
        __syncthreads();
    }
    int q = part * kBaNormalThreads + tid;
    const int q_rhs = (nup + 31) / 32 * 32;  // the warps after the entries
    if (q >= q_rhs) {
        const int c = q - q_rhs;
        if (c < nc - 1) {
            double gc = 0.0, ku = 0.0;
#pragma unroll 4
            for (int pt = 0; pt < np; pt++) {
                gc += s_gc[pt * (nc - 1) + c];
                ku += s_ku[pt * (nc - 1) + c];
            }
            out[nup + nc + c] = -gc + ku;
        }
        return;
    }
    if (q >= nup) return;
    int i, j, f_lo = 0, f_hi = 0, ai = 0, aj = 0;  // h sums frames [f_lo, f_hi) at local parameters ai, aj
    const int n_same = 21 * (F - 1);
    if (q < n_same) {  // two parameters of one pose
        const int f = q / 21;
        int r = q % 21, a = 0;
        while (r >= 6 - a) { r -= 6 - a; a++; }
        i = 6 * f + a;
        j = i + r;
        f_lo = f + 1;
        f_hi = f + 2;
        ai = a;
        aj = a + r;
    } else if (q < n_same + nc) {  // with the focal length
        i = q - n_same;
        j = nc - 1;
        aj = 6;
        if (i == nc - 1) {
            ai = 6;
            f_hi = F;
        } else {
            ai = i % 6;
            f_lo = i / 6 + 1;
            f_hi = f_lo + 1;
        }
    } else {  // of two poses: no observation has both
        q -= n_same + nc;
        int pair = q / 36, fi = 0;
        while (pair >= F - 2 - fi) { pair -= F - 2 - fi; fi++; }
        i = 6 * fi + q % 36 / 6;
        j = 6 * (fi + 1 + pair) + q % 6;
    }
    double h = 0.0;
    if (f_hi > f_lo)
        for (int pt = 0; pt < np; pt++) {
            float hp = 0.f;  // this point's terms in FP32
            for (int f = f_lo; f < f_hi; f++) {
                const float* J = s_J + (pt * F + f) * 16;
                hp += s_w[pt * F + f] * (J[ai] * J[aj] + J[8 + ai] * J[8 + aj]);
            }
            h += widen(hp);
        }
    double sch = 0.0;  // each point's dot product in FP32, the sum in FP64
    const float *Ki = s_K + 3 * i, *Vj = s_V + 3 * j;
#pragma unroll 4
    for (int pt = 0; pt < np; pt++, Ki += 3 * nc, Vj += 3 * nc)
        sch += widen(Ki[0] * Vj[0] + Ki[1] * Vj[1] + Ki[2] * Vj[2]);
    out[i * nc - i * (i - 1) / 2 + (j - i)] = h - sch;
    if (i == j) out[nup + i] = h;
}

// Fixed-order sum of the chunk partials: a block of 16 x 8 threads takes 16
// values; each of the 8 rows sums a contiguous segment of the chunks, then the 8
// segment sums are added in order. Many small blocks: the sums are FP64.
__global__ void __launch_bounds__(128) k_ba_reduce(const double* __restrict__ partial, int nb, int stride,
                                                   int n_values, double* __restrict__ tot) {
    __shared__ double s[8][17];
    const int v = blockIdx.x * 16 + threadIdx.x;
    const int seg = (nb + 7) / 8, b0 = threadIdx.y * seg, b1 = min(nb, b0 + seg);
    double a = 0.0;
    if (v < n_values)
#pragma unroll 8
        for (int b = b0; b < b1; b++) a += partial[(int64_t)b * stride + v];
    s[threadIdx.y][threadIdx.x] = a;
    __syncthreads();
    if (threadIdx.y == 0 && v < n_values) {
        double t = 0.0;
        for (int r = 0; r < 8; r++) t += s[r][threadIdx.x];
        tot[v] = t;
    }
}

// The current state's robust cost from the points' costs: sums of 32 points in
// order, then eight contiguous segments of those in order (an order of its own,
// whatever the chunks are); eight warps of the solving CTA, none of those that
// back-substitute at the same time.
__device__ double ba_cost_sum(const double* __restrict__ cost, int64_t P, double* s_part /* [8] */) {
    const int64_t n32 = ceil_div(P, 32), seg = (n32 + 7) / 8;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int w = (warp & 3) == 3 ? -1 : (warp / 4 - 1) * 3 + (warp & 3);  // warps 4-6, 8-10, 12, 13
    if (w >= 0 && w < 8) {
        const int64_t g0 = w * seg, g1 = min(n32, g0 + seg);
        double a = 0.0;
        for (int64_t b = g0; b < g1; b += 32) {  // lane l sums group b + l, then the groups join in order
            double t = 0.0;
            if (b + lane < g1)
#pragma unroll 8
                for (int k = 0; k < 32; k++) {
                    const int64_t p = (b + lane) * 32 + k;
                    if (p < P) t += cost[p];
                }
            const int m = (int)min((int64_t)32, g1 - b);
            for (int l = 0; l < m; l++) a += __shfl_sync(0xffffffffu, t, l);
        }
        if (lane == 0) s_part[w] = a;
    }
    __syncthreads();
    double t = 0.0;
    for (int r = 0; r < 8; r++) t += s_part[r];
    return t;
}

// Fixed-order sum of the trial-cost block partials (one CTA).
__global__ void k_ba_sum(const double* __restrict__ part, int nb, double* __restrict__ out) {
    __shared__ double s[256];
    double a = 0.0;
    for (int b = threadIdx.x; b < nb; b += blockDim.x) a += part[b];
    s[threadIdx.x] = a;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h) s[threadIdx.x] += s[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = s[0];
}

// T <- exp(d^) T for d = (rho, phi), in FP64: entry e of the 12 (R row-major | t).
// Each thread forms what its own entry needs: FP64 instructions take 64 cycles of
// their scheduler each, whether one lane runs them or all.
__device__ __forceinline__ void ba_retract_entry(const float* Rt, const double* d, int e, float* out) {
    const double wx = d[3], wy = d[4], wz = d[5];
    const double th2 = wx * wx + wy * wy + wz * wz, th = sqrt(th2);
    double A, B, Cc;
    if (th < 1e-4) {
        A = 1.0 - th2 / 6.0; B = 0.5 - th2 / 24.0; Cc = 1.0 / 6.0 - th2 / 120.0;
    } else {
        double sn, cs;
        sincos(th, &sn, &cs);
        A = sn / th; B = (1.0 - cs) / th2; Cc = (th - sn) / (th2 * th);
    }
    const int r = e < 9 ? e / 3 : e - 9;  // row r of K = d^ and of K^2, of dR = I + A K + B K^2 and V = I + B K + C K^2
    const double k0 = r == 0 ? 0.0 : r == 1 ? wz : -wy, k1 = r == 0 ? -wz : r == 1 ? 0.0 : wx;
    const double k2 = r == 0 ? wy : r == 1 ? -wx : 0.0;
    const double q0 = k0 * 0.0 + k1 * wz + k2 * -wy, q1 = k0 * -wz + k1 * 0.0 + k2 * wx, q2 = k0 * wy + k1 * -wx + k2 * 0.0;
    const double i0 = r == 0 ? 1.0 : 0.0, i1 = r == 1 ? 1.0 : 0.0, i2 = r == 2 ? 1.0 : 0.0;
    const double dR0 = i0 + A * k0 + B * q0, dR1 = i1 + A * k1 + B * q1, dR2 = i2 + A * k2 + B * q2;
    if (e < 9) {
        const int c = e % 3;
        out[e] = (float)(dR0 * Rt[c] + dR1 * Rt[3 + c] + dR2 * Rt[6 + c]);
    } else {
        const double V0 = i0 + B * k0 + Cc * q0, V1 = i1 + B * k1 + Cc * q1, V2 = i2 + B * k2 + Cc * q2;
        out[e] = (float)(dR0 * Rt[9] + dR1 * Rt[10] + dR2 * Rt[11] + V0 * d[0] + V1 * d[1] + V2 * d[2]);
    }
}

// One CTA: damping, L D L^T factorisation and solves (FP64), then the trial
// cameras. A dependent FP64 operation takes 66 cycles, a division 390, and a warp's
// FP64 instruction holds its quarter of the SM for 64, so the factorisation is a
// race of its longest chain (update a column, divide by its pivot, 43 times)
// against the trailing updates:
//   - right-looking on the lower triangle, every entry in its thread's registers,
//     dealt column by column so that whole warps finish early;
//   - warp 0 owns none, and neither do the other warps of its quarter of the SM: it
//     takes column k + 1 from its owners - who publish it updated by the columns
//     before k - applies column k, publishes it and divides, while the others apply
//     column k to the columns from k + 2;
//   - one barrier per column among these;
//   - warp 11 follows them without the barrier: row k of L and of L y = rhs need the
//     columns before k only, so forward substitution ends with the factorisation. A row
//     takes it as long as a column takes the others (1040 cycles alone, 1200 beside two
//     warps of owners; beside three, with four in the other quarters, 1240).
// A row's dot product is summed by a fixed tree over lanes (xor 16, 8, 4, 2, 1). Back
// substitution is a chain of rows through that tree from the newest term, always in lane
// 0, to its root; the tree's other branches end one row earlier, so three helping warps
// on the other quarters sum them a row ahead and hand them over in shared memory: seven
// dependent operations a row and no shuffles, 715 cycles against 1000. Branches in a row
// cost more than the operations that they leave out (levels without terms: 200 cycles a
// row), hence rows of up to 32 and of more terms as loops of their own.
// 43 x 43: 88 -> 72 us with both substitutions in one warp after the factorisation, 50 us
// like this (init 2.5, columns 25, back substitution 14.5, trial cameras and cost 5).
constexpr int kBaSolveThreads = 480;
constexpr int kBaForward = 11;  // the substituting warp
constexpr int kBaEntries = kBaMaxNc * (kBaMaxNc + 1) / 2;
constexpr int kBaOwners = 320;  // warps 1-3, 5-7, 9, 10, 13, 14: three entries a thread, two warps beside warp 11
constexpr int kBaPerThread = (kBaEntries + kBaOwners - 1) / kBaOwners;

// Values handed from warp to warp of the solving CTA: the value itself tells whether it
// is there, an empty place holds a signalling NaN, which no FP64 operation returns. The
// warps of a CTA all run, so a wait ends; it is bounded all the same.
constexpr int kBaEmpty = 0x7ff45a5a;  // its high word
constexpr int kBaWaits = 1 << 16;
__device__ __forceinline__ double ba_look(const double* place) { return *reinterpret_cast<const volatile double*>(place); }
__device__ __forceinline__ bool ba_empty(double v) { return __double2hiint(v) == kBaEmpty; }
__device__ __forceinline__ void ba_hand(double* place, double v) { *reinterpret_cast<volatile double*>(place) = v; }

__global__ void __launch_bounds__(kBaSolveThreads) k_ba_solve(const double* __restrict__ tot,
                                                               const double* __restrict__ cost, int64_t P, int F,
                                                               const float* __restrict__ lam_p,
                                                               const float* __restrict__ poses,
                                                               const float* __restrict__ fl_p,
                                                               double* __restrict__ dc, double* __restrict__ cost_cur,
                                                               float* __restrict__ poses_t, float* __restrict__ fl_t,
                                                               int* __restrict__ fail) {
    __shared__ double U[kBaMaxNc][kBaMaxNc + 2];  // published columns, unscaled: row k holds column k's rows k..
    __shared__ double L[kBaMaxNc][kBaMaxNc + 2];  // unit lower triangle
    __shared__ double y[kBaMaxNc], s_rhs[kBaMaxNc], s_z[kBaMaxNc];
    __shared__ double s_branch[kBaMaxNc][5];  // back substitution: sums of a row's tree beside its newest term's path
    __shared__ double s_dinv[kBaMaxNc];
    __shared__ double s_part[8];
    __shared__ int s_bad;
    const int nc = ba_nc(F), nup = ba_nup(nc);
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) s_bad = 0;
    if (tid < nc) {
        s_rhs[tid] = tot[nup + nc + tid];
        y[tid] = s_dinv[tid] = __hiloint2double(kBaEmpty, 0);
    }
    if (tid < nc * 5) s_branch[0][tid] = tid < (nc - 2) * 5 ? __hiloint2double(kBaEmpty, 0) : 0.0;  // (row nc - 2: one term)
    const double lam = *lam_p;
    double a[kBaPerThread];
    int ei[kBaPerThread], ej[kBaPerThread];  // row and column of each entry, column -1: none
#pragma unroll
    for (int s = 0; s < kBaPerThread; s++) {
        const int warp = tid >> 5;
        const int q = (warp - warp / 4 - 1 - (warp > kBaForward)) * 32 + lane + s * kBaOwners;
        ei[s] = ej[s] = -1;
        a[s] = 0.0;
        if ((warp & 3) && warp != kBaForward && q < nup) {
            up_ij(q, nc, ej[s], ei[s]);  // upper-triangle entry (column, row)
            a[s] = tot[q];
            if (ei[s] == ej[s]) a[s] += lam * tot[nup + ei[s]] + 1e-9;
            if (ej[s] <= 1) U[ej[s]][ei[s]] = a[s];  // columns 0 and 1 have no earlier updates to wait for
        }
    }
    __syncthreads();
    auto pivot = [&](int k, double d) {
        // d > 0 by its bits (an FP64 comparison costs as much as an addition)
        const int hi = __double2hiint(d);
        const bool pos = hi >= 0 && (hi | __double2loint(d)) != 0 &&
                         (hi < 0x7ff00000 || (hi == 0x7ff00000 && __double2loint(d) == 0));
        if (!pos) s_bad = 1;
        const double r = pos ? 1.0 / d : 0.0;
        __threadfence_block();  // the column is there for who sees its pivot
        ba_hand(&s_dinv[k], r);
    };
    if (tid == 0) pivot(0, U[0][0]);
    __syncthreads();
    const int hi = lane + 32;
    double y0 = 0.0, y1 = 0.0;  // the substituting warp: lane l holds y_l and y_{l + 32} of L y = rhs
    auto forward_row = [&](int k, auto wide) {
        bool wait = true;  // for column k - 1
        for (int n = 0; n < kBaWaits && wait; n++) wait = __any_sync(0xffffffffu, ba_empty(ba_look(&s_dinv[k - 1])));
        if (wait) s_bad = 1;
        __threadfence_block();
        // no branches: a lane past the row forms the last term again and leaves it out
        const double rhs = s_rhs[k];
        const int j0 = min(lane, k - 1), j1 = min(hi, k - 1);
        const double c0 = __dmul_rn(U[j0][k], s_dinv[j0]);
        L[k][j0] = c0;
        double t = __dmul_rn(lane < k ? c0 : 0.0, y0);
        if constexpr (decltype(wide)::value) {
            const double c1 = __dmul_rn(U[j1][k], s_dinv[j1]);
            L[k][j1] = c1;
            t = __fma_rn(hi < k ? c1 : 0.0, y1, t);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t = __dadd_rn(t, __shfl_xor_sync(0xffffffffu, t, o));
        const double v = __dsub_rn(rhs, t);
        if (lane == k) y0 = v;
        if (hi == k) y1 = v;
    };
    const bool substitutes = tid >> 5 == kBaForward;
    if (substitutes) {
        if (lane == 0) y0 = s_rhs[0];
        int k = 1;
        for (; k < min(nc, 33); k++) forward_row(k, std::false_type());
        for (; k < nc; k++) forward_row(k, std::true_type());
        if (lane < nc) s_z[lane] = y0;
        if (hi < nc) s_z[hi] = y1;
    } else {
        auto column = [&](int k, auto wide) {  // wide: more than 32 rows left
            const double dinv = s_dinv[k];
            if (tid < 32) {  // (the other warps of its quarter own no entry)
                // column k + 1, rows k + 1 + lane and + 32: the diagonal entry is lane 0's first
                const int c = k + 1, i0 = min(c + lane, nc - 1), i1 = min(i0 + 32, nc - 1);
                const double p = U[k][c];
                const double v = U[c][i0] - U[k][i0] * p * dinv;
                double v1 = 0.0;
                if constexpr (decltype(wide)::value) v1 = U[c][i1] - U[k][i1] * p * dinv;
                __syncwarp();
                if (c + lane < nc) U[c][c + lane] = v;
                if (decltype(wide)::value && c + lane + 32 < nc) U[c][c + lane + 32] = v1;
                __syncwarp();
                if (lane == 0) pivot(c, v);
            } else {
#pragma unroll
                for (int s = 0; s < kBaPerThread; s++)
                    if (ej[s] > k + 1) {
                        a[s] -= U[k][ei[s]] * U[k][ej[s]] * dinv;
                        if (ej[s] == k + 2) U[k + 2][ei[s]] = a[s];
                    }
            }
            asm volatile("bar.sync 1, %0;" ::"n"(kBaSolveThreads - 32) : "memory");  // all but the substituting warp
        };
        int k = 0;
        for (; k + 33 < nc; k++) column(k, std::true_type());
        for (; k + 1 < nc; k++) column(k, std::false_type());
    }
    __syncthreads();
    if (tid < nc) s_z[tid] = __dmul_rn(s_z[tid], s_dinv[tid]);
    __syncthreads();
    // L^T x = D^-1 y, x in y[]: row i's terms j > i start at lane 0 with j = i + 1
    if (substitutes) {  // every lane the same
        double x = s_z[nc - 1], z = s_z[nc > 1 ? nc - 2 : 0], l1 = nc > 1 ? L[nc - 1][nc - 2] : 0.0;
        if (lane == 0) ba_hand(&y[nc - 1], x);
        auto row = [&](int i, auto wide) {  // wide: more than 32 terms
            const int next = max(i - 1, 0);
            double t = __dmul_rn(l1, x);
            double l33 = 0.0, x33 = 0.0, br[5];
            if constexpr (decltype(wide)::value) l33 = L[i + 33][i], x33 = ba_look(&y[i + 33]);
            l1 = L[next + 1][next];
            const double zi = z;
            z = s_z[next];
            bool wait = true;
            for (int n = 0; n < kBaWaits && wait; n++) {
                wait = false;
#pragma unroll
                for (int s = 0; s < 5; s++) br[s] = ba_look(&s_branch[i][s]);
#pragma unroll
                for (int s = 0; s < 5; s++) wait |= ba_empty(br[s]);
                wait = __any_sync(0xffffffffu, wait);
            }
            if (wait) s_bad = 1;
            if constexpr (decltype(wide)::value) t = __fma_rn(l33, x33, t);
#pragma unroll
            for (int s = 0; s < 5; s++) t = __dadd_rn(t, br[s]);
            x = __dsub_rn(zi, t);
            if (lane == 0) ba_hand(&y[i], x);
        };
        int i = nc - 2;
        for (; i >= max(nc - 33, 0); i--) row(i, std::false_type());
        for (; i >= 0; i--) row(i, std::true_type());
    } else if (tid < 96) {
        auto branches = [&](int i, auto wide) {
            const int m = nc - 1 - i, j = i + 1 + lane;
            const bool has0 = lane > 0 && lane < m, has1 = decltype(wide)::value && lane > 0 && hi < m;
            const double l0 = has0 ? L[j][i] : 0.0, l1 = has1 ? L[j + 32][i] : 0.0;
            double x0 = 0.0, x1 = 0.0;
            bool wait = true;
            for (int n = 0; n < kBaWaits && wait; n++) {
                if (has0) x0 = ba_look(&y[j]);
                if (has1) x1 = ba_look(&y[j + 32]);
                wait = __any_sync(0xffffffffu, ba_empty(x0) || ba_empty(x1));
            }
            if (wait) s_bad = 1;
            double t = __dmul_rn(l0, x0);
            if constexpr (decltype(wide)::value) t = __fma_rn(l1, x1, t);
#pragma unroll
            for (int s = 0; s < 5; s++) {
                const int o = 16 >> s;
                if (lane == o) ba_hand(&s_branch[i][s], t);
                if (o > 1) t = __dadd_rn(t, __shfl_xor_sync(0xffffffffu, t, o));
            }
        };
        int i = nc - 3 - (tid >> 5);
        for (; i >= max(nc - 33, 0); i -= 3) branches(i, std::false_type());
        for (; i >= 0; i -= 3) branches(i, std::true_type());
    }
    const double total = ba_cost_sum(cost, P, s_part);
    __syncthreads();
    const bool bad = s_bad;
    if (bad)
        for (int c = tid; c < nc; c += blockDim.x) y[c] = 0.0;
    __syncthreads();
    for (int c = tid; c < nc; c += blockDim.x) dc[c] = y[c];
    if (tid == 0) {
        *cost_cur = total;
        if (bad) atomicExch(fail, 1);
    }
    if (tid < 12 * F) {  // trial camera state
        const int f = tid / 12, e = tid % 12;
        if (f == 0)
            poses_t[e] = poses[e];
        else
            ba_retract_entry(poses + 12 * f, y + 6 * (f - 1), e, poses_t + 12 * f);
    }
    if (tid == blockDim.x - 1) *fl_t = (float)((double)*fl_p + y[nc - 1]);
}

// Trial points and the trial state's robust cost: a CTA takes 256 observations and
// the points they belong to (a point shared by two CTAs is stepped by both, to the
// same value): one thread per point and coordinate forms the right-hand side from
// the stored coupling rows, one per point the step, one per observation the trial
// residual; the costs are summed by a fixed tree.
constexpr int kBaStepThreads = 256;
constexpr int ba_step_points(int F) { return (kBaStepThreads + F - 2) / F + 1; }  // most points 256 observations touch
constexpr int kBaStepPts = ba_step_points(2);

__global__ void __launch_bounds__(kBaStepThreads) k_ba_step(const float2* __restrict__ obs,
                                                            const float4* __restrict__ pts, float cx, float cy, int F,
                                                            int64_t P, const float* __restrict__ e_cur,
                                                            const float* __restrict__ thr_p, float delta, BaPoints in,
                                                            const double* __restrict__ dc,
                                                            const float* __restrict__ poses_t,
                                                            const float* __restrict__ fl_t, float4* __restrict__ pts_t,
                                                            double* __restrict__ partial) {
    __shared__ float4 s_X[kBaStepPts];  // trial points
    __shared__ double s_rhs[kBaStepPts][3];
    __shared__ double s_dc[kBaMaxNc];
    __shared__ double s_cost[kBaStepThreads];
    __shared__ float s_pose[12 * kBaMaxF];
    extern __shared__ float s_K[];  // [points][Nc][3]
    const int nc = ba_nc(F), tid = threadIdx.x;
    const int64_t n = P * F, i0 = (int64_t)blockIdx.x * kBaStepThreads;
    const int64_t p0 = i0 / F, p1 = (min(i0 + kBaStepThreads, n) - 1) / F;  // the points of these observations
    const int np = (int)(p1 - p0) + 1;
    for (int i = tid; i < 12 * F; i += kBaStepThreads) s_pose[i] = poses_t[i];
    for (int i = tid; i < nc; i += kBaStepThreads) s_dc[i] = dc[i];
#pragma unroll 8
    for (int i = tid; i < np * nc * 3; i += kBaStepThreads) s_K[i] = in.K[p0 * nc * 3 + i];
    __syncthreads();
    for (int i = tid; i < np * 3; i += kBaStepThreads) {
        const int k = i % 3;
        double r = in.g[p0 * 3 + i];
        const float* K = s_K + i / 3 * nc * 3 + k;
#pragma unroll 4
        for (int c = 0; c < nc; c++) r += widen(K[3 * c]) * s_dc[c];
        s_rhs[i / 3][k] = r;
    }
    __syncthreads();
    for (int i = tid; i < np; i += kBaStepThreads) {
        const double* S = in.Hinv + (p0 + i) * 6;
        const double* r = s_rhs[i];
        const double dx = -(S[0] * r[0] + S[1] * r[1] + S[2] * r[2]);
        const double dy = -(S[1] * r[0] + S[3] * r[1] + S[4] * r[2]);
        const double dz = -(S[2] * r[0] + S[4] * r[1] + S[5] * r[2]);
        const float4 X = pts[p0 + i];
        const float4 Xt = make_float4((float)(X.x + dx), (float)(X.y + dy), (float)(X.z + dz), 0.f);
        s_X[i] = Xt;
        pts_t[p0 + i] = Xt;
    }
    __syncthreads();
    double c = 0.0;
    if (i0 + tid < n) {
        const int64_t ob = i0 + tid;
        BaObs o;
        ba_observe(s_pose + 12 * (int)(ob % F), s_X[ob / F - p0], *fl_t, cx, cy, obs[ob], o);
        c = ba_cost(o.e, e_cur[ob] <= *thr_p, delta);
    }
    s_cost[tid] = c;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (tid < h) s_cost[tid] += s_cost[tid + h];
        __syncthreads();
    }
    if (tid == 0) partial[blockIdx.x] = s_cost[0];
}

__global__ void __launch_bounds__(256) k_ba_trial_cost(const float2* __restrict__ obs,
                                                        const float* __restrict__ poses_t,
                                                        const float4* __restrict__ pts_t,
                                                        const float* __restrict__ fl_t, float cx, float cy, int F,
                                                        int64_t P, const float* __restrict__ e_cur,
                                                        const float* __restrict__ thr_p, float delta,
                                                        double* __restrict__ partial) {
    __shared__ double s[256];
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double c = 0.0;
    if (i < P * F) {
        BaObs o;
        ba_observe(poses_t + 12 * (i % F), pts_t[i / F], *fl_t, cx, cy, obs[i], o);
        c = ba_cost(o.e, e_cur[i] <= *thr_p, delta);
    }
    s[threadIdx.x] = c;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h) s[threadIdx.x] += s[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = s[0];
}

__global__ void k_ba_accept(const double* __restrict__ trial_total, const double* __restrict__ cost_cur,
                            int F, int64_t P, const float* __restrict__ poses_t, const float4* __restrict__ pts_t,
                            const float* __restrict__ fl_t, float* __restrict__ poses, float4* __restrict__ pts,
                            float* __restrict__ fl, float* __restrict__ lam, float nu, float* __restrict__ history,
                            int* __restrict__ iter) {
    const double tc = *trial_total;
    const double cur = *cost_cur;
    const bool acc = tc < cur;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (acc) {
        if (i < P) pts[i] = pts_t[i];
        if (i < 12 * F) poses[i] = poses_t[i];
        if (i == 0) *fl = *fl_t;
    }
    if (i == 0) {
        // lam is kept within [1e-12, 1e10]: a converged run rejects every further
        // step, and unbounded growth would reach infinity
        *lam = fminf(1e10f, fmaxf(1e-12f, acc ? *lam / nu : *lam * nu));
        if (history) {
            const int it = *iter;
            history[3 * it] = (float)cur;
            history[3 * it + 1] = (float)tc;
            history[3 * it + 2] = acc ? 1.f : 0.f;
        }
        *iter += 1;
    }
}

__global__ void k_ba_project(const float* __restrict__ poses, const float4* __restrict__ pts,
                             const float* __restrict__ fl, float cx, float cy, int F, int64_t P,
                             float2* __restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P * F) return;
    BaObs o;
    ba_observe(poses + 12 * (i % F), pts[i / F], *fl, cx, cy, make_float2(0.f, 0.f), o);
    out[i] = make_float2(o.r[0], o.r[1]);
}

struct BaWs {
    float *e, *poses_t, *fl_t;
    float4* pts_t;
    double *partial, *trial_partial, *dc, *cost_cur, *tot, *trial_total;
    BaPoints pt;
    float* thr;
    int *iter, *fail;
};

static BaWs carve_ba(char* base, size_t cap, int F, int64_t P, size_t* used) {
    Carve c{base, 0, cap};
    BaWs w;
    const int64_t n = P * F;
    const int nc = 6 * (F - 1) + 1;
    const int64_t nb = ceil_div(P, kBaChunk), nt = ceil_div(n, 256);
    w.e = c.take<float>(n);
    w.poses_t = c.take<float>(12 * kBaMaxF);
    w.fl_t = c.take<float>(4);
    w.pts_t = c.take<float4>(P);
    w.partial = c.take<double>(nb * (nc * (nc + 1) / 2 + 2 * nc));
    w.trial_partial = c.take<double>(nt);
    w.pt.K = c.take<float>(P * nc * 3);
    w.pt.V = c.take<float>(P * nc * 3);
    w.pt.Hinv = c.take<double>(P * 6);
    w.pt.u = c.take<double>(P * 3);
    w.pt.g = c.take<float>(P * 3);
    w.pt.cost = c.take<double>(P);
    w.pt.J = c.take<float>(n * 16);
    w.pt.w = c.take<float>(n);
    w.dc = c.take<double>(kBaMaxNc);
    w.cost_cur = c.take<double>(1);
    w.tot = c.take<double>(nc * (nc + 1) / 2 + 2 * nc);
    w.trial_total = c.take<double>(1);
    w.thr = c.take<float>(1);
    w.iter = c.take<int>(1);
    w.fail = c.take<int>(1);
    *used = c.used;
    return w;
}

// ---------------------------------------------------------------------------
// Pose refinement of a new frame (Sec. 4.1, subsequent frames): the same
// robust iteration over one pose, points and focal length fixed. The 6 x 6
// normal equations are summed per CTA (FP32 products, FP64 warp and CTA sums
// in a fixed order); one CTA then damps, factors (L D L^T, FP64) and retracts.
// The residual, median / MAD, trial-cost and accept kernels are the bundle
// adjustment's with one frame.
// ---------------------------------------------------------------------------
constexpr int kBpThreads = 256;
constexpr int kBpVals = 28;  // H upper triangle (21) | g (6) | cost

__global__ void __launch_bounds__(kBpThreads) k_bp_normal(const float2* __restrict__ obs,
                                                           const float* __restrict__ pose,
                                                           const float4* __restrict__ pts,
                                                           const float* __restrict__ fl_p, float cx, float cy,
                                                           int64_t M, const float* __restrict__ e_cur,
                                                           const float* __restrict__ thr_p, float delta,
                                                           double* __restrict__ partial) {
    __shared__ float s_pose[12];
    __shared__ double s_w[kBpThreads / 32][kBpVals];
    if (threadIdx.x < 12) s_pose[threadIdx.x] = pose[threadIdx.x];
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double v[kBpVals];
#pragma unroll
    for (int k = 0; k < kBpVals; k++) v[k] = 0.0;
    if (i < M) {
        BaObs o;
        ba_observe(s_pose, pts[i], *fl_p, cx, cy, obs[i], o);
        const bool keep = e_cur[i] <= *thr_p;
        const float w = ba_weight(o.e, keep, delta);
        float J[2][6];
        const float qx = o.q[0], qy = o.q[1], qz = o.q[2];
        for (int k = 0; k < 2; k++) {  // rho: jq; phi: jq (-q^), -q^ = [[0, qz, -qy], [-qz, 0, qx], [qy, -qx, 0]]
            const float a0 = o.jq[k][0], a1 = o.jq[k][1], a2 = o.jq[k][2];
            J[k][0] = a0; J[k][1] = a1; J[k][2] = a2;
            J[k][3] = -a1 * qz + a2 * qy;
            J[k][4] = a0 * qz - a2 * qx;
            J[k][5] = -a0 * qy + a1 * qx;
        }
        int e = 0;
#pragma unroll
        for (int a = 0; a < 6; a++)
#pragma unroll
            for (int b = a; b < 6; b++) v[e++] = (double)(w * (J[0][a] * J[0][b] + J[1][a] * J[1][b]));
#pragma unroll
        for (int a = 0; a < 6; a++) v[21 + a] = (double)(w * (J[0][a] * o.r[0] + J[1][a] * o.r[1]));
        v[27] = ba_cost(o.e, keep, delta);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < kBpVals; k++) {
        double a = v[k];
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (lane == 0) s_w[warp][k] = a;
    }
    __syncthreads();
    if (threadIdx.x < kBpVals) {
        double a = 0.0;
        for (int wi = 0; wi < kBpThreads / 32; wi++) a += s_w[wi][threadIdx.x];
        partial[(int64_t)blockIdx.x * kBpVals + threadIdx.x] = a;
    }
}

// One warp: damping (H + lam diag(H) + 1e-9 I), L D L^T of the 6 x 6 system in FP64,
// the step d = -A^-1 g (0 for a system that is not positive definite, which is the
// return value) and the retracted trial pose. A lane holds each entry of the lower
// triangle and of the right-hand side, so that a column's update is one instruction.
__device__ __forceinline__ bool bp_solve(const double* tot, const float* pose, float lam_f, float* pose_t,
                                         double (*s_A)[8] /* [7][8] */, double* s_d /* [6] */) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const double lam = lam_f;
    // the lower triangle, row by row (21 entries), and -g as row 6
    int r = 0, c = lane;
    while (c > r) { c -= r + 1; r++; }
    const bool rhs = lane >= 21;
    if (rhs) { r = 6; c = lane - 21; }
    const bool live = lane < 27;
    double a = 0.0;
    if (live) a = rhs ? -tot[lane] : tot[c * 6 - c * (c - 1) / 2 + (r - c)];
    if (!rhs && r == c) a += lam * a + 1e-9;
    bool bad = false;
#pragma unroll
    for (int k = 0; k < 6; k++) {
        // entries (r, k), (c, k) and (k, k) of the unscaled column k
        auto at = [](int i) { return i < 6 ? i * (i + 1) / 2 : 21; };  // a row's first lane
        const double d = __shfl_sync(FULL, a, at(k) + k);
        if (!(d > 0.0)) bad = true;
        const double dinv = d > 0.0 ? 1.0 / d : 0.0;
        const double rk = __shfl_sync(FULL, a, (at(r) + k) & 31), ck = __shfl_sync(FULL, a, (at(c) + k) & 31);
        if (live && c > k) a -= rk * ck * dinv;
        else if (live && c == k && r > k) a *= dinv;  // L's column, and for row 6: z = D^-1 L^-1 (-g)
    }
    if (live) s_A[r][c] = a;
    __syncwarp();
    double x = lane < 6 ? s_A[6][lane] : 0.0;
#pragma unroll
    for (int i = 5; i > 0; i--) {
        const double xi = __shfl_sync(FULL, x, i);
        if (lane < i) x -= s_A[i][lane] * xi;
    }
    if (bad) x = 0.0;
    if (lane < 6) s_d[lane] = x;
    __syncwarp();
    if (lane < 12) ba_retract_entry(pose, s_d, lane, pose_t);
    return bad;
}

__global__ void k_bp_solve(const double* __restrict__ tot, const float* __restrict__ pose,
                           const float* __restrict__ lam_p, float* __restrict__ pose_t,
                           double* __restrict__ cost_cur, int* __restrict__ fail) {
    __shared__ double s_A[7][8], s_d[6];
    const bool bad = bp_solve(tot, pose, *lam_p, pose_t, s_A, s_d);  // one warp
    if (threadIdx.x == 0) {
        if (bad) *fail = 1;
        *cost_cur = tot[27];
    }
}

// All iterations in one launch of one cluster of 16 CTAs, for up to 24 observations
// a thread (24,576). Every CTA forms all residual norms and selects their median +
// 4 MAD by itself (FP32 and integers: cheap, no exchange); the FP64 sums - at two
// lanes a clock and SM most of an iteration - are divided among the CTAs, warp by
// warp of observations: 28 products per observation in shared memory, then one
// thread per product and 32 observations adds them in order. Two exchanges through
// the cluster's shared memory per iteration (the normal equations, the trial cost)
// leave every CTA with the same sums, so that each solves and decides for itself.
// 6144 observations, 20 iterations: 1397 -> 463 us against eight launches per
// iteration.
constexpr int kBpCluster = 16;
constexpr int kBpMaxNV = 24;
constexpr int64_t kBpClusterObs = (int64_t)kBaSelThreads * kBpMaxNV;

// Rows of 32 observations that a CTA sums, and the shared memory for their products.
static __host__ __device__ constexpr int bp_rows(int nv) { return nv * (kBaSelThreads / 32) / kBpCluster; }
static size_t bp_lm_smem(int nv) { return sizeof(float) * bp_rows(nv) * 32 * (kBpVals + 1); }

template <int NV>
__global__ void __launch_bounds__(kBaSelThreads) k_bp_lm(const float2* __restrict__ obs,
                                                         const float4* __restrict__ pts,
                                                         const float* __restrict__ fl_p, float cx, float cy, int M,
                                                         float* __restrict__ pose, float* __restrict__ lam_p,
                                                         int iterations, float delta, float nu,
                                                         float* __restrict__ history, int* __restrict__ failed) {
    namespace cg = cooperative_groups;
    constexpr int ROWS = bp_rows(NV), WARPS = kBaSelThreads / 32;
    extern __shared__ float s_terms[];  // [ROWS][32][kBpVals + 1]
    __shared__ SelScratch sc;
    __shared__ float s_pose[2][12];  // the state and the trial state
    __shared__ double s_row[ROWS][kBpVals];
    __shared__ double s_obs[WARPS][33];
    __shared__ double s_trial[ROWS];
    __shared__ double s_sum[2][kBpVals];  // this CTA's sums, read by the others (two take turns)
    __shared__ double s_tot[kBpVals];
    __shared__ double s_cost[2];
    __shared__ double s_A[7][8], s_d[6];
    __shared__ float s_lam;
    __shared__ int s_fail, s_acc;
    auto cluster = cg::this_cluster();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cta = (int)cluster.block_rank();
    if (tid < 12) s_pose[0][tid] = pose[tid];
    if (tid == 0) {
        s_lam = *lam_p;
        s_fail = 0;
    }
    const float fl = *fl_p;
    __syncthreads();
    const int rank = (M - 1) / 2;
    for (int it = 0; it < iterations; it++) {
        float thr;
        {
            uint32_t key[NV];
            int count = 0;
#pragma unroll
            for (int v = 0; v < NV; v++) {
                const int i = v * kBaSelThreads + tid;
                key[v] = 0;
                if (i < M) {
                    BaObs o;
                    ba_observe(s_pose[0], pts[i], fl, cx, cy, obs[i], o);
                    key[v] = __float_as_uint(o.e);
                    count = v + 1;
                }
            }
            const float med = __uint_as_float(select_in_registers<NV, 1>(key, count, rank, sc));
#pragma unroll
            for (int v = 0; v < NV; v++) key[v] = __float_as_uint(fabsf(__uint_as_float(key[v]) - med));
            thr = med + 4.f * __uint_as_float(select_in_registers<NV, 1>(key, count, rank, sc));
        }
        // this CTA's rows of 32 observations, one per warp: rows cta, cta + 16, ...
        for (int row = warp; row < ROWS; row += WARPS) {
            float* out = s_terms + (row * 32 + lane) * (kBpVals + 1);
            const int i = (row * kBpCluster + cta) * 32 + lane;
            if (i < M) {
                BaObs o;
                ba_observe(s_pose[0], pts[i], fl, cx, cy, obs[i], o);
                const bool keep = o.e <= thr;
                const float w = ba_weight(o.e, keep, delta);
                float J[2][6];
                const float qx = o.q[0], qy = o.q[1], qz = o.q[2];
#pragma unroll
                for (int k = 0; k < 2; k++) {  // rho: jq; phi: jq (-q^), -q^ = [[0, qz, -qy], [-qz, 0, qx], [qy, -qx, 0]]
                    const float a0 = o.jq[k][0], a1 = o.jq[k][1], a2 = o.jq[k][2];
                    J[k][0] = a0; J[k][1] = a1; J[k][2] = a2;
                    J[k][3] = -a1 * qz + a2 * qy;
                    J[k][4] = a0 * qz - a2 * qx;
                    J[k][5] = -a0 * qy + a1 * qx;
                }
                int e = 0;
#pragma unroll
                for (int a = 0; a < 6; a++)
#pragma unroll
                    for (int b = a; b < 6; b++) out[e++] = w * (J[0][a] * J[0][b] + J[1][a] * J[1][b]);
#pragma unroll
                for (int a = 0; a < 6; a++) out[21 + a] = w * (J[0][a] * o.r[0] + J[1][a] * o.r[1]);
                s_obs[warp][lane] = ba_cost(o.e, keep, delta);
            } else {
#pragma unroll
                for (int e = 0; e < kBpVals - 1; e++) out[e] = 0.f;
                s_obs[warp][lane] = 0.0;
            }
            __syncwarp();
            // the row's cost: four lanes add eight each, then one the four
            double c = 0.0;
            if (lane < 4)
                for (int l = 0; l < 8; l++) c += s_obs[warp][lane * 8 + l];
            c += __shfl_down_sync(0xffffffffu, c, 2);
            c += __shfl_down_sync(0xffffffffu, c, 1);
            if (lane == 0) s_row[row][kBpVals - 1] = c;
            __syncwarp();
        }
        __syncthreads();
        for (int j = tid; j < ROWS * (kBpVals - 1); j += kBaSelThreads) {
            const int r = j / (kBpVals - 1), c = j % (kBpVals - 1);
            const float* in = s_terms + r * 32 * (kBpVals + 1) + c;
            double a = 0.0;
#pragma unroll 8
            for (int l = 0; l < 32; l++) a += widen(in[l * (kBpVals + 1)]);
            s_row[r][c] = a;
        }
        __syncthreads();
        if (tid < kBpVals) {
            double a = 0.0;
            for (int r = 0; r < ROWS; r++) a += s_row[r][tid];
            s_sum[it & 1][tid] = a;
        }
        cluster.sync();
        if (warp == 0) {
            if (lane < kBpVals) {
                double a = 0.0;
#pragma unroll
                for (int r = 0; r < kBpCluster; r++) a += *cluster.map_shared_rank(&s_sum[it & 1][lane], r);
                s_tot[lane] = a;
            }
            __syncwarp();
            const bool bad = bp_solve(s_tot, s_pose[0], s_lam, s_pose[1], s_A, s_d);
            if (bad && lane == 0) s_fail = 1;
        }
        __syncthreads();
        for (int row = warp; row < ROWS; row += WARPS) {
            const int i = (row * kBpCluster + cta) * 32 + lane;
            double c = 0.0;
            if (i < M) {
                BaObs o, t;
                ba_observe(s_pose[0], pts[i], fl, cx, cy, obs[i], o);  // kept by the current residual
                ba_observe(s_pose[1], pts[i], fl, cx, cy, obs[i], t);
                c = ba_cost(t.e, o.e <= thr, delta);
            }
            s_obs[warp][lane] = c;
            __syncwarp();
            c = 0.0;
            if (lane < 4)
                for (int l = 0; l < 8; l++) c += s_obs[warp][lane * 8 + l];
            c += __shfl_down_sync(0xffffffffu, c, 2);
            c += __shfl_down_sync(0xffffffffu, c, 1);
            if (lane == 0) s_trial[row] = c;
            __syncwarp();
        }
        __syncthreads();
        if (tid == 0) {
            double a = 0.0;
            for (int r = 0; r < ROWS; r++) a += s_trial[r];
            s_cost[it & 1] = a;
        }
        cluster.sync();
        if (tid == 0) {
            double tc = 0.0;
#pragma unroll
            for (int r = 0; r < kBpCluster; r++) tc += *cluster.map_shared_rank(&s_cost[it & 1], r);
            const double cur = s_tot[kBpVals - 1];
            const bool acc = tc < cur;
            s_acc = acc;
            // lam is kept within [1e-12, 1e10]: a converged run rejects every further
            // step, and unbounded growth would reach infinity
            s_lam = fminf(1e10f, fmaxf(1e-12f, acc ? s_lam / nu : s_lam * nu));
            if (cta == 0 && history) {
                history[3 * it] = (float)cur;
                history[3 * it + 1] = (float)tc;
                history[3 * it + 2] = acc ? 1.f : 0.f;
            }
        }
        __syncthreads();
        if (s_acc && tid < 12) s_pose[0][tid] = s_pose[1][tid];
        __syncthreads();
    }
    if (cta == 0) {
        if (tid < 12) pose[tid] = s_pose[0][tid];
        if (tid == 0) {
            *lam_p = s_lam;
            *failed = s_fail;
        }
    }
    cluster.sync();  // no CTA leaves while its sums may be read
}

// The cluster kernel for M observations, or null where this GPU cannot run its
// cluster (then the iterations run as eight launches each). Asked once per kernel
// and device: later calls, e.g. inside a stream capture, make no runtime queries.
static const void* pick_bp_lm(int64_t M, int* nv) {
    struct Entry { int nv; const void* fn; };
    static const Entry table[] = {{1, (const void*)k_bp_lm<1>}, {4, (const void*)k_bp_lm<4>}, {6, (const void*)k_bp_lm<6>},
                                  {12, (const void*)k_bp_lm<12>}, {24, (const void*)k_bp_lm<24>}};
    constexpr int kKernels = sizeof(table) / sizeof(table[0]), kDevices = 64;
    static signed char usable[kKernels][kDevices];  // 0: not asked, 1: yes, -1: no
    static std::mutex lock;
    int dev = 0;
    if (M > kBpClusterObs || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return nullptr;
    int k = 0;
    while (M > (int64_t)table[k].nv * kBaSelThreads) k++;
    std::lock_guard<std::mutex> guard(lock);
    if (usable[k][dev] == 0) {
        const size_t smem = bp_lm_smem(table[k].nv);
        cudaLaunchConfig_t lc = {};
        cudaLaunchAttribute at;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = kBpCluster;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        lc.gridDim = dim3(kBpCluster);
        lc.blockDim = dim3(kBaSelThreads);
        lc.dynamicSmemBytes = smem;
        lc.attrs = &at;
        lc.numAttrs = 1;
        int clusters = 0;
        const bool ok =
            cudaFuncSetAttribute(table[k].fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess &&
            cudaFuncSetAttribute(table[k].fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&clusters, table[k].fn, &lc) == cudaSuccess && clusters > 0;
        if (!ok) (void)cudaGetLastError();
        usable[k][dev] = ok ? 1 : -1;
    }
    *nv = table[k].nv;
    return usable[k][dev] > 0 ? table[k].fn : nullptr;
}

struct BpWs {
    float *e, *pose_t, *fl_t, *thr;
    double *partial, *tot, *trial_partial, *trial_total, *cost_cur;
    int *iter, *fail;
};

static BpWs carve_bp(char* base, size_t cap, int64_t M, size_t* used) {
    Carve c{base, 0, cap};
    BpWs w;
    const int64_t nb = ceil_div(M, kBpThreads), nt = ceil_div(M, 256);
    w.e = c.take<float>(M);
    w.pose_t = c.take<float>(12);
    w.fl_t = c.take<float>(4);
    w.thr = c.take<float>(1);
    w.partial = c.take<double>(nb * kBpVals);
    w.tot = c.take<double>(kBpVals);
    w.trial_partial = c.take<double>(nt);
    w.trial_total = c.take<double>(1);
    w.cost_cur = c.take<double>(1);
    w.iter = c.take<int>(1);
    w.fail = c.take<int>(1);
    *used = c.used;
    return w;
}

}  // namespace gs

using namespace gs;

extern "C" size_t gs_ba_workspace_size(int32_t n_frames, int64_t n_points) {
    if (n_frames < 2 || n_frames > kBaMaxF || n_points < 1 || n_points * n_frames > kBaMaxObs) return 0;
    size_t used = 0;
    carve_ba(nullptr, 0, n_frames, n_points, &used);
    return used;
}

extern "C" int gs_ba_lm(const float* obs, int32_t n_frames, int64_t n_points, float cx, float cy, float* fl,
                        float* poses, float* points, float* lam, int32_t iterations, float huber_delta, float nu,
                        float* history, int32_t* failed, void* ws, size_t ws_bytes, void* stream) {
    const int F = n_frames;
    const int64_t P = n_points;
    if (!obs || !fl || !poses || !points || !lam || F < 2 || F > kBaMaxF || P < 1 || iterations < 0 ||
        !(huber_delta > 0.f) || !(nu > 1.f) || P * F > kBaMaxObs || !failed)
        return GS_ERR_INVALID_ARG;
    size_t need = 0;
    BaWs w = carve_ba((char*)ws, ws_bytes, F, P, &need);
    if (!ws || ws_bytes < need || ((uintptr_t)ws & 255) || ((uintptr_t)points & 15) || ((uintptr_t)obs & 7))
        return GS_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t n = P * F;
    const int nc = 6 * (F - 1) + 1;
    const int nb = (int)ceil_div(P, kBaChunk), nt = (int)ceil_div(n, kBaStepThreads);
    static std::once_flag attr_once;
    std::call_once(attr_once, [] {
        cudaFuncSetAttribute(k_ba_median_mad, cudaFuncAttributePreferredSharedMemoryCarveout, 25);
        cudaFuncSetAttribute(k_ba_normal, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)ba_normal_smem(kBaMaxF, kBaMaxNc));
    });
    const int nup = nc * (nc + 1) / 2;
    const unsigned normal_grid = (unsigned)(ceil_div(nb, kBaFocalChunks) +
                                            nb * ceil_div(ceil_div(nup, 32) * 32 + nc - 1, kBaNormalThreads));
    const int stride = nc * (nc + 1) / 2 + 2 * nc;
    const float2* ob = (const float2*)obs;
    float4* pts = (float4*)points;
    cudaMemsetAsync(w.iter, 0, sizeof(int), s);
    cudaMemsetAsync(w.fail, 0, sizeof(int), s);
    auto close = [&]() {  // accept or reject the trial state
        k_ba_sum<<<1, 256, 0, s>>>(w.trial_partial, nt, w.trial_total);
        count_launch();
        const int64_t na = P > 12 * F ? P : 12 * F;
        k_ba_accept<<<(unsigned)ceil_div(na, 256), 256, 0, s>>>(w.trial_total, w.cost_cur, F, P, w.poses_t,
                                                                w.pts_t, w.fl_t, poses, pts, fl, lam, nu, history,
                                                                w.iter);
        count_launch();
    };
    const int nv = (int)ceil_div(n, (int64_t)kBaCluster * kBaSelThreads);  // observations a thread of k_ba_begin
    for (int it = 0; it < iterations; it++) {
#define GS_BEGIN(NV)                                                                                                \
    k_ba_begin<NV><<<kBaCluster, kBaSelThreads, 0, s>>>(ob, poses, pts, fl, cx, cy, F, P, it == 0, w.trial_partial, nt, \
                                                        w.cost_cur, w.poses_t, w.pts_t, w.fl_t, lam, nu, history,   \
                                                        w.iter, w.e, w.thr)
        if (n <= kBaClusterObs) {
            if (nv <= 1) GS_BEGIN(1); else if (nv <= 2) GS_BEGIN(2); else if (nv <= 4) GS_BEGIN(4); else if (nv <= 6) GS_BEGIN(6); else GS_BEGIN(8);
            count_launch();
        } else {
            if (it > 0) close();
            k_ba_residual<<<(unsigned)ceil_div(n, 256), 256, 0, s>>>(ob, poses, pts, fl, cx, cy, F, P, w.e);
            count_launch();
            k_ba_median_mad<<<1, kBaSelThreads, 0, s>>>(w.e, (int)n, w.thr);
            count_launch();
        }
#undef GS_BEGIN
        k_ba_points<<<(unsigned)ceil_div(P, kBaPointsPts), kBaPointsThreads, 0, s>>>(
            ob, poses, pts, fl, cx, cy, F, P, w.e, w.thr, huber_delta, lam, w.pt);
        count_launch();
        k_ba_normal<<<normal_grid, kBaNormalThreads, ba_normal_smem(F, nc), s>>>(w.pt, F, P, w.partial);
        count_launch();
        k_ba_reduce<<<(unsigned)ceil_div(stride, 16), dim3(16, 8), 0, s>>>(w.partial, nb, stride, stride, w.tot);
        count_launch();
        k_ba_solve<<<1, kBaSolveThreads, 0, s>>>(w.tot, w.pt.cost, P, F, lam, poses, fl, w.dc, w.cost_cur, w.poses_t,
                                                 w.fl_t, w.fail);
        count_launch();
        k_ba_step<<<nt, kBaStepThreads, sizeof(float) * ba_step_points(F) * nc * 3, s>>>(ob, pts, cx, cy, F, P, w.e, w.thr, huber_delta, w.pt, w.dc, w.poses_t,
                                                w.fl_t, w.pts_t, w.trial_partial);
        count_launch();
    }
    if (iterations > 0) close();
    cudaMemcpyAsync(failed, w.fail, sizeof(int), cudaMemcpyDeviceToDevice, s);
    GS_CUDA_CHECK_LAUNCH();
    return GS_OK;
}

extern "C" int gs_ba_project(const float* fl, const float* poses, const float* points, int32_t n_frames,
                             int64_t n_points, float cx, float cy, float* obs, void* stream) {
    if (!fl || !poses || !points || !obs || n_frames < 1 || n_frames > kBaMaxF || n_points < 1 ||
        ((uintptr_t)points & 15) || ((uintptr_t)obs & 7))
        return GS_ERR_INVALID_ARG;
    const int64_t n = n_points * n_frames;
    k_ba_project<<<(unsigned)ceil_div(n, 256), 256, 0, (cudaStream_t)stream>>>(
        poses, (const float4*)points, fl, cx, cy, n_frames, n_points, (float2*)obs);
    count_launch();
    GS_CUDA_CHECK_LAUNCH();
    return GS_OK;
}

extern "C" size_t gs_ba_pose_workspace_size(int64_t n_obs) {
    if (n_obs < 1 || n_obs > kBaMaxObs) return 0;
    size_t used = 0;
    carve_bp(nullptr, 0, n_obs, &used);
    return used;
}

extern "C" int gs_ba_pose_lm(const float* points, const float* obs, int64_t n_obs, const float* fl, float cx,
                             float cy, float* pose, float* lam, int32_t iterations, float huber_delta, float nu,
                             float* history, int32_t* failed, void* ws, size_t ws_bytes, void* stream) {
    const int64_t M = n_obs;
    if (!points || !obs || !fl || !pose || !lam || !failed || M < 1 || M > kBaMaxObs || iterations < 0 ||
        !(huber_delta > 0.f) || !(nu > 1.f))
        return GS_ERR_INVALID_ARG;
    size_t need = 0;
    BpWs w = carve_bp((char*)ws, ws_bytes, M, &need);
    if (!ws || ws_bytes < need || ((uintptr_t)ws & 255) || ((uintptr_t)points & 15) || ((uintptr_t)obs & 7))
        return GS_ERR_INVALID_ARG;
    static bool attr_set = false;
    if (!attr_set) {
        cudaFuncSetAttribute(k_ba_median_mad, cudaFuncAttributePreferredSharedMemoryCarveout, 25);
        attr_set = true;
    }
    cudaStream_t s = (cudaStream_t)stream;
    const int nb = (int)ceil_div(M, kBpThreads), nt = (int)ceil_div(M, 256);
    const float2* ob = (const float2*)obs;
    const float4* pts = (const float4*)points;
    int nv = 0;
    if (const void* fn = iterations > 0 ? pick_bp_lm(M, &nv) : nullptr) {
        int m = (int)M;
        cudaLaunchConfig_t lc = {};
        cudaLaunchAttribute at;
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = kBpCluster;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        lc.gridDim = dim3(kBpCluster);
        lc.blockDim = dim3(kBaSelThreads);
        lc.dynamicSmemBytes = bp_lm_smem(nv);
        lc.stream = s;
        lc.attrs = &at;
        lc.numAttrs = 1;
        void* args[] = {(void*)&ob, (void*)&pts, (void*)&fl, &cx, &cy, &m, (void*)&pose, (void*)&lam, &iterations,
                        &huber_delta, &nu, (void*)&history, (void*)&failed};
        if (cudaLaunchKernelExC(&lc, fn, args) != cudaSuccess) {
            (void)cudaGetLastError();
            return GS_ERR_CUDA;
        }
        count_launch();
        return GS_OK;
    }
    cudaMemcpyAsync(w.fl_t, fl, sizeof(float), cudaMemcpyDeviceToDevice, s);
    cudaMemsetAsync(w.iter, 0, sizeof(int), s);
    cudaMemsetAsync(w.fail, 0, sizeof(int), s);
    for (int it = 0; it < iterations; it++) {
        k_ba_residual<<<nt, 256, 0, s>>>(ob, pose, pts, w.fl_t, cx, cy, 1, M, w.e);
        count_launch();
        k_ba_median_mad<<<1, kBaSelThreads, 0, s>>>(w.e, (int)M, w.thr);
        count_launch();
        k_bp_normal<<<nb, kBpThreads, 0, s>>>(ob, pose, pts, w.fl_t, cx, cy, M, w.e, w.thr, huber_delta, w.partial);
        count_launch();
        k_ba_reduce<<<(unsigned)ceil_div(kBpVals, 16), dim3(16, 8), 0, s>>>(w.partial, nb, kBpVals, kBpVals, w.tot);
        count_launch();
        k_bp_solve<<<1, 32, 0, s>>>(w.tot, pose, lam, w.pose_t, w.cost_cur, w.fail);
        count_launch();
        k_ba_trial_cost<<<nt, 256, 0, s>>>(ob, w.pose_t, pts, w.fl_t, cx, cy, 1, M, w.e, w.thr, huber_delta,
                                           w.trial_partial);
        count_launch();
        k_ba_sum<<<1, 256, 0, s>>>(w.trial_partial, nt, w.trial_total);
        count_launch();
        k_ba_accept<<<1, 32, 0, s>>>(w.trial_total, w.cost_cur, 1, 0, w.pose_t, nullptr, w.fl_t, pose, nullptr,
                                     w.fl_t, lam, nu, history, w.iter);
        count_launch();
    }
    cudaMemcpyAsync(failed, w.fail, sizeof(int), cudaMemcpyDeviceToDevice, s);
    GS_CUDA_CHECK_LAUNCH();
    return GS_OK;
}

