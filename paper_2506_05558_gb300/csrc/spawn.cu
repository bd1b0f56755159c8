// Direct spawn sampling (Sec. 4.2): per-pixel spawn probability from the norm
// of the Laplacian-of-Gaussian response of the input image (Eq. 1), the same
// quantity on the current render as a penalty (Eq. 2), their clamped
// difference (Eq. 3), a Bernoulli mask drawn with a counter-based generator,
// and, for every spawning pixel, a new Gaussian at the supplied depth with the
// expected nearest-neighbour scale s = z / (2 f sqrt(P_L)).
//
// k_spawn_maps forms the maps and the mask (one bit per pixel, 32 pixels of a row
// to a word), the words' counts are scanned in pixel order in one launch, and
// k_spawn_rows writes the spawned rows. A 1080p proposal with its maps takes 64 us;
// with a word per pixel, its scan in three launches and P_L formed twice it took 235.
#include <algorithm>
#include <cmath>
#include <cuda.h>
#include <mutex>

#include "common.cuh"

namespace gs {

constexpr int kSpMaxR = 8;
constexpr int kSpMaxTaps = (2 * kSpMaxR + 1) * (2 * kSpMaxR + 1);

struct LogTaps {
    int R;
    float w[kSpMaxTaps];
};

// A CTA takes 64 x 16 pixels, a thread 4 x 2 of them: the values of an input row that
// it loads, 128 bits at a time, serve both its output rows, and up to radius 3 (sigma
// 1) the rows are unrolled, so that each tap is the FMA's constant operand. Each pixel
// adds its taps row by row, left to right. The picture and then the render pass
// through the same shared tile, which leaves room for eleven CTAs per SM.
// 1080p, sigma = 1, two images: 610M FMAs, 16 us at the FP32 peak; 42 us, bound by issue
// (68% of slots; the draws and the staging are half of them) and by 1.5 waves of CTAs.
// One pixel per thread with tap loads took 95 us, and as much again for P_L when the
// rows were written.
constexpr int kSpW = 64, kSpH = 16;
constexpr int kSpThreads = 128;
constexpr int kSpMaxHeight = 65535 * kSpH;  // a grid's y extent

template <int R>
struct SpTile {
    static constexpr int kPad = (R + 3) / 4 * 4;  // columns left and right of the tile
    static constexpr int kRows = kSpH + 2 * R;
    static constexpr int kVec = (4 + 2 * kPad) / 4;  // 128-bit loads per input row and thread
    static constexpr int kPitch = kSpW + 2 * kPad;
    static constexpr size_t kBytes = sizeof(float) * 3 * kRows * kPitch;
};

// The tile with its halo, borders replicated. vec: the width is a multiple of 4 and
// the image 16-byte aligned, so that four columns are inside or outside together.
template <int R>
__device__ __forceinline__ void stage_tile(const float* __restrict__ img, int W, int H, int x0, int y0, bool vec,
                                           float* s) {
    using T = SpTile<R>;
    const int64_t plane = (int64_t)W * H;
    if (vec) {
        constexpr int kCols = T::kPitch / 4;
#pragma unroll 4
        for (int i = threadIdx.x; i < T::kRows * kCols; i += kSpThreads) {
            const int r = i / kCols, x = x0 - T::kPad + 4 * (i % kCols);
            const float* row = img + (int64_t)min(max(y0 - R + r, 0), H - 1) * W;
#pragma unroll
            for (int ch = 0; ch < 3; ch++) {
                float4 f;
                if (x >= 0 && x < W) {
                    f = *reinterpret_cast<const float4*>(row + ch * plane + x);
                } else {
                    f.x = row[ch * plane + (x < 0 ? 0 : W - 1)];
                    f.y = f.z = f.w = f.x;
                }
                reinterpret_cast<float4*>(s)[ch * T::kRows * kCols + i] = f;
            }
        }
    } else {
        for (int i = threadIdx.x; i < 3 * T::kRows * T::kPitch; i += kSpThreads) {
            const int r = i / T::kPitch, x = x0 - T::kPad + i % T::kPitch;
            s[i] = img[r / T::kRows * plane + (int64_t)min(max(y0 - R + r % T::kRows, 0), H - 1) * W +
                       min(max(x, 0), W - 1)];
        }
    }
}

// min(|LoG response|, 1) of this thread's 2 x 4 pixels.
template <int R>
__device__ __forceinline__ void log_norms(const float* s, const LogTaps& k, float (&out)[2][4]) {
    using T = SpTile<R>;
    constexpr int N = 2 * R + 1;
    const int gx = threadIdx.x % (kSpW / 4), gy = threadIdx.x / (kSpW / 4);
    float a[3][2][4];
#pragma unroll
    for (int ch = 0; ch < 3; ch++) {
#pragma unroll
        for (int o = 0; o < 2; o++)
#pragma unroll
            for (int p = 0; p < 4; p++) a[ch][o][p] = 0.f;
        const float* base = s + (ch * T::kRows + 2 * gy) * T::kPitch + 4 * gx;
        // input row r is tap row r of the upper output row and r - 1 of the lower
        auto row = [&](int r) {
            float v[4 * T::kVec];
#pragma unroll
            for (int q = 0; q < T::kVec; q++) {
                const float4 f = reinterpret_cast<const float4*>(base + r * T::kPitch)[q];
                v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
            }
            if (r < N)
#pragma unroll
                for (int i = 0; i < N; i++)
#pragma unroll
                    for (int p = 0; p < 4; p++) a[ch][0][p] += k.w[r * N + i] * v[T::kPad - R + i + p];
            if (r > 0)
#pragma unroll
                for (int i = 0; i < N; i++)
#pragma unroll
                    for (int p = 0; p < 4; p++) a[ch][1][p] += k.w[(r - 1) * N + i] * v[T::kPad - R + i + p];
        };
        if constexpr (R <= 3) {
#pragma unroll
            for (int r = 0; r <= N; r++) row(r);
        } else {
#pragma unroll 1
            for (int r = 0; r <= N; r++) row(r);
        }
    }
#pragma unroll
    for (int o = 0; o < 2; o++)
#pragma unroll
        for (int p = 0; p < 4; p++) {
            const float a0 = a[0][o][p], a1 = a[1][o][p], a2 = a[2][o][p];
            out[o][p] = fminf(sqrtf(a0 * a0 + a1 * a1 + a2 * a2), 1.f);
        }
}

// vec: the width is a multiple of 4 and the images, depth and the maps are 16-byte
// aligned.
// mask (direct sampling; the learned proposal only needs the maps): one word per 32
// pixels of a row; p_l_spawn: P_L of the spawning pixels only, or null. Clears the
// scan's words for the launch that follows.
template <int R>
__global__ void __launch_bounds__(kSpThreads) k_spawn_maps(const float* __restrict__ image,
                                                           const float* __restrict__ render,
                                                           const float* __restrict__ depth, int W, int H,
                                                           const __grid_constant__ LogTaps taps, uint2 key,
                                                           uint32_t frame, bool vec, float* __restrict__ p_l,
                                                           float* __restrict__ p_pen, float* __restrict__ p_s,
                                                           uint32_t* __restrict__ mask,
                                                           float* __restrict__ p_l_spawn,
                                                           uint32_t* __restrict__ scan_words, int n_scan_words) {
    extern __shared__ __align__(16) float s_tile[];
    const int x0 = blockIdx.x * kSpW, y0 = blockIdx.y * kSpH;
    for (int64_t i = ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * kSpThreads + threadIdx.x; i < n_scan_words;
         i += (int64_t)gridDim.x * gridDim.y * kSpThreads)
        scan_words[i] = 0;
    float pl[2][4], pp[2][4];
    stage_tile<R>(image, W, H, x0, y0, vec, s_tile);
    __syncthreads();
    log_norms<R>(s_tile, taps, pl);
    if (render) {
        __syncthreads();
        stage_tile<R>(render, W, H, x0, y0, vec, s_tile);
        __syncthreads();
        log_norms<R>(s_tile, taps, pp);
    }
    const int gx = threadIdx.x % (kSpW / 4), gy = threadIdx.x / (kSpW / 4);
    const int x = x0 + 4 * gx;
#pragma unroll
    for (int o = 0; o < 2; o++) {
        const int y = y0 + 2 * gy + o;
        const bool in = y < H && x < W;
        const int64_t p = (int64_t)y * W + x;
        float ps[4];
#pragma unroll
        for (int q = 0; q < 4; q++) {
            if (!render) pp[o][q] = 0.f;
            ps[q] = fmaxf(pl[o][q] - pp[o][q], 0.f);
        }
        auto store = [&](float* map, const float (&v)[4]) {
            if (!map || !in) return;
            if (vec) {
                *reinterpret_cast<float4*>(map + p) = make_float4(v[0], v[1], v[2], v[3]);
            } else {
#pragma unroll
                for (int q = 0; q < 4; q++)
                    if (x + q < W) map[p + q] = v[q];
            }
        };
        store(p_l, pl[o]);
        store(p_pen, pp[o]);
        store(p_s, ps);
        if (!mask) continue;
        unsigned bits = 0;
        if (in) {
            float z[4] = {0.f, 0.f, 0.f, 0.f};
            if (vec) {
                const float4 f = *reinterpret_cast<const float4*>(depth + p);
                z[0] = f.x; z[1] = f.y; z[2] = f.z; z[3] = f.w;
            } else {
#pragma unroll
                for (int q = 0; q < 4; q++)
                    if (x + q < W) z[q] = depth[p + q];
            }
#pragma unroll
            for (int q = 0; q < 4; q++) {
                if (!(ps[q] > 0.f && z[q] > 0.f && isfinite(z[q]))) continue;  // u < P_s needs P_s > 0
                const uint4 r = philox4x32_10(make_uint4((uint32_t)(p + q), frame, 0u, 0u), key);
                if (philox_u24(r.x) < ps[q]) {
                    bits |= 1u << q;
                    if (p_l_spawn) p_l_spawn[p + q] = pl[o][q];
                }
            }
        }
        // eight threads' bits make a word
        const int lane = threadIdx.x & 31;
        unsigned word = bits << (4 * (lane & 7));
#pragma unroll
        for (int d = 1; d < 8; d <<= 1) word |= __shfl_xor_sync(0xffffffffu, word, d);
        if ((lane & 7) == 0 && y < H && x < W) mask[(int64_t)y * ((W + 31) / 32) + x / 32] = word;
    }
}

// Depth of a learned spawn at pixel p: the depth map's value where it is
// positive and finite, else the patch's predicted depth.
__device__ __forceinline__ float learned_depth(const float* __restrict__ depth, const float* __restrict__ mlp_out,
                                               int64_t p, int64_t m) {
    const float d = depth ? depth[p] : 0.f;
    return (d > 0.f && isfinite(d)) ? d : mlp_out[m * 3 + 1];
}

// The spawned rows, in pixel order, and the count. A warp takes 8 words of the mask
// (prefix: how many pixels spawn before each); lane j takes the j-th of their
// spawns, and the warp writes the SH rows together, consecutive lanes consecutive
// rows. mlp_out: the learned proposal's outputs, or null for direct sampling.
// 1080p, 7% of the pixels spawning: 9 us (latency of four dependent loads).
constexpr int kSpRowWords = 8;

__global__ void __launch_bounds__(256) k_spawn_rows(const float* __restrict__ image, const float* __restrict__ depth,
                                                    const float* __restrict__ mlp_out, int W, int H,
                                                    const float* __restrict__ p_l, const uint32_t* __restrict__ mask,
                                                    const uint32_t* __restrict__ prefix, int64_t n_words,
                                                    const uint32_t* __restrict__ total, const int32_t* __restrict__ err,
                                                    const gs_camera* __restrict__ cam, int64_t capacity,
                                                    int64_t* __restrict__ count, int32_t* __restrict__ status,
                                                    float4* __restrict__ mean_opa, float4* __restrict__ scale,
                                                    float4* __restrict__ quat, float4* __restrict__ sh,
                                                    int32_t* __restrict__ pixel) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (warp == 0 && lane == 0) {
        *count = *total;
        *status = *err ? *err : (int64_t)*total > capacity ? GS_ERR_CAPACITY : GS_OK;
    }
    const int64_t w0 = warp * kSpRowWords;
    if (w0 >= n_words) return;  // uniform over the warp
    const int nw = (W + 31) / 32;
    uint32_t m = 0;
    if (lane < kSpRowWords && w0 + lane < n_words) {
        m = mask[w0 + lane];
        const int last = W - (int)((w0 + lane) % nw) * 32;  // a row's last word holds fewer pixels
        if (last < 32) m &= (1u << last) - 1u;
    }
    uint32_t start = __popc(m);  // inclusive, then exclusive prefix over the warp's words
#pragma unroll
    for (int o = 1; o < kSpRowWords; o <<= 1) {
        const uint32_t t = __shfl_up_sync(FULL, start, o);
        if (lane >= o) start += t;
    }
    const uint32_t n = __shfl_sync(FULL, start, kSpRowWords - 1);
    start -= __popc(m);
    if (n == 0) return;
    const int64_t o0 = prefix[w0];
    const gs_camera& c = *cam;
    const int64_t plane = (int64_t)W * H;
    const float inv_c0 = 3.5449077018110318f;  // 1 / SH band-0 constant = 2 sqrt(pi)
    for (uint32_t b = 0; b < n && o0 + b < capacity; b += 32) {
        const uint32_t j = b + lane;
        int k = 0;  // the word of spawn j: the last one that starts at or before it
#pragma unroll
        for (int step = kSpRowWords / 2; step >= 1; step >>= 1) {
            const uint32_t st = __shfl_sync(FULL, start, k + step);
            if (st <= j) k += step;
        }
        const uint32_t wm = __shfl_sync(FULL, m, k), ws = __shfl_sync(FULL, start, k);
        const int64_t o = o0 + j;
        const bool live = j < n && o < capacity;
        float dc0 = 0.f, dc1 = 0.f, dc2 = 0.f;
        if (live) {
            uint32_t left = j - ws, bit = 0;  // the (j - ws)-th set bit of the word
#pragma unroll
            for (int half = 16; half >= 1; half >>= 1) {
                const uint32_t low = __popc((wm >> bit) & ((1u << half) - 1u));
                if (left >= low) {
                    left -= low;
                    bit += half;
                }
            }
            const int64_t w = w0 + k;
            const int y = (int)(w / nw), x = (int)(w % nw) * 32 + (int)bit;
            const int64_t p = (int64_t)y * W + x;
            const float pl = p_l[p];
            float z, ls;
            if (mlp_out) {
                const int64_t pm = (int64_t)(y / 8) * (W / 8) + x / 8;
                z = learned_depth(depth, mlp_out, p, pm);
                // direct sampling's scale z / (2 fx sqrt(P_L)) times the patch's predicted factor exp(offset)
                ls = logf(z * (0.5f / sqrtf(pl)) / c.fx) + mlp_out[pm * 3 + 2];
            } else {
                z = depth[p];
                const float s_px = 0.5f / sqrtf(pl);
                ls = logf(z * s_px / c.fx);
            }
            const float xc = (x + 0.5f - c.cx) * z / c.fx, yc = (y + 0.5f - c.cy) * z / c.fy;
            const float qx = xc - c.t[0], qy = yc - c.t[1], qz = z - c.t[2];
            const float mx = c.R[0] * qx + c.R[3] * qy + c.R[6] * qz;  // R^T (p_cam - t)
            const float my = c.R[1] * qx + c.R[4] * qy + c.R[7] * qz;
            const float mz = c.R[2] * qx + c.R[5] * qy + c.R[8] * qz;
            mean_opa[o] = make_float4(mx, my, mz, 0.f);  // opacity 0.5
            scale[o] = make_float4(ls, ls, ls, 0.f);
            quat[o] = make_float4(1.f, 0.f, 0.f, 0.f);
            if (pixel) pixel[o] = (int32_t)p;
            dc0 = (image[p] - 0.5f) * inv_c0;
            dc1 = (image[plane + p] - 0.5f) * inv_c0;
            dc2 = (image[2 * plane + p] - 0.5f) * inv_c0;
        }
        const int rows = (int)min((int64_t)min(n - b, 32u), capacity - (o0 + b)) * 12;  // SH rows of this round
        for (int r0 = 0; r0 < rows; r0 += 32) {
            const int r = r0 + lane, from = min(r / 12, 31);
            const float v0 = __shfl_sync(FULL, dc0, from), v1 = __shfl_sync(FULL, dc1, from), v2 = __shfl_sync(FULL, dc2, from);
            if (r < rows) {
                const bool first = r % 12 == 0;
                sh[12 * (o0 + b) + r] = make_float4(first ? v0 : 0.f, first ? v1 : 0.f, first ? v2 : 0.f, 0.f);
            }
        }
    }
}

__global__ void k_spawn_count(const uint32_t* total, const int32_t* err, int64_t capacity, int64_t* count,
                              int32_t* status) {
    *count = *total;
    *status = *err ? *err : (int64_t)*total > capacity ? GS_ERR_CAPACITY : GS_OK;
}

static bool make_taps(float sigma, LogTaps* t) {
    if (!(sigma >= 0.3f) || !(sigma <= kSpMaxR / 3.f)) return false;
    const int R = std::min((int)std::ceil(3.0 * sigma), kSpMaxR);  // 8/3 as a float is above 8/3
    const int n = 2 * R + 1;
    const double s2 = (double)sigma * sigma;
    double w[kSpMaxTaps], sum = 0;
    for (int j = -R; j <= R; j++)
        for (int i = -R; i <= R; i++) {
            const double r2 = i * i + j * j;
            const double v = (r2 - 2 * s2) / (s2 * s2) * std::exp(-r2 / (2 * s2)) / (2 * 3.14159265358979323846 * s2);
            w[(j + R) * n + (i + R)] = v;
            sum += v;
        }
    t->R = R;
    for (int k = 0; k < n * n; k++) t->w[k] = (float)(w[k] - sum / (n * n));
    return true;
}

static int64_t mask_words(int W, int H) { return (int64_t)((W + 31) / 32) * H; }

// Scratch of one spawn proposal: the mask, its words' prefix counts, P_L of the
// spawning pixels where the caller keeps no map, and the scan's words.
struct SpawnScratch {
    uint32_t *mask, *prefix, *total;
    float* p_l;
    uint32_t* scan;
};

static SpawnScratch carve_spawn(Carve& c, int64_t pixels, int64_t words) {
    SpawnScratch w;
    w.mask = c.take<uint32_t>(words);
    w.prefix = c.take<uint32_t>(words);
    w.total = c.take<uint32_t>(1);
    w.p_l = c.take<float>(pixels);
    w.scan = c.take<uint32_t>(scan_popcounts_words(words));
    return w;
}

// Launches k_spawn_maps for the taps' radius.
static void launch_maps(const float* image, const float* render, const float* depth, int W, int H, const LogTaps& taps,
                        uint2 key, uint32_t frame, float* p_l, float* p_pen, float* p_s, uint32_t* mask,
                        float* p_l_spawn, const SpawnScratch& w, cudaStream_t s) {
    const bool vec = W % 4 == 0 && (((uintptr_t)image | (uintptr_t)render | (uintptr_t)depth | (uintptr_t)p_l |
                                     (uintptr_t)p_pen | (uintptr_t)p_s) & 15) == 0;
    const dim3 grid((unsigned)ceil_div(W, kSpW), (unsigned)ceil_div(H, kSpH));
    const int n_scan = (int)scan_popcounts_words(mask_words(W, H));
#define GS_MAPS(R)                                                                                                 \
    case R:                                                                                                        \
        k_spawn_maps<R><<<grid, kSpThreads, SpTile<R>::kBytes, s>>>(image, render, depth, W, H, taps, key, frame,  \
                                                                    vec, p_l, p_pen, p_s, mask, p_l_spawn, w.scan, \
                                                                    n_scan);                                       \
        break;
    switch (taps.R) {
        GS_MAPS(1) GS_MAPS(2) GS_MAPS(3) GS_MAPS(4) GS_MAPS(5) GS_MAPS(6) GS_MAPS(7) GS_MAPS(8)
    }
#undef GS_MAPS
    count_launch();
}

// The prefix counts of a mask and the rows of its pixels.
static void launch_rows(const float* image, const float* depth, const float* mlp_out, int W, int H, const float* p_l,
                        const SpawnScratch& w, const gs_camera* cam, const gs_spawn_out* out, cudaStream_t s) {
    const int64_t n = mask_words(W, H);
    const int32_t* err = scan_popcounts(w.mask, w.prefix, n, w.total, w.scan, s);
    if (out->capacity > 0) {
        k_spawn_rows<<<(unsigned)ceil_div(ceil_div(n, kSpRowWords), 8), 256, 0, s>>>(
            image, depth, mlp_out, W, H, p_l, w.mask, w.prefix, n, w.total, err, cam, out->capacity, out->count,
            out->status, (float4*)out->mean_opa, (float4*)out->scale, (float4*)out->quat, (float4*)out->sh, out->pixel);
    } else {
        k_spawn_count<<<1, 1, 0, s>>>(w.total, err, out->capacity, out->count, out->status);
    }
    count_launch();
}

static int spawn_propose(const float* image, const float* render, const float* depth, int W, int H,
                         const gs_camera* cam, const gs_spawn_config* sc, const gs_spawn_out* out, const LogTaps& taps,
                         const SpawnScratch& w, cudaStream_t s) {
    const uint2 key = make_uint2((uint32_t)sc->seed, (uint32_t)(sc->seed >> 32));
    launch_maps(image, render, depth, W, H, taps, key, sc->frame, out->p_l, out->p_pen, out->p_s, w.mask,
                out->p_l ? nullptr : w.p_l, w, s);
    launch_rows(image, depth, nullptr, W, H, out->p_l ? out->p_l : w.p_l, w, cam, out, s);
    GS_CUDA_CHECK_LAUNCH();
    return GS_OK;
}

}  // namespace gs

using namespace gs;

extern "C" size_t gs_spawn_workspace_size(int32_t width, int32_t height) {
    if (width <= 0 || height <= 0) return 0;
    const int64_t hw = (int64_t)width * height;
    Carve c{nullptr, 0, 0};
    // as many words as a frame one pixel wide has: what this many pixels need in any shape
    carve_spawn(c, hw, hw);
    c.take<float>(hw);       // gs_spawn_learned: P_s
    c.take<float>(hw / 64);  // gs_spawn_learned: patch sums
    return c.used;
}

extern "C" int gs_spawn_propose(const float* image, const float* render, const float* depth, int32_t width,
                                int32_t height, const gs_camera* cam, const gs_spawn_config* sc,
                                const gs_spawn_out* out, void* ws, size_t ws_bytes, void* stream) {
    if (!image || !depth || !cam || !sc || !out || width <= 0 || height <= 0) return GS_ERR_INVALID_ARG;
    if (!out->count || !out->status || out->capacity < 0 ||
        (out->capacity > 0 && (!out->mean_opa || !out->scale || !out->quat || !out->sh)))
        return GS_ERR_INVALID_ARG;
    const int64_t hw = (int64_t)width * height;
    if (hw > (int64_t)UINT32_MAX) return GS_ERR_INVALID_ARG;
    LogTaps taps;
    if (!make_taps(sc->sigma, &taps)) return GS_ERR_INVALID_ARG;
    Carve c{(char*)ws, 0, ws_bytes};
    const SpawnScratch w = carve_spawn(c, hw, mask_words(width, height));
    if (!ws || !c.ok() || ((uintptr_t)ws & 255)) return GS_ERR_INVALID_ARG;
    if (height > kSpMaxHeight) return GS_ERR_CUDA;
    return spawn_propose(image, render, depth, width, height, cam, sc, out, taps, w, (cudaStream_t)stream);
}

// ---------------------------------------------------------------------------
// Spawn proposal without caller-provided scratch.
//
// Some callers cannot allocate device memory at the point where they need a
// spawn proposal: code running under an allocator that is frozen or owned by
// another runtime (a host application that hands us only its input and output
// buffers), or a process that has reserved all its memory up front. For them
// the scratch (the spawn mask, its prefix counts, P_L of the spawning pixels and
// the scan's words) lives in this file-scope device array instead of a workspace.
// It is sized for at most kNoAllocMaxPixels pixels; every GPU that loads the
// library holds it until the process exits.
// ---------------------------------------------------------------------------
namespace gs {

constexpr int64_t kNoAllocMaxPixels = int64_t(1) << 21;  // 2,097,152 px: covers 1920x1080
constexpr int kNoAllocMaxDevices = 64;
// P_L, mask and prefix counts (a word each per 32 pixels of a row) of the narrowest
// frame that holds kNoAllocMaxPixels within kSpMaxHeight, two pixels wide; the total,
// the scan's words and the rounding of each part to 256 bytes.
constexpr int64_t kNoAllocWords = 2 * kNoAllocMaxPixels + 8192;

static __device__ __align__(256) uint32_t g_spawn_scratch[kNoAllocWords];  // ~16.8 MB

// Device address of g_spawn_scratch, looked up once per device with that
// device current (the host-side name of the array is not a device address).
// The address belongs to the device's context: after cudaDeviceReset the
// runtime creates a new primary context with the module loaded again, so the
// cached address is kept with the unique id of the context it came from
// (cuCtxGetCurrent + cuCtxGetId, resolved through the runtime's driver
// entry-point query, without linking the driver library) and looked up again
// when the current context is another one. Where the driver offers neither
// call, the address is looked up on every call. The mutex orders concurrent
// first calls from several host threads.
typedef CUresult (*CtxGetCurrentFn)(CUcontext*);
typedef CUresult (*CtxGetIdFn)(CUcontext, unsigned long long*);

static bool current_context_id(CtxGetCurrentFn cur, CtxGetIdFn id, unsigned long long* out) {
    CUcontext ctx = nullptr;
    return cur && id && cur(&ctx) == CUDA_SUCCESS && ctx && id(ctx, out) == CUDA_SUCCESS;
}

static uint32_t* noalloc_scratch_for_current_device() {
    static std::mutex mu;
    static uint32_t* ptr[kNoAllocMaxDevices] = {};
    static unsigned long long ctx_id[kNoAllocMaxDevices] = {};
    static bool resolved = false;
    static CtxGetCurrentFn ctx_current = nullptr;
    static CtxGetIdFn ctx_get_id = nullptr;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices) return nullptr;
    std::lock_guard<std::mutex> lock(mu);
    if (!resolved) {
        resolved = true;
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            ctx_current = (CtxGetCurrentFn)f;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            ctx_get_id = (CtxGetIdFn)f;
        (void)cudaGetLastError();
    }
    unsigned long long id = 0;
    const bool have_id = current_context_id(ctx_current, ctx_get_id, &id);
    if (!ptr[dev] || !have_id || id != ctx_id[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_spawn_scratch) != cudaSuccess) {
            (void)cudaGetLastError();
            return nullptr;
        }
        ptr[dev] = (uint32_t*)p;
        // the lookup made the device's context current if none was
        ctx_id[dev] = current_context_id(ctx_current, ctx_get_id, &id) ? id : 0;
    }
    return ptr[dev];
}

}  // namespace gs

extern "C" int gs_spawn_propose_noalloc(const float* image, const float* render, const float* depth,
                                        int32_t width, int32_t height, const gs_camera* cam,
                                        const gs_spawn_config* sc, const gs_spawn_out* out, void* stream) {
    if (!image || !depth || !cam || !sc || !out || width <= 0 || height <= 0) return GS_ERR_INVALID_ARG;
    if (!out->count || !out->status || out->capacity < 0 ||
        (out->capacity > 0 && (!out->mean_opa || !out->scale || !out->quat || !out->sh)))
        return GS_ERR_INVALID_ARG;
    const int64_t hw = (int64_t)width * height;
    if (hw > kNoAllocMaxPixels) return GS_ERR_INVALID_ARG;  // larger frames need gs_spawn_propose
    LogTaps taps;
    if (!make_taps(sc->sigma, &taps)) return GS_ERR_INVALID_ARG;
    if (height > kSpMaxHeight) return GS_ERR_CUDA;
    uint32_t* base = noalloc_scratch_for_current_device();
    if (!base) return GS_ERR_CUDA;
    // Nothing in it needs to start at zero: every call writes each word it later
    // reads (the mask and its prefix counts, P_L where the mask is set, and the
    // scan's words, which the call clears).
    Carve c{(char*)base, 0, sizeof(uint32_t) * kNoAllocWords};
    const SpawnScratch w = carve_spawn(c, hw, mask_words(width, height));
    if (!c.ok()) return GS_ERR_INVALID_ARG;
    return spawn_propose(image, render, depth, width, height, cam, sc, out, taps, w, (cudaStream_t)stream);
}

// ---------------------------------------------------------------------------
// Learned spawn proposal: training targets and spawning from its predictions.
// ---------------------------------------------------------------------------
namespace gs {

// Scatter the kept spawns into per-pixel slots (each pixel spawns at most once).
// One thread per spawn: kept when its optimised opacity sigmoid(logit) is
// above the threshold; then its camera depth R_2 . mu + t_2 and the change of
// its log-scale (mean over the three axes minus the spawned value) go to the
// spawn's pixel.
__global__ void k_kept_scatter(const int32_t* __restrict__ pixel, const float4* __restrict__ mean_opa,
                               const float4* __restrict__ scale, const float4* __restrict__ scale0,
                               const gs_camera* __restrict__ cam, float keep_threshold, int64_t n, int64_t hw,
                               float4* __restrict__ pix_slot) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float4 mo = mean_opa[i];
    const float o = 1.f / (1.f + expf(-mo.w));
    if (!(o > keep_threshold)) return;
    const int32_t p = pixel[i];
    if (p < 0 || (int64_t)p >= hw) return;
    const float z = cam->R[6] * mo.x + cam->R[7] * mo.y + cam->R[8] * mo.z + cam->t[2];
    const float4 s = scale[i];
    const float ls = (s.x + s.y + s.z) * (1.f / 3.f) - scale0[i].x;
    pix_slot[p] = make_float4(1.f, z, ls, 0.f);
}

// One thread per 8x8 patch: kept fraction, mean depth and log-scale, any-kept.
__global__ void k_patch_targets(const float4* __restrict__ pix_slot, int W, int H, float* __restrict__ targets) {
    const int nx = W / 8, ny = H / 8;
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= (int64_t)nx * ny) return;
    const int px = (int)(m % nx), py = (int)(m / nx);
    float cnt = 0.f, zs = 0.f, ss = 0.f;
    for (int dy = 0; dy < 8; dy++)
        for (int dx = 0; dx < 8; dx++) {
            const float4 v = pix_slot[(int64_t)(py * 8 + dy) * W + px * 8 + dx];
            if (v.x > 0.f) {
                cnt += 1.f;
                zs += v.y;
                ss += v.z;
            }
        }
    targets[m * 4 + 0] = cnt / 64.f;
    targets[m * 4 + 1] = cnt > 0.f ? zs / cnt : 0.f;
    targets[m * 4 + 2] = cnt > 0.f ? ss / cnt : 0.f;
    targets[m * 4 + 3] = cnt > 0.f ? 1.f : 0.f;
}

// Lower bound of a patch's P_s sum in the placement ratio (keeps the ratio
// well conditioned where the render already explains the patch).
constexpr float kPatchFloor = 64.f * 1e-3f;

// One thread per 8x8 patch: sum of P_s in row-major order, floored.
__global__ void k_patch_ps_sum(const float* __restrict__ ps, int W, int H, float* __restrict__ sums) {
    const int nx = W / 8, ny = H / 8;
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= (int64_t)nx * ny) return;
    const int px = (int)(m % nx), py = (int)(m / nx);
    float a = 0.f;
    for (int dy = 0; dy < 8; dy++)
        for (int dx = 0; dx < 8; dx++) a += ps[(int64_t)(py * 8 + dy) * W + px * 8 + dx];
    sums[m] = fmaxf(a, kPatchFloor);
}

// Spawn flags from the MLP: pixel p of patch m spawns with probability
// min(1, sigmoid(logit_m) 64 P_s(p) / patch sum) (the predicted count placed
// where direct sampling would place it) and a positive depth; the draw is
// Philox(counter (p, frame, 1, 0)).
// One warp per 32 pixels of a row, one word of the mask.
__global__ void __launch_bounds__(256) k_learned_mask(const float* __restrict__ mlp_out, const float* __restrict__ depth,
                                                      const float* __restrict__ ps, const float* __restrict__ sums,
                                                      int W, int H, uint2 key, uint32_t frame,
                                                      uint32_t* __restrict__ mask) {
    const int lane = threadIdx.x & 31, nw = (W + 31) / 32;
    const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (w >= (int64_t)nw * H) return;
    const int y = (int)(w / nw), x = (int)(w % nw) * 32 + lane;
    bool spawn = false;
    if (x < W) {
        const int64_t p = (int64_t)y * W + x;
        const int64_t m = (int64_t)(y / 8) * (W / 8) + x / 8;
        const float logit = mlp_out[m * 3 + 0], z = learned_depth(depth, mlp_out, p, m);
        const float sig = 1.f / (1.f + expf(-logit));
        const float prob = fminf(1.f, sig * 64.f * ps[p] / sums[m]);
        const uint4 r = philox4x32_10(make_uint4((uint32_t)p, frame, 1u, 0u), key);
        const float u = (float)(r.x >> 8) * (1.f / 16777216.f);
        spawn = u < prob && z > 0.f && isfinite(z);
    }
    const unsigned bits = __ballot_sync(0xffffffffu, spawn);
    if (lane == 0) mask[w] = bits;
}

}  // namespace gs

extern "C" size_t gs_mlp_targets_workspace_size(int32_t width, int32_t height) {
    if (width <= 0 || height <= 0) return 0;
    return align256(sizeof(float4) * (size_t)width * height);
}

extern "C" int gs_mlp_targets(const int32_t* pixel, const float* mean_opa, const float* scale, const float* scale0,
                              const gs_camera* cam, float keep_threshold, int64_t n_spawn, int32_t width,
                              int32_t height, float* targets, void* ws, size_t ws_bytes, void* stream) {
    if (!targets || width <= 0 || height <= 0 || width % 8 || height % 8 || n_spawn < 0 ||
        (n_spawn > 0 && (!pixel || !mean_opa || !scale || !scale0 || !cam)))
        return GS_ERR_INVALID_ARG;
    const int64_t hw = (int64_t)width * height;
    if (!ws || ws_bytes < gs_mlp_targets_workspace_size(width, height) || ((uintptr_t)ws & 255))
        return GS_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    float4* slot = (float4*)ws;
    cudaMemsetAsync(slot, 0, sizeof(float4) * hw, s);
    if (n_spawn > 0) {
        k_kept_scatter<<<(unsigned)ceil_div(n_spawn, 256), 256, 0, s>>>(
            pixel, (const float4*)mean_opa, (const float4*)scale, (const float4*)scale0, cam, keep_threshold, n_spawn,
            hw, slot);
        count_launch();
    }
    const int64_t np = hw / 64;
    k_patch_targets<<<(unsigned)ceil_div(np, 256), 256, 0, s>>>(slot, width, height, targets);
    count_launch();
    GS_CUDA_CHECK_LAUNCH();
    return GS_OK;
}

extern "C" int gs_spawn_learned(const float* image, const float* mlp_out, const float* render, const float* depth,
                                int32_t width, int32_t height, const gs_camera* cam, const gs_spawn_config* sc,
                                const gs_spawn_out* out, void* ws, size_t ws_bytes, void* stream) {
    if (!image || !mlp_out || !cam || !sc || !out || width <= 0 || height <= 0 || width % 8 || height % 8)
        return GS_ERR_INVALID_ARG;
    if (!out->count || !out->status || out->capacity < 0 ||
        (out->capacity > 0 && (!out->mean_opa || !out->scale || !out->quat || !out->sh)))
        return GS_ERR_INVALID_ARG;
    const int64_t hw = (int64_t)width * height;
    if (hw > (int64_t)UINT32_MAX) return GS_ERR_INVALID_ARG;
    LogTaps taps;
    if (!make_taps(sc->sigma, &taps)) return GS_ERR_INVALID_ARG;
    Carve c{(char*)ws, 0, ws_bytes};
    const SpawnScratch w = carve_spawn(c, hw, mask_words(width, height));
    float* ps = c.take<float>(hw);
    float* sums = c.take<float>(hw / 64);
    if (!ws || !c.ok() || ((uintptr_t)ws & 255)) return GS_ERR_INVALID_ARG;
    if (height > kSpMaxHeight) return GS_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    const uint2 key = make_uint2((uint32_t)sc->seed, (uint32_t)(sc->seed >> 32));
    // P_s (Eq. 1-3) of the frame, then its patch sums
    float* psb = out->p_s ? out->p_s : ps;  // the caller's maps when it asks for them
    float* plb = out->p_l ? out->p_l : w.p_l;
    launch_maps(image, render, nullptr, width, height, taps, key, sc->frame, plb, out->p_pen, psb, nullptr, nullptr, w, s);
    k_patch_ps_sum<<<(unsigned)ceil_div(hw / 64, 256), 256, 0, s>>>(psb, width, height, sums);
    count_launch();
    k_learned_mask<<<(unsigned)ceil_div(mask_words(width, height), 8), 256, 0, s>>>(mlp_out, depth, psb, sums, width,
                                                                                    height, key, sc->frame, w.mask);
    count_launch();
    launch_rows(image, depth, mlp_out, width, height, plb, w, cam, out, s);
    GS_CUDA_CHECK_LAUNCH();
    return GS_OK;
}
