// Front-to-back alpha compositing (K5) and its adjoint (K6).
//
// Two pairs of kernels. 16 x 16 tiles in launches large enough to fill the GPU
// with them take k_blocks_fwd and k_rows_bwd (further down); the other tile sizes
// and small launches take k_render_fwd and k_render_bwd, described here:
//
// One CTA of TILE x TILE threads per tile (TILE = 8, 16 or 32), one pixel per
// thread; each warp owns an 8x4 block of pixels so a small splat touches few
// warps. Each tile's depth-ordered list is walked in batches staged in shared
// memory (128-bit loads of the projected rows). While staging, each Gaussian
// gets the bounding box of the region where its alpha can reach alpha_min; a
// warp tests 32 staged boxes against its 8x4 block with one ballot and
// evaluates only the hits, so Gaussians that cannot touch any of its pixels
// cost nothing. The forward stops a CTA when every pixel's transmittance has
// terminated. The adjoint recomputes the blending state back to front from
// T_final and n_contrib, records per pixel and Gaussian two scalars in a
// per-warp table, forms each Gaussian's 9 partial derivatives from the table
// (sums over the warp's pixels in a fixed order), sums the warps in a fixed
// order and writes ONE partial per (tile, Gaussian) pair to the pair's
// emission slot. No atomics touch gradients: bit-reproducible.
//
// Scheduling: either one CTA per tile (grid order), or persistent CTAs (as
// many as fit on the SMs) that pull tiles from a global counter in the order
// gs_sort produced (largest pair list first), which evens out the tail when
// views of very different sizes and densities share one launch. The counter
// only hands out work; every loop is bounded by the tile count.
#include "common.cuh"

namespace gs {

template <int TILE>
struct Geom {
    static constexpr int kThreads = TILE * TILE;
    static constexpr int kWarps = kThreads / 32;
    static constexpr int kWX = TILE / 8;  // 8x4 warp blocks per tile row
};

struct TileInfo {
    int view, px, py, W, H;
    bool inside;
    int64_t pix;         // pixel index within all views
    int64_t plane;       // H*W of the view
    int64_t color_base;  // index of this pixel's red value in the colour buffer
};

template <int TILE>
__device__ __forceinline__ TileInfo tile_info(const gs_frame& f, int tile) {
    TileInfo t;
    t.view = view_of_tile(f, tile);
    const int local = tile - f.tile_base[t.view];
    const int tx = local % f.tiles_x[t.view], ty = local / f.tiles_x[t.view];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int lx = (w % Geom<TILE>::kWX) * 8 + (lane & 7);
    const int ly = (w / Geom<TILE>::kWX) * 4 + (lane >> 3);
    t.px = tx * TILE + lx;
    t.py = ty * TILE + ly;
    t.W = f.width[t.view];
    t.H = f.height[t.view];
    t.inside = t.px < t.W && t.py < t.H;
    t.plane = (int64_t)t.W * t.H;
    t.pix = f.pix_base[t.view] + (int64_t)t.py * t.W + t.px;
    t.color_base = 3 * f.pix_base[t.view] + (int64_t)t.py * t.W + t.px;
    return t;
}

// Staged form of a projected Gaussian: exponent coefficients in base 2,
// e = A dx^2 + B dx dy + C dy^2 = -(a dx^2 + 2 b dx dy + c dy^2)/2 * log2(e),
// and the bounding box (x0, y0, x1, y1) of the ellipse where o exp(-q/2) can
// reach alpha_min (q = d^T conic d <= 2 ln(o / alpha_min)); the box is widened
// by 0.1% + 0.01 px so that FP32 evaluation never finds a hit outside it.
__device__ __forceinline__ void stage(const float2* __restrict__ mean2d, const float4* __restrict__ conic_opa,
                                      const float4* __restrict__ rgb_depth, uint32_t idx, float alpha_min, float2& xy,
                                      float4& abco, float4& rgb, float4& box) {
    xy = mean2d[idx];
    const float4 co = conic_opa[idx];
    abco = make_float4(-0.5f * kLog2e * co.x, -kLog2e * co.y, -0.5f * kLog2e * co.z, co.w);
    rgb = rgb_depth[idx];
    const float det = co.x * co.z - co.y * co.y;
    if (!(co.w >= alpha_min)) {
        box = make_float4(1e30f, 1e30f, -1e30f, -1e30f);  // can never reach alpha_min
    } else if (!(det > 0.f)) {
        box = make_float4(-1e30f, -1e30f, 1e30f, 1e30f);  // degenerate conic: never skip
    } else {
        const float t = 2.f * logf(co.w / alpha_min);
        const float hx = sqrtf(fmaxf(t * co.z / det, 0.f)) * 1.001f + 0.01f;
        const float hy = sqrtf(fmaxf(t * co.x / det, 0.f)) * 1.001f + 0.01f;
        box = make_float4(xy.x - hx, xy.y - hy, xy.x + hx, xy.y + hy);
    }
}

struct WarpBlock {
    float x0, y0, x1, y1;  // pixel-centre extent of this warp's 8x4 block
    __device__ __forceinline__ bool hits(const float4& b) const {
        return b.x <= x1 && b.z >= x0 && b.y <= y1 && b.w >= y0;
    }
};

__device__ __forceinline__ WarpBlock warp_block(const TileInfo& ti) {
    const int lane = threadIdx.x & 31;
    WarpBlock wb;
    wb.x0 = (float)(ti.px - (lane & 7)) + 0.5f;
    wb.y0 = (float)(ti.py - (lane >> 3)) + 0.5f;
    wb.x1 = wb.x0 + 7.f;
    wb.y1 = wb.y0 + 3.f;
    return wb;
}

// Exponent (base 2) of the Gaussian at offset (dx, dy). The same rounding
// sequence is used forward and backward so both take identical decisions.
__device__ __forceinline__ float exponent2(const float4& abco, float dx, float dy) {
    return __fmaf_rn(__fmul_rn(abco.x, dx), dx,
                     __fmaf_rn(__fmul_rn(abco.z, dy), dy, __fmul_rn(__fmul_rn(abco.y, dx), dy)));
}

// Next tile for this CTA: its own (grid schedule, first call only: tile
// blockIdx.x, or entry blockIdx.x of the work order in the ordered-grid
// schedule) or the next entry of the work order (persistent schedule, with
// the counter). Returns -1 when done.
__device__ __forceinline__ int next_tile(const uint32_t* __restrict__ order, uint32_t* counter, int n_tiles,
                                         bool first, int* s_item) {
    if (!counter) return first ? (order ? (int)order[blockIdx.x] : (int)blockIdx.x) : -1;
    if (threadIdx.x == 0) {
        const uint32_t it = atomicAdd(counter, 1u);
        *s_item = it < (uint32_t)n_tiles ? (int)order[it] : -1;
    }
    __syncthreads();
    const int t = *s_item;
    __syncthreads();
    return t;
}

// DEPTH: also accumulate the depth integral sum_i alpha_i T_i z_i per pixel.
// COUNT (measurement only, never the timed instantiation): also count, into
// counts[0..2], the warp hits the ballot passes (each one runs the compositing
// step on all 32 lanes), the lane evaluations of pixels not yet terminated at
// those hits, and the evaluations that composite (alpha >= alpha_min, before
// termination) - the work the definition requires.
template <int TILE, int FB, bool DEPTH, bool COUNT = false>
__global__ void __launch_bounds__(TILE * TILE) k_render_fwd(gs_frame f, gs_config cfg,
                                                            const uint32_t* __restrict__ range,
                                                            const uint32_t* __restrict__ src,
                                                            const float2* __restrict__ mean2d,
                                                            const float4* __restrict__ conic_opa,
                                                            const float4* __restrict__ rgb_depth,
                                                            float* __restrict__ color, float* __restrict__ t_final,
                                                            int32_t* __restrict__ n_contrib,
                                                            float* __restrict__ depth_out,
                                                            const uint32_t* __restrict__ order, uint32_t* counter,
                                                            int n_tiles, unsigned long long* counts) {
    constexpr int NT = Geom<TILE>::kThreads;
    unsigned long long n_hit = 0, n_eval = 0, n_comp = 0;
    __shared__ float2 s_xy[FB];
    __shared__ float4 s_abco[FB];
    __shared__ float4 s_rgb[FB];
    __shared__ float4 s_box[FB];
    __shared__ int s_item;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    for (int tile = next_tile(order, counter, n_tiles, true, &s_item); tile >= 0;
         tile = next_tile(order, counter, n_tiles, false, &s_item)) {
        const TileInfo ti = tile_info<TILE>(f, tile);
        const WarpBlock wb = warp_block(ti);
        const float px = ti.px + 0.5f, py = ti.py + 0.5f;
        const uint32_t start = range[2 * tile], end = range[2 * tile + 1];
        float T = 1.f, cr = 0.f, cg = 0.f, cb = 0.f, cz = 0.f;
        int last = 0;
        bool done = !ti.inside;
        for (uint32_t b0 = start; b0 < end; b0 += FB) {
            if (__syncthreads_count(done) == NT) break;
            for (int j = threadIdx.x; j < FB; j += NT)
                if (b0 + j < end)
                    stage(mean2d, conic_opa, rgb_depth, src[b0 + j], cfg.alpha_min, s_xy[j], s_abco[j], s_rgb[j],
                          s_box[j]);
            __syncthreads();
            const int cnt = min((uint32_t)FB, end - b0);
            int lastk = -1;  // staged index of this batch's last composited Gaussian
            for (int k0 = 0; k0 < cnt; k0 += 32) {
                if (__all_sync(FULL, done)) break;
                const int kk = k0 + lane;
                unsigned m = __ballot_sync(FULL, kk < cnt && wb.hits(s_box[kk < cnt ? kk : 0]));
                // predicated: every lane runs the same instructions, the
                // pixel's state changes only where the Gaussian composites
                auto composite = [&](int k, const float2 xy, const float4 abco, const float4 c) {
                    const float e = exponent2(abco, px - xy.x, py - xy.y);
                    const float og = __fmul_rn(abco.w, fast_exp2(e));
                    const float alpha = fminf(cfg.alpha_max, og);
                    const bool ok = !done && !(e > 0.f) && alpha >= cfg.alpha_min;
                    const float aT = __fmul_rn(alpha, T);  // the blending weight
                    const float nT = __fsub_rn(T, aT);     // T (1 - alpha)
                    const bool term = ok && nT < cfg.t_min;
                    const bool acc = ok && !term;
                    if (COUNT) {
                        n_hit += 1;
                        n_eval += !done;
                        n_comp += acc;
                    }
                    done = done || term;
                    const float w = acc ? aT : 0.f;
                    cr += w * c.x; cg += w * c.y; cb += w * c.z;
                    if (DEPTH) cz += w * c.w;
                    T = acc ? nT : T;
                    lastk = acc ? k : lastk;
                };
                // two hits per round (warp-uniform): both Gaussians' shared
                // loads are issued before the first composites, in order
                while (m) {
                    const int ka = k0 + __ffs(m) - 1;
                    m &= m - 1;
                    const bool two = m != 0;
                    const int kb = two ? k0 + __ffs(m) - 1 : ka;
                    m &= m - 1;
                    const float2 xya = s_xy[ka], xyb = s_xy[kb];
                    const float4 aba = s_abco[ka], abb = s_abco[kb];
                    const float4 ca = s_rgb[ka], cb2 = s_rgb[kb];
                    composite(ka, xya, aba, ca);
                    if (two) composite(kb, xyb, abb, cb2);
                }
            }
            if (lastk >= 0) last = (int)(b0 - start) + lastk + 1;
        }
        if (ti.inside) {
            color[ti.color_base] = cr + T * cfg.bg[0];
            color[ti.color_base + ti.plane] = cg + T * cfg.bg[1];
            color[ti.color_base + 2 * ti.plane] = cb + T * cfg.bg[2];
            t_final[ti.pix] = T;
            n_contrib[ti.pix] = last;
            if (DEPTH) depth_out[ti.pix] = cz;
        }
        __syncthreads();  // shared buffers are reused by the next tile
    }
    if (COUNT) {
        for (int o = 16; o > 0; o >>= 1) {
            n_eval += __shfl_xor_sync(FULL, n_eval, o);
            n_comp += __shfl_xor_sync(FULL, n_comp, o);
        }
        if (lane == 0) {
            atomicAdd(&counts[0], n_hit);  // every lane counted the warp's hits; lane 0 reports them once
            atomicAdd(&counts[1], n_eval);
            atomicAdd(&counts[2], n_comp);
        }
    }
}

// Long lists in launches of k_rows_bwd (further down). Its one warp per tile takes 0.116 us
// for each entry that a pixel composites, with an SM to itself, and k_render_bwd's eight
// 0.072, so that uneven launches ended with single warps at their longest lists. Tiles
// with more than kLongMean times the mean list (uniform scenes have up to 4.5 times) go to
// k_render_bwd, launched to start when the last CTA of k_rows_bwd has started and the
// registers of the first ones are free: 100k Gaussians over a 720p view and 20k more in
// 60 x 60 px of it, 901 us without and 604 with it (604 by k_render_bwd for all tiles);
// 400k in 60 clusters over a 1080p view 386 and 295 (413); 200k all over a 720p view, no
// long list, 82 and 85. Three CTAs per SM: with two, 400k Gaussians in 200 x 200 px of two
// 1080p views took 2000 us instead of 1340. Each CTA looks through all ranges, so launches of more than kLongTiles
// tiles do without: four 1080p views with such clusters take 1.05 to 1.4 times k_render_bwd's time.
constexpr int kLongMean = 8, kLongTiles = 16384, kLongCtas = 3 * 152;
constexpr uint32_t kLongMin = 1024;
__device__ __forceinline__ uint32_t long_list(const int64_t* __restrict__ count, int64_t capacity, float share) {
    return max(kLongMin, __float2uint_rz(__fmul_rn((float)(uint32_t)min(*count, capacity), share)));
}

// Launches that overlap: the next one may start when every CTA of this one has called
// launch_next or ended; wait_for_last returns when the one before has ended.
__device__ __forceinline__ void launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_last() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The tiles with long lists, dealt to the CTAs in turn: this CTA's to s_mine; their number.
constexpr int kLongMine = (kLongTiles / kLongMean + kLongCtas - 1) / kLongCtas;
template <int NT>
__device__ __forceinline__ int my_long_tiles(const uint32_t* __restrict__ range, int n_tiles, uint32_t len, int* s_mine) {
    constexpr int NW = NT / 32, kWords = kLongTiles / 32, kPer = kWords / NT, kAhead = 8;
    __shared__ unsigned s_mask[kWords];  // a bit per tile
    __shared__ int s_count[NW], s_n;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    unsigned any = 0;
#pragma unroll 1
    for (int t0 = 0; t0 < n_tiles; t0 += kAhead * NT) {
        uint32_t a[kAhead], b[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; k++) {
            const int t = min(t0 + k * NT + (int)threadIdx.x, n_tiles - 1);
            a[k] = range[2 * t];
            b[k] = range[2 * t + 1];
        }
#pragma unroll
        for (int k = 0; k < kAhead; k++) {
            const int t = t0 + k * NT + threadIdx.x;
            const unsigned m = __ballot_sync(FULL, t < n_tiles && b[k] - a[k] > len);
            if (lane == 0) s_mask[t / 32] = m;
            any |= m;
        }
    }
    if (threadIdx.x == 0) s_n = 0;
    if (!__syncthreads_or(any != 0)) return 0;
    // a tile's rank: the long ones of the words before its own, then of its word
    const int w0 = threadIdx.x * kPer, w1 = min(w0 + kPer, (n_tiles + 31) / 32);
    int mine = 0;
    for (int q = w0; q < w1; q++) mine += __popc(s_mask[q]);
    int rank = mine;  // inclusive over the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(FULL, rank, o);
        if (lane >= o) rank += u;
    }
    if (lane == 31) s_count[w] = rank;
    __syncthreads();
    rank -= mine;
    for (int q = 0; q < w; q++) rank += s_count[q];
    for (int q = w0; q < w1; q++)
        for (unsigned m = s_mask[q]; m; m &= m - 1, rank++)
            if (rank % (int)gridDim.x == (int)blockIdx.x) {
                const int i = atomicAdd(&s_n, 1);
                if (i < kLongMine) s_mine[i] = 32 * q + __ffs(m) - 1;
            }
    __syncthreads();
    return min(s_n, kLongMine);
}

// Compositing adjoint. Per pixel (one lane) and Gaussian, back to front: the
// transmittance in front of it, dL/dalpha and from it the two scalars that all
// nine gradient terms of the (tile, Gaussian) pair are built from - dpow =
// dL/d(exponent) and the blending weight. Rather than a 9-value warp reduction
// per Gaussian, each warp keeps the scalars of its last kBwdHits Gaussians in a
// shared table (row = Gaussian, column = pixel) and, when full, four lanes per
// Gaussian form sum(dpow), sum(dpow dx), ..., sum(w dL/dc) over eight pixels
// each and combine in a fixed order: about a third fewer instructions per hit.
constexpr int kBwdHits = 8;  // hits per table flush (4 lanes per hit, 8 pixels each)

// LONG: the tiles of a launch of k_rows_bwd that are not for it: those with long lists,
// beside it, and when it has ended those that it marked (again: a byte per tile).
template <int TILE, int BB, bool LONG = false>
__global__ void __launch_bounds__(TILE * TILE) k_render_bwd(gs_frame f, gs_config cfg,
                                                            const uint32_t* __restrict__ range,
                                                            const uint32_t* __restrict__ src,
                                                            const uint32_t* __restrict__ emit,
                                                            const float2* __restrict__ mean2d,
                                                            const float4* __restrict__ conic_opa,
                                                            const float4* __restrict__ rgb_depth,
                                                            const float* __restrict__ t_final,
                                                            const int32_t* __restrict__ n_contrib,
                                                            const float* __restrict__ dL_dcolor,
                                                            float4* __restrict__ part0, float4* __restrict__ part1,
                                                            float* __restrict__ part2, int64_t capacity,
                                                            const uint32_t* __restrict__ order, uint32_t* counter,
                                                            int n_tiles, const int64_t* __restrict__ count,
                                                            float share, uint8_t* again) {
    constexpr int NT = Geom<TILE>::kThreads;
    constexpr int NW = Geom<TILE>::kWarps;
    __shared__ float2 s_xy[BB];
    __shared__ float4 s_abco[BB];
    __shared__ float4 s_rgb[BB];
    __shared__ float4 s_box[BB];
    __shared__ uint32_t s_emit[BB];
    __shared__ float s_part[NW][BB][9];
    __shared__ uint32_t s_hit[NW][BB / 32];  // which Gaussians each warp wrote
    // per warp: the last HB hits' per-pixel adjoint scalars (row = hit, column =
    // pixel) and each pixel's colour gradient
    __shared__ float2 s_tdw[NW][kBwdHits][33];  // (dpow, weight)
    __shared__ float4 s_pix[NW][32];
    __shared__ int s_max;
    __shared__ int s_item;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const float inv_log2e = 1.f / kLog2e;
    __shared__ int s_mine[LONG ? kLongMine : 1];
    __shared__ unsigned s_again[NW];
    int mine = 0, word = NW;
    unsigned bits = 0;
    int64_t at = 0, seen = blockIdx.x;  // tiles at + i gridDim.x are in s_again; the next to look at
    if (LONG && share > 0.f) mine = my_long_tiles<NT>(range, n_tiles, long_list(count, capacity, share), s_mine);
    auto next_long = [&]() {
        if (mine > 0) return s_mine[--mine];
        for (;;) {
            if (bits) {
                const int i = 32 * (word - 1) + __ffs(bits) - 1;
                bits &= bits - 1;
                return (int)(at + (int64_t)i * gridDim.x);
            }
            if (word < NW) {
                bits = s_again[word++];
                continue;
            }
            if (seen >= n_tiles) return -1;
            wait_for_last();  // every CTA comes here: this launch ends no sooner than the one that it overlaps
            __syncthreads();
            at = seen;
            const int64_t t = at + (int64_t)threadIdx.x * gridDim.x;
            unsigned is = 0;
            if (t < n_tiles) asm volatile("ld.relaxed.gpu.global.u8 %0, [%1];" : "=r"(is) : "l"(again + t) : "memory");
            const unsigned m = __ballot_sync(FULL, is != 0);
            if (lane == 0) s_again[w] = m;
            __syncthreads();
            seen += (int64_t)NT * gridDim.x;
            word = 0;
        }
    };
    for (int tile = LONG ? next_long() : next_tile(order, counter, n_tiles, true, &s_item); tile >= 0;
         tile = LONG ? next_long() : next_tile(order, counter, n_tiles, false, &s_item)) {
        const TileInfo ti = tile_info<TILE>(f, tile);
        const WarpBlock wb = warp_block(ti);
        const float px = ti.px + 0.5f, py = ti.py + 0.5f;
        const uint32_t start = range[2 * tile];
        float Tf = 1.f, gr = 0.f, gg = 0.f, gb = 0.f;
        int nc = 0;
        if (ti.inside) {
            Tf = t_final[ti.pix];
            nc = n_contrib[ti.pix];
            gr = dL_dcolor[ti.color_base];
            gg = dL_dcolor[ti.color_base + ti.plane];
            gb = dL_dcolor[ti.color_base + 2 * ti.plane];
        }
        if (threadIdx.x == 0) s_max = 0;
        __syncthreads();
        const int warp_nc = __reduce_max_sync(FULL, (unsigned)nc);
        if (lane == 0) atomicMax(&s_max, warp_nc);
        __syncthreads();
        const int n_list = s_max;
        // pairs past every pixel's last contributor: their emission slots are gathered per
        // Gaussian like all others
        const uint32_t len = range[2 * tile + 1] - start;
        for (uint32_t j = (uint32_t)n_list + threadIdx.x; j < len; j += NT) {
            const uint32_t e = emit[start + j];
            if ((int64_t)e < capacity) part2[e] = __uint_as_float(kNoPartial);
        }
        // gS = sum over channels of dL/dC_ch times the colour composited behind the
        // current Gaussian plus the background seen through T_final: dL/dalpha needs
        // only this dot product, so one scalar replaces three running colours
        float T = Tf, gS = Tf * (gr * cfg.bg[0] + gg * cfg.bg[1] + gb * cfg.bg[2]);
        s_pix[w][lane] = make_float4(gr, gg, gb, 0.f);
        int nh = 0;    // hits recorded in this warp's table (warp-uniform)
        int myk = 0;   // the staged index of hit (lane % HB) of the table
        // Sums over the warp's 32 pixels of the 9 gradient terms of each recorded
        // hit: lanes r, r + HB, ... share hit r, each summing 32 / L pixels from the
        // table, then combine in a fixed order; the first writes the CTA partial.
        auto flush = [&]() {
            __syncwarp();
            const int r = lane % kBwdHits, part = lane / kBwdHits;
            const bool act = r < nh;
            float S[9];
#pragma unroll
            for (int c = 0; c < 9; c++) S[c] = 0.f;
            float4 abco = make_float4(0.f, 0.f, 0.f, 1.f);
            if (act) {
                const float2 xy = s_xy[myk];
                abco = s_abco[myk];
                // pixel p = 8 part + i sits at (x0 + i, y0 + part): the same floats as the
                // compositing pass's pixel centres, so dx is identical; dy is constant over
                // this lane's row, so the dy terms follow from sum(d) and sum(d dx)
                static_assert(kBwdHits == 8, "one pixel row per lane");
                const float dy = (wb.y0 + (float)part) - xy.y;
#pragma unroll
                for (int i = 0; i < kBwdHits; i++) {
                    const int pp = part * kBwdHits + i;
                    const float dx = (wb.x0 + (float)i) - xy.x;
                    const float2 dw = s_tdw[w][r][pp];
                    const float d = dw.x, wv = dw.y;
                    const float4 pc = s_pix[w][pp];
                    const float t1 = d * dx;
                    S[0] += d; S[1] += t1; S[3] += t1 * dx;
                    S[6] += wv * pc.x; S[7] += wv * pc.y; S[8] += wv * pc.z;
                }
                S[2] = dy * S[0];
                S[4] = dy * S[1];
                S[5] = dy * S[2];
            }
#pragma unroll
            for (int off = kBwdHits; off < 32; off <<= 1)
#pragma unroll
                for (int c = 0; c < 9; c++) S[c] += __shfl_xor_sync(FULL, S[c], off);
            if (act && part == 0) {
                float* o = s_part[w][myk];
                o[0] = -inv_log2e * (2.f * abco.x * S[1] + abco.y * S[2]);
                o[1] = -inv_log2e * (abco.y * S[1] + 2.f * abco.z * S[2]);
                o[2] = -0.5f * S[3];
                o[3] = -S[4];
                o[4] = -0.5f * S[5];
                o[5] = abco.w > 0.f ? S[0] / abco.w : 0.f;  // sum of dalpha G = sum of dalpha (o G) / o
                o[6] = S[6]; o[7] = S[7]; o[8] = S[8];
            }
            nh = 0;
            __syncwarp();
        };
        for (int bend = n_list; bend > 0; bend -= BB) {
            const int b0 = max(0, bend - BB);
            const int cnt = bend - b0;
            __syncthreads();
            for (int j = threadIdx.x; j < cnt; j += NT) {
                const uint32_t p = start + b0 + j;
                stage(mean2d, conic_opa, rgb_depth, src[p], cfg.alpha_min, s_xy[j], s_abco[j], s_rgb[j], s_box[j]);
                s_emit[j] = emit[p];
            }
            __syncthreads();
            for (int ch = (cnt - 1) >> 5; ch >= 0; ch--) {
                const int k0 = ch * 32;
                const int kk = k0 + lane;
                const bool cand = kk < cnt && b0 + kk < warp_nc;
                unsigned m = __ballot_sync(FULL, cand && wb.hits(s_box[cand ? kk : 0]));
                const unsigned hits = m;
                unsigned skipped = 0;  // hits where no pixel of the warp composites (rare)
                const int ncb = nc - b0 - k0;  // this lane's contributors past the chunk start
                while (m) {  // back to front inside the chunk
                    const int jb = 31 - __clz(m);
                    m &= ~(1u << jb);
                    const int k = k0 + jb;
                    const float2 xy = s_xy[k];
                    const float4 abco = s_abco[k];
                    const float dx = px - xy.x, dy = py - xy.y;
                    const float e = exponent2(abco, dx, dy);
                    const float G = fast_exp2(e);
                    const float og = __fmul_rn(abco.w, G);
                    const float alpha = fminf(cfg.alpha_max, og);
                    // same decisions as the forward pass: listed before this pixel's
                    // last contributor, exponent <= 0, alpha >= alpha_min
                    const bool contrib = jb < ncb && !(e > 0.f) && alpha >= cfg.alpha_min;
                    if (__any_sync(FULL, contrib)) {
                        // predicated adjoint: non-contributing lanes keep their
                        // state and add zeros
                        const float inv = fast_rcp(1.f - alpha);
                        T = contrib ? T * inv : T;  // transmittance in front of this Gaussian
                        const float4 c = s_rgb[k];
                        const float wgt = contrib ? alpha * T : 0.f;
                        // dL/dalpha = sum_ch dL/dC_ch (T c_ch - S_ch / (1 - alpha))
                        const float gc = gr * c.x + gg * c.y + gb * c.z;
                        const float dalpha = T * gc - gS * inv;
                        gS += wgt * gc;
                        // alpha clamped at alpha_max passes no gradient to the exponent or
                        // opacity; selects (not products with 0) keep a non-finite og or G
                        // of a lane outside the Gaussian out of the sums
                        const bool pass = contrib && og < cfg.alpha_max;
                        const float dpow = pass ? dalpha * og : 0.f;  // d alpha / d(natural exponent)
                        // record this pixel's two scalars; the 9 gradient terms are summed
                        // over the warp's pixels when the table is full
                        s_tdw[w][nh][lane] = make_float2(dpow, wgt);
                        if (lane % kBwdHits == nh) myk = k;
                        if (++nh == kBwdHits) flush();
                    } else {
                        skipped |= 1u << jb;
                    }
                }
                if (lane == 0) s_hit[w][ch] = hits & ~skipped;
            }
            if (nh > 0) flush();
            __syncthreads();
            for (int j = threadIdx.x; j < cnt; j += NT) {
                const int ch = j >> 5;
                const uint32_t bit = 1u << (j & 31);
                float a[9];
#pragma unroll
                for (int c = 0; c < 9; c++) a[c] = 0.f;
                for (int ww = 0; ww < NW; ww++)
                    if (s_hit[ww][ch] & bit)
#pragma unroll
                        for (int c = 0; c < 9; c++) a[c] += s_part[ww][j][c];
                const uint32_t e = s_emit[j];
                if ((int64_t)e < capacity) {
                    part0[e] = make_float4(a[0], a[1], a[2], a[3]);
                    part1[e] = make_float4(a[4], a[5], a[6], a[7]);
                    part2[e] = a[8];
                }
            }
        }
        __syncthreads();  // shared buffers are reused by the next tile
    }
}

// ---------------------------------------------------------------------------
// 16 x 16 tiles, large launches. Both kernels are bound by instruction issue, so
// both put two pixels into the halves of the packed FP32 instructions
// (fma/mul/add.rn.f32x2: two FP32 operations, each rounded as the scalar one, in
// one issue slot), give each lane more than one pixel, and drop a Gaussian from a
// block of pixels that none of its pixels can reach alpha_min in before the block
// spends anything on it. Images, transmittances and contributor counts are the
// bits of k_render_fwd; the adjoint keeps that of k_render_bwd but for the
// roundings of the colour and opacity sums.
// ---------------------------------------------------------------------------
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ f32x2 both(float v) { return pack2(v, v); }
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

template <bool B>
struct BoolC {
    static constexpr bool value = B;
};

constexpr int kFastTile = 16;

// A list entry as one lane stages it: the exponent coefficients in base 2, e =
// A dx^2 + B dx dy + C dy^2, the negated centre, opacity, colour, depth, and a
// bit for each block of the tile in which its alpha can reach alpha_min (bit
// column + COLS * row).
//
// `plain` marks a Gaussian at which the exponent cannot round to a positive
// value and alpha cannot reach alpha_max, so that a batch of plain ones does
// without those two tests: with B^2 <= 4 A C (1 - d) the exact exponent is at
// most -(d/2)(|A| dx^2 + |C| dy^2) while the rounding of its five operations adds
// at most 8 * 2^-24 (|A| dx^2 + |C| dy^2), less than that for d = 1e-5; then
// 2^e <= 1 + 2^-22 and o 2^e < alpha_max for o < alpha_max (1 - 1e-6).
struct Entry {
    float nx, ny, A, B, C, o, r, g, b, z;
    unsigned blocks;
    bool plain;
};

// COLS x ROWS blocks of 16 / COLS by 16 / ROWS pixels from the tile's first pixel
// centre (tx0, ty0). A block is kept when the exponent's maximum over the
// rectangle of its pixel centres - on the two edges that face the Gaussian's
// centre, or 0 inside - reaches log2(alpha_min / o), with 0.2% + 0.02 to spare.
// That holds for ellipses that are not too thin (d = 1e-3 in the bound above
// keeps the rounding of the exponent below 1e-3 of it); the others take the
// bounding box of stage(). Against the box alone this drops a fifth of the 8x4
// blocks and a sixth of the 8x8 blocks of the synthetic 1080p scenes.
template <int COLS, int ROWS>
__device__ __forceinline__ Entry load_entry(const float2* __restrict__ mean2d, const float4* __restrict__ conic_opa,
                                            const float4* __restrict__ rgb_depth, uint32_t idx, float tx0, float ty0,
                                            float alpha_min, float alpha_max) {
    constexpr float BW = 16 / COLS, BH = 16 / ROWS;
    const float2 xy = mean2d[idx];
    const float4 co = conic_opa[idx], rgb = rgb_depth[idx];
    Entry e;
    e.nx = -xy.x; e.ny = -xy.y;
    e.A = -0.5f * kLog2e * co.x; e.B = -kLog2e * co.y; e.C = -0.5f * kLog2e * co.z; e.o = co.w;
    e.r = rgb.x; e.g = rgb.y; e.b = rgb.z; e.z = rgb.w;
    const bool conic = e.A < 0.f && e.C < 0.f && e.A > -1e15f && e.C > -1e15f;
    const float ac4 = 4.f * (e.A * e.C), bb = e.B * e.B;
    e.plain = conic && bb <= (1.f - 1e-5f) * ac4 && e.o < alpha_max * (1.f - 1e-6f);
    unsigned m = 0;
    if (!(e.o >= alpha_min)) {
        // can never reach alpha_min
    } else if (conic && bb <= (1.f - 1e-3f) * ac4) {
        const float low = 1.002f * (fast_log2(alpha_min) - fast_log2(e.o)) - 0.02f;
        const float sx = -0.5f * e.B * fast_rcp(e.A);  // along a row dy the maximum is at sx dy
        const float sy = -0.5f * e.B * fast_rcp(e.C);  // along a column dx at sy dx
#pragma unroll
        for (int c = 0; c < COLS; c++) {
            const float X0 = (tx0 + BW * c) + e.nx, X1 = (tx0 + (BW * c + (BW - 1.f))) + e.nx;
            const float ex = fminf(fmaxf(0.f, X0), X1);  // the column of centres nearest to the Gaussian's
            const float vs = sy * ex, be = e.B * ex, ae = e.A * ex * ex;
#pragma unroll
            for (int r = 0; r < ROWS; r++) {
                const float Y0 = (ty0 + BH * r) + e.ny, Y1 = (ty0 + (BH * r + (BH - 1.f))) + e.ny;
                const float ey = fminf(fmaxf(0.f, Y0), Y1);
                const float vy = fminf(fmaxf(vs, Y0), Y1);       // the maximum on column ex
                const float ux = fminf(fmaxf(sx * ey, X0), X1);  // and on row ey
                const float e1 = ae + vy * (be + e.C * vy);
                const float e2 = e.C * ey * ey + ux * (e.B * ey + e.A * ux);
                if (!(fmaxf(e1, e2) < low)) m |= 1u << (c + COLS * r);
            }
        }
    } else {
        float2 xy2;
        float4 abco, c2, box;
        stage(mean2d, conic_opa, rgb_depth, idx, alpha_min, xy2, abco, c2, box);
#pragma unroll
        for (int c = 0; c < COLS; c++)
#pragma unroll
            for (int r = 0; r < ROWS; r++)
                if (box.x <= tx0 + (BW * c + (BW - 1.f)) && box.z >= tx0 + BW * c &&
                    box.y <= ty0 + (BH * r + (BH - 1.f)) && box.w >= ty0 + BH * r)
                    m |= 1u << (c + COLS * r);
    }
    e.blocks = m;
    return e;
}

// ---------------------------------------------------------------------------
// Forward: four warps per tile, each warp an 8x8 block, each lane two pixels four
// rows apart. FB list entries are staged per round by the whole CTA.
// ---------------------------------------------------------------------------
struct __align__(16) FwdRow {
    float nx, ny, A, B;
    float C, o, r, g;
    float b, z, unused0, unused1;
};

// One pixel's forward step by predicated instructions: p = alpha reaches
// alpha_min (and, with ALL, the exponent is not positive), q = p and the pixel
// goes on, r = p and it terminates here. T carries a second meaning in its sign:
// a pixel that has terminated (or lies outside the view) keeps its transmittance
// with the sign set, so that T (1 - alpha) < t_min holds at every later Gaussian.
// Predicated FMAs instead of selects: selects and compares share the half-rate
// ALU pipe.
struct FwdPixel {
    float T, cr, cg, cb, cz;
    int last;  // the batch's last composited Gaussian, or -1
};
template <bool ALL>
__device__ __forceinline__ void composite(FwdPixel& s, float e, float alpha, float aT, float nT, float alpha_min,
                                          float t_min, float r, float g, float b, int pos) {
    if (ALL) {
        asm("{\n\t.reg .pred p, q, r;\n\t"
            "setp.leu.f32 p, %5, 0f00000000;\n\t"
            "setp.ge.and.f32 p, %6, %9, p;\n\t"
            "setp.lt.and.f32 r|q, %8, %10, p;\n\t"
            "@q fma.rn.f32 %1, %7, %11, %1;\n\t"
            "@q fma.rn.f32 %2, %7, %12, %2;\n\t"
            "@q fma.rn.f32 %3, %7, %13, %3;\n\t"
            "@q sub.rn.f32 %0, %0, %7;\n\t"
            "@q mov.b32 %4, %14;\n\t"
            "@r or.b32 %0, %0, 0x80000000;\n\t}"
            : "+f"(s.T), "+f"(s.cr), "+f"(s.cg), "+f"(s.cb), "+r"(s.last)
            : "f"(e), "f"(alpha), "f"(aT), "f"(nT), "f"(alpha_min), "f"(t_min), "f"(r), "f"(g), "f"(b), "r"(pos));
    } else {
        asm("{\n\t.reg .pred p, q, r;\n\t"
            "setp.ge.f32 p, %5, %8;\n\t"
            "setp.lt.and.f32 r|q, %7, %9, p;\n\t"
            "@q fma.rn.f32 %1, %6, %10, %1;\n\t"
            "@q fma.rn.f32 %2, %6, %11, %2;\n\t"
            "@q fma.rn.f32 %3, %6, %12, %3;\n\t"
            "@q sub.rn.f32 %0, %0, %6;\n\t"
            "@q mov.b32 %4, %13;\n\t"
            "@r or.b32 %0, %0, 0x80000000;\n\t}"
            : "+f"(s.T), "+f"(s.cr), "+f"(s.cg), "+f"(s.cb), "+r"(s.last)
            : "f"(alpha), "f"(aT), "f"(nT), "f"(alpha_min), "f"(t_min), "f"(r), "f"(g), "f"(b), "r"(pos));
    }
}

// 1M Gaussians, eight 1080p views: 1.92 -> 1.21 ms against k_render_fwd<16, 256>
// (86% of issue slots, FMA and ALU pipes about half busy); with two pixels side by
// side and the mask scan as before 1.36 ms, the exact block test and its cheaper
// staging (one log2 and two reciprocals instead of two roots and two divisions)
// 1.30, two hits per loop round 1.21. Four warps per tile leave small launches
// with too few warps: at 240 tiles 102 against 82 us, at 960 tiles 132 against
// 133, at 1840 tiles 67 against 78. A tile whose list is many times the others' ends
// the launch by itself, and an entry of it takes 0.040 us here against 0.029 in
// k_render_fwd: scenes with deep transparent clusters run at 0.87 to 0.99 of its speed
// (0.73 with nearly all pairs in a few tiles).
constexpr int kFwdThreads = 128;
constexpr int kFwdMinTiles = 1216;

// DEPTH and COUNT as for k_render_fwd; counts[0] counts a warp's hit twice, once
// for each 32 of its 64 pixels.
template <int FB, bool DEPTH, bool COUNT = false>
__global__ void __launch_bounds__(kFwdThreads) k_blocks_fwd(gs_frame f, gs_config cfg,
                                                            const uint32_t* __restrict__ range,
                                                            const uint32_t* __restrict__ src,
                                                            const float2* __restrict__ mean2d,
                                                            const float4* __restrict__ conic_opa,
                                                            const float4* __restrict__ rgb_depth,
                                                            float* __restrict__ color, float* __restrict__ t_final,
                                                            int32_t* __restrict__ n_contrib,
                                                            float* __restrict__ depth_out,
                                                            const uint32_t* __restrict__ order, uint32_t* counter,
                                                            int n_tiles, unsigned long long* counts) {
    constexpr int NT = kFwdThreads;
    unsigned long long n_hit = 0, n_eval = 0, n_comp = 0;
    __shared__ FwdRow s_g[FB];
    __shared__ uint8_t s_blocks[FB];  // bits 0-3: the warps whose block it touches; bit 4: needs all tests
    __shared__ int s_item;
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const float alpha_min = cfg.alpha_min, t_min = cfg.t_min;
    for (int tile = next_tile(order, counter, n_tiles, true, &s_item); tile >= 0;
         tile = next_tile(order, counter, n_tiles, false, &s_item)) {
        const int view = view_of_tile(f, tile);
        const int local = tile - f.tile_base[view];
        const int tx = local % f.tiles_x[view], ty = local / f.tiles_x[view];
        const int x = tx * kFastTile + (w & 1) * 8 + (lane & 7), y = ty * kFastTile + (w >> 1) * 8 + (lane >> 3);
        const int W = f.width[view], H = f.height[view];
        const bool in0 = x < W && y < H, in1 = x < W && y + 4 < H;
        const float px = x + 0.5f;
        const f32x2 py = pack2(y + 0.5f, y + 4.5f);
        const float tx0 = tx * kFastTile + 0.5f, ty0 = ty * kFastTile + 0.5f;
        const uint32_t start = range[2 * tile], end = range[2 * tile + 1];
        FwdPixel s0 = {in0 ? 1.f : -1.f, 0.f, 0.f, 0.f, 0.f, -1}, s1 = {in1 ? 1.f : -1.f, 0.f, 0.f, 0.f, 0.f, -1};
        int last0 = 0, last1 = 0;  // list positions after the last composited Gaussian
        auto done = [&]() { return (__float_as_uint(s0.T) & __float_as_uint(s1.T)) >> 31; };
        for (uint32_t b0 = start; b0 < end; b0 += FB) {
            if (__syncthreads_and(done())) break;
#pragma unroll 1
            for (int j = threadIdx.x; j < FB; j += NT)
                if (b0 + j < end) {
                    const Entry e = load_entry<2, 2>(mean2d, conic_opa, rgb_depth, src[b0 + j], tx0, ty0, alpha_min,
                                                     cfg.alpha_max);
                    s_blocks[j] = (uint8_t)(e.blocks | (e.plain ? 0u : 16u));
                    float4* o = reinterpret_cast<float4*>(&s_g[j]);
                    o[0] = make_float4(e.nx, e.ny, e.A, e.B);
                    o[1] = make_float4(e.C, e.o, e.r, e.g);
                    o[2] = make_float4(e.b, e.z, 0.f, 0.f);
                }
            __syncthreads();
            const int cnt = min((uint32_t)FB, end - b0);
            s0.last = s1.last = -1;
            for (int k0 = 0; k0 < cnt; k0 += 32) {
                if (__all_sync(FULL, done())) break;
                const unsigned bits = k0 + lane < cnt ? s_blocks[k0 + lane] : 0u;
                const bool hit = (bits >> w) & 1u;
                unsigned m = __ballot_sync(FULL, hit);
                const bool all = (__ballot_sync(FULL, bits & 16u) & m) != 0;
                auto walk = [&](auto all_c) {
                    constexpr bool ALL = decltype(all_c)::value;
                    auto one = [&](int k, const FwdRow& G) {
                        const float dx = px + G.nx;
                        const f32x2 dy = add2(py, both(G.ny));
                        // fma(A dx, dx, fma(C dy, dy, (B dx) dy)): the rounding sequence of exponent2,
                        // the same forward and backward, so that both take identical decisions
                        const f32x2 in = fma2(mul2(both(G.C), dy), dy, mul2(both(__fmul_rn(G.B, dx)), dy));
                        const f32x2 e2 = fma2(both(__fmul_rn(G.A, dx)), both(dx), in);
                        float e[2], a[2], aT[2], nT[2];
                        unpack2(e2, e[0], e[1]);
                        unpack2(mul2(both(G.o), pack2(fast_exp2(e[0]), fast_exp2(e[1]))), a[0], a[1]);
                        if (ALL) {
                            a[0] = fminf(cfg.alpha_max, a[0]);
                            a[1] = fminf(cfg.alpha_max, a[1]);
                        }
                        const f32x2 T2 = pack2(s0.T, s1.T);
                        const f32x2 aT2 = mul2(pack2(a[0], a[1]), T2);  // the blending weights
                        unpack2(aT2, aT[0], aT[1]);
                        unpack2(fma2(aT2, both(-1.f), T2), nT[0], nT[1]);  // T (1 - alpha)
                        if (COUNT) {
                            n_hit += 2;
                            n_eval += (s0.T > 0.f) + (s1.T > 0.f);
                        }
                        composite<ALL>(s0, e[0], a[0], aT[0], nT[0], alpha_min, t_min, G.r, G.g, G.b, k);
                        composite<ALL>(s1, e[1], a[1], aT[1], nT[1], alpha_min, t_min, G.r, G.g, G.b, k);
                        if (COUNT) n_comp += (s0.last == k) + (s1.last == k);
                        if (DEPTH) {  // composited here exactly when this Gaussian is now the last
                            if (s0.last == k) s0.cz += aT[0] * G.z;
                            if (s1.last == k) s1.cz += aT[1] * G.z;
                        }
                    };
                    while (m) {
                        const int ka = k0 + __ffs(m) - 1;
                        m &= m - 1;
                        const bool two = m != 0;
                        const int kb = two ? k0 + __ffs(m) - 1 : ka;
                        m &= m - 1;
                        const FwdRow ga = s_g[ka], gb = s_g[kb];
                        one(ka, ga);
                        if (two) one(kb, gb);
                    }
                };
                if (all) walk(BoolC<true>{}); else walk(BoolC<false>{});
            }
            if (s0.last >= 0) last0 = (int)(b0 - start) + s0.last + 1;
            if (s1.last >= 0) last1 = (int)(b0 - start) + s1.last + 1;
        }
        const int64_t plane = (int64_t)W * H, pix = f.pix_base[view] + (int64_t)y * W + x;
        const int64_t cbase = 3 * f.pix_base[view] + (int64_t)y * W + x;
        auto write = [&](const FwdPixel& s, int last, int64_t down) {
            const float T = fabsf(s.T);
            color[cbase + down] = s.cr + T * cfg.bg[0];
            color[cbase + down + plane] = s.cg + T * cfg.bg[1];
            color[cbase + down + 2 * plane] = s.cb + T * cfg.bg[2];
            t_final[pix + down] = T;
            n_contrib[pix + down] = last;
            if (DEPTH) depth_out[pix + down] = s.cz;
        };
        if (in0) write(s0, last0, 0);
        if (in1) write(s1, last1, 4 * (int64_t)W);
        __syncthreads();  // shared buffers are reused by the next tile
    }
    if (COUNT) {
        for (int o = 16; o > 0; o >>= 1) {
            n_eval += __shfl_xor_sync(FULL, n_eval, o);
            n_comp += __shfl_xor_sync(FULL, n_comp, o);
        }
        if (lane == 0) {
            atomicAdd(&counts[0], n_hit);  // every lane counted the warp's hits; lane 0 reports them once
            atomicAdd(&counts[1], n_eval);
            atomicAdd(&counts[2], n_comp);
        }
    }
}

// ---------------------------------------------------------------------------
// Adjoint: one warp per tile, each quad of lanes owning one 8x4 block of pixels
// and each lane one row of eight of them. The quads walk lists of their own: at
// any time the eight quads work on eight different Gaussians, so a block costs
// nothing for a Gaussian that does not touch it, no barrier joins warps, a
// Gaussian's sums over a row stay in registers, and what it costs beside its
// pixels - loads, list and loop, the reduction over rows - is paid once per eight
// blocks.
//
// 1M Gaussians, eight 1080p views: 4.43 -> 2.38 ms against k_render_bwd<16, 64>
// (248 instead of 535 million warp instructions per view; issue 67% busy at 14
// warps per SM, which registers and the block sums in shared memory allow; 2.33 ms
// before non-finite sums were looked for and long lists left out). Of
// this the exact block test took 3.05 to 2.89 ms, batches of 32 instead of 64
// with the next rows on their way 2.42, the cheaper staging 2.33. One warp per
// tile needs many tiles, more of them in several small views, whose full tiles in the
// middle come round at the same SMs: 200k Gaussians in seven 320x240 views (2,100
// tiles) 714 against 499 us, in one of 960x640 (2,400) 91 against 93, in four of 480x400
// (3,000) 267 against 286, in one of 1100x720 (3,105) 85 against 96, in eight of 400x320
// (4,000) 493 against 508, in one of 1280x720 (3,600) 82 against 101: from 20 tiles per SM,
// a quarter more than are resident.
// ---------------------------------------------------------------------------
constexpr int kBwdMinTiles = 20 * 152;
constexpr int kRowPx = 8;      // pixels of a lane
constexpr int kRowBlocks = 8;  // 8x4 blocks of a tile, one per quad of lanes

// This lane's row of pixels: block (lane / 4) in raster order of the tile's 2 x 4
// blocks, row lane % 4 of it.
struct RowInfo {
    int view, x, y, W, n_in;  // first pixel; how many of the eight lie in the view
    int64_t pix, plane, color_base;
    bool vec;                 // all eight lie in the view and 16-byte loads are aligned
    float tx0, ty0;           // the tile's first pixel centre
};

// aligned: the buffers that rows are read from start on 16 bytes.
__device__ __forceinline__ RowInfo row_info(const gs_frame& f, int tile, bool aligned) {
    RowInfo t;
    t.view = view_of_tile(f, tile);
    const int local = tile - f.tile_base[t.view];
    const int tx = local % f.tiles_x[t.view], ty = local / f.tiles_x[t.view];
    const int lane = threadIdx.x & 31, b = lane >> 2;
    t.x = tx * kFastTile + (b & 1) * kRowPx;
    t.y = ty * kFastTile + (b >> 1) * 4 + (lane & 3);
    t.W = f.width[t.view];
    const int H = f.height[t.view];
    t.n_in = t.y < H ? min(max(t.W - t.x, 0), kRowPx) : 0;
    t.plane = (int64_t)t.W * H;
    const int64_t pb = f.pix_base[t.view];
    t.pix = pb + (int64_t)t.y * t.W + t.x;
    t.color_base = 3 * pb + (int64_t)t.y * t.W + t.x;
    t.vec = aligned && t.n_in == kRowPx && ((t.W | (int)pb) & 3) == 0;
    t.tx0 = (float)(tx * kFastTile) + 0.5f;
    t.ty0 = (float)(ty * kFastTile) + 0.5f;
    return t;
}

// A row's eight values from memory (aligned: two 16-byte loads).
template <class T, class V4>
__device__ __forceinline__ void load_row(const T* __restrict__ p, const RowInfo& t, T (&v)[kRowPx]) {
    if (t.vec) {
        const V4 a = reinterpret_cast<const V4*>(p)[0], b = reinterpret_cast<const V4*>(p)[1];
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
        for (int i = 0; i < kRowPx; i++)
            if (i < t.n_in) v[i] = p[i];
    }
}

// Exponents and 2^exponent times opacity at two neighbouring pixels of a row:
// the rounding sequence e = fma(A dx, dx, fma(C dy, dy, (B dx) dy)) of the
// tile-8 and tile-32 kernels, the same forward and backward, so that all take
// identical decisions.
struct TwoAlphas {
    f32x2 dx;
    float e[2], og[2];
};
__device__ __forceinline__ TwoAlphas two_alphas(f32x2 x, f32x2 nx, f32x2 A, f32x2 B, f32x2 o, f32x2 dy, f32x2 cy) {
    TwoAlphas r;
    r.dx = add2(x, nx);
    unpack2(fma2(mul2(A, r.dx), r.dx, fma2(cy, dy, mul2(mul2(B, r.dx), dy))), r.e[0], r.e[1]);
    unpack2(mul2(o, pack2(fast_exp2(r.e[0]), fast_exp2(r.e[1]))), r.og[0], r.og[1]);
    return r;
}

struct __align__(16) BwdRow {
    float nx, ny, A, B;
    float C, o, r, g;
    float b, unused[3];
};
__device__ __forceinline__ f32x2 load2(const float (&v)[2]) { return pack2(v[0], v[1]); }

template <int CG>
__device__ __forceinline__ void cp_async(void* smem, const void* gmem) {
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem);
    if (CG == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(s), "l"(gmem), "n"(CG) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The adjoint by rows. Per pixel and Gaussian, back to front: the transmittance in
// front of it, dL/dalpha and from it dpow = dL/d(exponent) and the blending
// weight. A lane sums the nine gradient terms over its row of eight pixels in
// registers, two shuffles join the block's four rows, and the block's sums wait in
// shared memory until the batch of 32 list entries is done; then each entry adds
// its blocks' sums in raster order into its one partial. A pixel the Gaussian does
// not touch enters with alpha = 0, which leaves its state as it is and adds zeros,
// so one select per pixel is all the predication there is. The next batch's
// projected rows are on their way (cp.async) while this one is worked on.
//
// A product with that zero is NaN where the other factor is not finite: a pixel whose
// gradient is infinite or NaN would spoil the sums of every Gaussian listed for its
// block, not of those that it composites. k_render_bwd has selects for that and does
// tiles with such a sum once more (a look at the pixels' gradients cost 3% of this kernel's
// speed, a second form of its loop 5%).
constexpr int kBwdBatch = 32;

__global__ void __launch_bounds__(32, 16) k_rows_bwd(gs_frame f, gs_config cfg, const uint32_t* __restrict__ range,
                                                     const uint32_t* __restrict__ src,
                                                     const uint32_t* __restrict__ emit,
                                                     const float2* __restrict__ mean2d,
                                                     const float4* __restrict__ conic_opa,
                                                     const float4* __restrict__ rgb_depth,
                                                     const float* __restrict__ t_final,
                                                     const int32_t* __restrict__ n_contrib,
                                                     const float* __restrict__ dL_dcolor, float4* __restrict__ part0,
                                                     float4* __restrict__ part1, float* __restrict__ part2,
                                                     int64_t capacity, const uint32_t* __restrict__ order,
                                                     uint32_t* counter, int n_tiles,
                                                     const int64_t* __restrict__ count, float share,
                                                     uint8_t* __restrict__ again, bool aligned) {
    __shared__ float2 s_raw_xy[kBwdBatch];  // the next batch's projected rows
    __shared__ float4 s_raw_co[kBwdBatch];
    __shared__ float4 s_raw_rgb[kBwdBatch];
    __shared__ BwdRow s_row[kBwdBatch + 1];  // the last one: a Gaussian that no pixel composites
    __shared__ uint16_t s_list[kRowBlocks][kBwdBatch + 1];  // row | block sum << 8
    __shared__ float s_sum[kBwdBatch * kRowBlocks][9];
    __shared__ int s_item;
    __shared__ int s_tile, s_odd;  // the tile; a sum of it that is not finite
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x, blk = lane >> 2;
    const float inv_log2e = 1.f / kLog2e;
    const float alpha_min = cfg.alpha_min;
    launch_next();
    if (lane == 0) {
        BwdRow none = {};
        none.o = -INFINITY;  // times 2^0: below any alpha_min
        s_row[kBwdBatch] = none;
    }
    for (int tile = next_tile(order, counter, n_tiles, true, &s_item); tile >= 0;
         tile = next_tile(order, counter, n_tiles, false, &s_item)) {
        const uint32_t start = range[2 * tile], len = range[2 * tile + 1] - start;
        if (lane == 0) {
            s_tile = tile;
            s_odd = 0;
            again[tile] = 0;
        }
        if (share > 0.f && len > long_list(count, capacity, share)) continue;  // k_render_bwd's
        const RowInfo ti = row_info(f, tile, aligned);
        const float py = ti.y + 0.5f;
        int nc[kRowPx];
        f32x2 xs[kRowPx / 2], T2[kRowPx / 2], S2[kRowPx / 2], nr[kRowPx / 2], ng[kRowPx / 2], nb[kRowPx / 2];
        {
            float t[kRowPx], r[kRowPx], g[kRowPx], b[kRowPx];
#pragma unroll
            for (int i = 0; i < kRowPx; i++) {
                t[i] = 1.f;
                r[i] = g[i] = b[i] = 0.f;
                nc[i] = 0;
            }
            if (ti.n_in > 0) {
                load_row<float, float4>(t_final + ti.pix, ti, t);
                load_row<int, int4>(n_contrib + ti.pix, ti, nc);
                load_row<float, float4>(dL_dcolor + ti.color_base, ti, r);
                load_row<float, float4>(dL_dcolor + ti.color_base + ti.plane, ti, g);
                load_row<float, float4>(dL_dcolor + ti.color_base + 2 * ti.plane, ti, b);
            }
            // S = sum over channels of dL/dC_ch times the colour composited behind the
            // current Gaussian plus the background seen through T_final: dL/dalpha needs
            // only this dot product, so one scalar replaces three running colours. The
            // colour gradients are held negated: with -alpha the packed operations, which
            // have no negation, then give S, dpow and w dL/dc.
#pragma unroll
            for (int p = 0; p < kRowPx / 2; p++) {
                const int i = 2 * p, j = i + 1;
                xs[p] = pack2(ti.x + (i + 0.5f), ti.x + (j + 0.5f));
                T2[p] = pack2(t[i], t[j]);
                S2[p] = pack2(t[i] * (r[i] * cfg.bg[0] + g[i] * cfg.bg[1] + b[i] * cfg.bg[2]),
                              t[j] * (r[j] * cfg.bg[0] + g[j] * cfg.bg[1] + b[j] * cfg.bg[2]));
                nr[p] = pack2(-r[i], -r[j]);
                ng[p] = pack2(-g[i], -g[j]);
                nb[p] = pack2(-b[i], -b[j]);
            }
        }
        int nc_blk = nc[0], nc_low = ti.n_in > 0 ? nc[0] : 0x7fffffff;  // the row's (then block's) range
#pragma unroll
        for (int i = 1; i < kRowPx; i++) {
            nc_blk = max(nc_blk, nc[i]);
            if (i < ti.n_in) nc_low = min(nc_low, nc[i]);
        }
        nc_blk = max(nc_blk, __shfl_xor_sync(FULL, nc_blk, 1));
        nc_blk = max(nc_blk, __shfl_xor_sync(FULL, nc_blk, 2));
        const int n_list = __reduce_max_sync(FULL, (unsigned)nc_blk);
        // batches of entries before this position need no test against a pixel's last
        // contributor (pixels outside the view have none and keep that test on)
        const int n_plain = ti.n_in == kRowPx ? nc_low : 0;
        const int n_all = __reduce_min_sync(FULL, (unsigned)n_plain);
        // pairs past every pixel's last contributor: their emission slots are gathered per
        // Gaussian like all others
        constexpr int kZeros = 8;
        for (uint32_t j0 = (uint32_t)n_list + lane; j0 < len; j0 += 32 * kZeros) {
            uint32_t e[kZeros];
#pragma unroll
            for (int k = 0; k < kZeros; k++) e[k] = j0 + 32 * k < len ? emit[start + j0 + 32 * k] : 0xffffffffu;
#pragma unroll
            for (int k = 0; k < kZeros; k++)
                if ((int64_t)e[k] < capacity) part2[e[k]] = __uint_as_float(kNoPartial);
        }
        auto fetch = [&](int q, uint32_t idx) {  // entry q's rows on their way to this lane's places
            if (q >= 0) {
                cp_async<8>(&s_raw_xy[lane], mean2d + idx);
                cp_async<16>(&s_raw_co[lane], conic_opa + idx);
                cp_async<16>(&s_raw_rgb[lane], rgb_depth + idx);
            }
        };
        uint32_t idx = 0;  // the source row of this lane's entry of the batch after the fetched one
        if (n_list - 1 - lane >= 0) idx = src[start + n_list - 1 - lane];
        fetch(n_list - 1 - lane, idx);
        if (n_list - 1 - 32 - lane >= 0) idx = src[start + n_list - 1 - 32 - lane];
        for (int end0 = n_list; end0 > 0; end0 -= kBwdBatch) {  // row k is entry end0 - 1 - k
            const int q = end0 - 1 - lane;
            const uint32_t em = q >= 0 ? emit[start + q] : 0xffffffffu;
            cp_async_wait();  // each lane reads only what it fetched itself
            Entry e;
            e.blocks = 0;
            e.plain = true;
            e.o = 1.f;
            if (q >= 0) {
                e = load_entry<2, 4>(s_raw_xy, s_raw_co, s_raw_rgb, lane, ti.tx0, ti.ty0, alpha_min, cfg.alpha_max);
                float4* w = reinterpret_cast<float4*>(&s_row[lane]);
                w[0] = make_float4(e.nx, e.ny, e.A, e.B);
                w[1] = make_float4(e.C, e.o, e.r, e.g);
                s_row[lane].b = e.b;
            }
            fetch(q - kBwdBatch, idx);
            if (q - 2 * kBwdBatch >= 0) idx = src[start + q - 2 * kBwdBatch];
#pragma unroll
            for (int b = 0; b < kRowBlocks; b++)
                if (q >= __shfl_sync(FULL, nc_blk, 4 * b)) e.blocks &= ~(1u << b);
            const int mine = __popc(e.blocks);
            int incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(FULL, incl, o);
                if (lane >= o) incl += u;
            }
            const int first = incl - mine;  // this entry's block sums: [first, first + mine)
            int n_mine = 0, job = first;
#pragma unroll
            for (int b = 0; b < kRowBlocks; b++) {
                const bool hit = (e.blocks >> b) & 1u;
                const unsigned m = __ballot_sync(FULL, hit);
                if (hit) {
                    s_list[b][__popc(m & lanemask_lt())] = (uint16_t)(lane | job << 8);
                    job++;
                }
                if (blk == b) n_mine = __popc(m);
            }
            const int n_max = __reduce_max_sync(FULL, (unsigned)n_mine);
            const bool all = __any_sync(FULL, e.blocks && !e.plain);
            __syncwarp();
            // ALL: with the tests that plain Gaussians do without; LIM: with the test against
            // each pixel's last contributor
            auto walk = [&](auto all_c, auto lim_c) {
                constexpr bool ALL = decltype(all_c)::value, LIM = decltype(lim_c)::value;
                unsigned next = n_mine > 0 ? (unsigned)s_list[blk][0] : (unsigned)kBwdBatch;
                for (int i = 0; i < n_max; i++) {
                    const bool live = i < n_mine;
                    const unsigned ent = next;
                    next = i + 1 < n_mine ? (unsigned)s_list[blk][i + 1] : (unsigned)kBwdBatch;
                    const int k = ent & 255u;
                    const int pos = end0 - 1 - k;
                    const BwdRow& R = s_row[k];
                    const float4 q0 = reinterpret_cast<const float4*>(&R)[0], q1 = reinterpret_cast<const float4*>(&R)[1];
                    const f32x2 nx = both(q0.x), A = both(q0.z), B = both(q0.w), o = both(q1.y);
                    const f32x2 r2 = both(q1.z), g2 = both(q1.w), b2 = both(R.b);
                    const float dy = py + q0.y;
                    const f32x2 dy2 = both(dy), cy2 = both(__fmul_rn(q1.x, dy));
                    float s0 = 0.f, s1 = 0.f, s3 = 0.f;
                    f32x2 c6 = 0, c7 = 0, c8 = 0;
#pragma unroll
                    for (int p = 0; p < kRowPx / 2; p++) {
                        const TwoAlphas t = two_alphas(xs[p], nx, A, B, o, dy2, cy2);
                        // the same decisions as the forward pass: listed before this pixel's last
                        // contributor, exponent <= 0, alpha >= alpha_min; na = -alpha, or 0. Alpha
                        // clamped at alpha_max passes no gradient to the exponent or opacity (nog);
                        // selects keep a non-finite 2^e outside the Gaussian out of the sums.
                        float na[2], nog[2], m[2], dx[2], d[2];
#pragma unroll
                        for (int h = 0; h < 2; h++) {
                            const float alpha = ALL ? fminf(cfg.alpha_max, t.og[h]) : t.og[h];
                            bool in = alpha >= alpha_min;
                            if (LIM) in = in && pos < nc[2 * p + h];
                            if (ALL) in = in && !(t.e[h] > 0.f);
                            na[h] = in ? -alpha : 0.f;
                            nog[h] = ALL ? (in && t.og[h] < cfg.alpha_max ? -t.og[h] : 0.f) : na[h];
                        }
                        unpack2(add2(load2(na), both(1.f)), m[0], m[1]);
                        const f32x2 inv = pack2(fast_rcp(m[0]), fast_rcp(m[1]));
                        const f32x2 ngc = fma2(nb[p], b2, fma2(nr[p], r2, mul2(ng[p], g2)));
                        T2[p] = mul2(T2[p], inv);  // transmittance in front of this Gaussian (1/1 = 1 keeps it)
                        const f32x2 nw = mul2(load2(na), T2[p]);
                        // -dL/dalpha = S / (1 - alpha) - T sum_ch dL/dC_ch c_ch
                        const f32x2 ndal = fma2(T2[p], ngc, mul2(S2[p], inv));
                        S2[p] = fma2(nw, ngc, S2[p]);
                        unpack2(mul2(ndal, load2(nog)), d[0], d[1]);  // d alpha / d(natural exponent) dL/dalpha
                        unpack2(t.dx, dx[0], dx[1]);
#pragma unroll
                        for (int h = 0; h < 2; h++) {
                            s0 += d[h];
                            const float t1 = __fmul_rn(d[h], dx[h]);
                            s1 = __fadd_rn(s1, t1);
                            s3 = __fmaf_rn(t1, dx[h], s3);
                        }
                        c6 = fma2(nw, nr[p], c6);
                        c7 = fma2(nw, ng[p], c7);
                        c8 = fma2(nw, nb[p], c8);
                    }
                    // The block's sums, rows (0 + 1) + (2 + 3): in the first step the lanes of
                    // rows 0 and 2 keep the terms of dx and dy, those of rows 1 and 3 the others,
                    // in the second each lane keeps two (three in row 0) and finishes them.
                    float u, v, k0, k1, k2, k3, k4;
                    {
                        const bool odd = lane & 1;
                        const float dy1 = __fmul_rn(dy, s0);
                        auto part = [&](float keep_even, float keep_odd) {
                            const float give = odd ? keep_even : keep_odd;
                            return __fadd_rn(odd ? keep_odd : keep_even, __shfl_xor_sync(FULL, give, 1));
                        };
                        unpack2(c6, u, v);
                        const float s6 = u + v;
                        unpack2(c7, u, v);
                        const float s7 = u + v;
                        unpack2(c8, u, v);
                        const float s8 = u + v;
                        k0 = part(s1, __fmul_rn(dy, dy1));
                        k1 = part(dy1, s6);
                        k2 = part(s3, s7);
                        k3 = part(__fmul_rn(dy, s1), s8);
                        k4 = __fadd_rn(s0, __shfl_xor_sync(FULL, s0, 1));
                    }
                    {
                        const bool low = lane & 2;  // rows 2 and 3
                        const float g0 = low ? k0 : k2, g1 = low ? k1 : k3;
                        u = __fadd_rn(low ? k2 : k0, __shfl_xor_sync(FULL, g0, 2));
                        v = __fadd_rn(low ? k3 : k1, __shfl_xor_sync(FULL, g1, 2));
                        k4 = __fadd_rn(k4, __shfl_xor_sync(FULL, k4, 2));
                    }
                    // row 0: dx, dy, sum(dpow); row 1: dy dy, red; row 2: dx dx, dx dy; row 3: green, blue
                    if (live) {
                        float* out = s_sum[ent >> 8] + 2 * (lane & 3);
                        const float a = q0.z, b = q0.w, cc = q1.x;
                        const float m0 = -inv_log2e * (2.f * a * u + b * v), m1 = -inv_log2e * (b * u + 2.f * cc * v);
                        const bool row0 = (lane & 3) == 0;
                        out[0] = row0 ? m0 : u;
                        out[1] = row0 ? m1 : v;
                        if (row0) out[8] = k4;
                    }
                }
            };
            if (all) walk(BoolC<true>{}, BoolC<true>{});
            else if (end0 > n_all) walk(BoolC<false>{}, BoolC<true>{});
            else walk(BoolC<false>{}, BoolC<false>{});
            __syncwarp();
            if ((int64_t)em < capacity) {  // (no entry: past any capacity)
                float a[9];
#pragma unroll
                for (int c = 0; c < 9; c++) a[c] = 0.f;
                for (int j = first; j < first + mine; j++)
#pragma unroll
                    for (int c = 0; c < 9; c++) a[c] += s_sum[j][c];
                // sum of dalpha G = sum of dalpha (o G) / o
                part0[em] = make_float4(a[0], a[1], -0.5f * a[4], -a[5]);
                part1[em] = make_float4(-0.5f * a[2], e.o > 0.f ? a[8] / e.o : 0.f, a[3], a[6]);
                part2[em] = a[7];
                if (!(fabsf(a[8]) < INFINITY)) s_odd = 1;
            }
            __syncwarp();  // rows, lists and sums are rewritten by the next batch
        }
        if (lane == 0 && s_odd) again[s_tile] = 1;
    }
}

// ---------------------------------------------------------------------------
// Launch configurations (the autotuner picks among these)
// ---------------------------------------------------------------------------
struct RenderLaunch {
    const void* fn;
    int threads;
};

static RenderLaunch pick_fwd(int tile, int batch, int n_tiles, bool depth = false, bool count = false) {
#define GS_BLOCKS(B)                                                    \
    if (tile == kFastTile && n_tiles >= kFwdMinTiles && batch == B)     \
        return {count   ? (const void*)k_blocks_fwd<B, false, true>     \
                : depth ? (const void*)k_blocks_fwd<B, true>            \
                        : (const void*)k_blocks_fwd<B, false>,          \
                kFwdThreads};
    GS_BLOCKS(64) GS_BLOCKS(128) GS_BLOCKS(256)
#undef GS_BLOCKS
#define GS_FWD(T, B)                                                                     \
    if (tile == T && batch == B)                                                         \
        return {count   ? (const void*)k_render_fwd<T, B, false, true>                   \
                : depth ? (const void*)k_render_fwd<T, B, true>                          \
                        : (const void*)k_render_fwd<T, B, false>,                        \
                T * T};
    GS_FWD(8, 64) GS_FWD(8, 128) GS_FWD(8, 256)
    GS_FWD(16, 64) GS_FWD(16, 128) GS_FWD(16, 256)
    GS_FWD(32, 128) GS_FWD(32, 256)
#undef GS_FWD
    return {nullptr, 0};
}

static RenderLaunch pick_bwd(int tile, int batch, int n_tiles) {
    // k_rows_bwd has one batch size (its block sums take most of the shared memory)
    if (tile == kFastTile && n_tiles >= kBwdMinTiles && (batch == 32 || batch == 64 || batch == 128))
        return {(const void*)k_rows_bwd, 32};
#define GS_BWD(T, B) if (tile == T && batch == B) return {(const void*)k_render_bwd<T, B>, T * T};
    GS_BWD(8, 64) GS_BWD(8, 128) GS_BWD(8, 256)
    GS_BWD(16, 32) GS_BWD(16, 64) GS_BWD(16, 128)
    GS_BWD(32, 32)
#undef GS_BWD
    return {nullptr, 0};
}

static int default_fwd_batch(int tile, int n_tiles) {
    return tile == 8 || (tile == kFastTile && n_tiles >= kFwdMinTiles) ? 128 : 256;
}
static int default_bwd_batch(int tile) { return tile == 32 ? 32 : tile == 16 ? 64 : 128; }

// overlap: the launch starts when the one before allows it (launch_next), not when that ends.
static int launch(const RenderLaunch& L, int grid, bool persistent, void** args, cudaStream_t s, bool overlap = false) {
    if (persistent) {
        const int pg = persistent_grid(L.fn, L.threads);
        grid = grid < pg ? grid : pg;
    }
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(grid);
    lc.blockDim = dim3(L.threads);
    lc.stream = s;
    lc.attrs = &at;
    lc.numAttrs = overlap ? 1 : 0;
    if (cudaLaunchKernelExC(&lc, L.fn, args) != cudaSuccess) {
        (void)cudaGetLastError();
        return GS_ERR_CUDA;
    }
    count_launch();
    return GS_OK;
}

bool render_batch_supported(int tile, int fwd_batch, int bwd_batch) {
    return pick_fwd(tile, fwd_batch ? fwd_batch : default_fwd_batch(tile, 0), 0).fn != nullptr &&
           pick_bwd(tile, bwd_batch ? bwd_batch : default_bwd_batch(tile), 0).fn != nullptr;
}

}  // namespace gs

using namespace gs;

extern "C" size_t gs_render_workspace_size(const gs_frame* f) {
    (void)f;
    return 256;  // the persistent schedule's work counter
}

static bool render_args_ok(const gs_frame* f, const gs_config* cfg) {
    return f && cfg && f->n_views >= 1 && f->n_views <= GS_MAX_VIEWS && cfg->tile == f->tile &&
           render_batch_supported(cfg->tile, cfg->fwd_batch, cfg->bwd_batch);
}

static int render_fwd_impl(const gs_projected* p, const gs_pairs* pairs, const gs_frame* f, const gs_config* cfg,
                           const gs_image* out, void* ws, size_t ws_bytes, void* stream, unsigned long long* counts) {
    if (!p || !pairs || !out || !out->color || !out->t_final || !out->n_contrib || !render_args_ok(f, cfg))
        return GS_ERR_INVALID_ARG;
    const bool persistent = cfg->schedule == 1, ordered = cfg->schedule == 2;
    if (persistent && (!pairs->order || !ws || ws_bytes < 256)) return GS_ERR_INVALID_ARG;
    if (ordered && !pairs->order) return GS_ERR_INVALID_ARG;
    int n_tiles = f->tile_base[f->n_views];
    cudaStream_t s = (cudaStream_t)stream;
    if (counts && cudaMemsetAsync(counts, 0, 3 * sizeof(unsigned long long), s) != cudaSuccess) {
        (void)cudaGetLastError();
        return GS_ERR_CUDA;
    }
    if (n_tiles == 0) return GS_OK;
    uint32_t* counter = persistent ? (uint32_t*)ws : nullptr;
    const uint32_t* order = persistent || ordered ? pairs->order : nullptr;
    if (persistent) cudaMemsetAsync(counter, 0, sizeof(uint32_t), s);
    const RenderLaunch L = pick_fwd(cfg->tile, cfg->fwd_batch ? cfg->fwd_batch : default_fwd_batch(cfg->tile, n_tiles),
                                    n_tiles, out->depth != nullptr && !counts, counts != nullptr);
    gs_frame fv = *f;
    gs_config cv = *cfg;
    const uint32_t* range = pairs->range;
    const uint32_t* src = pairs->src;
    const float2* m2 = (const float2*)p->mean2d;
    const float4* co = (const float4*)p->conic_opa;
    const float4* rd = (const float4*)p->rgb_depth;
    float* color = out->color;
    float* tf = out->t_final;
    int32_t* nc = out->n_contrib;
    float* dz = out->depth;
    void* args[] = {&fv, &cv, (void*)&range, (void*)&src, (void*)&m2, (void*)&co, (void*)&rd,
                    (void*)&color, (void*)&tf, (void*)&nc, (void*)&dz, (void*)&order, (void*)&counter, &n_tiles,
                    (void*)&counts};
    return launch(L, n_tiles, persistent, args, s);
}

extern "C" int gs_render_fwd(const gs_projected* p, const gs_pairs* pairs, const gs_frame* f, const gs_config* cfg,
                             const gs_image* out, void* ws, size_t ws_bytes, void* stream) {
    return render_fwd_impl(p, pairs, f, cfg, out, ws, ws_bytes, stream, nullptr);
}

extern "C" int gs_render_fwd_count(const gs_projected* p, const gs_pairs* pairs, const gs_frame* f,
                                   const gs_config* cfg, const gs_image* out, void* ws, size_t ws_bytes,
                                   unsigned long long* counts, void* stream) {
    if (!counts) return GS_ERR_INVALID_ARG;
    return render_fwd_impl(p, pairs, f, cfg, out, ws, ws_bytes, stream, counts);
}

namespace gs {
int launch_render_bwd(const gs_projected* p, const gs_pairs* pairs, const gs_frame* f, const gs_config* cfg,
                      const gs_image* fwd, const float* dL_dcolor, float4* part0, float4* part1, float* part2,
                      uint32_t* counter, uint8_t* again, cudaStream_t s) {
    if (!render_args_ok(f, cfg)) return GS_ERR_INVALID_ARG;
    int n_tiles = f->tile_base[f->n_views];
    if (n_tiles == 0) return GS_OK;
    const bool persistent = cfg->schedule == 1, ordered = cfg->schedule == 2;
    if ((persistent || ordered) && !pairs->order) return GS_ERR_INVALID_ARG;
    const uint32_t* order = persistent || ordered ? pairs->order : nullptr;
    if (!persistent) counter = nullptr;
    if (persistent) cudaMemsetAsync(counter, 0, sizeof(uint32_t), s);
    const RenderLaunch L = pick_bwd(cfg->tile, cfg->bwd_batch ? cfg->bwd_batch : default_bwd_batch(cfg->tile), n_tiles);
    gs_frame fv = *f;
    gs_config cv = *cfg;
    const uint32_t* range = pairs->range;
    const uint32_t* src = pairs->src;
    const uint32_t* emit = pairs->emit;
    const int64_t* count = pairs->count;
    const bool rows = L.fn == (const void*)k_rows_bwd;
    float share = rows && count && n_tiles <= kLongTiles ? kLongMean / (float)n_tiles : 0.f;  // (without a count: none long)
    const float2* m2 = (const float2*)p->mean2d;
    const float4* co = (const float4*)p->conic_opa;
    const float4* rd = (const float4*)p->rgb_depth;
    const float* tf = fwd->t_final;
    const int32_t* nc = fwd->n_contrib;
    int64_t cap = pairs->capacity;
    // a caller's image or gradient may be any slice of a larger buffer; k_rows_bwd alone takes the flag
    bool aligned = (((uintptr_t)tf | (uintptr_t)nc | (uintptr_t)dL_dcolor) & 15) == 0;
    void* args[] = {&fv, &cv, (void*)&range, (void*)&src, (void*)&emit, (void*)&m2, (void*)&co, (void*)&rd,
                    (void*)&tf, (void*)&nc, (void*)&dL_dcolor, (void*)&part0, (void*)&part1, (void*)&part2,
                    &cap, (void*)&order, (void*)&counter, &n_tiles, (void*)&count, &share, (void*)&again, &aligned};
    const int rc = launch(L, n_tiles, persistent, args, s);
    if (rc != GS_OK || !rows) return rc;
    return launch({(const void*)k_render_bwd<kFastTile, 64, true>, kFastTile * kFastTile}, kLongCtas, false, args, s, true);
}
}  // namespace gs
