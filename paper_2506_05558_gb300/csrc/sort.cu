// Per-tile duplication and depth ordering (K2-K4).
//
// Design: instead of one radix sort of 64-bit (tile, depth) keys over all P
// pairs, the V visible (view, Gaussian) items are first sorted by their 32-bit
// fp32 depth bits (stable), their pairs are then emitted in that order, and a
// stable sort on the global tile index alone (ceil(log2 tiles) bits, 2 passes
// at 1080p x 8 views) yields each tile's list in (depth bits, item index)
// order. gs_sort uses single-pass kernels: each scan is one launch (chunks with
// decoupled look-back) and each radix sort one launch per 8-bit digit (tiles with
// decoupled look-back), the digits counted by the kernel that writes the keys; the
// tile sort carries every pair's (item, emission slot) and its last pass writes
// them to the output lists. 8 views of 1080p, 1M Gaussians (5.8M visible items, 15.8M
// pairs): 659 us in a graph, of which the passes over items take 188 and those over
// pairs 230 (970, 274 and 333 with separate scans, histograms, and values gathered from
// global memory in sorted order). Element counts are read from device memory, so the
// whole sort is enqueued without a host sync and can be captured in a CUDA
// graph. The reduce-then-scan scan and radix sort below serve the library's
// other compactions and sorts (anchors).
#include "common.cuh"

namespace gs {

// ---------------------------------------------------------------------------
// Device-wide exclusive scan (reduce, scan of block sums, down-sweep).
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;

struct LoadU32 {
    const uint32_t* p;
    __device__ uint32_t operator()(int64_t i) const { return p[i]; }
};
__device__ __forceinline__ int64_t valid_count(int64_t n_max, const uint32_t* n_dev) {
    return n_dev ? min(n_max, (int64_t)*n_dev) : n_max;
}

// Block-wide exclusive scan of one value per thread; returns the block total.
template <int NT>
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t& excl) {
    constexpr int NW = NT / 32;
    __shared__ uint32_t warp_off[NW];
    __shared__ uint32_t s_total;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t inc = v;  // inclusive scan within the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) warp_off[w] = inc;
    __syncthreads();
    if (w == 0) {
        const uint32_t t = lane < NW ? warp_off[lane] : 0u;
        uint32_t ti = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, ti, o);
            if (lane >= o) ti += u;
        }
        if (lane < NW) warp_off[lane] = ti - t;
        if (lane == NW - 1) s_total = ti;
    }
    __syncthreads();
    excl = warp_off[w] + inc - v;
    const uint32_t total = s_total;
    __syncthreads();  // the shared words may be reused by the next call
    return total;
}

template <class Load>
__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(Load load, int64_t n_max, const uint32_t* n_dev,
                                                              uint32_t* partial) {
    const int64_t n = valid_count(n_max, n_dev);
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    uint32_t s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; k++)
        if (base + k < n) s += load(base + k);
    uint32_t excl;
    uint32_t tot = block_exclusive_scan<kScanThreads>(s, excl);
    if (threadIdx.x == 0) partial[blockIdx.x] = tot;
}

// Single CTA: exclusive scan of nb block sums in place; total -> *total.
__global__ void __launch_bounds__(1024) k_scan_top(uint32_t* partial, int64_t nb, uint32_t* total) {
    const int64_t per = (nb + 1023) / 1024;
    const int64_t b0 = (int64_t)threadIdx.x * per;
    uint32_t s = 0;
    for (int64_t i = b0; i < b0 + per && i < nb; i++) s += partial[i];
    uint32_t excl;
    uint32_t tot = block_exclusive_scan<1024>(s, excl);
    uint32_t run = excl;
    for (int64_t i = b0; i < b0 + per && i < nb; i++) {
        uint32_t t = partial[i];
        partial[i] = run;
        run += t;
    }
    if (threadIdx.x == 0 && total) *total = tot;
}

template <class Load>
__global__ void __launch_bounds__(kScanThreads) k_scan_down(Load load, uint32_t* out, int64_t n_max,
                                                            const uint32_t* n_dev, const uint32_t* partial) {
    const int64_t n = valid_count(n_max, n_dev);
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    uint32_t s = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; k++) {
        v[k] = base + k < n ? load(base + k) : 0u;
        s += v[k];
    }
    uint32_t excl;
    block_exclusive_scan<kScanThreads>(s, excl);
    uint32_t run = excl + partial[blockIdx.x];
#pragma unroll
    for (int k = 0; k < kScanItems; k++) {
        if (base + k < n_max) out[base + k] = run;
        run += v[k];
    }
}

size_t scan_workspace_bytes(int64_t n_max) { return align256(sizeof(uint32_t) * (ceil_div(n_max, kScanTile) + 1)); }

template <class Load>
static void scan_exclusive(Load load, uint32_t* out, int64_t n_max, const uint32_t* n_dev, uint32_t* total, void* ws,
                           cudaStream_t s) {
    const int64_t nb = ceil_div(n_max, kScanTile);
    uint32_t* partial = (uint32_t*)ws;
    if (nb == 0) return;
    k_scan_reduce<<<(unsigned)nb, kScanThreads, 0, s>>>(load, n_max, n_dev, partial);
    count_launch();
    k_scan_top<<<1, 1024, 0, s>>>(partial, nb, total);
    count_launch();
    k_scan_down<<<(unsigned)nb, kScanThreads, 0, s>>>(load, out, n_max, n_dev, partial);
    count_launch();
}

void scan_exclusive_u32(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* total, void* ws, cudaStream_t s) {
    scan_exclusive(LoadU32{in}, out, n, nullptr, total, ws, s);
}

// ---------------------------------------------------------------------------
// LSD radix sort, 8-bit digits, stable.
//
// Each CTA owns 4096 consecutive keys. The histogram pass counts digits with
// shared-memory atomics into per-warp sub-histograms. The scatter pass ranks
// keys within each warp (peers by one ballot per digit bit, running per-warp digit
// counts in shared memory), turns warp counts into block-local digit offsets,
// places keys and values in shared memory in sorted order and then writes
// each digit's run to its global offset with consecutive threads on
// consecutive addresses.
// ---------------------------------------------------------------------------
constexpr int kRadixThreads = 256;
constexpr int kRadixWarps = kRadixThreads / 32;
constexpr int kRadixIters = 16;                                 // 32-key rounds per warp
constexpr int kRadixTile = kRadixThreads * kRadixIters;         // 4096 keys per CTA
constexpr int kRadixWarpSpan = 32 * kRadixIters;                // 512 keys per warp

int64_t radix_blocks(int64_t n_max) { return ceil_div(n_max, kRadixTile); }

// Per-CTA digit histogram, stored digit-major: hist[d * nb + block].
__global__ void __launch_bounds__(kRadixThreads) k_radix_hist(const uint32_t* __restrict__ keys, int64_t n_max,
                                                              const uint32_t* n_dev, int shift, uint32_t* hist,
                                                              int64_t nb) {
    __shared__ uint32_t h[kRadixWarps][256];
    const int w = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < kRadixWarps * 256; i += kRadixThreads) (&h[0][0])[i] = 0;
    __syncthreads();
    const int64_t n = valid_count(n_max, n_dev);
    const int64_t b0 = (int64_t)blockIdx.x * kRadixTile;
    if (b0 < n) {
        uint32_t k[kRadixIters];
#pragma unroll
        for (int it = 0; it < kRadixIters; it++) {
            const int64_t idx = b0 + it * kRadixThreads + threadIdx.x;
            k[it] = idx < n ? keys[idx] : 0u;
        }
#pragma unroll
        for (int it = 0; it < kRadixIters; it++)
            if (b0 + it * kRadixThreads + threadIdx.x < n) atomicAdd(&h[w][(k[it] >> shift) & 255u], 1u);
    }
    __syncthreads();
    uint32_t s = 0;
#pragma unroll
    for (int q = 0; q < kRadixWarps; q++) s += h[q][threadIdx.x];
    hist[(int64_t)threadIdx.x * nb + blockIdx.x] = s;
}

// vin == nullptr: the values are the keys' input positions (0, 1, 2, ...).
__global__ void __launch_bounds__(kRadixThreads, 3) k_radix_scatter(const uint32_t* __restrict__ kin,
                                                                 const uint32_t* __restrict__ vin,
                                                                 uint32_t* __restrict__ kout,
                                                                 uint32_t* __restrict__ vout, int64_t n_max,
                                                                 const uint32_t* n_dev, int shift,
                                                                 const uint32_t* __restrict__ hist, int64_t nb) {
    __shared__ uint32_t cnt[kRadixWarps][256];  // per-warp digit counts, then each warp's offset within the digit
    __shared__ uint32_t goff[256];              // global offset of this CTA's run of each digit
    __shared__ uint32_t dstart[256];            // block-local start of each digit
    __shared__ uint32_t s_k[kRadixTile];
    __shared__ uint32_t s_v[kRadixTile];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t n = valid_count(n_max, n_dev);
    const int64_t b0 = (int64_t)blockIdx.x * kRadixTile;
    if (b0 >= n) return;  // uniform over the CTA
    for (int i = threadIdx.x; i < kRadixWarps * 256; i += kRadixThreads) (&cnt[0][0])[i] = 0;
    goff[threadIdx.x] = hist[(int64_t)threadIdx.x * nb + blockIdx.x];
    __syncthreads();
    const int64_t base = b0 + (int64_t)w * kRadixWarpSpan;
    // this lane's keys are kin[base + lane + 32 it] for 32 it < rem
    const int64_t rem = n - base - lane;
    const uint32_t* kp = kin + base + lane;
    uint32_t kk[kRadixIters], rank[kRadixIters];  // values are loaded after ranking (fewer registers)
#pragma unroll
    for (int it = 0; it < kRadixIters; it++) kk[it] = 32 * it < rem ? kp[32 * it] : 0u;
#pragma unroll
    for (int it = 0; it < kRadixIters; it++) {
        const bool valid = 32 * it < rem;
        const unsigned d = valid ? (kk[it] >> shift) & 255u : 256u;
        // lanes holding the same digit: one ballot per bit of the 9-bit label
        // (256 marks a missing key), all in registers
        unsigned peers = 0xffffffffu;
#pragma unroll
        for (int b = 0; b < 9; b++) {
            const bool bit = (d >> b) & 1u;
            const unsigned bal = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? bal : ~bal;
        }
        const unsigned lower = peers & lanemask_lt();
        const uint32_t before = valid ? cnt[w][d] : 0u;
        __syncwarp();
        if (valid && lower == 0) cnt[w][d] = before + __popc(peers);
        __syncwarp();
        rank[it] = valid ? before + __popc(lower) : 0xFFFFFFFFu;
    }
    __syncthreads();
    uint32_t tot = 0;  // thread t handles digit t
#pragma unroll
    for (int q = 0; q < kRadixWarps; q++) {
        const uint32_t c = cnt[q][threadIdx.x];
        cnt[q][threadIdx.x] = tot;
        tot += c;
    }
    uint32_t ex;
    block_exclusive_scan<kRadixThreads>(tot, ex);
    dstart[threadIdx.x] = ex;
    __syncthreads();
    uint32_t vv[kRadixIters];
    const uint32_t* vp = vin ? vin + base + lane : nullptr;
#pragma unroll
    for (int it = 0; it < kRadixIters; it++)
        vv[it] = 32 * it < rem ? (vp ? vp[32 * it] : (uint32_t)(base + lane + 32 * it)) : 0u;
#pragma unroll
    for (int it = 0; it < kRadixIters; it++) {
        if (rank[it] != 0xFFFFFFFFu) {
            const unsigned d = (kk[it] >> shift) & 255u;
            const uint32_t pos = dstart[d] + cnt[w][d] + rank[it];
            s_k[pos] = kk[it];
            s_v[pos] = vv[it];
        }
    }
    __syncthreads();
    const int cnt_block = (int)min((int64_t)kRadixTile, n - b0);
    for (int i = threadIdx.x; i < cnt_block; i += kRadixThreads) {
        const uint32_t k = s_k[i];
        const unsigned d = (k >> shift) & 255u;
        const uint32_t dest = goff[d] + (uint32_t)i - dstart[d];
        if ((int64_t)dest < n) {  // always true for a consistent histogram; guards the scatter
            kout[dest] = k;
            vout[dest] = s_v[i];
        }
    }
}

bool radix_sort_pairs(uint32_t* ka, uint32_t* va, uint32_t* kb, uint32_t* vb, int64_t n_max, const uint32_t* n_dev,
                      int bits, uint32_t* hist, void* scan_ws, cudaStream_t s, bool va_is_position) {
    const int64_t nb = radix_blocks(n_max);
    bool in_b = false;
    if (nb == 0) return false;
    for (int shift = 0; shift < bits; shift += 8) {
        uint32_t* ki = in_b ? kb : ka;
        const uint32_t* vi = in_b ? vb : (va_is_position && shift == 0 ? nullptr : va);
        uint32_t* ko = in_b ? ka : kb;
        uint32_t* vo = in_b ? va : vb;
        k_radix_hist<<<(unsigned)nb, kRadixThreads, 0, s>>>(ki, n_max, n_dev, shift, hist, nb);
        count_launch();
        scan_exclusive(LoadU32{hist}, hist, 256 * nb, nullptr, nullptr, scan_ws, s);
        k_radix_scatter<<<(unsigned)nb, kRadixThreads, 0, s>>>(ki, vi, ko, vo, n_max, n_dev, shift, hist, nb);
        count_launch();
        in_b = !in_b;
    }
    return in_b;
}

// ---------------------------------------------------------------------------
// Single-pass scans and one-sweep radix passes with decoupled look-back (the
// scheme of Merrill & Garland's single-pass prefix scan and of Adinets &
// Merrill's Onesweep radix sort). CTAs take consecutive tiles of the input by
// ticket (an atomic counter), so every tile below a CTA's own belongs to a CTA
// that started earlier. Each CTA publishes its tile's aggregate at once, then
// walks back over the earlier tiles' words - adding aggregates until it meets
// an inclusive prefix - and publishes its own inclusive prefix. A CTA only
// ever waits for earlier tiles to publish their aggregate, which they do
// before waiting on anything, so the waits always end; each poll loop is
// still bounded (kSpinLimit polls), after which the CTA records
// GS_ERR_TIMEOUT in an error word and carries on with the prefix it has.
// Look-back words are 64-bit: flag in bits 62-63, a 32-bit count below.
// ---------------------------------------------------------------------------
constexpr uint64_t kLbAgg = 1ull << 62, kLbPre = 2ull << 62, kLbFlags = 3ull << 62;
constexpr int kSpinLimit = 1 << 22;
constexpr int kMaxPasses = 4;

__device__ __forceinline__ uint64_t lb_load(const uint64_t* p) {
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void lb_store(uint64_t* p, uint64_t v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Look-back words of a radix pass, per digit (256 of each kind in a row): one per
// tile, and two per group of kLbGroup tiles, the group's sum with the number of
// tiles that have added to it (atomicAdd) and the inclusive prefix at its end. At
// most kLbGroup - 1 tile words and the words of the groups in flight lie between a
// tile and the nearest prefix. A walk over single tiles has up to 608 words to add in a
// first wave of CTAs, at eight a round of L2 latency; the passes over 5.8M items
// took 70 us with it and 66 with groups.
constexpr int kLbGroup = 16;
constexpr int kLbGroupShift = 40;  // count of tiles in a group's sum
constexpr uint64_t kLbGroupFull = (uint64_t)kLbGroup << kLbGroupShift;

struct LbWords {
    uint64_t *tile, *sum, *pre;
};
__host__ __device__ __forceinline__ int64_t lb_groups(int64_t tiles) { return (tiles + kLbGroup - 1) / kLbGroup; }
__host__ __device__ __forceinline__ LbWords lb_words(uint64_t* w, int64_t tiles) {
    return {w, w + 256 * tiles, w + 256 * (tiles + lb_groups(tiles))};
}

// Zeroes the words that `tile` is the first to need (256 threads).
__device__ __forceinline__ void lb_zero(const LbWords& w, int64_t tile) {
    w.tile[tile * 256 + threadIdx.x] = 0;
    if (tile % kLbGroup == 0) {
        w.sum[tile / kLbGroup * 256 + threadIdx.x] = 0;
        w.pre[tile / kLbGroup * 256 + threadIdx.x] = 0;
    }
}

// Publishes this thread's digit count `tot` of the tile.
__device__ __forceinline__ void lb_publish(const LbWords& w, int64_t tile, uint32_t tot) {
    lb_store(w.tile + tile * 256 + threadIdx.x, kLbAgg | tot);
    atomicAdd((unsigned long long*)w.sum + tile / kLbGroup * 256 + threadIdx.x, (1ull << kLbGroupShift) | tot);
}

// The exclusive prefix of this thread's digit at `tile`; the last tile of a group
// publishes the group's inclusive prefix.
constexpr int kLbWin = 4;
__device__ __forceinline__ uint32_t look_back(const LbWords& w, int64_t tile, uint32_t tot, int32_t* err) {
    const int64_t g = tile / kLbGroup;
    uint32_t excl = 0;
    int spins = 0;
    for (int64_t j = g - 1; j >= 0;) {  // groups before this one
        uint64_t p[kLbWin], v[kLbWin];
#pragma unroll
        for (int q = 0; q < kLbWin; q++) {
            p[q] = j - q >= 0 ? lb_load(w.pre + (j - q) * 256 + threadIdx.x) : kLbPre;
            v[q] = j - q >= 0 ? lb_load(w.sum + (j - q) * 256 + threadIdx.x) : 0;
        }
        int used = 0;
        bool found = false, open = false;
#pragma unroll
        for (int q = 0; q < kLbWin; q++) {
            if (found || open) continue;
            if (p[q] & kLbPre) {
                excl += (uint32_t)p[q];
                found = true;
            } else if (v[q] >= kLbGroupFull) {
                excl += (uint32_t)v[q];
                used++;
            } else {
                open = true;  // not all of its tiles have published; read it again
            }
        }
        if (found) break;
        j -= used;
        if (open && ++spins > kSpinLimit) {
            if (err) atomicExch(err, GS_ERR_TIMEOUT);
            return excl;
        }
    }
    for (int64_t j = g * kLbGroup; j < tile;) {  // tiles of the group
        uint64_t v[kLbWin];
#pragma unroll
        for (int q = 0; q < kLbWin; q++) v[q] = j + q < tile ? lb_load(w.tile + (j + q) * 256 + threadIdx.x) : 0;
        bool open = false;
        int used = 0;
#pragma unroll
        for (int q = 0; q < kLbWin; q++) {
            if (open || j + q >= tile) continue;
            if (v[q] & kLbAgg) {
                excl += (uint32_t)v[q];
                used++;
            } else {
                open = true;
            }
        }
        j += used;
        if (open && ++spins > kSpinLimit) {
            if (err) atomicExch(err, GS_ERR_TIMEOUT);
            return excl;
        }
    }
    if (tile % kLbGroup == kLbGroup - 1) lb_store(w.pre + g * 256 + threadIdx.x, kLbPre | (uint32_t)(excl + tot));
    return excl;
}

// Exclusive prefix of tile `tile` in one row of words, by a whole CTA of NT threads:
// thread t reads the word of tile
// j - t, so each round covers NT earlier tiles (the walk back from a tile is
// about as long as the number of CTAs in flight, so it must cover many tiles
// per round). Called by every thread; returns the prefix in every thread.
template <int NT>
__device__ __forceinline__ uint32_t look_back_cta(const uint64_t* words, int64_t tile, int32_t* err) {
    constexpr int NW = NT / 32;
    __shared__ unsigned s_min[NW];
    __shared__ uint32_t s_sum[NW];
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t excl = 0;
    int64_t j = tile - 1;
    int spins = 0;
    while (j >= 0) {  // uniform over the CTA
        const int64_t jj = j - threadIdx.x;
        const uint64_t v = jj >= 0 ? lb_load(words + jj) : kLbPre;  // before tile 0: an empty prefix
        // nearest inclusive prefix among the NT words
        const unsigned wm = __reduce_min_sync(FULL, (v & kLbPre) ? (unsigned)threadIdx.x : (unsigned)NT);
        if (lane == 0) s_min[w] = wm;
        __syncthreads();
        unsigned first = NT;
#pragma unroll
        for (int q = 0; q < NW; q++) first = min(first, s_min[q]);
        const bool need = (unsigned)threadIdx.x <= first;
        if (__syncthreads_or(need && (v & kLbFlags) == 0)) {  // a needed tile is not published yet
            if (++spins > kSpinLimit) {
                if (err && threadIdx.x == 0) atomicExch(err, GS_ERR_TIMEOUT);
                break;
            }
            continue;
        }
        const uint32_t ws = __reduce_add_sync(FULL, need ? (uint32_t)v : 0u);
        if (lane == 0) s_sum[w] = ws;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NW; q++) excl += s_sum[q];
        __syncthreads();  // s_min / s_sum are rewritten by the next round
        if (first < (unsigned)NT) break;
        j -= NT;
    }
    return excl;
}

// Control words of one single-pass scan or one radix sort, zeroed by the
// caller before the first kernel that uses them.
struct ScanCtl {
    uint32_t ticket;
};
struct SortCtl {
    uint32_t count[kMaxPasses][256];  // digit counts of every pass, then their exclusive sums
    uint32_t ticket[kMaxPasses];
    uint32_t hist_done;
};

// A load that stays where it is written: the compiler sinks plain loads to
// their uses, one latency each.
__device__ __forceinline__ uint32_t load_now(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint2 load_now2(const uint2* p) {
    uint2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}

// Exclusive scan of load(0..n-1) into out[0..n), total -> *total. Each CTA
// takes one contiguous chunk: it sums the chunk, publishes the sum, looks
// back over the earlier chunks (all CTAs of the grid run at once, so the walk
// covers at most a round or two of the CTA-wide window), then scans the chunk
// tile by tile (its second read mostly hits L2).
template <class Load>
__global__ void __launch_bounds__(kScanThreads) k_scan_single(Load load, uint32_t* __restrict__ out, int64_t n,
                                                              int64_t chunk, ScanCtl* ctl, uint64_t* words, uint32_t* total,
                                                              int32_t* err) {
    // each tile passes through shared memory so that global loads and stores
    // are coalesced while each thread scans 8 consecutive values (one padding
    // word per 32 keeps the per-thread reads free of bank conflicts)
    __shared__ uint32_t s_v[kScanTile + kScanTile / 32];
    __shared__ uint32_t s_tile;
    if (threadIdx.x == 0) s_tile = atomicAdd(&ctl->ticket, 1u);
    __syncthreads();
    const int64_t c = s_tile;
    const int64_t c0 = c * chunk;
    if (c0 >= n) return;  // uniform over the CTA
    const int64_t c1 = min(c0 + chunk, n);
    uint32_t sum = 0;
#pragma unroll 2
    for (int64_t i0 = c0; i0 < c1; i0 += kScanTile) {
        uint32_t part[kScanItems];
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            const int64_t i = i0 + k * kScanThreads + threadIdx.x;
            part[k] = i < c1 ? load(i) : 0u;
        }
#pragma unroll
        for (int k = 0; k < kScanItems; k++) sum += part[k];
    }
    uint32_t unused;
    const uint32_t agg = block_exclusive_scan<kScanThreads>(sum, unused);
    uint64_t* mine = words + c;
    uint32_t run = 0;
    if (c == 0) {
        if (threadIdx.x == 0) lb_store(mine, kLbPre | agg);
    } else {
        if (threadIdx.x == 0) lb_store(mine, kLbAgg | agg);
        run = look_back_cta<kScanThreads>(words, c, err);
        if (threadIdx.x == 0) lb_store(mine, kLbPre | (uint32_t)(run + agg));
    }
    if (threadIdx.x == 0 && total && c1 >= n) *total = run + agg;
    for (int64_t t0 = c0; t0 < c1; t0 += kScanTile) {
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            const int i = k * kScanThreads + threadIdx.x;
            s_v[i + (i >> 5)] = t0 + i < c1 ? load(t0 + i) : 0u;
        }
        __syncthreads();
        uint32_t v[kScanItems];
        uint32_t tsum = 0;
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            const int i = threadIdx.x * kScanItems + k;
            v[k] = s_v[i + (i >> 5)];
            tsum += v[k];
        }
        uint32_t excl;
        const uint32_t tagg = block_exclusive_scan<kScanThreads>(tsum, excl);
        uint32_t r = run + excl;
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            const int i = threadIdx.x * kScanItems + k;
            s_v[i + (i >> 5)] = r;
            r += v[k];
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            const int i = k * kScanThreads + threadIdx.x;
            if (t0 + i < c1) out[t0 + i] = s_v[i + (i >> 5)];
        }
        run += tagg;
        __syncthreads();  // s_v is rewritten by the next tile
    }
}

// CTAs of the single-pass scan: four per SM (each CTA's two walks over its
// chunk are latency-bound, so shorter chunks finish sooner), each with one
// chunk of whole tiles.
static int64_t scan_ctas() {
    static int sms = 0;
    if (sms == 0) {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        sms = v > 0 ? v : 152;
    }
    return 4 * (int64_t)sms;
}

template <class Load>
static void scan_single(Load load, uint32_t* out, int64_t n, uint32_t* total, ScanCtl* ctl, uint64_t* words,
                        int32_t* err, cudaStream_t s) {
    const int64_t tiles = ceil_div(n, kScanTile);
    if (tiles == 0) return;
    const int64_t g = tiles < scan_ctas() ? tiles : scan_ctas();
    const int64_t chunk = ceil_div(tiles, g) * kScanTile;
    k_scan_single<<<(unsigned)ceil_div(n, chunk), kScanThreads, 0, s>>>(load, out, n, chunk, ctl, words, total, err);
    count_launch();
}

struct LoadPopcount {
    const uint32_t* words;
    __device__ uint32_t operator()(int64_t i) const { return (uint32_t)__popc(words[i]); }
};

size_t scan_popcounts_words(int64_t n) { return 64 + 2 * ceil_div(n, kScanTile); }

int32_t* scan_popcounts(const uint32_t* words, uint32_t* out, int64_t n, uint32_t* total, uint32_t* ws, cudaStream_t s) {
    int32_t* err = (int32_t*)ws + 32;
    scan_single(LoadPopcount{words}, out, n, total, (ScanCtl*)ws, (uint64_t*)(ws + 64), err, s);
    return err;
}

// Digit counts of every pass of a radix sort, gathered by the kernel that writes the
// keys in s_h and added up over its CTAs; the last of n_ctas to add turns the sums
// into each digit's global start. 256 threads.
__device__ __forceinline__ void add_digit_counts(const uint32_t (*s_h)[256], int passes, SortCtl* ctl, int64_t n_ctas) {
    __shared__ bool s_last;
    __syncthreads();
    for (int p = 0; p < passes; p++) {
        const uint32_t c = s_h[p][threadIdx.x];
        if (c) atomicAdd(&ctl->count[p][threadIdx.x], c);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&ctl->hist_done, 1u) == (uint32_t)(n_ctas - 1);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (int p = 0; p < passes; p++) {
        const uint32_t c = atomicAdd(&ctl->count[p][threadIdx.x], 0u);  // read past L1
        uint32_t ex;
        block_exclusive_scan<256>(c, ex);
        ctl->count[p][threadIdx.x] = ex;
    }
}

// Keys per CTA of a pass over at most n_max keys: 16 rounds of 32 per warp, or 8 where
// even those tiles are about one round of the resident CTAs (three per SM), and a
// pass takes as long as one tile does (the sort of 150K items and 410K pairs: 86 us
// against 96; of 1M and 2M, where only the items' passes take it: 148 against 150).
constexpr int64_t kFewKeys = 1 << 20;
static int onesweep_tile(int64_t n_max) { return n_max <= kFewKeys ? kRadixTile / 2 : kRadixTile; }
static int64_t onesweep_blocks(int64_t n_max) { return ceil_div(n_max, onesweep_tile(n_max)); }

// Digit counts of given keys, and the first pass's look-back words zeroed; a CTA counts
// two of the passes' smaller tiles.
__global__ void __launch_bounds__(256) k_onesweep_hist(const uint32_t* __restrict__ keys, int64_t n, int passes,
                                                       SortCtl* ctl, LbWords words, int64_t blocks) {
    __shared__ uint32_t s_h[kMaxPasses][256];
    for (int i = threadIdx.x; i < kMaxPasses * 256; i += 256) (&s_h[0][0])[i] = 0;
    __syncthreads();
    const int64_t t0 = (int64_t)blockIdx.x * kRadixTile;
    uint32_t k[kRadixIters];
#pragma unroll
    for (int it = 0; it < kRadixIters; it++) {
        const int64_t i = t0 + it * 256 + threadIdx.x;
        k[it] = i < n ? keys[i] : 0u;
    }
#pragma unroll
    for (int it = 0; it < kRadixIters; it++)
        if (t0 + it * 256 + threadIdx.x < n)
            for (int p = 0; p < passes; p++) atomicAdd(&s_h[p][(k[it] >> (8 * p)) & 255u], 1u);
    for (int64_t b = blockIdx.x; b < blocks; b += gridDim.x) lb_zero(words, b);
    add_digit_counts(s_h, passes, ctl, gridDim.x);
}

// 16 bytes to shared memory, of which the first `bytes` are read.
__device__ __forceinline__ void cp_async16(void* dst, const void* src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One 8-bit digit pass; values of type V travel with the keys. With out_x / out_y set
// (V = uint2), the last pass writes the two halves of each value to separate arrays.
// words: this pass's look-back words; next: the next pass's, zeroed here for this
// tile (or null).
// Bound by the latency of its stages (ticket, load, rank, scan, look back, write: 27,000
// cycles a tile, three or four tiles per SM at a time) and by shared memory: the values come in by asynchronous copies while the keys are ranked (peers of a key
// by an OR of lane bits per digit: 13 instructions a round, 50 by nine ballots, and
// match.any was slower than both), and the sorted order fetches them from shared
// memory. 5.8M items: 45 us a pass (70 before), 15.8M pairs: 115 (166).
template <class V, int ITERS>
__global__ void __launch_bounds__(kRadixThreads, 3) k_onesweep_pass(
    const uint32_t* __restrict__ kin, const V* __restrict__ vin, uint32_t* __restrict__ kout, V* __restrict__ vout,
    uint32_t* __restrict__ out_x, uint32_t* __restrict__ out_y, int64_t n_max, const uint32_t* n_dev, int pass,
    SortCtl* ctl, LbWords words, LbWords next, int32_t* err) {
    constexpr int kTile = kRadixThreads * ITERS, kSpan = 32 * ITERS;  // keys per CTA and per warp
    __shared__ uint16_t cnt[kRadixWarps][256];  // keys so far per warp and digit, then the warp's first place in the tile
    __shared__ uint32_t goff[256];              // global minus tile-local start of each digit
    __shared__ uint32_t s_k[kTile];        // the sorted tile's keys
    __shared__ uint16_t s_i[kTile];        // and their places in the input
    __shared__ __align__(16) V s_v[kTile];  // the input's values
    __shared__ uint32_t s_tile;
    // while ranking: lanes whose key of this round has the digit, per warp
    uint32_t(*mask)[256] = reinterpret_cast<uint32_t(*)[256]>(s_k);
    static_assert(kTile >= kRadixWarps * 256);
    const int shift = 8 * pass;
    if (threadIdx.x == 0) s_tile = atomicAdd(&ctl->ticket[pass], 1u);
    for (int i = threadIdx.x; i < kRadixWarps * 256; i += kRadixThreads) {
        (&cnt[0][0])[i] = 0;
        (&mask[0][0])[i] = 0;
    }
    __syncthreads();
    const int64_t tile = s_tile;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t n = valid_count(n_max, n_dev);
    const int64_t b0 = tile * kTile;
    if (b0 >= n) return;  // uniform over the CTA
    if (next.tile) lb_zero(next, tile);
    const int64_t base = b0 + (int64_t)w * kSpan;
    const int rem = (int)min(n - base, (int64_t)kSpan) - lane;
    const uint32_t* kp = kin + base + lane;
    const int cnt_block = (int)min((int64_t)kTile, n - b0);
    // the values travel to shared memory while the keys are ranked
    constexpr int kPer = 16 / (int)sizeof(V);
#pragma unroll
    for (int i = threadIdx.x * kPer; i < kTile; i += kRadixThreads * kPer)
        if (i < cnt_block) cp_async16(s_v + i, vin + b0 + i, min((cnt_block - i) * (int)sizeof(V), 16));
    uint32_t kk[ITERS], rank[ITERS];
#pragma unroll
    for (int it = 0; it < ITERS; it++) kk[it] = 32 * it < rem ? load_now(kp + 32 * it) : 0u;
#pragma unroll
    for (int it = 0; it < ITERS; it++) {
        const bool valid = 32 * it < rem;
        const unsigned d = (kk[it] >> shift) & 255u;
        if (valid) atomicOr(&mask[w][d], 1u << lane);
        __syncwarp();
        const uint32_t m = mask[w][d], before = cnt[w][d];
        __syncwarp();
        const unsigned lower = m & lanemask_lt();
        if (valid && lower == 0) {
            mask[w][d] = 0;
            cnt[w][d] = (uint16_t)(before + __popc(m));
        }
        __syncwarp();
        rank[it] = before + __popc(lower);
    }
    __syncthreads();
    uint32_t tot = 0;  // thread t handles digit t
#pragma unroll
    for (int q = 0; q < kRadixWarps; q++) tot += cnt[q][threadIdx.x];
    lb_publish(words, tile, tot);
    uint32_t ex;
    block_exclusive_scan<kRadixThreads>(tot, ex);
    uint32_t place = ex;
#pragma unroll
    for (int q = 0; q < kRadixWarps; q++) {
        const uint32_t c = cnt[q][threadIdx.x];
        cnt[q][threadIdx.x] = (uint16_t)place;
        place += c;
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < ITERS; it++) {
        if (32 * it < rem) {
            const uint32_t pos = cnt[w][(kk[it] >> shift) & 255u] + rank[it];
            s_k[pos] = kk[it];
            s_i[pos] = (uint16_t)(w * kSpan + lane + 32 * it);
        }
    }
    goff[threadIdx.x] = ctl->count[pass][threadIdx.x] + look_back(words, tile, tot, err) - ex;
    cp_async_wait();
    __syncthreads();
#pragma unroll 4
    for (int i = threadIdx.x; i < cnt_block; i += kRadixThreads) {
        const uint32_t k = s_k[i];
        const V v = s_v[s_i[i]];
        const uint32_t dest = goff[(k >> shift) & 255u] + (uint32_t)i;
        if ((int64_t)dest < n) {  // always true for consistent counts; guards the scatter after a timeout
            kout[dest] = k;
            if constexpr (sizeof(V) == 8) {
                if (out_x) {
                    out_x[dest] = v.x;
                    out_y[dest] = v.y;
                    continue;
                }
            }
            vout[dest] = v;
        }
    }
}

// Look-back words that a radix pass over n_max keys or fewer needs at most: the tiles
// halve at kFewKeys, so that many keys have more of them than somewhat more keys do, and
// a workspace sized for the largest sort of several has to hold the others too.
static int64_t onesweep_words(int64_t n_max) {
    const int64_t few = onesweep_blocks(n_max < kFewKeys ? n_max : kFewKeys), all = onesweep_blocks(n_max);
    const int64_t tiles = few > all ? few : all;
    return 256 * (tiles + 2 * lb_groups(tiles));
}

// Stable LSD sort of (key, value) pairs on key bits [0, bits), one launch per 8 of
// them; ctl->count holds the digits' starts and the words of wa that the tiles need
// are zero (k_onesweep_hist, or the kernel that wrote the keys). (ka, va) hold the
// input, (kb, vb) are the alternates. With out_x set (V = uint2), the last pass
// writes the values' two halves to out_x / out_y instead of va / vb. Returns true
// when the sorted keys (and values, unless split) end in (kb, vb). wa / wb:
// onesweep_words(n_max) words each.
template <class V>
static bool onesweep_passes(uint32_t* ka, V* va, uint32_t* kb, V* vb, int64_t n_max, const uint32_t* n_dev, int bits,
                            SortCtl* ctl, uint64_t* wa, uint64_t* wb, int32_t* err, cudaStream_t s,
                            uint32_t* out_x = nullptr, uint32_t* out_y = nullptr) {
    const int64_t nb = onesweep_blocks(n_max);
    const auto kernel = onesweep_tile(n_max) == kRadixTile ? k_onesweep_pass<V, kRadixIters>
                                                           : k_onesweep_pass<V, kRadixIters / 2>;
    const int passes = (bits + 7) / 8;
    bool in_b = false;
    for (int p = 0; p < passes; p++) {
        const bool last = p + 1 == passes;
        const LbWords w = lb_words((p & 1) ? wb : wa, nb);
        const LbWords wn = last ? LbWords{} : lb_words((p & 1) ? wa : wb, nb);
        kernel<<<(unsigned)nb, kRadixThreads, 0, s>>>(
            in_b ? kb : ka, in_b ? vb : va, in_b ? ka : kb, in_b ? va : vb, last ? out_x : nullptr,
            last ? out_y : nullptr, n_max, n_dev, p, ctl, w, wn, err);
        count_launch();
        in_b = !in_b;
    }
    return in_b;
}

// ---------------------------------------------------------------------------
// gs_sort stages
// ---------------------------------------------------------------------------
// count[0] = number of pairs; n_eff = min(count, capacity); status (a
// look-back timeout recorded in *err so far takes precedence)
__device__ __forceinline__ void pair_count(uint32_t t, int64_t capacity, int64_t* count, uint32_t* n_eff,
                                           int32_t* status, const int32_t* err) {
    const int32_t e = atomicAdd((int32_t*)err, 0);
    *count = t;
    *n_eff = (uint32_t)min((int64_t)t, capacity);
    *status = e ? e : (int64_t)t > capacity ? GS_ERR_CAPACITY : GS_OK;
}
__global__ void k_no_pairs(int64_t* count, int32_t* status) {
    *count = 0;
    *status = GS_OK;
}

// The two prefixes of a chunk in the words of a scan of pairs, as look_back_cta.
template <int NT>
__device__ __forceinline__ uint2 look_back_cta2(const uint64_t* wa, const uint64_t* wb, int64_t tile, int32_t* err) {
    constexpr int NW = NT / 32;
    __shared__ unsigned s_min[NW];
    __shared__ uint2 s_sum[NW];
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint2 excl = make_uint2(0, 0);
    int64_t j = tile - 1;
    int spins = 0;
    while (j >= 0) {  // uniform over the CTA
        const int64_t jj = j - threadIdx.x;
        const uint64_t a = jj >= 0 ? lb_load(wa + jj) : kLbPre;
        const uint64_t b = jj >= 0 ? lb_load(wb + jj) : kLbPre;
        const unsigned wm = __reduce_min_sync(FULL, (a & b & kLbPre) ? (unsigned)threadIdx.x : (unsigned)NT);
        if (lane == 0) s_min[w] = wm;
        __syncthreads();
        unsigned first = NT;
#pragma unroll
        for (int q = 0; q < NW; q++) first = min(first, s_min[q]);
        const bool need = (unsigned)threadIdx.x <= first;
        // behind the first pair of prefixes, the two words must be of one kind: a sum and a
        // prefix are read again
        const bool open = need && ((a & kLbFlags) == 0 || (a & kLbFlags) != (b & kLbFlags));
        if (__syncthreads_or(open)) {
            if (++spins > kSpinLimit) {
                if (err && threadIdx.x == 0) atomicExch(err, GS_ERR_TIMEOUT);
                break;
            }
            continue;
        }
        const uint32_t sa = __reduce_add_sync(FULL, need ? (uint32_t)a : 0u);
        const uint32_t sb = __reduce_add_sync(FULL, need ? (uint32_t)b : 0u);
        if (lane == 0) s_sum[w] = make_uint2(sa, sb);
        __syncthreads();
#pragma unroll
        for (int q = 0; q < NW; q++) {
            excl.x += s_sum[q].x;
            excl.y += s_sum[q].y;
        }
        __syncthreads();  // s_min / s_sum are rewritten by the next round
        if (first < (unsigned)NT) break;
        j -= NT;
    }
    return excl;
}

// Everything the depth sort needs of the items, in one launch: each item's first pair
// slot (exclusive sum of n_tiles in item order: each item's pairs occupy offset[item]
// .. offset[item] + n_tiles - 1, so that the adjoint's per-item runs of the Gaussians
// of one view are adjacent), the visible items with their depth keys in item order,
// their count, the keys' digit counts, the zeroed words of the sort's first pass and
// empty tile ranges.
// Chunks and look-back as in k_scan_single, with a word for each of the two sums.
// SINGLE: a chunk is one tile of 2048 items, read and scanned once.
// 8M items: 77 us against 72 + 32 + 19 for two scans and a histogram of the keys; the
// depths' 16-byte stride alone reads 128 MB.
template <bool SINGLE>
__global__ void __launch_bounds__(kScanThreads) k_scan_items(const int32_t* __restrict__ n_tiles,
                                                             const float4* __restrict__ rgb_depth, int64_t n,
                                                             int64_t chunk, uint32_t* __restrict__ offset,
                                                             uint32_t* __restrict__ key, uint32_t* __restrict__ val,
                                                             uint32_t* __restrict__ n_vis, ScanCtl* ctl,
                                                             uint64_t* words_v, uint64_t* words_t, SortCtl* sort,
                                                             LbWords sort_words, int64_t sort_tiles,
                                                             uint32_t* __restrict__ range, int64_t n_range,
                                                             int32_t* err) {
    constexpr int kPad = kScanTile + kScanTile / 32;
    __shared__ uint32_t s_t[kPad];  // tiles of each item, then its first slot
    __shared__ uint32_t s_v[kPad];  // visible items before it
    __shared__ uint32_t s_h[kMaxPasses][256];
    __shared__ uint32_t s_tile;
    if (threadIdx.x == 0) s_tile = atomicAdd(&ctl->ticket, 1u);
    for (int p = 0; p < kMaxPasses; p++) s_h[p][threadIdx.x] = 0;
    for (int64_t t = blockIdx.x; t < sort_tiles; t += gridDim.x) lb_zero(sort_words, t);
    for (int64_t i = (int64_t)blockIdx.x * kScanThreads + threadIdx.x; i < n_range; i += (int64_t)gridDim.x * kScanThreads)
        range[i] = 0;
    __syncthreads();
    const int64_t c = s_tile, c0 = c * chunk, c1 = min(c0 + chunk, n);  // c < gridDim.x = chunks
    uint32_t agg_v = 0, agg_t = 0;
    uint2 run = make_uint2(0, 0);
    auto look = [&]() {  // publishes the chunk's sums and finds those of the chunks before it
        if (threadIdx.x == 0) {
            lb_store(words_v + c, (c == 0 ? kLbPre : kLbAgg) | agg_v);
            lb_store(words_t + c, (c == 0 ? kLbPre : kLbAgg) | agg_t);
        }
        if (c > 0) {
            run = look_back_cta2<kScanThreads>(words_v, words_t, c, err);
            if (threadIdx.x == 0) {
                lb_store(words_v + c, kLbPre | (uint32_t)(run.x + agg_v));
                lb_store(words_t + c, kLbPre | (uint32_t)(run.y + agg_t));
            }
        }
        if (threadIdx.x == 0 && c1 >= n) *n_vis = run.x + agg_v;
    };
    if constexpr (!SINGLE) {
        uint32_t vis = 0, sum = 0;
        for (int64_t i0 = c0; i0 < c1; i0 += kScanTile) {
            int32_t t[kScanItems];
#pragma unroll
            for (int k = 0; k < kScanItems; k++) {
                const int64_t i = i0 + k * kScanThreads + threadIdx.x;
                t[k] = i < c1 ? (int32_t)load_now((const uint32_t*)n_tiles + i) : 0;
            }
#pragma unroll
            for (int k = 0; k < kScanItems; k++) {
                vis += t[k] > 0;
                sum += max(t[k], 0);
            }
        }
        uint32_t unused;
        agg_v = block_exclusive_scan<kScanThreads>(vis, unused);
        agg_t = block_exclusive_scan<kScanThreads>(sum, unused);
        look();
    }
    for (int64_t t0 = c0; t0 < c1; t0 += kScanTile) {
        uint32_t vis_bits = 0;
        uint32_t own[kScanItems];  // tiles of the items this thread writes out, then their depth bits
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            const int i = k * kScanThreads + threadIdx.x;
            own[k] = t0 + i < c1 ? load_now((const uint32_t*)n_tiles + t0 + i) : 0u;
        }
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            const int i = k * kScanThreads + threadIdx.x;
            s_t[i + (i >> 5)] = (uint32_t)max((int)own[k], 0);
            if ((int)own[k] > 0) vis_bits |= 1u << k;
            // depth > near_z > 0: the bits are monotone
            own[k] = (int)own[k] > 0 ? load_now((const uint32_t*)(rgb_depth + t0 + i) + 3) : 0u;
        }
        __syncthreads();
        uint32_t t[kScanItems], tv = 0, tt = 0;
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            const int i = threadIdx.x * kScanItems + k;
            t[k] = s_t[i + (i >> 5)];
            tv += t[k] > 0;
            tt += t[k];
        }
        uint32_t rv, rt;
        const uint32_t gv = block_exclusive_scan<kScanThreads>(tv, rv);
        const uint32_t gt = block_exclusive_scan<kScanThreads>(tt, rt);
        if constexpr (SINGLE) {
            agg_v = gv;
            agg_t = gt;
            look();
        }
        rv += run.x;
        rt += run.y;
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            const int i = threadIdx.x * kScanItems + k;
            s_t[i + (i >> 5)] = rt;
            s_v[i + (i >> 5)] = rv;
            rt += t[k];
            rv += t[k] > 0;
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kScanItems; k++) {
            const int i = k * kScanThreads + threadIdx.x;
            if (t0 + i >= c1) continue;
            const uint32_t pos = s_v[i + (i >> 5)];
            offset[t0 + i] = s_t[i + (i >> 5)];
            if (vis_bits >> k & 1) {
                const uint32_t d = own[k];
                key[pos] = d;
                val[pos] = (uint32_t)(t0 + i);
#pragma unroll
                for (int p = 0; p < kMaxPasses; p++) atomicAdd(&s_h[p][(d >> (8 * p)) & 255u], 1u);
            }
        }
        run.x += gv;
        run.y += gt;
        __syncthreads();  // s_t and s_v are rewritten by the next tile
    }
    add_digit_counts(s_h, kMaxPasses, sort, gridDim.x);
}

// Pairs are laid out in depth order (what the stable tile sort needs): one per tile of
// each visible item's rect, item after item. k_pair_positions finds where the pairs of
// every 32 sorted items begin, and k_duplicate writes them.
// item / n by a multiplication: with magic = floor(2^32 / n) the estimate is at most one low.
__device__ __forceinline__ uint32_t view_magic(uint32_t n) {
    return n > 1 ? (uint32_t)(0x100000000ull / n) : 0xFFFFFFFFu;
}
__device__ __forceinline__ uint32_t view_of(uint32_t item, uint32_t n, uint32_t magic) {
    const uint32_t v = __umulhi(item, magic);
    return v + (item - v * n >= n);
}

struct ItemRect {
    uint32_t x0, y0, wx, cnt, tx, base;
};
__device__ __forceinline__ ItemRect item_rect(const ushort4 r, const gs_frame& f, uint32_t v) {
    ItemRect q;
    q.tx = (uint32_t)f.tiles_x[v];
    q.base = (uint32_t)f.tile_base[v];
    const uint32_t ty = (uint32_t)f.tiles_y[v];
    // rect is clamped to the view's grid by gs_project; re-clamp so foreign input cannot index past it
    q.x0 = min((uint32_t)r.x, q.tx);
    const uint32_t x1 = max(min((uint32_t)r.z, q.tx), q.x0);
    q.y0 = min((uint32_t)r.y, ty);
    const uint32_t y1 = max(min((uint32_t)r.w, ty), q.y0);
    q.wx = max(x1 - q.x0, 1u);
    q.cnt = (x1 - q.x0) * (y1 - q.y0);
    return q;
}

// A CTA takes one contiguous chunk of the sorted items, an eighth per warp: it counts
// their pairs, finds its first position by look-back (all CTAs run at once) and
// writes the first position of each group of 32 items, and for every kDupPairs
// positions the group that holds the first of them; the last CTA the pair count.
// 5.8M items: 48 us, bound by the gather of their rects (86 for a scan that
// gathered twice and wrote a word per item).
constexpr int kDupThreads = 256;
constexpr int kDupPairs = 1024;  // the span that a CTA of k_duplicate writes is a multiple of it

__global__ void __launch_bounds__(kDupThreads) k_pair_positions(
    const uint32_t* __restrict__ sorted_item, const uint32_t* n_vis, const ushort4* __restrict__ rect, int64_t n,
    const __grid_constant__ gs_frame f, int64_t capacity, uint32_t* __restrict__ group_off,
    uint32_t* __restrict__ first_group, ScanCtl* ctl, uint64_t* words, int64_t* count, uint32_t* n_eff, int32_t* status,
    int32_t* err) {
    const unsigned FULL = 0xffffffffu;
    __shared__ uint32_t s_tile;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_tile = atomicAdd(&ctl->ticket, 1u);
    __syncthreads();
    const int64_t c = s_tile, nv = *n_vis;
    const int64_t per_warp = (((nv + gridDim.x - 1) / gridDim.x + kDupThreads - 1) / kDupThreads) * 32;
    const int64_t i0 = min((c * (kDupThreads / 32) + warp) * per_warp, nv), i1 = min(i0 + per_warp, nv);
    const uint32_t n32 = (uint32_t)n, magic = view_magic(n32);  // item < 2^32 (checked by gs_sort)
    constexpr int U = 8;                                        // items in flight per lane
    uint32_t sum = 0;
    for (int64_t i = i0 + lane; i - lane < i1; i += 32 * U) {
        uint32_t it[U];
        ushort4 r[U];
#pragma unroll
        for (int q = 0; q < U; q++) it[q] = i + 32 * q < i1 ? load_now(sorted_item + i + 32 * q) : 0u;
#pragma unroll
        for (int q = 0; q < U; q++) {
            const uint2 v = load_now2((const uint2*)rect + it[q]);
            r[q] = make_ushort4(v.x & 0xFFFFu, v.x >> 16, v.y & 0xFFFFu, v.y >> 16);
        }
        uint32_t mine = 0;  // lane q: the position of group q within the warp's pairs
#pragma unroll
        for (int q = 0; q < U; q++) {
            if (lane == q) mine = sum;
            sum += __reduce_add_sync(FULL, i + 32 * q < i1 ? item_rect(r[q], f, view_of(it[q], n32, magic)).cnt : 0u);
        }
        if (lane < U && i - lane + 32 * lane < i1) group_off[(i - lane) / 32 + lane] = mine;
    }
    uint32_t base;
    const uint32_t agg = block_exclusive_scan<kDupThreads>(lane == 0 ? sum : 0u, base);
    base = __shfl_sync(FULL, base, 0);
    uint32_t run = 0;
    if (threadIdx.x == 0) lb_store(words + c, (c == 0 ? kLbPre : kLbAgg) | agg);
    if (c > 0) {
        run = look_back_cta<kDupThreads>(words, c, err);
        if (threadIdx.x == 0) lb_store(words + c, kLbPre | (uint32_t)(run + agg));
    }
    if (threadIdx.x == 0 && c == gridDim.x - 1) pair_count(run + agg, capacity, count, n_eff, status, err);
    base += run;
    __syncwarp();
    const int64_t g0 = i0 / 32, g1 = (i1 + 31) / 32;  // i0 is a multiple of 32, or nv
    for (int64_t g = g0 + lane; i0 < i1 && g - lane < g1; g += 32) {
        const bool in = g < g1;
        const uint32_t off = in ? base + group_off[g] : 0u;
        const uint32_t end = in ? (g + 1 < g1 ? base + group_off[g + 1] : base + sum) : 0u;
        __syncwarp();  // a lane's neighbour reads its word before it is replaced
        if (!in) continue;
        group_off[g] = off;
        for (int64_t r = ((int64_t)off + kDupPairs - 1) / kDupPairs; r * kDupPairs < min((int64_t)end, capacity); r++)
            first_group[r] = (uint32_t)g;
    }
}

// Writes the pairs, one contiguous span of positions per CTA (rects differ too much in
// size for spans of items): each pair's tile, its item and its emission slot (the item's first slot, offset, plus the pair's index
// in the item). Also counts the tiles' digits and zeroes the words that the pair sort's
// first pass needs. A warp takes 32 consecutive items and writes their pairs together,
// consecutive lanes consecutive positions whatever the rect sizes. 15.8M pairs: 139 us
// with the digit counts (125 + 29 for a warp per group in grid order, and a histogram);
// about 170 instructions per 32 pairs and the gathers of rect and offset.
__global__ void __launch_bounds__(kDupThreads, 5) k_duplicate(
    const uint32_t* __restrict__ sorted_item, const uint32_t* n_vis, const ushort4* __restrict__ rect, int64_t n,
    const __grid_constant__ gs_frame f, const uint32_t* n_eff, const uint32_t* __restrict__ group_off,
    const uint32_t* __restrict__ first_group, const uint32_t* __restrict__ offset, uint32_t* __restrict__ pkey,
    uint2* __restrict__ psrc, int passes, SortCtl* sort, LbWords sort_words, int sort_tile) {
    const unsigned FULL = 0xffffffffu;
    __shared__ uint32_t s_h[kMaxPasses][256];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int p = 0; p < kMaxPasses; p++) s_h[p][threadIdx.x] = 0;
    __syncthreads();
    const int64_t nv = *n_vis, n_pairs = *n_eff, n_groups = (nv + 31) / 32;
    const uint32_t n32 = (uint32_t)n, magic = view_magic(n32);
    const int64_t spans = (n_pairs + kDupPairs - 1) / kDupPairs;
    const int64_t span = (spans + gridDim.x - 1) / gridDim.x * kDupPairs;
    const int64_t p0 = blockIdx.x * span, p1 = min(p0 + span, n_pairs);
    for (int64_t t = (p0 + sort_tile - 1) / sort_tile; t * sort_tile < p1; t++) lb_zero(sort_words, t);
    if (p0 < p1) {
        // the loads of a warp's next two groups are in flight while it writes one
        int64_t g = first_group[p0 / kDupPairs] + warp;
        constexpr int kStep = kDupThreads / 32;
        auto off_of = [&](int64_t k) -> int64_t { return k < n_groups ? (int64_t)load_now(group_off + k) : p1; };
        auto item_of = [&](int64_t k) { return k * 32 + lane < nv ? load_now(sorted_item + k * 32 + lane) : 0u; };
        int64_t off = off_of(g), off1 = off_of(g + kStep);
        uint32_t item = item_of(g), item1 = item_of(g + kStep);
        uint2 rc = load_now2((const uint2*)rect + item);
        uint32_t slot0 = load_now(offset + item);
        for (; off < p1; g += kStep) {
            const int64_t off2 = off_of(g + 2 * kStep);
            const uint32_t item2 = item_of(g + 2 * kStep);
            const uint2 rc1 = load_now2((const uint2*)rect + item1);
            const uint32_t slot1 = load_now(offset + item1);
            ItemRect q = item_rect(make_ushort4(rc.x & 0xFFFFu, rc.x >> 16, rc.y & 0xFFFFu, rc.y >> 16), f,
                                   view_of(item, n32, magic));
            if (g * 32 + lane >= nv) q.cnt = 0;
            const uint32_t t0 = q.base + q.y0 * q.tx + q.x0;  // the rect's first tile
            const float inv = __fdividef(1.f, (float)q.wx);
            uint32_t start = q.cnt;                           // inclusive, then exclusive prefix
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(FULL, start, o);
                if (lane >= o) start += t;
            }
            const uint32_t total = __shfl_sync(FULL, start, 31);
            start -= q.cnt;
            const unsigned some = __ballot_sync(FULL, q.cnt > 0);
            const uint32_t first = off < p0 ? (uint32_t)(p0 - off) : 0u;
            const uint32_t last = (uint32_t)min((int64_t)total, p1 - off);
            for (uint32_t b = first; b < last; b += 32) {
                const uint32_t j = b + lane;
                // the item of pair j: the last one with pairs that starts at or before it
                const bool in = q.cnt > 0 && start > b && start < b + 32;
                const unsigned begins = __reduce_or_sync(FULL, in ? 1u << (start - b) : 0u);
                const unsigned before = __ballot_sync(FULL, q.cnt > 0 && start <= b);
                int L = __popc(before) + __popc(begins & (lanemask_lt() | (1u << lane))) - 1;
                if (some & (some + 1)) L = __fns(some, 0, L + 1);  // items without pairs in between (foreign rects)
                const uint32_t st = __shfl_sync(FULL, start, L);
                const uint32_t it = __shfl_sync(FULL, item, L), sl = __shfl_sync(FULL, slot0, L);
                const uint32_t aw = __shfl_sync(FULL, q.wx, L);
                const float ai = __shfl_sync(FULL, inv, L);
                const uint32_t at = __shfl_sync(FULL, t0, L), atx = __shfl_sync(FULL, q.tx, L);
                if (j < last) {
                    const uint32_t local = j - st;
                    // below 2^16, (local + 1/2) / aw is at least 2^-17 of itself away from a whole number
                    const uint32_t yy = local < 65536u ? (uint32_t)(((float)local + 0.5f) * ai) : local / aw;
                    const uint32_t t = at + yy * atx + (local - yy * aw);
                    pkey[off + j] = t;
                    psrc[off + j] = make_uint2(it, sl + local);
                    for (int p = 0; p < passes; p++) atomicAdd(&s_h[p][(t >> (8 * p)) & 255u], 1u);
                }
            }
            off = off1; off1 = off2;
            item = item1; item1 = item2;
            rc = rc1;
            slot0 = slot1;
        }
    }
    add_digit_counts(s_h, passes, sort, gridDim.x);
}

// Tile ranges of the sorted pairs (the last tile-sort pass wrote each sorted
// pair's item and emission slot); eight keys per thread and round, two loads:
// 15.8M pairs in 19 us (35 with a key and its two neighbours per thread).
__global__ void __launch_bounds__(256) k_tile_ranges(const uint32_t* __restrict__ skey, const uint32_t* n_eff,
                                                     uint32_t* __restrict__ range, int64_t n_tiles,
                                                     const int32_t* err, int32_t* status) {
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i0 == 0 && *err) *status = *err;
    const int64_t cnt = *n_eff;
    for (int64_t p = 8 * i0; p < cnt; p += 8 * (int64_t)gridDim.x * blockDim.x) {  // grid-stride: few CTAs
        uint32_t t[8];
        if (p + 8 <= cnt) {  // the buffer is 256-byte aligned
            const uint4 a = reinterpret_cast<const uint4*>(skey + p)[0], b = reinterpret_cast<const uint4*>(skey + p)[1];
            t[0] = a.x; t[1] = a.y; t[2] = a.z; t[3] = a.w;
            t[4] = b.x; t[5] = b.y; t[6] = b.z; t[7] = b.w;
        } else {
#pragma unroll
            for (int q = 0; q < 8; q++) t[q] = p + q < cnt ? skey[p + q] : 0xFFFFFFFFu;
        }
        uint32_t prev = p > 0 ? skey[p - 1] : 0xFFFFFFFFu;  // no tile
#pragma unroll
        for (int q = 0; q < 8; q++) {
            if (p + q < cnt && t[q] != prev && t[q] < n_tiles) {  // a tile, unless a wait timed out
                range[2 * (int64_t)t[q]] = (uint32_t)(p + q);
                if (prev < n_tiles) range[2 * (int64_t)prev + 1] = (uint32_t)(p + q);
            }
            if (p + q == cnt - 1 && t[q] < n_tiles) range[2 * (int64_t)t[q] + 1] = (uint32_t)cnt;
            prev = t[q];
        }
    }
}

// Work order of the persistent schedule: tiles by decreasing pair count.
__global__ void k_tile_order_keys(const uint32_t* __restrict__ range, int64_t n_tiles, uint32_t* __restrict__ key,
                                  uint32_t* __restrict__ val) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_tiles) return;
    const uint32_t len = range[2 * t + 1] - range[2 * t];
    key[t] = 0xFFFFu - min(len, 0xFFFFu);
    val[t] = (uint32_t)t;
}

__global__ void k_copy_u32(const uint32_t* __restrict__ a, uint32_t* __restrict__ b, int64_t n, const int32_t* err,
                           int32_t* status) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0 && *err) *status = *err;
    if (i < n) b[i] = a[i];
}

// ---------------------------------------------------------------------------
// The whole of gs_sort in one CTA, for frames whose items, pairs and tiles fit its
// shared memory: offsets and compaction, depth sort (8-bit passes in shared memory, those
// whose digit all keys share skipped), pairs in depth order, one counting pass over the
// tiles that writes the lists, ranges and work order. 1000 items, 2000 pairs, 16 tiles:
// 18 us against 51 for the general path's eleven launches of 3-10 us of latency (in a
// graph); at 4096 items and 12,600 pairs 34 against 58, with the gap closing by the
// 2 us that another 1000 items or pairs cost one CTA, about where its arrays end.
// ---------------------------------------------------------------------------
constexpr int kSmThreads = 1024, kSmWarps = kSmThreads / 32;
constexpr int kSmItems = 4096, kSmPairs = 24576, kSmTiles = 256;
struct SmallSmem {
    uint32_t key[2][kSmItems];  // depth bits; then each sorted item's first pair
    uint16_t val[2][kSmItems];
    uint32_t off[kSmItems];
    uint32_t mask[kSmWarps][256];
    uint16_t cnt[kSmWarps][256];
    uint16_t p_item[kSmPairs];
    uint8_t p_tile[kSmPairs], p_local[kSmPairs];  // tile; index in the item's rect
    uint32_t len[kSmTiles];
};

// First place of each (warp, digit) in the sorted order from the counts in s.cnt; the
// digit's total and start to thread d < 256. All threads.
__device__ __forceinline__ void small_places(SmallSmem& s, uint32_t& tot, uint32_t& start) {
    const int t = threadIdx.x;
    tot = 0;
    if (t < 256) {
#pragma unroll 8
        for (int q = 0; q < kSmWarps; q++) tot += s.cnt[q][t];
    }
    block_exclusive_scan<kSmThreads>(tot, start);
    if (t < 256) {
        uint32_t place = start;
#pragma unroll 8
        for (int q = 0; q < kSmWarps; q++) {
            const uint32_t c = s.cnt[q][t];
            s.cnt[q][t] = (uint16_t)place;
            place += c;
        }
    }
    __syncthreads();
}

// The place of a warp's key with digit d among its (warp, digit)'s keys, which have
// s.cnt[w][d] before them: the lanes before it with the same digit, the count moved on.
__device__ __forceinline__ uint32_t small_rank(SmallSmem& s, int w, unsigned d, bool valid) {
    if (valid) atomicOr(&s.mask[w][d], 1u << (threadIdx.x & 31));
    __syncwarp();
    const uint32_t m = s.mask[w][d], before = s.cnt[w][d];
    __syncwarp();
    const unsigned lower = m & lanemask_lt();
    if (valid && lower == 0) {
        s.mask[w][d] = 0;
        s.cnt[w][d] = (uint16_t)(before + __popc(m));
    }
    __syncwarp();
    return before + __popc(lower);
}

__global__ void __launch_bounds__(kSmThreads, 1) k_sort_small(
    const int32_t* __restrict__ n_tiles, const float4* __restrict__ rgb_depth, const ushort4* __restrict__ rect,
    int64_t n, const __grid_constant__ gs_frame f, int n_items, int tiles, int64_t capacity, uint32_t* __restrict__ offset,
    uint32_t* __restrict__ src, uint32_t* __restrict__ emit, uint32_t* __restrict__ range, uint32_t* __restrict__ order,
    int64_t* __restrict__ count, int32_t* __restrict__ status) {
    extern __shared__ __align__(16) uint8_t s_raw[];
    SmallSmem& s = *reinterpret_cast<SmallSmem*>(s_raw);
    const unsigned FULL = 0xffffffffu;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    constexpr int kPer = kSmItems / kSmThreads;
    for (int i = t; i < kSmWarps * 256; i += kSmThreads) {
        (&s.mask[0][0])[i] = 0;
        (&s.cnt[0][0])[i] = 0;
    }
    // 1. offsets in item order, visible items with their depths
    uint32_t nv;
    {
        uint32_t nt[kPer], vis = 0, sum = 0, depth[kPer];
#pragma unroll
        for (int k = 0; k < kPer; k++) nt[k] = kPer * t + k < n_items ? (uint32_t)max(n_tiles[kPer * t + k], 0) : 0u;
#pragma unroll
        for (int k = 0; k < kPer; k++) {
            depth[k] = nt[k] > 0 ? __float_as_uint(rgb_depth[kPer * t + k].w) : 0u;
            vis += nt[k] > 0;
            sum += nt[k];
        }
        uint32_t pos, slot;
        nv = block_exclusive_scan<kSmThreads>(vis, pos);
        block_exclusive_scan<kSmThreads>(sum, slot);
#pragma unroll
        for (int k = 0; k < kPer; k++) {
            if (kPer * t + k >= n_items) break;
            offset[kPer * t + k] = slot;
            s.off[kPer * t + k] = slot;
            slot += nt[k];
            if (nt[k] > 0) {
                s.key[0][pos] = depth[k];
                s.val[0][pos++] = (uint16_t)(kPer * t + k);
            }
        }
    }
    __syncthreads();
    // 2. stable sort by depth bits; a warp takes a contiguous span
    int in = 0;
    {
        const int span = (int)((nv + kSmThreads - 1) / kSmThreads) * 32, b0 = w * span + lane;
        for (int shift = 0; shift < 32; shift += 8) {
            uint32_t kk[kPer], rank[kPer];
#pragma unroll
            for (int k = 0; k < kPer; k++) {
                const bool valid = 32 * k < span && b0 + 32 * k < (int)nv;
                kk[k] = valid ? s.key[in][b0 + 32 * k] : 0u;
                rank[k] = small_rank(s, w, (kk[k] >> shift) & 255u, valid);
            }
            __syncthreads();
            uint32_t tot, start;
            small_places(s, tot, start);
            const bool same = __syncthreads_or(t < 256 && nv > 0 && tot == nv);
            if (!same) {
#pragma unroll
                for (int k = 0; k < kPer; k++)
                    if (32 * k < span && b0 + 32 * k < (int)nv) {
                        const uint32_t pos = s.cnt[w][(kk[k] >> shift) & 255u] + rank[k];
                        s.key[in ^ 1][pos] = kk[k];
                        s.val[in ^ 1][pos] = s.val[in][b0 + 32 * k];
                    }
                in ^= 1;
            }
            __syncthreads();
            for (int i = t; i < kSmWarps * 256; i += kSmThreads) (&s.cnt[0][0])[i] = 0;
            __syncthreads();
        }
    }
    // 3. pairs in depth order: first pair of each sorted item, then a warp writes 32 items' pairs together
    const uint32_t n32 = (uint32_t)n, magic = view_magic(n32);
    uint32_t* first = s.key[in];
    uint32_t total;
    {
        uint32_t c[kPer], sum = 0, pos;
#pragma unroll
        for (int k = 0; k < kPer; k++) {
            c[k] = 0;
            if (kPer * t + k < (int)nv) {
                const uint32_t item = s.val[in][kPer * t + k];
                c[k] = item_rect(rect[item], f, view_of(item, n32, magic)).cnt;
            }
            sum += c[k];
        }
        total = block_exclusive_scan<kSmThreads>(sum, pos);
#pragma unroll
        for (int k = 0; k < kPer; k++) {
            if (kPer * t + k < (int)nv) first[kPer * t + k] = pos;
            pos += c[k];
        }
    }
    const uint32_t n_eff = (uint32_t)min((int64_t)total, capacity);
    if (t == 0) {
        *count = total;
        *status = (int64_t)total > capacity ? GS_ERR_CAPACITY : GS_OK;
    }
    __syncthreads();
    for (int g = w; g * 32 < (int)nv; g += kSmWarps) {
        const int at = g * 32 + lane;
        const bool have = at < (int)nv;
        const uint32_t item = have ? s.val[in][at] : 0u;
        const ItemRect q = item_rect(rect[item], f, view_of(item, n32, magic));
        const uint32_t cnt = have ? q.cnt : 0u, start = have ? first[at] : 0xFFFFFFFFu;
        const uint32_t t0 = q.base + q.y0 * q.tx + q.x0;
        const uint32_t lo = __shfl_sync(FULL, start, 0);
        const uint32_t hi = min(__reduce_max_sync(FULL, have ? start + cnt : 0u), n_eff);
        for (uint32_t b = lo; b < hi; b += 32) {
            const uint32_t j = b + lane;
            int L = 0;  // the last item that starts at or before pair j (its pairs reach past j: empty items start later)
#pragma unroll
            for (int step = 16; step >= 1; step >>= 1) {
                const uint32_t st = __shfl_sync(FULL, start, L + step);
                if (L + step < 32 && st <= j) L += step;
            }
            const uint32_t st = __shfl_sync(FULL, start, L), it = __shfl_sync(FULL, item, L);
            const uint32_t aw = __shfl_sync(FULL, q.wx, L), at0 = __shfl_sync(FULL, t0, L);
            const uint32_t atx = __shfl_sync(FULL, q.tx, L);
            if (j < hi) {
                const uint32_t local = j - st, yy = local / aw;
                s.p_item[j] = (uint16_t)it;
                s.p_local[j] = (uint8_t)local;
                s.p_tile[j] = (uint8_t)(at0 + yy * atx + (local - yy * aw));
            }
        }
    }
    __syncthreads();
    // 4. stable counting sort by tile, written to the lists
    const int span = (int)((n_eff + kSmThreads - 1) / kSmThreads) * 32, p0 = w * span, p1 = min(p0 + span, (int)n_eff);
    for (int p = p0 + lane; p < p1; p += 32) atomicAdd(&s.mask[w][s.p_tile[p]], 1u);
    __syncthreads();
    for (int i = t; i < kSmWarps * 256; i += kSmThreads) {
        (&s.cnt[0][0])[i] = (uint16_t)(&s.mask[0][0])[i];
        (&s.mask[0][0])[i] = 0;
    }
    __syncthreads();
    uint32_t tot, start;
    small_places(s, tot, start);
    if (t < tiles) {
        range[2 * t] = tot ? start : 0u;
        range[2 * t + 1] = tot ? start + tot : 0u;
        s.len[t] = min(tot, 0xFFFFu);
    }
    for (int p = p0; p < p1; p += 32) {
        const bool valid = p + lane < p1;
        const uint32_t item = valid ? s.p_item[p + lane] : 0u, local = valid ? s.p_local[p + lane] : 0u;
        const uint32_t dest = small_rank(s, w, valid ? s.p_tile[p + lane] : 0u, valid);
        if (valid) {
            src[dest] = item;
            emit[dest] = s.off[item] + local;
        }
    }
    // 5. work order: tiles by decreasing pair count
    if (order) {
        __syncthreads();
        if (t < tiles) {
            uint32_t r = 0;
            for (int u = 0; u < tiles; u++) r += s.len[u] > s.len[t] || (s.len[u] == s.len[t] && u < t);
            order[r] = (uint32_t)t;
        }
    }
}

// The rule: what the CTA's arrays hold (a rect has at most its view's tiles).
static bool small_fits(int64_t n, int64_t n_items, int64_t n_tiles, int64_t capacity) {
    const int64_t most = n * n_tiles < capacity ? n * n_tiles : capacity;
    return n_items <= kSmItems && n_tiles <= kSmTiles && most <= kSmPairs;
}

struct SortWs {
    uint32_t *vk0, *vv0, *vk1, *vv1, *group_off, *first_group, *pk0, *pk1, *misc;
    uint2 *psrc, *psrc2;
    uint32_t *tk0, *tv0, *tk1, *tv1;
    // zeroed together at the start of every call: counts, control words of the two
    // scans and the three sorts, and the scans' look-back words
    size_t zero_bytes;
    ScanCtl* scan_ctl;     // [2]
    SortCtl* sort_ctl;     // [3]
    uint64_t* scan_words;  // [2][scan tiles], then [duplication CTAs]
    uint64_t *wa, *wb;     // radix look-back words (zeroed by the kernels)
};

// One chunk per CTA, all of them resident, at least 1024 items each. Fewer CTAs look back
// over fewer words, more of them gather faster: 152K, 750K and 5.8M visible items
// took 5 and 6 us less and 4 us more of a sort with at most 304 than with 608.
static int64_t dup_ctas(int64_t n_items) {
    const int64_t g = ceil_div(n_items, 1024), most = n_items < ((int64_t)4 << 20) ? scan_ctas() / 2 : scan_ctas();
    return g < most ? g : most;
}

static SortWs carve_sort(char* base, size_t cap_bytes, int64_t n_items, int64_t capacity, int64_t n_tiles,
                         size_t* used) {
    Carve c{base, 0, cap_bytes};
    SortWs w;
    const size_t z0 = c.used;
    w.misc = c.take<uint32_t>(8);
    w.scan_ctl = c.take<ScanCtl>(2);
    w.sort_ctl = c.take<SortCtl>(3);
    w.scan_words = c.take<uint64_t>(2 * ceil_div(n_items, kScanTile) + dup_ctas(n_items));
    w.zero_bytes = c.used - z0;
    w.vk0 = c.take<uint32_t>(n_items);
    w.vv0 = c.take<uint32_t>(n_items);
    w.vk1 = c.take<uint32_t>(n_items);
    w.vv1 = c.take<uint32_t>(n_items);
    w.group_off = c.take<uint32_t>(ceil_div(n_items, 32));
    w.first_group = c.take<uint32_t>(ceil_div(capacity, kDupPairs));
    w.pk0 = c.take<uint32_t>(capacity);
    w.pk1 = c.take<uint32_t>(capacity);
    w.psrc = c.take<uint2>(capacity);
    w.psrc2 = c.take<uint2>(capacity);
    w.tk0 = c.take<uint32_t>(n_tiles);
    w.tv0 = c.take<uint32_t>(n_tiles);
    w.tk1 = c.take<uint32_t>(n_tiles);
    w.tv1 = c.take<uint32_t>(n_tiles);
    int64_t words = onesweep_words(n_items);  // the most that one of the three sorts needs
    for (const int64_t k : {capacity, n_tiles})
        if (onesweep_words(k) > words) words = onesweep_words(k);
    w.wa = c.take<uint64_t>(words);
    w.wb = c.take<uint64_t>(words);
    *used = c.used;
    return w;
}

static int bits_for(int64_t v) {
    int b = 0;
    while (b < 32 && ((int64_t)1 << b) < v) b++;
    return b < 1 ? 1 : b;
}

}  // namespace gs

using namespace gs;

extern "C" size_t gs_sort_workspace_size(int64_t n, const gs_frame* f, int64_t capacity) {
    if (!f || n < 0 || capacity < 0) return 0;
    size_t used = 0;
    carve_sort(nullptr, 0, n * f->n_views, capacity, f->tile_base[f->n_views], &used);
    return used;
}

extern "C" int gs_sort(const gs_projected* p, int64_t n, const gs_frame* f, const gs_pairs* out, void* ws,
                       size_t ws_bytes, void* stream) {
    if (!p || !f || !out || n < 0 || f->n_views < 1 || f->n_views > GS_MAX_VIEWS) return GS_ERR_INVALID_ARG;
    const int64_t n_items = n * f->n_views;
    if (n_items > (int64_t)UINT32_MAX || out->capacity < 0 || out->capacity > (int64_t)UINT32_MAX - 1)
        return GS_ERR_INVALID_ARG;
    if (!out->count || !out->status || !out->range || (out->capacity > 0 && (!out->src || !out->emit)) ||
        (n_items > 0 && !out->offset))
        return GS_ERR_INVALID_ARG;
    size_t need = 0;
    const int64_t n_tiles_all = f->tile_base[f->n_views];
    SortWs w = carve_sort((char*)ws, ws_bytes, n_items, out->capacity, n_tiles_all, &need);
    if (!ws || ws_bytes < need || ((uintptr_t)ws & 255)) return GS_ERR_INVALID_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t n_tiles_total = f->tile_base[f->n_views];
    uint32_t* n_vis = w.misc;        // visible item count
    uint32_t* n_eff = w.misc + 2;    // pairs actually stored
    int32_t* err = (int32_t*)(w.misc + 3);  // GS_ERR_TIMEOUT from a look-back wait
    if (n_items > 0 && small_fits(n, n_items, n_tiles_total, out->capacity)) {
        if (cudaFuncSetAttribute(k_sort_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmallSmem)) !=
            cudaSuccess) {
            (void)cudaGetLastError();
            return GS_ERR_CUDA;
        }
        k_sort_small<<<1, kSmThreads, sizeof(SmallSmem), s>>>(
            p->n_tiles, (const float4*)p->rgb_depth, (const ushort4*)p->rect, n, *f, (int)n_items, (int)n_tiles_total,
            out->capacity, out->offset, out->src, out->emit, out->range, out->order, out->count, out->status);
        count_launch();
        GS_CUDA_CHECK_LAUNCH();
        return GS_OK;
    }
    if (n_items == 0) {
        cudaMemsetAsync(out->range, 0, sizeof(uint32_t) * 2 * n_tiles_total, s);
        k_no_pairs<<<1, 1, 0, s>>>(out->count, out->status);
        count_launch();
        GS_CUDA_CHECK_LAUNCH();
        return GS_OK;
    }
    cudaMemsetAsync(w.misc, 0, w.zero_bytes, s);
    // 1. emission slots, and the visible items (in item order) with their depth keys
    const int64_t scan_tiles = ceil_div(n_items, kScanTile);
    // two CTAs per SM: fewer words to look back over than with four (148 against 154 us of sort at 1M
    // items); a tile each where that is enough (84 against 86 us at 200K)
    const int64_t scan_tiles_per = scan_tiles <= scan_ctas() / 2 ? 1 : ceil_div(scan_tiles, scan_ctas() / 2);
    const int64_t chunk = scan_tiles_per * kScanTile;
    const int64_t item_blocks = onesweep_blocks(n_items);
    const auto scan_items = scan_tiles_per == 1 ? k_scan_items<true> : k_scan_items<false>;
    scan_items<<<(unsigned)ceil_div(n_items, chunk), kScanThreads, 0, s>>>(
        p->n_tiles, (const float4*)p->rgb_depth, n_items, chunk, out->offset, w.vk0, w.vv0, n_vis, &w.scan_ctl[0],
        w.scan_words, w.scan_words + scan_tiles, &w.sort_ctl[0], lb_words(w.wa, item_blocks), item_blocks,
        out->range, 2 * n_tiles_total, err);
    count_launch();
    // 2. stable sort of visible items by depth bits
    const bool in1 = onesweep_passes<uint32_t>(w.vk0, w.vv0, w.vk1, w.vv1, n_items, n_vis, 32, &w.sort_ctl[0], w.wa,
                                               w.wb, err, s);
    // 3. pair positions in depth order; the pair count
    const uint32_t* sorted_item = in1 ? w.vv1 : w.vv0;
    k_pair_positions<<<(unsigned)dup_ctas(n_items), kDupThreads, 0, s>>>(
        sorted_item, n_vis, (const ushort4*)p->rect, n, *f, out->capacity, w.group_off, w.first_group, &w.scan_ctl[1],
        w.scan_words + 2 * scan_tiles, out->count, n_eff, out->status, err);
    count_launch();
    // 4. one (tile, emission slot) pair per tile of each visible item's rect; stable sort by global tile
    //    index carrying each pair's (item, emission slot), the last pass writing them to src / emit;
    //    tile ranges
    if (out->capacity > 0) {
        const int tile_bits = bits_for(n_tiles_total);
        const int64_t dup_grid = ceil_div(out->capacity, kDupPairs);
        k_duplicate<<<(unsigned)(dup_grid < 5 * 152 ? dup_grid : 5 * 152), kDupThreads, 0, s>>>(
            sorted_item, n_vis, (const ushort4*)p->rect, n, *f, n_eff, w.group_off, w.first_group, out->offset, w.pk0,
            w.psrc, (tile_bits + 7) / 8, &w.sort_ctl[1], lb_words(w.wa, onesweep_blocks(out->capacity)),
            onesweep_tile(out->capacity));
        count_launch();
        const bool pin1 = onesweep_passes<uint2>(w.pk0, w.psrc, w.pk1, w.psrc2, out->capacity, n_eff, tile_bits,
                                                 &w.sort_ctl[1], w.wa, w.wb, err, s, out->src, out->emit);
        const int64_t rg = ceil_div(out->capacity, 8 * 256);
        k_tile_ranges<<<(unsigned)(rg < 152 * 8 ? rg : 152 * 8), 256, 0, s>>>(pin1 ? w.pk1 : w.pk0, n_eff, out->range,
                                                                             n_tiles_total, err, out->status);
        count_launch();
    }
    // 5. optional work order for the persistent render schedule
    if (out->order && n_tiles_total > 0) {
        k_tile_order_keys<<<(unsigned)ceil_div(n_tiles_total, 256), 256, 0, s>>>(out->range, n_tiles_total, w.tk0,
                                                                                  w.tv0);
        count_launch();
        k_onesweep_hist<<<(unsigned)radix_blocks(n_tiles_total), 256, 0, s>>>(
            w.tk0, n_tiles_total, 2, &w.sort_ctl[2], lb_words(w.wa, onesweep_blocks(n_tiles_total)),
            onesweep_blocks(n_tiles_total));
        count_launch();
        const bool t1 = onesweep_passes<uint32_t>(w.tk0, w.tv0, w.tk1, w.tv1, n_tiles_total, nullptr, 16,
                                                  &w.sort_ctl[2], w.wa, w.wb, err, s);
        k_copy_u32<<<(unsigned)ceil_div(n_tiles_total, 256), 256, 0, s>>>(t1 ? w.tv1 : w.tv0, out->order,
                                                                           n_tiles_total, err, out->status);
        count_launch();
    }
    GS_CUDA_CHECK_LAUNCH();
    return GS_OK;
}
