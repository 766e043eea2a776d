// False-alarm rates from a timeslide background (Sec. IX: the FAR of an event is
// the number of background events whose detection statistic is greater than the
// event's, divided by the background livetime).
//
// The background statistics are sorted in decreasing order on the device by an
// LSD radix sort of order-preserving 32-bit keys (4 passes of 8 bits, each pass
// stable: per-tile digit histograms, a scan of each digit's row over the tiles, and a
// scatter that adds up the digits before and ranks equal digits in input order).  The
// first pass reads the statistics, the last writes them.  Launches are sized by the
// capacity; only the tiles that hold keys do work.  Each foreground statistic x
// then gets count = #{background > x} by a 32-way search (one warp), and FAR = count / livetime.
// The background count may live on the device (as afg_batch_run writes it), so
// every kernel reads n = min(*n_dev, cap) itself and nothing synchronises.
// A handful of small kernels in a row: latency sets the time (0.93 million events: 330 us with the histogram
// scanned by one block (43 us of each pass) and four barriers per 256 keys of the scatter, 95 us now).
#include <stdint.h>

#include <algorithm>

#include "afg_internal.cuh"

namespace {

constexpr int RS_T = 256;              // threads per tile
constexpr int RS_ROUNDS = 8;           // keys per thread per tile
constexpr int RS_TILE = RS_T * RS_ROUNDS;
constexpr int RS_WARPS = RS_T / 32;

__device__ __forceinline__ int64_t dev_count(const int64_t *n_dev, int64_t cap) {
    const int64_t n = *n_dev;
    return n < 0 ? 0 : (n < cap ? n : cap);
}

// Ascending order of keys = decreasing order of statistics.
__device__ __forceinline__ uint32_t key_of(float v) {
    uint32_t b = __float_as_uint(v);
    b = (b & 0x80000000u) ? ~b : (b | 0x80000000u);  // ascending with v
    return ~b;                                        // descending with v
}

__device__ __forceinline__ float value_of(uint32_t k) {
    uint32_t b = ~k;
    b = (b & 0x80000000u) ? (b & 0x7fffffffu) : ~b;
    return __uint_as_float(b);
}

// tiles that hold keys
__device__ __forceinline__ int occupied_tiles(int64_t n) { return (int)((n + RS_TILE - 1) / RS_TILE); }

// The keys a pass reads: of the previous pass, or (keys null, first pass) of the statistics.
struct KeySource {
    const uint32_t *keys;
    const float *stat;
    const int64_t *idx;
    __device__ __forceinline__ uint32_t operator()(int64_t i) const {
        return keys ? keys[i] : key_of(stat[idx ? idx[i] : i]);
    }
};

// hist[d * n_eff + tile] = keys of the tile whose digit (at `shift`) is d, over the
// n_eff = ceil(n / RS_TILE) tiles that hold keys (blocks past them return at once)
__global__ void __launch_bounds__(RS_T) k_rs_hist(const KeySource src, const int64_t *n_dev, int64_t cap, int shift,
                                                  uint32_t *__restrict__ hist) {
    __shared__ uint32_t h[256];
    const int64_t n = dev_count(n_dev, cap);
    const int n_eff = occupied_tiles(n);
    if ((int)blockIdx.x >= n_eff) return;
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RS_TILE;
    uint32_t k[RS_ROUNDS];
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) {
        const int64_t i = base + r * RS_T + threadIdx.x;
        k[r] = i < n ? src(i) : 0u;
    }
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r)
        if (base + r * RS_T + threadIdx.x < n) atomicAdd(&h[(k[r] >> shift) & 255u], 1u);
    __syncthreads();
    hist[(size_t)threadIdx.x * n_eff + blockIdx.x] = h[threadIdx.x];
}

// grid (256): exclusive scan of digit d's row of n_eff tile counts in place, and its sum to total[d]
__global__ void __launch_bounds__(256) k_rs_scan(uint32_t *__restrict__ hist, const int64_t *n_dev, int64_t cap,
                                                 uint32_t *__restrict__ total) {
    __shared__ uint32_t wsum[2][8];
    const int n_eff = occupied_tiles(dev_count(n_dev, cap));
    uint32_t *a = hist + (size_t)blockIdx.x * n_eff;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint32_t carry = 0;
    int buf = 0;
    for (int c0 = 0; c0 < n_eff; c0 += 1024, buf ^= 1) {  // four consecutive entries a thread
        uint32_t v[4], x = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = c0 + 4 * t + k;
            v[k] = i < n_eff ? a[i] : 0u;
            x += v[k];
        }
        const uint32_t own = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[buf][warp] = x;
        __syncthreads();
        uint32_t before = carry + x - own;
        for (int w = 0; w < 8; ++w) {
            const uint32_t s = wsum[buf][w];
            if (w < warp) before += s;
            carry += s;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = c0 + 4 * t + k;
            if (i < n_eff) a[i] = before;
            before += v[k];
        }
    }
    if (t == 0) total[blockIdx.x] = carry;
}

// Stable scatter of one tile: warp w takes its 32 RS_ROUNDS consecutive keys, 32 a round; equal digits of a round
// are ranked by lane (match_any peers with lower lanes) behind the warp's count so far, then the warps' counts are
// added up per digit.  Writes keys, or (last pass, out set) the statistics themselves.
__global__ void __launch_bounds__(RS_T) k_rs_scatter(const KeySource src, uint32_t *__restrict__ kout,
                                                     float *__restrict__ out, const int64_t *n_dev, int64_t cap, int shift,
                                                     const uint32_t *__restrict__ hist,
                                                     const uint32_t *__restrict__ total) {
    __shared__ uint32_t wcnt[RS_WARPS][257];  // per-warp digit counts, then each warp's first place
    __shared__ uint32_t dsum[RS_WARPS];
    const int64_t n = dev_count(n_dev, cap);
    const int n_eff = occupied_tiles(n);
    if ((int)blockIdx.x >= n_eff) return;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    for (int i = lane; i < 257; i += 32) wcnt[warp][i] = 0;
    // keys of lower digits: exclusive sum of the 256 totals (thread t: digit t)
    const uint32_t dt = total[t];
    uint32_t x = dt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) dsum[warp] = x;
    uint32_t place = x - dt + hist[(size_t)t * n_eff + blockIdx.x];
    const int64_t base = (int64_t)blockIdx.x * RS_TILE + warp * (32 * RS_ROUNDS) + lane;
    uint32_t key[RS_ROUNDS], rank[RS_ROUNDS];
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) key[r] = base + 32 * r < n ? src(base + 32 * r) : 0u;
    const uint32_t lt = (1u << lane) - 1u;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) {
        const uint32_t d = base + 32 * r < n ? (key[r] >> shift) & 255u : 256u;  // 256: no key
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        rank[r] = wcnt[warp][d] + __popc(peers & lt);
        __syncwarp();
        if ((peers & lt) == 0) wcnt[warp][d] += __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    for (int w = 0; w < warp; ++w) place += dsum[w];
#pragma unroll
    for (int w = 0; w < RS_WARPS; ++w) {  // thread t: digit t
        const uint32_t c = wcnt[w][t];
        wcnt[w][t] = place;
        place += c;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r)
        if (base + 32 * r < n) {
            const uint32_t p = wcnt[warp][(key[r] >> shift) & 255u] + rank[r];
            if (out) out[p] = value_of(key[r]);
            else kout[p] = key[r];
        }
}

// count = #{sorted > x}: the first index whose value is <= x in the decreasing array.  One warp per x: each step
// splits the range in 33 at 32 probes.
__global__ void k_far_count(const float *__restrict__ sorted, const int64_t *n_dev, int64_t cap,
                            const float *__restrict__ fg, int64_t n_fg, double livetime, int64_t *__restrict__ n_above,
                            double *__restrict__ far) {
    const int64_t n = dev_count(n_dev, cap);
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * blockDim.x / 32;
    for (int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32; j < n_fg; j += warps) {
        const float x = fg[j];
        int64_t lo = 0, hi = n;  // the answer lies in [lo, hi]
        while (lo < hi) {
            const int64_t step = (hi - lo + 32) / 33, i = lo + step * (lane + 1) - 1;  // probes, in order
            const uint32_t above = __ballot_sync(0xffffffffu, i < hi && sorted[i] > x);
            const int c = __popc(above);  // the first c probes are above x
            const int64_t nhi = lo + step * (c + 1) - 1;
            lo += step * c;
            hi = c < 32 && nhi < hi ? nhi : hi;
        }
        if (lane == 0) {
            if (n_above) n_above[j] = lo;
            if (far) far[j] = (double)lo / livetime;
        }
    }
}

}  // namespace

int launch_far(afg_ctx *ctx, const float *bg_stat, const int64_t *bg_idx, const int64_t *n_bg_dev, int64_t bg_cap,
               double livetime_s, const float *fg, int64_t n_fg, int64_t *n_above, double *far, float *bg_sorted,
               cudaStream_t st) {
    const int n_tiles = (int)std::max<int64_t>(1, (bg_cap + RS_TILE - 1) / RS_TILE);
    const int64_t m = (int64_t)256 * n_tiles + 256;  // and the digits' totals
    void *wk = nullptr, *wh = nullptr, *ws = nullptr;
    int rc = afg_ws_reserve(ctx, WS_FAR_KEYS, (size_t)2 * std::max<int64_t>(bg_cap, 1) * sizeof(uint32_t), &wk);
    if (!rc) rc = afg_ws_reserve(ctx, WS_FAR_HIST, (size_t)m * sizeof(uint32_t), &wh);
    if (!rc && !bg_sorted) {
        rc = afg_ws_reserve(ctx, WS_FAR_SORTED, (size_t)std::max<int64_t>(bg_cap, 1) * sizeof(float), &ws);
        bg_sorted = static_cast<float *>(ws);
    }
    if (rc) return rc;
    uint32_t *ka = static_cast<uint32_t *>(wk), *kb = ka + std::max<int64_t>(bg_cap, 1);
    uint32_t *hist = static_cast<uint32_t *>(wh);
    uint32_t *total = hist + (int64_t)256 * n_tiles;
    {
        KScope ks(ctx, st, KK_FAR, 0.0, (double)bg_cap * (4.0 + 8.0 + 4.0 * 4 * 4 + 4.0) + n_fg * 20.0);
        KeySource src = {nullptr, bg_stat, bg_idx};
        for (int pass = 0; pass < 4; ++pass) {
            k_rs_hist<<<n_tiles, RS_T, 0, st>>>(src, n_bg_dev, bg_cap, 8 * pass, hist);
            k_rs_scan<<<256, 256, 0, st>>>(hist, n_bg_dev, bg_cap, total);
            k_rs_scatter<<<n_tiles, RS_T, 0, st>>>(src, ka, pass == 3 ? bg_sorted : nullptr, n_bg_dev, bg_cap, 8 * pass,
                                                   hist, total);
            src.keys = ka;
            std::swap(ka, kb);
        }
        if (n_fg > 0)
            k_far_count<<<(unsigned)std::min<int64_t>((n_fg + 7) / 8, 152 * 16), 256, 0, st>>>(
                bg_sorted, n_bg_dev, bg_cap, fg, n_fg, livetime_s, n_above, far);
    }
    AFG_LAUNCH_CHECK(ctx, "far (radix sort + rank count)");
    return AFG_OK;
}
