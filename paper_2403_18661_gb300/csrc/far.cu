// False-alarm rates from a timeslide background (Sec. IX: the FAR of an event is
// the number of background events whose detection statistic is greater than the
// event's, divided by the background livetime).
//
// The background statistics are sorted in decreasing order on the device by an
// LSD radix sort of order-preserving 32-bit keys, 4 stable passes of 8 bits.  One launch counts all four digits of
// every key; then one launch a pass ranks each tile's keys in input order and scatters them.  A tile's first places
// are the keys of lower digits (from the counts) plus those of its digit in the tiles before it, which it adds up
// from the sums the tiles publish (decoupled look-back, Merrill & Garland 2016).  The first pass reads the
// statistics, the last writes them.  Launches are sized by the capacity; only the tiles that hold keys do work.
// Each foreground statistic x then gets count = #{background > x} by a 32-way search (one warp; one thread's bisection
// where there are many) and FAR = count / livetime.  The background count may live on the device (as afg_batch_run writes it), so
// every kernel reads n = min(*n_dev, cap) itself and nothing synchronises.
// A handful of small kernels in a row: latency sets the time (0.93 million events: 330 us with the histogram scanned
// by one block and four barriers per 256 keys of the scatter; 97 us as histogram, row scan and scatter a pass, 13
// launches; 68 us now, 7 launches; 20,000 events 66 -> 34 us).
#include <stdint.h>

#include <algorithm>

#include "afg_internal.cuh"

namespace {

constexpr int RS_T = 512;              // threads per tile
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

// hist[p][d] += keys whose digit p is d, all four digits in one read; and the published sums of the tiles cleared.
// Blocks stride over the tiles (two an SM at most: every block adds up to 1024 counts to the same 4 KB).
__global__ void __launch_bounds__(RS_T) k_rs_hist(const KeySource src, const int64_t *n_dev, int64_t cap,
                                                  uint32_t *__restrict__ hist, unsigned long long *__restrict__ status) {
    __shared__ uint32_t h[4][256];
    const int64_t n = dev_count(n_dev, cap);
    const int n_eff = occupied_tiles(n), lane = threadIdx.x & 31;
    pdl_trigger();  // (launched plainly)
    if ((int)blockIdx.x >= n_eff) return;
#pragma unroll
    for (int p = 0; p < 4; ++p)
        if (threadIdx.x < 256) h[p][threadIdx.x] = 0;
    __syncthreads();
    for (int tile = blockIdx.x; tile < n_eff; tile += gridDim.x) {
        if (threadIdx.x < 256) status[(size_t)tile * 256 + threadIdx.x] = 0;
        const int64_t base = (int64_t)tile * RS_TILE;
        uint32_t k[RS_ROUNDS];
#pragma unroll
        for (int r = 0; r < RS_ROUNDS; ++r) {
            const int64_t i = base + r * RS_T + threadIdx.x;
            k[r] = i < n ? src(i) : 0u;
        }
#pragma unroll
        for (int r = 0; r < RS_ROUNDS; ++r) {
            const bool in = base + r * RS_T + threadIdx.x < n;
            if (in)
#pragma unroll
                for (int p = 0; p < 3; ++p) atomicAdd(&h[p][(k[r] >> (8 * p)) & 255u], 1u);
            // sign and most of the exponent: few values, so equal ones of a warp are added once
            const uint32_t d = in ? k[r] >> 24 : 256u, peers = __match_any_sync(0xffffffffu, d);
            if (in && !(peers & ((1u << lane) - 1u))) atomicAdd(&h[3][d], (uint32_t)__popc(peers));
        }
    }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const uint32_t c = threadIdx.x < 256 ? h[p][threadIdx.x] : 0u;
        if (c) atomicAdd(&hist[p * 256 + threadIdx.x], c);
    }
}

// A tile's published sum of a digit: one 64-bit word, so that no order between words matters.  Top four bits: which
// pass (1..4) wrote it, shifted by one, and whether it is the sum over all tiles up to this one; else the tile's own.
constexpr int ST_SHIFT = 60;
constexpr unsigned long long ST_VALUE = (1ull << ST_SHIFT) - 1;
constexpr int ST_LOOK = 4;                           // tiles read at a time
constexpr unsigned long long ST_WAIT_NS = 2000000000ull;

__device__ __forceinline__ unsigned long long timer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Lanes whose value (below 512) equals this lane's, by nine votes: match_any takes one step per distinct value, and
// the low digits have 32 (23.4 against 19.3 us a pass of 0.93 million keys).
__device__ __forceinline__ uint32_t digit_peers(uint32_t d) {
    uint32_t p = 0xffffffffu;
#pragma unroll
    for (int b = 0; b < 9; ++b) {
        const bool set = (d >> b) & 1u;
        const uint32_t v = __ballot_sync(0xffffffffu, set);
        p &= set ? v : ~v;
    }
    return p;
}

// One pass.  A tile is 4096 keys: with 2048 the look-back has twice the tiles to pass (92 us in all at 0.93 million
// keys with 1024), with 8192 fewer blocks share a small sort (20,000 keys: 46 us against 34).  Tiles are taken in
// the order the blocks start, so every tile before a block's own is running or done and the look-back ends; it
// gives up after 2 s all the same (err set; the places it then has are too low, never past the end).  Within a tile
// warp w takes its 32 RS_ROUNDS consecutive keys, 32 a round; equal digits of a round are ranked by lane (peers
// with lower lanes) behind the warp's count so far, then the warps' counts are added up per digit.  The tile is
// sorted in shared memory first, so that the writes are runs of a digit's keys (16 on average; single keys took 2.7
// us a pass longer).  Writes keys, or (last pass, out set) the statistics themselves.  hist null: the capacity is
// one tile, whose own counts are the totals.
__global__ void __launch_bounds__(RS_T) k_rs_pass(const KeySource src, uint32_t *__restrict__ kout,
                                                  float *__restrict__ out, const int64_t *n_dev, int64_t cap, int pass,
                                                  const uint32_t *hist, uint32_t *ticket, unsigned long long *status,
                                                  int *err) {
    __shared__ uint32_t wcnt[RS_WARPS][257];  // per-warp digit counts, then each warp's first slot in the tile
    __shared__ uint32_t skey[RS_TILE];
    __shared__ uint32_t gofs[256];            // first place of the tile's keys of a digit, less their first slot
    __shared__ uint32_t dsum[8], osum[8];
    __shared__ int s_tile;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, shift = 8 * pass;
    // (the counters were cleared before the launch of k_rs_hist, which this one comes after)
    if (t == 0) s_tile = hist ? (int)atomicAdd(&ticket[pass], 1u) : 0;
    for (int i = lane; i < 257; i += 32) wcnt[warp][i] = 0;
    pdl_wait();
    pdl_trigger();
    const int64_t n = dev_count(n_dev, cap);
    __syncthreads();
    const int tile = s_tile;
    if (tile >= occupied_tiles(n)) return;
    const bool digit = t < 256;  // thread t: digit t
    const uint32_t dt = hist && digit ? hist[pass * 256 + t] : 0u;
    const int64_t base = (int64_t)tile * RS_TILE + warp * (32 * RS_ROUNDS) + lane;
    uint32_t key[RS_ROUNDS], rank[RS_ROUNDS];  // rank: first the lanes with an equal digit
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) key[r] = base + 32 * r < n ? src(base + 32 * r) : 0u;
    const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) rank[r] = digit_peers(base + 32 * r < n ? (key[r] >> shift) & 255u : 256u);
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) {
        const uint32_t d = base + 32 * r < n ? (key[r] >> shift) & 255u : 256u;  // 256: no key
        const uint32_t peers = rank[r];
        rank[r] = wcnt[warp][d] + __popc(peers & lt);
        __syncwarp();
        if ((peers & lt) == 0) wcnt[warp][d] += __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    uint32_t own = 0;
    if (digit)
#pragma unroll
        for (int w = 0; w < RS_WARPS; ++w) own += wcnt[w][t];
    volatile unsigned long long *const sum = status + (size_t)tile * 256 + t;
    const unsigned long long tag = (unsigned long long)(pass + 1) << 1, all = (tag | 1) << ST_SHIFT;
    if (hist && digit) *sum = (tile ? tag << ST_SHIFT : all) | own;
    // keys of lower digits, in the tile and (from the totals) in all
    uint32_t x = own, y = dt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, x, o), v = __shfl_up_sync(0xffffffffu, y, o);
        if (lane >= o) {
            x += u;
            y += v;
        }
    }
    if (digit && lane == 31) {
        osum[warp] = x;
        dsum[warp] = y;
    }
    __syncthreads();
    if (digit) {
        uint32_t slot = x - own, place = y - dt;
        for (int w = 0; w < warp; ++w) {
            slot += osum[w];
            place += dsum[w];
        }
        const uint32_t first = slot;
        if (!hist) place = first;
#pragma unroll
        for (int w = 0; w < RS_WARPS; ++w) {
            const uint32_t c = wcnt[w][t];
            wcnt[w][t] = slot;
            slot += c;
        }
        // keys of the digit in the tiles before
        unsigned long long before = 0;
        if (tile) {
            const volatile unsigned long long *q = sum;
            unsigned long long t0 = 0;
            uint32_t spins = 0;
            for (int j = tile; j > 0;) {
                unsigned long long v[ST_LOOK];
#pragma unroll
                for (int i = 0; i < ST_LOOK; ++i) v[i] = j - i > 0 ? q[-256 * (i + 1)] : 0;
                int done = 0;
#pragma unroll
                for (int i = 0; i < ST_LOOK; ++i)
                    if (done == i && j > 0 && (v[i] >> (ST_SHIFT + 1)) == (unsigned long long)(pass + 1)) {
                        before += v[i] & ST_VALUE;
                        done = i + 1;
                        j = (v[i] >> ST_SHIFT) & 1 ? 0 : j - 1;
                    }
                q -= 256 * done;
                if (!done && (++spins & 1023u) == 0) {  // (the clock is read now and then)
                    const unsigned long long now = timer_ns();
                    if (!t0) t0 = now;
                    else if (now - t0 > ST_WAIT_NS) {
                        atomicExch(err, 1);
                        break;
                    }
                }
            }
            *sum = all | (before + own);
        }
        gofs[t] = place + (uint32_t)before - first;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r)
        if (base + 32 * r < n) skey[wcnt[warp][(key[r] >> shift) & 255u] + rank[r]] = key[r];
    __syncthreads();
    const int m = (int)min((int64_t)RS_TILE, n - (int64_t)tile * RS_TILE);
#pragma unroll
    for (int r = 0; r < RS_ROUNDS; ++r) {
        const int i = r * RS_T + t;
        if (i < m) {
            const uint32_t k = skey[i], p = gofs[(k >> shift) & 255u] + (uint32_t)i;
            if (out) out[p] = value_of(k);
            else kout[p] = k;
        }
    }
}

// count = #{sorted > x}: the first index whose value is <= x in the decreasing array, by bisection
__device__ __forceinline__ int64_t bisect(const float *sorted, int64_t n, float x) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (sorted[mid] > x) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// One warp per x: each step splits the range in 33 at 32 probes, which is where bisection ends as long as the probes
// above x are the first ones.  Positive NaN come before every number and are not above it: then each lane bisects.
__global__ void k_far_count(const float *sorted, const int64_t *n_dev, int64_t cap, const float *fg, int64_t n_fg,
                            double livetime, int64_t *__restrict__ n_above, double *__restrict__ far) {
    pdl_wait();
    const int64_t n = dev_count(n_dev, cap);
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * blockDim.x / 32;
    const float first = n > 0 ? sorted[0] : 0.f;  // (looked at after the search: its load waits for nothing)
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
        if (isnan(first)) lo = bisect(sorted, n, x);
        if (lane == 0) {
            if (n_above) n_above[j] = lo;
            if (far) far[j] = (double)lo / livetime;
        }
    }
}

// One thread per x.  A warp per x has a quarter of the dependent loads but as many loads in all as eight threads, so
// above about a warp an x that the GPU holds at once (8192) the loads bind it.  With the sort, 0.93 million background
// events: 4096 x 69 us either way, 65,536 101 us as warps and 77 so, a million 595 and 105 (4000 events, a million x: 541
// and 42).
__global__ void k_far_bisect(const float *sorted, const int64_t *n_dev, int64_t cap, const float *fg, int64_t n_fg,
                             double livetime, int64_t *n_above, double *far) {
    pdl_wait();
    const int64_t n = dev_count(n_dev, cap), threads = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n_fg; j += threads) {
        const int64_t c = bisect(sorted, n, fg[j]);
        if (n_above) n_above[j] = c;
        if (far) far[j] = (double)c / livetime;
    }
}

constexpr int64_t FAR_WARPS = 8192;  // foreground events searched by a warp each

}  // namespace

int launch_far(afg_ctx *ctx, const float *bg_stat, const int64_t *bg_idx, const int64_t *n_bg_dev, int64_t bg_cap,
               double livetime_s, const float *fg, int64_t n_fg, int64_t *n_above, double *far, float *bg_sorted,
               cudaStream_t st) {
    const int n_tiles = (int)std::max<int64_t>(1, (bg_cap + RS_TILE - 1) / RS_TILE);
    // per tile 256 published sums, then the four digits' totals and four tile counters (nothing for one tile); the keys
    // go back and forth between one buffer and bg_sorted: in all no more than two buffers and a histogram row a tile took
    const size_t m = n_tiles > 1 ? (size_t)n_tiles * 256 * 8 + 4 * 256 * 4 + 16 : 0;
    void *wk = nullptr, *wh = nullptr, *ws = nullptr;
    int rc = afg_ws_reserve(ctx, WS_FAR_KEYS, (size_t)std::max<int64_t>(bg_cap, 1) * sizeof(uint32_t), &wk);
    if (!rc && m) rc = afg_ws_reserve(ctx, WS_FAR_HIST, m, &wh);
    if (!rc && !bg_sorted) {
        rc = afg_ws_reserve(ctx, WS_FAR_SORTED, (size_t)std::max<int64_t>(bg_cap, 1) * sizeof(float), &ws);
        bg_sorted = static_cast<float *>(ws);
    }
    if (rc) return rc;
    uint32_t *keys[2] = {static_cast<uint32_t *>(wk), reinterpret_cast<uint32_t *>(bg_sorted)};
    unsigned long long *status = static_cast<unsigned long long *>(wh);
    uint32_t *hist = m ? reinterpret_cast<uint32_t *>(status + (size_t)n_tiles * 256) : nullptr;
    uint32_t *ticket = m ? hist + 4 * 256 : nullptr;
    {
        KScope ks(ctx, st, KK_FAR, 0.0, (double)bg_cap * (4.0 + 8.0 + 4.0 * 4 * 4 + 4.0) + n_fg * 20.0);
        KeySource src = {nullptr, bg_stat, bg_idx};
        if (m) {
            AFG_CUDA(ctx, cudaMemsetAsync(hist, 0, 4 * 256 * 4 + 16, st));
            k_rs_hist<<<std::min(n_tiles, 304), RS_T, 0, st>>>(src, n_bg_dev, bg_cap, hist, status);
        }
        for (int pass = 0; pass < 4; ++pass) {
            uint32_t *ko = keys[pass & 1];
            AFG_CUDA(ctx, launch_pdl(k_rs_pass, dim3(n_tiles), dim3(RS_T), 0, st, src, ko, pass == 3 ? bg_sorted : nullptr,
                                     n_bg_dev, bg_cap, pass, (const uint32_t *)hist, ticket, status, ctx->d_err));
            src.keys = ko;
        }
        if (n_fg > FAR_WARPS)
            AFG_CUDA(ctx, launch_pdl(k_far_bisect, dim3((unsigned)std::min<int64_t>((n_fg + 255) / 256, 152 * 16)), dim3(256), 0,
                                     st, (const float *)bg_sorted, n_bg_dev, bg_cap, fg, n_fg, livetime_s, n_above, far));
        else if (n_fg > 0)
            AFG_CUDA(ctx, launch_pdl(k_far_count, dim3((unsigned)std::min<int64_t>((n_fg + 7) / 8, 152 * 16)), dim3(256), 0, st,
                                     (const float *)bg_sorted, n_bg_dev, bg_cap, fg, n_fg, livetime_s, n_above, far));
    }
    AFG_LAUNCH_CHECK(ctx, "far (radix sort + rank count)");
    return AFG_OK;
}
