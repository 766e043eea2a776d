// Integration and clustering of the per-window outputs (Sec. II: the
// predictions are integrated with a 1 s top-hat filter; the maximum
// integrated value over an 8 s window is the detection statistic of a
// candidate).
//
//   statistic     stat[j] = (1/n_int) sum_{i<n_int} z[j+i], summed in index order
//   triggers      the cluster maxima (earliest index wins ties), compacted in increasing
//                 index order
//
// k_cluster does both for a tile of the series from one read of its logits: statistic of
// the tile and of h indices to each side, windowed maxima by doubling in shared memory
// (O(log h) an index), flags and their count; k_cluster_write turns the flags into indices.
// One launch for a series of one tile, two for longer ones (before: one launch for the
// statistic and one for each doubling, each a pass over memory: 10 launches and 75 us for
// 1.4 million windows at h = 64, now 2 and 15 us).  Long integrations may be a launch of their own
// before it (launch_integrate); clusters too long for a tile take the separate passes below.
#include <math.h>

#include <algorithm>

#include "afg_internal.cuh"

namespace {

__global__ void k_integrate(const float *__restrict__ z, int64_t n_out, int n_int, float *__restrict__ stat) {
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n_out) return;
    float s = 0.f;
    for (int i = 0; i < n_int; ++i) s += z[j + i];
    stat[j] = s / (float)n_int;
}

// ---- one tile: CL_N indices by CL_T threads.  Shared memory: logits of the tile and its halo, then two rows of
// CL_N + 2 h statistics (-inf outside the series).  With M_k[i] = max P[i .. i + 2^k) and 2^k <= h < 2^(k+1), each
// half-window is the union of two overlapping 2^k windows.
constexpr int CL_N = 1024, CL_T = 256;
constexpr int CL_H = 1024;    // largest half-width
constexpr int CL_INT = 1024;  // largest integration
constexpr int CL_SUMS = 8192; // tiles whose counts a writing block adds up itself

inline size_t cluster_smem(int h, int n_int) { return (size_t)(3 * (CL_N + 2 * h) + n_int) * sizeof(float); }

// Trigger indices of flag words (index 32 w + bit) from position `pos` on
__device__ __forceinline__ void put_triggers(uint32_t m, int64_t j, int64_t pos, int64_t *idx, int64_t cap) {
    for (; m; m &= m - 1, ++pos)
        if (pos < cap) idx[pos] = j + __ffs(m) - 1;
}

__device__ __forceinline__ float max_nan(float a, float b) {  // NaN if either is
    float d;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}

// z: logits, or (stat null, n_int 1) the statistic itself.
// NAN_STOPS (series of at most CL_DIRECT indices, half-widths up to CL_DIRECT_H): an index with a NaN within h of it
// is no trigger, and a side without any index is no condition; else NaNs count as -inf unless a whole side is NaN (then
// no trigger), and so do missing sides.
constexpr int64_t CL_DIRECT = 16384;
constexpr int CL_DIRECT_H = 256;

template <bool NAN_STOPS>
__global__ void __launch_bounds__(CL_T) k_cluster(const float *z, int64_t n_out, int n_int, int h,
                                                  float *__restrict__ stat, uint32_t *__restrict__ flags,
                                                  int *__restrict__ counts, int64_t *__restrict__ idx, int64_t cap,
                                                  int64_t *__restrict__ n_trig) {
    extern __shared__ float cs[];
    __shared__ uint32_t words[CL_N / 32];
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t j0 = (int64_t)blockIdx.x * CL_N;
    const int len = CL_N + 2 * h;
    float *zl = cs, *A = cs + len + n_int, *B = A + len;
    const int64_t n_win = n_out + n_int - 1;
    pdl_wait();  // the logits
    pdl_trigger();
    for (int i = tid; i < len + n_int - 1; i += CL_T) {
        const int64_t j = j0 - h + i;
        zl[i] = j >= 0 && j < n_win ? z[j] : 0.f;
    }
    __syncthreads();
    for (int i = tid; i < len; i += CL_T) {
        const int64_t j = j0 - h + i;
        float v = -INFINITY;
        if (j >= 0 && j < n_out) {
            float s = 0.f;
            for (int q = 0; q < n_int; ++q) s += zl[i + q];
            v = s / (float)n_int;
            if (stat && i >= h && i < h + CL_N) stat[j] = v;
        }
        A[i] = v;
    }
    __syncthreads();
    float own[CL_N / CL_T];
#pragma unroll
    for (int q = 0; q < CL_N / CL_T; ++q) own[q] = A[h + tid + q * CL_T];
    int w = 1, m = len;
    for (; 2 * w <= h; w *= 2) {
        m -= w;
        for (int i = tid; i < m; i += CL_T) B[i] = NAN_STOPS ? max_nan(A[i], A[i + w]) : fmaxf(A[i], A[i + w]);
        __syncthreads();
        float *t = A;
        A = B;
        B = t;
    }
#pragma unroll
    for (int q = 0; q < CL_N / CL_T; ++q) {
        const int i = tid + q * CL_T, p = i + h;
        bool f = j0 + i < n_out;
        if (h > 0 && NAN_STOPS) {
            const int64_t j = j0 + i;
            f = f && (j == 0 || own[q] > max_nan(A[p - h], A[p - w])) &&
                (j == n_out - 1 || own[q] >= max_nan(A[p + 1], A[p + h - w + 1]));
        } else if (h > 0) {
            f = f && own[q] > fmaxf(A[p - h], A[p - w]) && own[q] >= fmaxf(A[p + 1], A[p + h - w + 1]);
        }
        const uint32_t b = __ballot_sync(0xffffffffu, f);
        if (lane == 0) words[i >> 5] = b;
    }
    __syncthreads();
    if (tid < 32) {
        const uint32_t b = words[tid];
        int c = __popc(b);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, c, o);
            if (lane >= o) c += y;
        }
        if (gridDim.x == 1) {
            put_triggers(b, 32 * tid, c - __popc(b), idx, cap);
            if (tid == 31) *n_trig = c;
        } else {
            flags[(int64_t)blockIdx.x * 32 + tid] = b;
            if (tid == 31) counts[blockIdx.x] = c;
        }
    }
}

// grid (tiles): the tile's triggers behind those of the tiles before it.  counts: of every tile, added up here, or
// (scanned) already an exclusive sum with the total written.
__global__ void __launch_bounds__(CL_T) k_cluster_write(const uint32_t *flags, const int *counts,
                                                        int scanned, int64_t *__restrict__ idx, int64_t cap,
                                                        int64_t *__restrict__ n_trig) {
    __shared__ int64_t sum[CL_T / 32];
    const int tid = threadIdx.x, lane = tid & 31, t = blockIdx.x;
    int64_t s = 0;
    pdl_wait();  // flags and counts
    if (!scanned) {
        for (int i = tid; i < t; i += CL_T) s += counts[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) sum[tid >> 5] = s;
        __syncthreads();
    }
    if (tid >= 32) return;
    if (scanned) {
        s = counts[t];
    } else {
        s = 0;
        for (int i = 0; i < CL_T / 32; ++i) s += sum[i];
    }
    const uint32_t b = flags[(int64_t)t * 32 + tid];
    int c = __popc(b);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, c, o);
        if (lane >= o) c += y;
    }
    put_triggers(b, (int64_t)t * CL_N + 32 * tid, s + c - __popc(b), idx, cap);
    if (!scanned && tid == 31 && t == (int)gridDim.x - 1) *n_trig = s + c;
}

// ---- clustering: j is a trigger iff I[j] > max I[j-h .. j-1] and I[j] >= max I[j+1 .. j+h]
// (earliest index wins ties).  The statistic is padded with -inf on both sides (h each), so
// every window is full; M_k[i] = max P[i .. i + 2^k) is built by k doubling passes
// (2^k <= h < 2^(k+1)), and each half-window is the union of two overlapping 2^k windows.
constexpr int TB = 1024;  // indices per compaction block

__global__ void k_trig_pad(const float *__restrict__ I, int64_t n, int h, float *__restrict__ P) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n + 2 * (int64_t)h;
         i += (int64_t)gridDim.x * blockDim.x)
        P[i] = (i >= h && i < n + h) ? I[i - h] : -INFINITY;
}

__global__ void k_trig_double(const float *__restrict__ A, int64_t len, int64_t step, float *__restrict__ B) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < len; i += (int64_t)gridDim.x * blockDim.x)
        B[i] = fmaxf(A[i], A[i + step]);
}

// flags and per-block counts (M: level-k maxima of the padded statistic, or the statistic when h = 0)
__global__ void __launch_bounds__(TB) k_trig_flag(const float *__restrict__ I, const float *__restrict__ M,
                                                  int64_t n, int h, int64_t w, uint8_t *__restrict__ flag,
                                                  int *__restrict__ counts) {
    __shared__ int wc[TB / 32];
    const int64_t j = (int64_t)blockIdx.x * TB + threadIdx.x;
    int f = 0;
    if (j < n) {
        if (h == 0) {
            f = 1;
        } else {
            const int64_t p = j + h;  // padded index of j
            const float v = I[j];
            const float left = fmaxf(M[p - h], M[p - w]);
            const float right = fmaxf(M[p + 1], M[p + h - w + 1]);
            f = (v > left) && (v >= right);
        }
        flag[j] = (uint8_t)f;
    }
    const unsigned m = __ballot_sync(0xffffffffu, f);
    if ((threadIdx.x & 31) == 0) wc[threadIdx.x >> 5] = __popc(m);
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int i = 0; i < TB / 32; ++i) t += wc[i];
        counts[blockIdx.x] = t;
    }
}

// exclusive scan of the block counts (one block, fixed order) and the total
__global__ void __launch_bounds__(1024) k_trig_scan(int *__restrict__ counts, int nb, int64_t *__restrict__ n_trig) {
    __shared__ int64_t s[1024];
    __shared__ int64_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int c0 = 0; c0 < nb; c0 += 1024) {
        const int i = c0 + threadIdx.x;
        const int64_t v = i < nb ? counts[i] : 0;
        s[threadIdx.x] = v;
        __syncthreads();
        for (int o = 1; o < 1024; o <<= 1) {
            const int64_t t = threadIdx.x >= (unsigned)o ? s[threadIdx.x - o] : 0;
            __syncthreads();
            s[threadIdx.x] += t;
            __syncthreads();
        }
        if (i < nb) counts[i] = (int)(carry + s[threadIdx.x] - v);
        __syncthreads();
        if (threadIdx.x == 1023) carry += s[1023];
        __syncthreads();
    }
    if (threadIdx.x == 0) *n_trig = carry;
}

__global__ void __launch_bounds__(TB) k_trig_write(const uint8_t *__restrict__ flag, int64_t n,
                                                   const int *__restrict__ base, int64_t *__restrict__ idx,
                                                   int64_t cap) {
    __shared__ int wc[TB / 32];
    const int64_t j = (int64_t)blockIdx.x * TB + threadIdx.x;
    const int f = j < n ? flag[j] : 0;
    const unsigned m = __ballot_sync(0xffffffffu, f);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) wc[wid] = __popc(m);
    __syncthreads();
    int before = 0;
    for (int i = 0; i < wid; ++i) before += wc[i];
    if (f) {
        const int64_t pos = (int64_t)base[blockIdx.x] + before + __popc(m & ((1u << lane) - 1u));
        if (pos < cap) idx[pos] = j;
    }
}

}  // namespace

int launch_integrate(afg_ctx *ctx, const float *logits, int64_t n_win, int n_int, int cluster_half, float *stat,
                     int64_t *trig_idx, int64_t trig_cap, int64_t *n_trig, cudaStream_t st) {
    const int64_t n_out = n_win - n_int + 1;
    const int h = cluster_half;
    const int64_t tiles = (n_out + CL_N - 1) / CL_N;
    if (n_out > 0 && h <= CL_H && tiles <= 0x7fffffff) {
        // The statistic first: integrations past a tile's, and long ones where a tile would form the sums of h > 256
        // indices to each side again (1.4 million windows, 1024 each: 234 us apart or together at h = 256, 249 and 459 at
        // 1024; 128 each: 58 and 82).  Short integrations stay together, a launch less.
        const bool apart = n_int > CL_INT || (h > 256 && n_int >= 128);
        void *pf = nullptr, *pc = nullptr;
        if (tiles > 1) {
            int rc = afg_ws_reserve(ctx, WS_TRIG_FLAG, (size_t)tiles * 32 * sizeof(uint32_t), &pf);
            if (!rc) rc = afg_ws_reserve(ctx, WS_TRIG_COUNT, (size_t)tiles * sizeof(int), &pc);
            if (rc) return rc;
        }
        uint32_t *flags = static_cast<uint32_t *>(pf);
        int *counts = static_cast<int *>(pc);
        {
            KScope ks(ctx, st, KK_INTEGRATE, (double)n_out * n_int, (double)(n_win + n_out) * 4.0);
            if (apart) k_integrate<<<(unsigned)((n_out + 255) / 256), 256, 0, st>>>(logits, n_out, n_int, stat);
            const int ni = apart ? 1 : n_int;
            AFG_CUDA(ctx, launch_pdl(n_out <= CL_DIRECT && h <= CL_DIRECT_H ? k_cluster<true> : k_cluster<false>,
                                     dim3((unsigned)tiles), dim3(CL_T), cluster_smem(h, ni), st,
                                     (const float *)(apart ? stat : logits), n_out, ni, h, apart ? nullptr : stat, flags,
                                     counts, trig_idx, trig_cap, n_trig));
        }
        AFG_LAUNCH_CHECK(ctx, "k_cluster");
        if (tiles > 1) {
            KScope ks(ctx, st, KK_TRIGGERS, 0.0, (double)n_out / 8.0);
            const int scanned = tiles > CL_SUMS;
            if (scanned) k_trig_scan<<<1, 1024, 0, st>>>(counts, (int)tiles, n_trig);
            AFG_CUDA(ctx, launch_pdl(k_cluster_write, dim3((unsigned)tiles), dim3(CL_T), 0, st, (const uint32_t *)flags,
                                     (const int *)counts, scanned, trig_idx, trig_cap, n_trig));
        }
        AFG_LAUNCH_CHECK(ctx, "k_cluster_write");
        return AFG_OK;
    }
    {
        KScope ks(ctx, st, KK_INTEGRATE, (double)n_out * n_int, (double)(n_win + n_out) * 4.0);
        k_integrate<<<(unsigned)((n_out + 255) / 256), 256, 0, st>>>(logits, n_out, n_int, stat);
    }
    AFG_LAUNCH_CHECK(ctx, "k_integrate");
    if (n_out <= 0) {
        AFG_CUDA(ctx, cudaMemsetAsync(n_trig, 0, sizeof(int64_t), st));
        return AFG_OK;
    }
    int k = 0;
    while (h > 0 && ((int64_t)2 << k) <= h) ++k;  // 2^k <= h < 2^(k+1)
    const int64_t w = h > 0 ? ((int64_t)1 << k) : 0;
    const int64_t N = n_out + 2 * (int64_t)h;
    const int nb = (int)((n_out + TB - 1) / TB);
    void *pa = nullptr, *pb = nullptr, *pf = nullptr, *pc = nullptr;
    int rc = afg_ws_reserve(ctx, WS_TRIG_A, (size_t)N * sizeof(float), &pa);
    if (!rc && h > 0) rc = afg_ws_reserve(ctx, WS_TRIG_B, (size_t)N * sizeof(float), &pb);
    if (!rc) rc = afg_ws_reserve(ctx, WS_TRIG_FLAG, (size_t)n_out, &pf);
    if (!rc) rc = afg_ws_reserve(ctx, WS_TRIG_COUNT, (size_t)nb * sizeof(int), &pc);
    if (rc) return rc;
    float *A = static_cast<float *>(pa), *B = static_cast<float *>(pb);
    const unsigned g = (unsigned)std::min<int64_t>((N + 255) / 256, 152 * 32);
    {
        KScope ks(ctx, st, KK_TRIGGERS, 0.0, (double)n_out * 4.0 * (3 + 2 * k));
        const float *M = stat;
        if (h > 0) {
            k_trig_pad<<<g, 256, 0, st>>>(stat, n_out, h, A);
            int64_t len = N;
            for (int l = 1; l <= k; ++l) {  // M_l[i] = max(M_{l-1}[i], M_{l-1}[i + 2^(l-1)])
                const int64_t step = (int64_t)1 << (l - 1);
                len -= step;
                k_trig_double<<<g, 256, 0, st>>>(A, len, step, B);
                std::swap(A, B);
            }
            M = A;
        }
        uint8_t *flag = static_cast<uint8_t *>(pf);
        int *counts = static_cast<int *>(pc);
        k_trig_flag<<<nb, TB, 0, st>>>(stat, M, n_out, h, w, flag, counts);
        k_trig_scan<<<1, 1024, 0, st>>>(counts, nb, n_trig);
        k_trig_write<<<nb, TB, 0, st>>>(flag, n_out, counts, trig_idx, trig_cap);
    }
    AFG_LAUNCH_CHECK(ctx, "k_triggers");
    return AFG_OK;
}
