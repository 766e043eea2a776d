// The 16-channel one-stage network in FP32 (Sec. II network, Sec. IX: kernel length 3, global pooling), whole
// windows at a time: one window per cluster of two CTAs, its activations in shared memory from the stem to the logit.
//
// CTA r of a cluster owns positions [r W/2, (r + 1) W/2): a block's input X and its hidden activation H, 16 channels
// each, in 198 KB.  A thread takes 4 positions of all 16 channels (64 sums), so that a layer reads each activation
// three times and its weights as broadcasts, 96 packed FMAs per 15 shared-memory reads.  GroupNorm: channel sums and
// then the centred squares over the CTA, combined with the other CTA's (Chan, Golub and LeVeque's update of mean and
// centred sum) through distributed shared memory, with the neighbour's boundary row for the halo: one cluster barrier
// per layer.
//
// Bound by the FP32 pipe (9 k clocks a layer of 16 -> 16 channels, 3 taps, 1536 positions).  3601 windows: 6.0 ms as
// one launch per convolution and GroupNorm (each activation written and read through memory, the stem with integer
// divisions per output), 1.89 ms here.  The FMA pipe is 57 % busy: reductions and the cluster barrier
// stand between the layers' sums.  Four CTAs of a quarter each, two on an SM: 2.2 ms at best (more reductions per
// position, and 74 of 76 clusters fit).
#include <algorithm>

#include "afg_internal.cuh"

namespace {

constexpr int T32_T = 384;                 // threads: 4 positions each
constexpr int T32_HALF = 4 * T32_T;        // positions of a CTA at most
constexpr int T32_C = 16;
constexpr int T32_LD = T32_HALF + 8;       // row: 4 slots (the last is position -1), positions, position W/2
constexpr int T32_WARPS = T32_T / 32;
constexpr int T32_KMAX = 7;

struct T32Smem {
    float x[T32_C * T32_LD], h[T32_C * T32_LD];
    float raw[2][2 * T32_LD];              // samples of this window and the next, position t at 4 + t (|halo| <= 3)
    float w[3 * T32_C * T32_C];            // weights of the current layer, [tap][in][out] (stem: [in][tap][out])
    float red[2][T32_WARPS * T32_C];       // warps' channel sums
    float peer[2][3 * T32_C];              // from the other CTA, by layer parity: mean, centred sum, boundary row
};

struct T32Args {
    const float *y;
    int64_t n_y, y_stride, first, stride, shift, n_win;
    float *logits;
    const float *stem, *sg, *sb;           // stem weights [16][2][k], gamma, beta
    const float *conv[2 * 64], *gamma[2 * 64], *beta[2 * 64];
    const float *fc_w, *fc_b;
    int n_conv, k, half, lcg;              // convolutions after the stem, stem taps, W / 2, log2 channels per group
    float eps;
};

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void st_peer(float *local, uint32_t rank, float v) {  // the same variable of CTA `rank`
    uint32_t a = (uint32_t)__cvta_generic_to_shared(local), p;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(p) : "r"(a), "r"(rank));
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(p), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}

// Sums over the warp of 16 per-lane values: lanes l and l + 16 end with the total of value l.
__device__ __forceinline__ float reduce16(float (&v)[16], int lane) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < o; ++i) {
            const float send = up ? v[i] : v[i + o], keep = up ? v[i + o] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 16);
}
// Channel lane & 15's total over the CTA from the warps' sums, then over its group
__device__ __forceinline__ float group_total(const float *red, int lane, int lcg) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < T32_WARPS; ++w) s += red[w * T32_C + (lane & 15)];
    for (int o = 1; o < (1 << lcg); o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

__global__ void __launch_bounds__(T32_T, 1) k_tiny32(const T32Args a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T32Smem &sm = *reinterpret_cast<T32Smem *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t rank = cluster_rank();
    const int half = a.half, t0 = 4 * tid, pad = a.k / 2;
    const bool live = t0 < half;  // (half is a multiple of 16: a thread's 4 positions are all in or all out)
    const float cnt = (float)half * (float)(1 << a.lcg);  // values of a group in one CTA
    const int64_t n_clusters = gridDim.x / 2;

    // samples [-pad, half + pad) of this CTA's half of window win, zero outside the window
    auto fetch = [&](int64_t win, float *raw) {
        const int64_t start = a.first + win * a.stride;
        for (int i = tid; i < 2 * (half + 2 * pad); i += T32_T) {
            const int ci = i >= half + 2 * pad, t = i - ci * (half + 2 * pad) - pad, g = (int)rank * half + t;
            float *dst = raw + ci * T32_LD + 4 + t;
            if (g < 0 || g >= 2 * half) {
                *dst = 0.f;
                continue;
            }
            int64_t p = start + g;
            const float *row = a.y;
            if (ci) {
                p += a.shift;
                if (p >= a.n_y) p -= a.n_y;
                row += a.y_stride;
            }
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(row + p)
                         : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto load_weights = [&](const float *w) {
        for (int i = tid; i < 3 * T32_C * T32_C / 4; i += T32_T)
            reinterpret_cast<float4 *>(sm.w)[i] = __ldg(reinterpret_cast<const float4 *>(w) + i);
    };
    auto load_stem = [&]() {
        for (int i = tid; i < 2 * a.k * T32_C; i += T32_T) sm.w[i] = a.stem[(i % T32_C) * 2 * a.k + i / T32_C];
    };

    int buf = 0;
    uint32_t layer = 0;  // parity of the exchange slots, over all windows
    int64_t win = blockIdx.x / 2;
    if (win < a.n_win) {
        fetch(win, sm.raw[0]);
        load_stem();
    }
    // outer halo columns stay zero for good: position -1 of CTA 0, position half of CTA 1
    if (tid < T32_C) {
        const int s = tid * T32_LD + (rank == 0 ? 3 : 4 + half);
        sm.x[s] = 0.f;
        sm.h[s] = 0.f;
    }
    cluster_sync_all();  // both CTAs have started: their shared memory may be written
    for (; win < a.n_win; win += n_clusters, buf ^= 1) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        if (win + n_clusters < a.n_win) fetch(win + n_clusters, sm.raw[buf ^ 1]);
        float2 acc[8][4];
        // layer 0: stem -> X; odd: X -> H; even: H -> X with X added
        for (int l = 0; l <= a.n_conv; ++l, ++layer) {
            const bool to_h = (l & 1) != 0;
#pragma unroll
            for (int c = 0; c < 8; ++c)
#pragma unroll
                for (int p = 0; p < 4; ++p) acc[c][p] = make_float2(0.f, 0.f);
            if (live && l == 0) {
                for (int ci = 0; ci < 2; ++ci) {
                    const float *xr = sm.raw[buf] + ci * T32_LD + 4 + t0 - pad;
                    for (int r = 0; r < a.k; ++r) {
                        const float4 *wp = reinterpret_cast<const float4 *>(sm.w + (ci * a.k + r) * T32_C);
#pragma unroll
                        for (int p = 0; p < 4; ++p) {
                            const float2 xx = make_float2(xr[r + p], xr[r + p]);
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                const float4 w4 = wp[c];
                                acc[2 * c][p] = __ffma2_rn(xx, make_float2(w4.x, w4.y), acc[2 * c][p]);
                                acc[2 * c + 1][p] = __ffma2_rn(xx, make_float2(w4.z, w4.w), acc[2 * c + 1][p]);
                            }
                        }
                    }
                }
            } else if (live) {
                const float *in = (to_h ? sm.x : sm.h) + 4 + t0;
#pragma unroll 2
                for (int ci = 0; ci < T32_C; ++ci) {
                    const float *row = in + ci * T32_LD;
                    const float4 m = *reinterpret_cast<const float4 *>(row);
                    const float x[6] = {row[-1], m.x, m.y, m.z, m.w, row[4]};
#pragma unroll
                    for (int r = 0; r < 3; ++r) {
                        const float4 *wp = reinterpret_cast<const float4 *>(sm.w + (r * T32_C + ci) * T32_C);
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const float4 w4 = wp[c];
#pragma unroll
                            for (int p = 0; p < 4; ++p) {
                                const float2 xx = make_float2(x[r + p], x[r + p]);
                                acc[2 * c][p] = __ffma2_rn(xx, make_float2(w4.x, w4.y), acc[2 * c][p]);
                                acc[2 * c + 1][p] = __ffma2_rn(xx, make_float2(w4.z, w4.w), acc[2 * c + 1][p]);
                            }
                        }
                    }
                }
            }
            // ---- GroupNorm statistics: mean over the CTA, centred squares over the CTA, then both CTAs
            const float *gam = l ? a.gamma[l - 1] : a.sg, *bet = l ? a.beta[l - 1] : a.sb;
            const float g1 = __ldg(gam + (lane & 15)), b1 = __ldg(bet + (lane & 15));
            float v[16];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const float2 s = __fadd2_rn(__fadd2_rn(acc[c][0], acc[c][1]), __fadd2_rn(acc[c][2], acc[c][3]));
                v[2 * c] = s.x;
                v[2 * c + 1] = s.y;
            }
            float t = reduce16(v, lane);
            if (lane < 16) sm.red[0][warp * T32_C + lane] = t;
            __syncthreads();  // (also: every read of the weights and of the layer's input is done)
            if (l < a.n_conv) load_weights(a.conv[l]);
            else load_stem();  // of the next window
            const float mean = group_total(sm.red[0], lane, a.lcg) / cnt;  // of channel lane & 15's group
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const float m0 = __shfl_sync(0xffffffffu, mean, 2 * c), m1 = __shfl_sync(0xffffffffu, mean, 2 * c + 1);
                const float2 nm = make_float2(-m0, -m1);
                float2 s = make_float2(0.f, 0.f);
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const float2 d = __fadd2_rn(acc[c][p], nm);
                    s = __ffma2_rn(d, d, s);
                }
                v[2 * c] = live ? s.x : 0.f;
                v[2 * c + 1] = live ? s.y : 0.f;
            }
            t = reduce16(v, lane);
            if (lane < 16) sm.red[1][warp * T32_C + lane] = t;
            // the boundary row the other CTA needs: its neighbour position's raw sums
            float *slot = sm.peer[layer & 1];
            const int edge = rank == 0 ? half - 4 : 0;
            if (t0 == edge && live) {
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float2 e = rank == 0 ? acc[c][3] : acc[c][0];
                    st_peer(slot + 2 * T32_C + 2 * c, rank ^ 1, e.x);
                    st_peer(slot + 2 * T32_C + 2 * c + 1, rank ^ 1, e.y);
                }
            }
            __syncthreads();
            const float m2 = group_total(sm.red[1], lane, a.lcg);
            if (warp == 0 && lane < 16) {
                st_peer(slot + lane, rank ^ 1, mean);
                st_peer(slot + T32_C + lane, rank ^ 1, m2);
            }
            cluster_sync_all();
            const float om = slot[lane & 15], d = mean - om;
            const float var = (m2 + slot[T32_C + (lane & 15)] + d * d * (0.5f * cnt)) / (2.f * cnt);
            const float sc = rsqrtf(var + a.eps) * g1, sh = b1 - 0.5f * (mean + om) * sc;
            // ---- normalise (+ residual), ReLU
            float *dst = to_h ? sm.h : sm.x;
            const bool res = l > 0 && !to_h;
            const bool last = l == a.n_conv;
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                const float s = __shfl_sync(0xffffffffu, sc, c), b = __shfl_sync(0xffffffffu, sh, c);
                if (!live) continue;
                float o[4];
#pragma unroll
                for (int p = 0; p < 4; ++p) o[p] = fmaf((c & 1) ? acc[c / 2][p].y : acc[c / 2][p].x, s, b);
                float4 *q = reinterpret_cast<float4 *>(dst + c * T32_LD + 4 + t0);
                if (res) {
                    const float4 r = *q;
                    o[0] += r.x;
                    o[1] += r.y;
                    o[2] += r.z;
                    o[3] += r.w;
                }
#pragma unroll
                for (int p = 0; p < 4; ++p) o[p] = fmaxf(o[p], 0.f);
                if (last) v[c] = (o[0] + o[1]) + (o[2] + o[3]);
                else *q = make_float4(o[0], o[1], o[2], o[3]);
            }
            if (warp == 0 && lane < 16 && !last) {  // inner halo column
                float *q = dst + lane * T32_LD + (rank == 0 ? 4 + half : 3);
                *q = fmaxf(fmaf(slot[2 * T32_C + lane], sc, sh) + (res ? *q : 0.f), 0.f);
            }
            if (!last) {
                __syncthreads();
                continue;
            }
            // ---- head: channel means over both CTAs, linear
#pragma unroll
            for (int c = 0; c < 16; ++c)
                if (!live) v[c] = 0.f;
            t = reduce16(v, lane);
            if (lane < 16) sm.red[0][warp * T32_C + lane] = t;
            __syncthreads();
            ++layer;
            slot = sm.peer[layer & 1];
            if (warp == 0) {
                t = group_total(sm.red[0], lane, 0);
                if (lane < 16) st_peer(slot + lane, rank ^ 1, t);
            }
            cluster_sync_all();
            if (warp == 0 && rank == 0) {
                float z = __ldg(a.fc_w + (lane & 15)) * ((t + slot[lane & 15]) / (float)(2 * half));
                float s = __ldg(a.fc_b);
#pragma unroll
                for (int c = 0; c < 16; ++c) s += __shfl_sync(0xffffffffu, z, c);
                if (lane == 0) a.logits[win] = s;
            }
        }
    }
    cluster_sync_all();  // no CTA leaves while the other may still write to it
}

}  // namespace

// The 16-channel one-stage networks whose window fits: stem stride 1 without pooling, at most 3072 positions.
bool net_tiny32_fits(const afg_ctx *ctx) {
    const afg_net &n = ctx->plan.net;
    const int W = ctx->cfg.win_len;
    return n.n_stages == 1 && n.widths[0] == T32_C && n.stem_stride == 1 && !n.stem_pool && n.stem_k <= T32_KMAX &&
           W % 32 == 0 && W <= 2 * T32_HALF && ctx->plan.convs.size() <= 1 + 2 * 64 && T32_C % n.groups == 0;
}

int launch_infer_tiny32(afg_ctx *ctx, const float *y, int64_t n_y, int64_t y_stride, int64_t first, int64_t stride,
                        int64_t n_win, int64_t shift, float *logits, cudaStream_t st) {
    const NetPlan &P = ctx->plan;
    const ConvLayer &S = P.convs[0];
    T32Args a = {};
    a.y = y;
    a.n_y = n_y;
    a.y_stride = y_stride;
    a.first = first;
    a.stride = stride;
    a.shift = shift;
    a.n_win = n_win;
    a.logits = logits;
    a.stem = S.wt;
    a.sg = S.gamma;
    a.sb = S.beta;
    a.n_conv = (int)P.convs.size() - 1;
    double flops = 2.0 * S.lout * S.cout * S.cin * S.k;
    for (int i = 0; i < a.n_conv; ++i) {
        const ConvLayer &C = P.convs[i + 1];
        a.conv[i] = C.wt;
        a.gamma[i] = C.gamma;
        a.beta[i] = C.beta;
        flops += 2.0 * C.lout * C.cout * C.k * C.cin;
    }
    a.fc_w = P.fc_w;
    a.fc_b = P.fc_b;
    a.k = S.k;
    a.half = ctx->cfg.win_len / 2;
    for (a.lcg = 0; (P.net.groups << a.lcg) < T32_C; ++a.lcg) {
    }
    a.eps = P.net.eps;
    int sms = 0;
    AFG_CUDA(ctx, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device));
    AFG_CUDA(ctx, cudaFuncSetAttribute(k_tiny32, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(T32Smem)));
    KScope ks(ctx, st, KK_TINY32, flops * n_win, 8.0 * n_win * ctx->cfg.win_len);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2u * (unsigned)std::min<int64_t>(n_win, std::max(1, sms / 2)));
    cfg.blockDim = dim3(T32_T);
    cfg.dynamicSmemBytes = sizeof(T32Smem);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    AFG_CUDA(ctx, cudaLaunchKernelEx(&cfg, k_tiny32, a));
    return AFG_OK;
}
