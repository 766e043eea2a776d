// FP32 1D ResNet with GroupNorm on the tensor cores (Sec. II network, widths 64..512): every
// convolution after the stem is an implicit GEMM of BF16 products whose sum is the FP32 product to 2^-26 or so.
//
// A float is the sum of three BF16 values (8 significant bits each: 24 in all), x = x1 + x2 + x3,
// x1 = bf16(x), x2 = bf16(x - x1), x3 = x - x1 - x2: exactly for |x| from 2^-110 to the largest float (x1 is
// held at the largest BF16 number), and to 2^-134, half of BF16's smallest, below.  The product of two floats is the
// nine products x_i w_j, each exact in FP32; the six with i + j <= 4 are formed, the other three are below 2^-26 of
// |x w|.  FP32 SIMT FMAs run at 80 TFLOP/s on this GPU, six BF16 products at 1950 / 6 = 325 (k_conv_fp32
// of net_fp32.cu, at 78 % of the FP32 pipe, and its GroupNorm took 73.4 ms for 1920 ResNet34 windows and
// 14.2 ms for 333; this path takes 23.9 and 4.44, and its logits are closer to 64-bit ones: norm of the difference
// over the norm, root mean square over 12 seeds, 2.0e-7 to 3.5e-7 for 1 to 200 windows against 6.4e-7 to 8.7e-7).
//
// Accumulation: the tensor core adds into FP32 but does not promise round-to-nearest, so no long sum is
// left to it.  Each stage (16 input channels x taps: 48 products a term) starts a fresh TMEM
// accumulator, the five small products first, so that the accumulator is at full size only for its last
// `taps` MMAs; the epilogue warps then add the stage's sums to FP32 registers with ordinary (nearest)
// adds, C_in / 16 of them in all against the 3 C_in roundings of an FMA chain.
//
// Layouts
//   activations  three BF16 planes, each chunk-major over all windows of a launch: [plane][C / 8][rows][8],
//                rows = n_win (L + 2) with a zero row before and after each window's, plus slack rows that
//                the last tile may read.  Input row h + r feeds tap r of output row h = w (L + 2) + t, so
//                a convolution is one GEMM over all rows; the two rows between windows compute unused
//                outputs.  A chunk is the no-swizzle K-major core-matrix layout of the tensor core.
//                Input of a stride-2 convolution: even padded rows, then odd ones, [plane][C / 8][2][rows][8],
//                rows = n_win (L_out + 1); taps 0, 1, 2 of h = w (L_out + 1) + t are even h, odd h, even h + 1.
//   raw          the convolution's output before GroupNorm, FP32 [C][hs] over the same rows h.
//   weights      BF16 planes in stage order: [slice][C_in / 16][plane][2][tap][128][8] (zero past C_out).
#include <algorithm>
#include <vector>

#include "afg_internal.cuh"
#include "tc_ptx.cuh"

namespace {

constexpr int SC_EPI_WARPS = 16;                // four per TMEM lane quarter
constexpr int SC_T = (SC_EPI_WARPS + 2) * 32;   // + producer and MMA issuer
constexpr int SC_KB = 16;                       // input channels per stage
constexpr int SC_MAX_STAGES = 4;
constexpr uint64_t SC_WAIT_NS = 2000000000ull;
constexpr int SC_SLACK = 264;                   // rows past the last that a tile may read (256 + 2, rounded up)
constexpr uint32_t SC_SMEM = 226 * 1024;

// MODE 0: 3 taps, stride 1; 1: 3 taps, stride 2; 2: 1 tap, stride 2 (the shortcut)
template <int TN, int MODE>
struct SplitGeo {
    static constexpr int TAPS = MODE == 2 ? 1 : 3;
    static constexpr int ROWS = MODE == 0 ? TN + 2 : MODE == 1 ? 2 * TN + 2 : TN;  // rows of a chunk in shared memory
    static constexpr uint32_t CHUNK = ROWS * 16;
    static constexpr uint32_t ACT = 6 * CHUNK;                 // 3 planes x 2 chunks
    static constexpr uint32_t W = 6 * TAPS * 128 * 16;         // 3 planes x 2 chunks x taps x 128 channels
    static constexpr uint32_t STAGE = ACT + W;
    static constexpr uint32_t TX = W + 6 * 16 * (MODE == 0 ? TN + 2 : MODE == 1 ? 2 * TN + 1 : TN);
    static constexpr int NS = (int)(SC_SMEM / STAGE) < SC_MAX_STAGES ? (int)(SC_SMEM / STAGE) : SC_MAX_STAGES;
    static constexpr uint32_t BYTES = NS * STAGE + 256;
    static_assert(NS >= 2, "at least two stages");
};

struct SplitConvArgs {
    const unsigned char *wimg;
    const __nv_bfloat16 *in;
    int64_t in_ps, in_cs, in_odd;  // elements from one plane, chunk to the next; from the even rows to the odd
    float *raw;
    int64_t hs;
    int cout, n_kb, slices, n_tiles;
    int *err;
};

__device__ __forceinline__ bool sc_wait(uint64_t *bar, uint32_t parity, int *abort_flag, int *err) {
    if (tc::mbar_wait(bar, parity, SC_WAIT_NS)) return true;
    atomicExch(err, 1);
    *(volatile int *)abort_flag = 1;
    return false;
}

// One tile: 128 output channels (TMEM lanes) x TN rows (columns).  Per stage the 6 TAPS MMAs of
// 128 x TN x 16 read 4 KB + 32 TN B of shared memory each, 96 B/clk at TN = 256, and 62 KB are copied in
// (27 B/clk): under the 128 B/clk of shared memory.  Narrower tiles are chosen by tile_rows.
template <int TN, int MODE>
__global__ void __launch_bounds__(SC_T, 1) k_conv_split(const SplitConvArgs a) {
    using G = SplitGeo<TN, MODE>;
    extern __shared__ __align__(1024) unsigned char sm[];
    uint64_t *full = reinterpret_cast<uint64_t *>(sm + G::NS * G::STAGE);
    uint64_t *empty = full + SC_MAX_STAGES;
    uint64_t *acc_full = empty + SC_MAX_STAGES;  // [2]
    uint64_t *acc_empty = acc_full + 2;          // [2]
    uint64_t *drain = acc_empty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drain + 1);
    int *abort_flag = reinterpret_cast<int *>(tmem_slot + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (tid == 0) {
        for (int i = 0; i < G::NS; ++i) {
            tc::mbar_init(&full[i], 1);
            tc::mbar_init(&empty[i], 1);
        }
        for (int b = 0; b < 2; ++b) {
            tc::mbar_init(&acc_full[b], 1);
            tc::mbar_init(&acc_empty[b], SC_EPI_WARPS);
        }
        tc::mbar_init(drain, 1);
        tc::fence_mbar_init();
        *abort_flag = 0;
    }
    if (warp == 1) {
        tc::tmem_alloc(tmem_slot, 512);
        tc::tmem_relinquish();
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tmem_slot;
    pdl_trigger();
    pdl_wait();  // (a programmatic dependent of the GroupNorm before: the set-up overlaps its tail)

    if (warp == 0) {
        // ------------------------------------------------------------ producer
        uint32_t k = 0;
        bool stop = false;
        for (int t = blockIdx.x; t < a.n_tiles && !stop; t += gridDim.x) {
            const int slice = t % a.slices;
            const int64_t h0 = (int64_t)(t / a.slices) * TN;
            for (int kb = 0; kb < a.n_kb; ++kb, ++k) {
                const int s = k % G::NS;
                unsigned char *wsm = sm + (size_t)s * G::STAGE, *act = wsm + G::W;
                int ok = 1;
                if (lane == 0) {
                    if (*(volatile int *)abort_flag ||
                        (k >= (uint32_t)G::NS && !sc_wait(&empty[s], ((k / G::NS) - 1) & 1, abort_flag, a.err))) {
                        ok = 0;
                    } else {
                        tc::mbar_expect_tx(&full[s], G::TX);
                        const unsigned char *src = a.wimg + ((size_t)slice * a.n_kb + kb) * G::W;
                        for (uint32_t o = 0; o < G::W; o += 12288) tc::bulk_load(wsm + o, src + o, 12288, &full[s]);
                    }
                }
                if (!__shfl_sync(0xffffffffu, ok, 0)) {
                    stop = true;
                    break;
                }
                if (lane < (MODE == 1 ? 12 : 6)) {  // lane = (odd, plane, chunk)
                    const int pc = lane % 6, odd = MODE == 2 ? 1 : lane / 6;
                    const __nv_bfloat16 *src = a.in + (pc >> 1) * a.in_ps + (int64_t)(2 * kb + (pc & 1)) * a.in_cs + h0 * 8 +
                                               (odd ? a.in_odd : 0);
                    unsigned char *dst = act + pc * G::CHUNK + (MODE == 1 && odd ? (TN + 2) * 16 : 0);
                    const uint32_t rows = MODE == 0 ? TN + 2 : (MODE == 1 && !odd) ? TN + 1 : TN;
                    tc::bulk_load(dst, src, rows * 16, &full[s]);
                }
            }
        }
        if (lane == 0 && *(volatile int *)abort_flag)  // gave up: no copy may still be in flight at the exit
            for (uint32_t j = k > (uint32_t)G::NS ? k - G::NS : 0; j < k; ++j)
                tc::mbar_wait(&full[j % G::NS], (j / G::NS) & 1, SC_WAIT_NS);
    } else if (warp == 1) {
        // ------------------------------------------------------------ MMA issuer
        if (lane == 0) {
            constexpr uint32_t idesc = tc::idesc_bf16_f32(128, TN);
            uint32_t k = 0;
            bool stop = false;
            for (int t = blockIdx.x; t < a.n_tiles && !stop; t += gridDim.x)
                for (int kb = 0; kb < a.n_kb; ++kb, ++k) {
                    const int s = k % G::NS, buf = k & 1;
                    if (*(volatile int *)abort_flag || !sc_wait(&full[s], (k / G::NS) & 1, abort_flag, a.err) ||
                        (k >= 2 && !sc_wait(&acc_empty[buf], ((k >> 1) - 1) & 1, abort_flag, a.err))) {
                        stop = true;
                        break;
                    }
                    tc::fence_after_sync();
                    const uint32_t wb = tc::smem_addr(sm + (size_t)s * G::STAGE), ab = wb + G::W;
                    const uint64_t wd0 = tc::desc_kmajor_noswizzle(wb, G::TAPS * 2048, 128);
                    const uint64_t ad0 = tc::desc_kmajor_noswizzle(ab, G::CHUNK, 128);
                    const uint32_t dt = tmem + (uint32_t)(buf * 256);
                    // planes (weight, activation) of the six products, smallest first
                    constexpr int PW[6] = {2, 0, 1, 1, 0, 0}, PA[6] = {0, 2, 1, 0, 1, 0};
#pragma unroll
                    for (int m = 0; m < 6; ++m)
#pragma unroll
                        for (int r = 0; r < G::TAPS; ++r) {
                            const uint32_t trow = MODE == 0 ? r : r == 1 ? TN + 2 : r == 2 ? 1 : 0;
                            tc::mma_bf16(dt, wd0 + (uint64_t)(PW[m] * G::TAPS * 256 + r * 128),
                                         ad0 + (uint64_t)(PA[m] * 2 * G::ROWS + trow), idesc, (m | r) ? 1u : 0u);
                        }
                    tc::mma_commit(&empty[s]);
                    tc::mma_commit(&acc_full[buf]);
                }
            if (*(volatile int *)abort_flag) {
                tc::mma_commit(drain);
                tc::mbar_wait(drain, 0, SC_WAIT_NS);
            }
        }
    } else {
        // ------------------------------------------------------------ epilogue
        // Warp e adds columns [COLS g, COLS (g + 1)), g = e / 4, of its 32 lanes, in the MMA fragment
        // layout: lane t holds channels t / 4 and 8 + t / 4 of each 16 at columns 2 (t % 4), + 1 of each
        // 8, so that a quad stores 32 contiguous bytes of a channel's row.
        constexpr int COLS = TN / 4, NB8 = COLS / 8;
        const int q = warp & 3, cg = (warp - 2) >> 2;
        const uint32_t tq = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(COLS * cg);
        float acc[2][NB8 * 4];
        uint32_t k = 0;
        bool stop = false;
        for (int t = blockIdx.x; t < a.n_tiles && !stop; t += gridDim.x) {
#pragma unroll
            for (int i = 0; i < NB8 * 4; ++i) acc[0][i] = acc[1][i] = 0.f;
            for (int kb = 0; kb < a.n_kb; ++kb, ++k) {
                const int buf = k & 1;
                if (!tc::mbar_wait_warp_tested(&acc_full[buf], (k >> 1) & 1, SC_WAIT_NS)) {
                    if (lane == 0) {
                        atomicExch(a.err, 1);
                        *(volatile int *)abort_flag = 1;
                    }
                    stop = true;
                    break;
                }
                tc::fence_after_sync();
                const uint32_t tb = tq + (uint32_t)(buf * 256);
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    // 32 columns at a time, then the 16 and the 8 that are left
                    const uint32_t th = tb + ((uint32_t)(16 * hf) << 16);
#pragma unroll
                    for (int b = 0; b < COLS / 32; ++b) {
                        uint32_t r[16];
                        tc::tmem_ld16x256b_x4_nowait(th + (uint32_t)(32 * b), r);
                        tc::tmem_wait_ld();
                        tc::tmem_regs_ready(r);
#pragma unroll
                        for (int i = 0; i < 16; ++i) acc[hf][16 * b + i] += __uint_as_float(r[i]);
                    }
                    if constexpr (COLS % 32 >= 16) {
                        constexpr int C0 = COLS / 32 * 32;
                        uint32_t r[8];
                        tc::tmem_ld16x256b_x2_nowait(th + C0, r);
                        tc::tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 8; ++i) asm volatile("" : "+r"(r[i]));  // (uses stay after the wait)
#pragma unroll
                        for (int i = 0; i < 8; ++i) acc[hf][C0 / 2 + i] += __uint_as_float(r[i]);
                    }
                    if constexpr (COLS % 16 == 8) {
                        constexpr int C0 = COLS / 16 * 16;
                        uint32_t r[4];
                        tc::tmem_ld16x256b_x1_nowait(th + C0, r);
                        tc::tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 4; ++i) asm volatile("" : "+r"(r[i]));
#pragma unroll
                        for (int i = 0; i < 4; ++i) acc[hf][C0 / 2 + i] += __uint_as_float(r[i]);
                    }
                }
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive(&acc_empty[buf]);
            }
            if (stop) break;
            const int c0 = (t % a.slices) * 128 + 32 * q;
            if (c0 < a.cout) {
                float *o = a.raw + (int64_t)(c0 + (lane >> 2)) * a.hs + (int64_t)(t / a.slices) * TN + COLS * cg +
                           2 * (lane & 3);
#pragma unroll
                for (int hf = 0; hf < 2; ++hf)
#pragma unroll
                    for (int i = 0; i < 2; ++i) {
                        float *oc = o + (int64_t)(16 * hf + 8 * i) * a.hs;
#pragma unroll
                        for (int g = 0; g < NB8; ++g)
                            *reinterpret_cast<float2 *>(oc + 8 * g) = make_float2(acc[hf][4 * g + 2 * i], acc[hf][4 * g + 2 * i + 1]);
                    }
            }
        }
    }
    tc::fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        tc::fence_after_sync();
        tc::tmem_dealloc(tmem, 512);
    }
}

// the three BF16 terms of two floats (lo in the low half of each word).  The first is at most the largest BF16 number: a
// float that rounds past it would leave x - inf.
__device__ __forceinline__ void split3(float lo, float hi, uint32_t &p1, uint32_t &p2, uint32_t &p3) {
    p1 = tc::pack_bf16x2_sat(lo, hi);
    lo -= __uint_as_float(p1 << 16);
    hi -= __uint_as_float(p1 & 0xffff0000u);
    p2 = tc::pack_bf16x2(lo, hi);
    lo -= __uint_as_float(p2 << 16);
    hi -= __uint_as_float(p2 & 0xffff0000u);
    p3 = tc::pack_bf16x2(lo, hi);
}

// Weight image of one convolution from wt [k][cin][cout] (the image is zeroed beforehand).
__global__ void k_split_weights(const float *__restrict__ wt, int cin, int cout, int k, __nv_bfloat16 *__restrict__ o) {
    const int n = k * cin * cout;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int co = i % cout, ci = i / cout % cin, r = i / cout / cin;
        const size_t blk = (size_t)(co / 128) * (cin / SC_KB) + ci / SC_KB;
        uint32_t b[3];
        split3(wt[i], 0.f, b[0], b[1], b[2]);
        for (int p = 0; p < 3; ++p)
            o[((((blk * 3 + p) * 2 + ci % SC_KB / 8) * k + r) * 128 + co % 128) * 8 + ci % 8] =
                __ushort_as_bfloat16((unsigned short)b[p]);
    }
}

// ---------------------------------------------------------------- planes
__device__ __forceinline__ float2 join3(uint32_t p1, uint32_t p2, uint32_t p3) {  // exact: the sum is the float
    return make_float2((__uint_as_float(p1 << 16) + __uint_as_float(p2 << 16)) + __uint_as_float(p3 << 16),
                       (__uint_as_float(p1 & 0xffff0000u) + __uint_as_float(p2 & 0xffff0000u)) +
                           __uint_as_float(p3 & 0xffff0000u));
}

// An activation: planes at p, plane and chunk strides in elements, split (even rows, then odd ones at
// `odd` elements) or plain, `rows` rows from one window to the next (of each half).
struct Planes {
    __nv_bfloat16 *p;
    int64_t ps, cs, odd;
    int rows;
};
__device__ __forceinline__ int64_t plane_row(const Planes &o, int64_t w, int r) {
    return o.odd ? ((r & 1) ? o.odd : 0) + (w * o.rows + (r >> 1)) * 8 : (w * o.rows + r) * 8;
}

// GroupNorm (+ residual, ReLU) of raw [C][hs] (window w, position t at row w hr + t) into planes.
// grid (parts, n_win): CTA (i, w) takes the channels [cp i, cp (i + 1)), whole groups of cg.  A unit is 32
// positions of one 8-channel chunk: lane = position, the 8 channels in registers (8 coalesced loads), so
// the three plane stores are 16 bytes a lane and contiguous over the warp.  REG: every warp holds its
// units (at most GN_U) in registers and reads raw once; else each pass reads it again.  The mean and
// the centred variance are two passes in a fixed order, as in k_groupnorm_st.
// Bound by memory: 4 B read + 6 B written (+ 6 B residual) per element.  Groups are independent, so a
// window is split over several CTAs; two fit an SM and hide each other's loads.  The residual's rows are fetched into L2
// while the statistics are formed.
// (Per sequence of 960 ResNet34 windows, 35 launches, 21 GB: 256 threads of 6 units at three CTAs an SM 5.51 ms, at
// two 5.04; 512 of 3 at two CTAs 4.25, with the residual fetched into L2 before the statistics 4.06, 76 % of the
// copy rate; 1024 of 3 4.91, 512 of 2 5.21.)
constexpr int GNS_T = 512;
constexpr int GNS_U = 3;

template <int GS, bool REG>
__global__ void __launch_bounds__(GNS_T, 2) k_gn_split(const float *raw, int64_t hs, int hr, int L,
                                                                 int cp, int lcg, const float *__restrict__ gamma,
                                                                 const float *__restrict__ beta, float eps,
                                                                 const Planes res, int relu, const Planes out) {
    constexpr int NV = 8 / GS;  // group parts in a chunk (1 where a group holds whole chunks)
    constexpr int NW = GNS_T / 32;
    extern __shared__ float part[];  // [units][NV]
    __shared__ float gmean[256];     // mean of the group of channel slot c / GS (cp / GS of them)
    __shared__ float grstd[256];
    __shared__ __align__(16) float scl[512], shf[512];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t w = gridDim.y - 1 - blockIdx.y;  // (what the convolution wrote last is still in L2: 333 windows -1 %)
    const int c0 = blockIdx.x * cp, nb = (L + 31) / 32, U = cp / 8 * nb, cg = 1 << lcg;
    const int per = (U + NW - 1) / NW, u0 = warp * per, u1 = min(U, u0 + per);
    const int ch0 = u0 / nb, b0 = u0 - ch0 * nb;  // chunk and 32-position block of the warp's first unit
    const int ng = cp >> lcg, gu = cg >= 8 ? cg / 8 * nb : nb;  // groups, and units a group spans
    const float inv = 1.0f / ((float)L * (float)cg);
    const float *src = raw + (int64_t)c0 * hs + w * hr;
    float v[REG ? GNS_U : 1][8];
    pdl_trigger();
    pdl_wait();

    // body(i, u, chunk, position) for the warp's units in order
    auto units = [&](auto body) {
        int ch = ch0, b = b0;
        if (REG) {
#pragma unroll
            for (int i = 0; i < GNS_U; ++i) {
                if (u0 + i < u1) body(i, u0 + i, ch, b * 32 + lane);
                if (++b == nb) {
                    b = 0;
                    ++ch;
                }
            }
        } else {
            for (int u = u0; u < u1; ++u) {
                body(0, u, ch, b * 32 + lane);
                if (++b == nb) {
                    b = 0;
                    ++ch;
                }
            }
        }
    };
    auto load = [&](int i, int ch, int t) {
        const float *s = src + (int64_t)ch * 8 * hs + t;
#pragma unroll
        for (int e = 0; e < 8; ++e) v[i][e] = t < L ? s[e * hs] : 0.f;
    };
    // sums of f(x, group slot) over each group: by unit, then over the group's units
    auto reduce = [&](auto f, auto fin) {
        units([&](int i, int u, int ch, int t) {
            if (!REG) load(i, ch, t);
#pragma unroll
            for (int j = 0; j < NV; ++j) {
                float s = 0.f;
#pragma unroll
                for (int e = 0; e < GS; ++e) s += f(v[i][j * GS + e], ch * NV + j);
                if (t >= L) s = 0.f;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                if (lane == 0) part[u * NV + j] = s;
            }
        });
        __syncthreads();
        for (int g = warp; g < ng; g += NW) {
            const int first = cg >= 8 ? g * gu : (g * cg / 8) * nb, j = cg >= 8 ? 0 : (g * cg % 8) / GS;
            float s = 0.f;
            for (int i = lane; i < gu; i += 32) s += part[(first + i) * NV + j];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            for (int q = lane; q < cg / GS; q += 32) fin(g * (cg / GS) + q, s);
        }
        __syncthreads();
    };
    if (REG) units([&](int i, int, int ch, int t) { load(i, ch, t); });
    static_assert(GNS_T >= 512, "one channel of an item a thread");
    const float gm = tid < cp ? __ldg(gamma + c0 + tid) : 0.f, bt = tid < cp ? __ldg(beta + c0 + tid) : 0.f;
    if (REG && res.p) units([&](int, int, int ch, int t) {
        if (t < L) {
            const __nv_bfloat16 *rp = res.p + (int64_t)(c0 / 8 + ch) * res.cs + plane_row(res, w, t + 1);
            asm volatile("prefetch.global.L2 [%0];" ::"l"(rp));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(rp + res.ps));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(rp + 2 * res.ps));
        }
    });
    reduce([](float x, int) { return x; }, [&](int q, float s) { gmean[q] = s * inv; });
    reduce(
        [&](float x, int q) {
            const float d = x - gmean[q];
            return d * d;
        },
        [&](int q, float s) { grstd[q] = rsqrtf(s * inv + eps); });
    if (tid < cp) {
        const float sc = grstd[tid / GS] * gm;
        scl[tid] = sc;
        shf[tid] = bt - gmean[tid / GS] * sc;
    }
    __syncthreads();

    units([&](int i, int, int ch, int t) {
        if (!REG) load(i, ch, t);
        if (t >= L) return;
        const int64_t chunk = c0 / 8 + ch;
        uint4 r1, r2, r3;
        if (res.p) {
            const __nv_bfloat16 *rp = res.p + chunk * res.cs + plane_row(res, w, t + 1);
            r1 = *reinterpret_cast<const uint4 *>(rp);
            r2 = *reinterpret_cast<const uint4 *>(rp + res.ps);
            r3 = *reinterpret_cast<const uint4 *>(rp + 2 * res.ps);
        }
        float y[8];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float4 sc = *reinterpret_cast<const float4 *>(scl + ch * 8 + 4 * h);
            const float4 sh = *reinterpret_cast<const float4 *>(shf + ch * 8 + 4 * h);
            y[4 * h] = fmaf(v[i][4 * h], sc.x, sh.x);
            y[4 * h + 1] = fmaf(v[i][4 * h + 1], sc.y, sh.y);
            y[4 * h + 2] = fmaf(v[i][4 * h + 2], sc.z, sh.z);
            y[4 * h + 3] = fmaf(v[i][4 * h + 3], sc.w, sh.w);
        }
        if (res.p) {
            const uint32_t a1[4] = {r1.x, r1.y, r1.z, r1.w}, a2[4] = {r2.x, r2.y, r2.z, r2.w};
            const uint32_t a3[4] = {r3.x, r3.y, r3.z, r3.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 r = join3(a1[e], a2[e], a3[e]);
                y[2 * e] += r.x;
                y[2 * e + 1] += r.y;
            }
        }
        if (relu)
#pragma unroll
            for (int e = 0; e < 8; ++e) y[e] = fmaxf(y[e], 0.f);
        uint32_t q1[4], q2[4], q3[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) split3(y[2 * e], y[2 * e + 1], q1[e], q2[e], q3[e]);
        __nv_bfloat16 *o = out.p + chunk * out.cs + plane_row(out, w, t + 1);
        *reinterpret_cast<uint4 *>(o) = make_uint4(q1[0], q1[1], q1[2], q1[3]);
        *reinterpret_cast<uint4 *>(o + out.ps) = make_uint4(q2[0], q2[1], q2[2], q2[3]);
        *reinterpret_cast<uint4 *>(o + 2 * out.ps) = make_uint4(q3[0], q3[1], q3[2], q3[3]);
    });
    for (int i = tid; i < cp / 8 * 6; i += GNS_T) {  // zero rows before and after the window
        const int ch = i / 6, pl = (i % 6) >> 1, r = (i & 1) ? L + 1 : 0;
        *reinterpret_cast<uint4 *>(out.p + pl * out.ps + (int64_t)(c0 / 8 + ch) * out.cs + plane_row(out, w, r)) =
            make_uint4(0, 0, 0, 0);
    }
}

// ---------------------------------------------------------------- stem
// Convolution (FP32, the FMA order of k_stem), GroupNorm, ReLU and max-pool of one window's channels, straight into
// planes.  grid (C0 / cp, n_win), 256 threads: CTA (i, w) takes the channels [cp i, cp (i + 1)), whole groups; a warp
// takes four channels and a run of positions, 32 a step, the samples in shared memory.  REG: the run is at most
// STS_U steps and its outputs stay in registers, so the convolution (2 k FMAs and, for four channels, 2 k
// shared-memory reads an output) is evaluated once; else three times (mean, centred variance, output).  Bound by the
// shared-memory reads: 718 us for 960 ResNet34 windows evaluated three times, 393 now; k_stem + k_groupnorm moved
// 2 MB a window through memory.
constexpr int STS_T = 256, STS_W = STS_T / 32;
constexpr int STS_K = 7;
constexpr int STS_U = 24;

template <bool REG>
__global__ void __launch_bounds__(STS_T, 1) k_stem_split(const float *__restrict__ y, int64_t n_y, int64_t y_stride,
                                                         int64_t first, int64_t stride, int64_t shift, int64_t w0,
                                                         const float *__restrict__ wt, const float *__restrict__ gamma,
                                                         const float *__restrict__ beta, int cp, int k, int s, int W,
                                                         int L0, int pool, int cg, float eps, const Planes out) {
    extern __shared__ float xs[];  // [2][W + 2 pad], then sums [warps per quad][cp], mean or shift [cp], scale [cp]
    const int pad = k / 2, Wp = W + 2 * pad, c0 = blockIdx.x * cp;
    const int wq = max(1, 4 * STS_W / cp);  // warps that share a quad's positions
    float *csum = xs + 2 * Wp, *shf = csum + wq * cp, *scl = shf + cp;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t start = first + (w0 + blockIdx.y) * stride;
    for (int t = tid; t < Wp; t += STS_T) {
        const int tt = t - pad;
        float a = 0.f, b = 0.f;
        if (tt >= 0 && tt < W) {
            a = y[start + tt];
            int64_t i1 = start + shift + tt;
            if (i1 >= n_y) i1 -= n_y;
            b = y[y_stride + i1];
        }
        xs[t] = a;
        xs[Wp + t] = b;
    }
    // the warp's first channels (local; more only where cp > 4 STS_W, never with REG) and its run of positions
    const int cl0 = warp / wq * 4, cls = STS_W / wq * 4, part = warp % wq;
    const int steps = (L0 + 31) / 32, per = (steps + wq - 1) / wq, s0 = part * per, s1 = min(steps, s0 + per);
    float wr[4][2][STS_K];
    auto weights = [&](int cl) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int r = 0; r < STS_K; ++r) wr[e][i][r] = r < k ? wt[((c0 + cl + e) * 2 + i) * k + r] : 0.f;
    };
    weights(cl0);
    auto conv = [&](int t, float (&z)[4]) {
#pragma unroll
        for (int e = 0; e < 4; ++e) z[e] = 0.f;
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int r = 0; r < STS_K; ++r)
                if (r < k) {
                    const float x = xs[i * Wp + t * s + r];
#pragma unroll
                    for (int e = 0; e < 4; ++e) z[e] = fmaf(wr[e][i][r], x, z[e]);
                }
    };
    float v[REG ? STS_U : 1][4];
    // body(i, step) over the warp's steps
    auto run = [&](auto body) {
        if (REG) {
#pragma unroll
            for (int i = 0; i < STS_U; ++i)
                if (s0 + i < s1) body(i, s0 + i);
        } else {
            for (int st = s0; st < s1; ++st) {
                conv(min(st * 32 + lane, L0 - 1), v[0]);
                body(0, st);
            }
        }
    };
    __syncthreads();
    if (REG) run([&](int i, int st) { conv(min(st * 32 + lane, L0 - 1), v[i]); });
    // two passes: channel sums of the values, then of their squared distance to the group mean (in shf)
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll 1
        for (int cl = cl0; cl < cp; cl += cls) {
        if (!REG) weights(cl);
        float m[4], a[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int e = 0; e < 4; ++e) m[e] = pass ? shf[cl + e] : 0.f;
        run([&](int i, int st) {
            if (st * 32 + lane < L0)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float d = v[i][e] - m[e];
                    a[e] = pass ? fmaf(d, d, a[e]) : a[e] + d;
                }
        });
#pragma unroll
        for (int e = 0; e < 4; ++e) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a[e] += __shfl_xor_sync(0xffffffffu, a[e], o);
            if (lane == 0) csum[part * cp + cl + e] = a[e];
        }
        }
        __syncthreads();
        for (int c = tid; c < cp; c += STS_T) {
            float t = 0.f;
            for (int i = c / cg * cg; i < (c / cg + 1) * cg; ++i)
                for (int q = 0; q < wq; ++q) t += csum[q * cp + i];
            t /= (float)L0 * (float)cg;
            if (pass == 0) {
                shf[c] = t;
            } else {
                const float sc = rsqrtf(t + eps) * gamma[c0 + c];
                scl[c] = sc;
                shf[c] = beta[c0 + c] - shf[c] * sc;
            }
        }
        __syncthreads();
    }
    const int Lo = pool ? (L0 + 2 - 3) / 2 + 1 : L0;
#pragma unroll 1
    for (int cl = cl0; cl < cp; cl += cls) {
    if (!REG) weights(cl);
    float sc[4], sh[4], carry[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        sc[e] = scl[cl + e];
        sh[e] = shf[cl + e];
        carry[e] = -INFINITY;
    }
    if (pool && s0 > 0) {  // the position before the run
        conv(min(s0 * 32, L0) - 1, carry);
#pragma unroll
        for (int e = 0; e < 4; ++e) carry[e] = fmaxf(fmaf(carry[e], sc[e], sh[e]), 0.f);
    }
    __nv_bfloat16 *oc = out.p + (int64_t)((c0 + cl) / 8) * out.cs + (cl & 4);
    run([&](int i, int st) {
        const int t = st * 32 + lane;
        float z[4], m[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            z[e] = t < L0 ? fmaxf(fmaf(v[i][e], sc[e], sh[e]), 0.f) : -INFINITY;
            if (pool) {
                float lo = __shfl_up_sync(0xffffffffu, z[e], 1);
                const float hi = __shfl_down_sync(0xffffffffu, z[e], 1);
                if (lane == 0) lo = carry[e];
                m[e] = fmaxf(fmaxf(lo, z[e]), hi);  // (stored by even lanes: hi is in the warp)
                carry[e] = __shfl_sync(0xffffffffu, z[e], 31);
            } else {
                m[e] = z[e];
            }
        }
        const int u = pool ? t >> 1 : t;
        if (t < L0 && u < Lo && (!pool || !(lane & 1))) {
            uint32_t p[3][2];
            split3(m[0], m[1], p[0][0], p[1][0], p[2][0]);
            split3(m[2], m[3], p[0][1], p[1][1], p[2][1]);
            const int64_t o = plane_row(out, blockIdx.y, u + 1);
#pragma unroll
            for (int q = 0; q < 3; ++q) *reinterpret_cast<uint2 *>(oc + q * out.ps + o) = make_uint2(p[q][0], p[q][1]);
        }
    });
    }
    for (int i = tid; i < cp / 8 * 6; i += STS_T)
        *reinterpret_cast<uint4 *>(out.p + ((i % 6) >> 1) * out.ps + (int64_t)(c0 / 8 + i / 6) * out.cs +
                                   plane_row(out, blockIdx.y, (i & 1) ? Lo + 1 : 0)) = make_uint4(0, 0, 0, 0);
}

// ---------------------------------------------------------------- head
// grid (n_win), block 256: logit = fc_b + sum_c fc_w[c] * mean_t x[t][c]; each thread sums 8 channels of
// a chunk over some of the rows
__global__ void k_head_split(const Planes x, int L, int C, const float *__restrict__ fc_w,
                             const float *__restrict__ fc_b, float *__restrict__ logits, int64_t w0) {
    __shared__ float part[256][9];
    __shared__ float term[512];
    const int tid = threadIdx.x, nch = C / 8, tpc = 256 / nch, ch = tid % nch, r0 = tid / nch;
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    pdl_wait();
    if (r0 < tpc)
        for (int r = r0; r < L; r += tpc) {
            const __nv_bfloat16 *p = x.p + (int64_t)ch * x.cs + plane_row(x, blockIdx.x, r + 1);
            const uint4 a = *reinterpret_cast<const uint4 *>(p), b = *reinterpret_cast<const uint4 *>(p + x.ps);
            const uint4 c = *reinterpret_cast<const uint4 *>(p + 2 * x.ps);
            const uint32_t a4[4] = {a.x, a.y, a.z, a.w}, b4[4] = {b.x, b.y, b.z, b.w}, c4[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 v = join3(a4[e], b4[e], c4[e]);
                s[2 * e] += v.x;
                s[2 * e + 1] += v.y;
            }
        }
#pragma unroll
    for (int e = 0; e < 8; ++e) part[tid][e] = s[e];
    __syncthreads();
    for (int c = tid; c < C; c += 256) {
        float t = 0.f;
        for (int g = 0; g < tpc; ++g) t += part[g * nch + c / 8][c % 8];
        term[c] = fc_w[c] * (t / (float)L);
    }
    __syncthreads();
    if (tid < 32) {
        float z = 0.f;
        for (int c = tid; c < C; c += 32) z += term[c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
        if (tid == 0) logits[w0 + blockIdx.x] = fc_b[0] + z;
    }
}

}  // namespace

// ---------------------------------------------------------------- plan
struct SplitPlan {
    std::vector<unsigned char *> wimg;  // indexed like NetPlan::convs (0 unused)
    void *mem = nullptr;
    int sms = 0;
    int64_t max_chunk = 1;  // windows per launch sequence at most
};

// Windows per launch sequence at most (1.4 GB of ResNet34 activations), and bytes of each of its five buffers, which
// hold fewer of the longest and widest windows.  Each of the 70 launches costs about 5 us whatever its size, and a short sequence leaves its last wave of tiles part empty; in a long one less of a layer's output is still in L2
// for the next: 1920 ResNet34 windows take 26.8 ms in sequences of at most 256, 24.5 of 512, 23.95 of 1024 and 24.8 of
// 2048; 7680 take 103.4, 98.5, 95.8 and 99.0, and 101.4 of 4096.
constexpr int64_t SPLIT_MAX_CHUNK = 1024;
constexpr int64_t SPLIT_MAX_BYTES = (int64_t)4 << 30;

static int mode_of(const ConvLayer &C) { return C.stride == 1 ? 0 : C.k == 3 ? 1 : 2; }
static int64_t conv_rows(const ConvLayer &C, int64_t nw) { return nw * (C.lout + (C.stride == 1 ? 2 : 1)); }

// Cycles of one stage of a tile of tn rows: its 6 taps MMAs at 4096 MACs a clock, or (tn < 256, where the weights'
// 4 KB an MMA are shared by fewer rows) their operand reads and the stage's copies at the 128 B/clk of shared memory.
static int64_t stage_cycles(int tn, int taps) {
    return std::max<int64_t>(6 * taps * tn / 2, (6 * taps * (4096 + 32 * tn) + 6 * taps * 2048 + 6 * 16 * tn) / 128);
}

// Output rows per tile.  Wide tiles cost the fewest cycles a row (9.0 at 256, 9.1 at 224, 9.8 at 192, 12 at 128, 19 at
// 64 with three taps); narrower ones fill the last wave, or shorten the only one: the width whose waves of one tile an
// SM take the fewest cycles, the wider one of equals.  Against 256, else 128 or 64 where half of the SMs had no tile:
// 152 ResNet34 windows 2.32 -> 2.20 ms, 333 4.71 -> 4.47; 960 the same.
static int tile_rows(const ConvLayer &C, int64_t nw, int sms) {
    const int64_t rows = conv_rows(C, nw), slices = (C.cout + 127) / 128;
    int best = 0;
    int64_t least = 0;
    for (int tn : {256, 224, 192, 128, 64}) {
        const int64_t waves = ((rows + tn - 1) / tn * slices + sms - 1) / sms, t = waves * stage_cycles(tn, C.k);
        if (!best || t < least) best = tn, least = t;
    }
    return best;
}

static Planes make_planes(__nv_bfloat16 *p, int64_t nw, int L, int C, bool split) {
    Planes o;
    o.p = p;
    o.rows = split ? L / 2 + 1 : L + 2;
    const int64_t r = nw * o.rows + SC_SLACK;
    o.odd = split ? r * 8 : 0;
    o.cs = (split ? 2 : 1) * r * 8;
    o.ps = (C / 8) * o.cs;
    return o;
}
// (whole tiles of any width)
static int64_t raw_stride(const ConvLayer &C, int64_t nw) { return (conv_rows(C, nw) + 224 + 255) / 256 * 256; }

// Bytes of each of the four activation buffers (three planes) and of the raw output of a sequence of nw windows
static void split_bytes(const NetPlan &P, int64_t nw, int64_t &planes, int64_t &raw) {
    planes = 3 * make_planes(nullptr, nw, P.l_after_stem, P.convs[0].cout, false).ps;
    raw = 0;
    for (size_t i = 1; i < P.convs.size(); ++i) {
        const ConvLayer &C = P.convs[i];
        for (bool split : {false, true})
            if (!split || C.lout % 2 == 0)
                planes = std::max(planes, 3 * make_planes(nullptr, nw, C.lout, C.cout, split).ps);
        raw = std::max(raw, (int64_t)C.cout * raw_stride(C, nw));
    }
    planes *= (int64_t)sizeof(__nv_bfloat16);
    raw *= (int64_t)sizeof(float);
}

static bool split_supported(const afg_ctx *ctx) {
    const NetPlan &P = ctx->plan;
    if (P.convs.size() < 2 || P.convs[0].k > STS_K || P.convs[0].cout % 64) return false;
    for (size_t i = 1; i < P.convs.size(); ++i) {
        const ConvLayer &C = P.convs[i];
        const int cg = C.cout / P.net.groups;
        if (C.cin % 64 || C.cout % 64 || C.cout > 512 || cg < 2 || (cg & (cg - 1))) return false;
        if (!((C.k == 3 && C.stride <= 2) || (C.k == 1 && C.stride == 2))) return false;
        if (C.stride == 2 && (C.lin % 2 || C.lout != C.lin / 2)) return false;
        if (C.lout < 1) return false;
    }
    return true;
}

// Weight images of the tensor-core FP32 path.  Left out (and the SIMT path kept) where the network's
// widths do not fit, where the context has a memory budget (the images and planes are larger than the
// SIMT path's buffers for small calls, and a call that fitted must still fit), or where the device has no
// room for them.
int net_split_prepare(afg_ctx *ctx) {
    NetPlan &P = ctx->plan;
    if (ctx->cfg.precision != AFG_FP32 || ctx->cfg.hbm_budget > 0 || !split_supported(ctx)) return AFG_OK;
    std::vector<size_t> off(P.convs.size());
    size_t total = 0;
    for (size_t i = 1; i < P.convs.size(); ++i) {
        const ConvLayer &C = P.convs[i];
        off[i] = total;
        total += (size_t)((C.cout + 127) / 128) * (C.cin / SC_KB) * 6 * C.k * 128 * 16;
    }
    void *d = nullptr;
    if (cudaMalloc(&d, total) != cudaSuccess) {
        cudaGetLastError();
        return AFG_OK;
    }
    SplitPlan *sp = new SplitPlan();
    sp->mem = d;
    ctx->splitplan = sp;
    ctx->bytes_held += (int64_t)total;
    AFG_CUDA(ctx, cudaMemset(d, 0, total));
    sp->max_chunk = SPLIT_MAX_CHUNK;
    for (int64_t planes, raw; sp->max_chunk > 1; sp->max_chunk = sp->max_chunk * 3 / 4) {
        split_bytes(P, sp->max_chunk, planes, raw);
        if (std::max(planes, raw) <= SPLIT_MAX_BYTES) break;
    }
    sp->wimg.resize(P.convs.size());
    for (size_t i = 1; i < P.convs.size(); ++i) {
        const ConvLayer &C = P.convs[i];
        sp->wimg[i] = static_cast<unsigned char *>(d) + off[i];
        k_split_weights<<<512, 256>>>(C.wt, C.cin, C.cout, C.k, reinterpret_cast<__nv_bfloat16 *>(sp->wimg[i]));
    }
    AFG_LAUNCH_CHECK(ctx, "k_split_weights");
    AFG_CUDA(ctx, cudaDeviceGetAttribute(&sp->sms, cudaDevAttrMultiProcessorCount, ctx->device));
#define AFG_SPLIT_ATTR(TN, MODE)                                                                          \
    AFG_CUDA(ctx, cudaFuncSetAttribute(k_conv_split<TN, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                       (int)SplitGeo<TN, MODE>::BYTES))
    AFG_SPLIT_ATTR(256, 0); AFG_SPLIT_ATTR(256, 1); AFG_SPLIT_ATTR(256, 2);
    AFG_SPLIT_ATTR(224, 0); AFG_SPLIT_ATTR(224, 1); AFG_SPLIT_ATTR(224, 2);
    AFG_SPLIT_ATTR(192, 0); AFG_SPLIT_ATTR(192, 1); AFG_SPLIT_ATTR(192, 2);
    AFG_SPLIT_ATTR(128, 0); AFG_SPLIT_ATTR(128, 1); AFG_SPLIT_ATTR(128, 2);
    AFG_SPLIT_ATTR(64, 0); AFG_SPLIT_ATTR(64, 1); AFG_SPLIT_ATTR(64, 2);
#undef AFG_SPLIT_ATTR
#define AFG_SPLIT_GN(GS)                                                                                              \
    AFG_CUDA(ctx, cudaFuncSetAttribute(k_gn_split<GS, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 192 * 1024))
    AFG_SPLIT_GN(2); AFG_SPLIT_GN(4); AFG_SPLIT_GN(8);
#undef AFG_SPLIT_GN
    AFG_CUDA(ctx, cudaFuncSetAttribute(k_stem_split<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 192 * 1024));
    AFG_CUDA(ctx, cudaFuncSetAttribute(k_stem_split<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 192 * 1024));
    return AFG_OK;
}

void net_split_release(afg_ctx *ctx) {
    if (!ctx->splitplan) return;
    if (ctx->splitplan->mem) cudaFree(ctx->splitplan->mem);
    delete ctx->splitplan;
    ctx->splitplan = nullptr;
}

bool net_split_available(const afg_ctx *ctx) { return ctx->splitplan != nullptr; }

// Windows per launch sequence for a call of n_win: equal shares
static int64_t split_chunk(const afg_ctx *ctx, int64_t n_win) {
    const int64_t n = (n_win + ctx->splitplan->max_chunk - 1) / ctx->splitplan->max_chunk;
    return (n_win + n - 1) / n;
}

// The workspaces of a launch sequence over nw windows: four activations in planes and one raw output.
static int split_reserve(afg_ctx *ctx, int64_t nw, __nv_bfloat16 *(&act)[4], float *&raw) {
    int64_t planes, rw;
    split_bytes(ctx->plan, nw, planes, rw);
    int rc = AFG_OK;
    for (int i = 0; i < 4 && !rc; ++i) rc = afg_ws_reserve(ctx, WS_ACT0 + i, (size_t)planes, (void **)&act[i]);
    if (!rc) rc = afg_ws_reserve(ctx, WS_RAW, (size_t)rw, (void **)&raw);
    return rc;
}

// The workspaces of a call of n_win windows, and so of any shorter one.  (Not those of its sequence: 1025 windows go in
// sequences of 513, but 1024 in one, and a call inside a caller's capture may not grow what a longer one left.)  Where
// the device has no room for them the sequences become shorter, for good.
static int split_fit(afg_ctx *ctx, int64_t n_win, __nv_bfloat16 *(&act)[4], float *&raw) {
    int64_t &most = ctx->splitplan->max_chunk;
    int rc;
    while ((rc = split_reserve(ctx, std::min(n_win, most), act, raw)) == AFG_ERR_OOM && most > 1) {
        most = std::max<int64_t>(1, std::min(most, n_win) / 2);
        for (int slot : {(int)WS_ACT0, (int)WS_ACT1, (int)WS_ACT2, (int)WS_ACT3, (int)WS_RAW}) afg_ws_release(ctx, slot);
    }
    return rc;
}

int net_split_reserve(afg_ctx *ctx, int64_t n_win) {
    __nv_bfloat16 *act[4];
    float *raw;
    return split_fit(ctx, std::max<int64_t>(1, n_win), act, raw);
}

static cudaError_t split_conv(afg_ctx *ctx, int i, const Planes &in, float *raw, int64_t nw, cudaStream_t st) {
    const ConvLayer &C = ctx->plan.convs[i];
    const SplitPlan &sp = *ctx->splitplan;
    const int tn = tile_rows(C, nw, sp.sms);
    SplitConvArgs a;
    a.wimg = sp.wimg[i];
    a.in = in.p;
    a.in_ps = in.ps;
    a.in_cs = in.cs;
    a.in_odd = in.odd;
    a.raw = raw;
    a.hs = raw_stride(C, nw);
    a.cout = C.cout;
    a.n_kb = C.cin / SC_KB;
    a.slices = (C.cout + 127) / 128;
    a.n_tiles = (int)((conv_rows(C, nw) + tn - 1) / tn) * a.slices;
    a.err = ctx->d_err;
    const unsigned grid = (unsigned)std::min(a.n_tiles, sp.sms);
    // algorithmic: 2 M N K FLOPs; the input and weights read and the output written once, in FP32
    KScope ks(ctx, st, KK_CONV_SPLIT, 2.0 * nw * C.lout * C.cout * (double)C.k * C.cin,
              4.0 * ((double)nw * ((double)C.lin * C.cin + (double)C.lout * C.cout) + (double)C.k * C.cin * C.cout));
#define AFG_SPLIT_CONV(TN, MODE) \
    case TN * 4 + MODE: return launch_pdl(k_conv_split<TN, MODE>, dim3(grid), dim3(SC_T), SplitGeo<TN, MODE>::BYTES, st, a);
    switch (tn * 4 + mode_of(C)) {
        AFG_SPLIT_CONV(256, 0) AFG_SPLIT_CONV(256, 1) AFG_SPLIT_CONV(256, 2)
        AFG_SPLIT_CONV(224, 0) AFG_SPLIT_CONV(224, 1) AFG_SPLIT_CONV(224, 2)
        AFG_SPLIT_CONV(192, 0) AFG_SPLIT_CONV(192, 1) AFG_SPLIT_CONV(192, 2)
        AFG_SPLIT_CONV(128, 0) AFG_SPLIT_CONV(128, 1) AFG_SPLIT_CONV(128, 2)
        AFG_SPLIT_CONV(64, 0) AFG_SPLIT_CONV(64, 1) AFG_SPLIT_CONV(64, 2)
    }
#undef AFG_SPLIT_CONV
    return cudaErrorInvalidValue;  // (not reached)
}

static cudaError_t split_gn(afg_ctx *ctx, int i, const float *raw, int64_t nw, const Planes &res, int relu, const Planes &out,
                     cudaStream_t st) {
    const ConvLayer &C = ctx->plan.convs[i];
    const int cg = C.cout / ctx->plan.net.groups, nb = (C.lout + 31) / 32;
    int cp = C.cout;  // channels per CTA: whole chunks and groups, halved until a CTA's units fit its registers
    while (cp / 8 * nb > GNS_U * (GNS_T / 32) && cp > 8 && cp > cg) cp /= 2;
    int lcg = 0;
    while ((1 << lcg) < cg) ++lcg;
    const int U = cp / 8 * nb, hr = C.lout + (C.stride == 1 ? 2 : 1);
    const bool reg = (U + GNS_T / 32 - 1) / (GNS_T / 32) <= GNS_U;
    KScope ks(ctx, st, KK_GROUPNORM, 0.0, (double)nw * C.lout * C.cout * 4.0 * (res.p ? 3.0 : 2.0));
    const dim3 grid(C.cout / cp, (unsigned)nw);
    const size_t sm = (size_t)U * (8 / std::min(cg, 8)) * sizeof(float);
#define AFG_GN(GS)                                                                                                        \
    launch_pdl(reg ? k_gn_split<GS, true> : k_gn_split<GS, false>, grid, dim3(GNS_T), sm, st, raw, raw_stride(C, nw), hr,  \
               C.lout, cp, lcg, (const float *)C.gamma, (const float *)C.beta, ctx->plan.net.eps, res, relu, out)
    return cg >= 8 ? AFG_GN(8) : cg == 4 ? AFG_GN(4) : AFG_GN(2);
#undef AFG_GN
}

// ---------------------------------------------------------------- forward
int launch_infer_split(afg_ctx *ctx, const float *y, int64_t n_y, int64_t y_stride, int64_t first, int64_t stride,
                       int64_t n_win, int64_t shift, float *logits, cudaStream_t st) {
    const NetPlan &P = ctx->plan;
    const ConvLayer &S = P.convs[0];
    const int W = ctx->cfg.win_len;
    __nv_bfloat16 *act[4];
    float *raw;
    int rc = split_fit(ctx, n_win, act, raw);
    if (rc) return rc;
    const int64_t chunk = split_chunk(ctx, n_win);
    const Planes none = {nullptr, 0, 0, 0, 0};
    for (int64_t w0 = 0; w0 < n_win; w0 += chunk) {
        const int nw = (int)std::min<int64_t>(chunk, n_win - w0);
        int ia = 0, ic = 2;  // the block's input and (where it cannot be written in place) its output
        Planes A = make_planes(act[ia], nw, P.l_after_stem, S.cout, false);
        {
            KScope ks(ctx, st, KK_STEM, 2.0 * nw * S.lout * S.cout * S.cin * S.k,
                      4.0 * nw * ((double)2 * W + (double)P.l_after_stem * S.cout));
            // channels per CTA: 32 (four a warp), fewer where that puts a warp's run of positions in registers, or a
            // whole group
            const int cg = S.cout / P.net.groups, steps = (S.lout + 31) / 32;
            int cp = std::max(4 * STS_W, cg);
            auto run = [&] {
                const int wq = std::max(1, 4 * STS_W / cp);
                return cp <= 4 * STS_W ? (steps + wq - 1) / wq : STS_U + 1;
            };
            while (run() > STS_U && cp > 8 && cp > cg) cp /= 2;
            const size_t sm = (size_t)(2 * (W + 2 * (S.k / 2)) + std::max(4 * STS_W, cp) + 2 * cp) * sizeof(float);
            const dim3 grid(S.cout / cp, nw);
#define AFG_STEM(REG)                                                                                                    \
    k_stem_split<REG><<<grid, STS_T, sm, st>>>(y, n_y, y_stride, first, stride, shift, w0, S.wt, S.gamma, S.beta, cp, S.k, \
                                               S.stride, W, S.lout, P.net.stem_pool, cg, P.net.eps, A)
            if (run() <= STS_U) AFG_STEM(true);
            else AFG_STEM(false);
#undef AFG_STEM
        }
        AFG_LAUNCH_CHECK(ctx, "k_stem_split");
        for (size_t b = 0; b < P.blocks.size(); ++b) {
            const BlockPlan &bp = P.blocks[b];
            const ConvLayer &c1 = P.convs[bp.c1], &c2 = P.convs[bp.c2];
            const bool split_out = b + 1 < P.blocks.size() && P.convs[P.blocks[b + 1].c1].stride == 2;
            const Planes B = make_planes(act[1], nw, c1.lout, c1.cout, false);
            AFG_CUDA(ctx, split_conv(ctx, bp.c1, A, raw, nw, st));
            AFG_CUDA(ctx, split_gn(ctx, bp.c1, raw, nw, none, 1, B, st));
            Planes res = A;
            if (bp.sc >= 0) {
                res = make_planes(act[3], nw, c2.lout, c2.cout, false);
                AFG_CUDA(ctx, split_conv(ctx, bp.sc, A, raw, nw, st));
                AFG_CUDA(ctx, split_gn(ctx, bp.sc, raw, nw, none, 0, res, st));
            }
            AFG_CUDA(ctx, split_conv(ctx, bp.c2, B, raw, nw, st));
            // the output replaces the residual (the same thread reads and writes an element) unless its layout differs
            if (bp.sc >= 0 || split_out) std::swap(ia, ic);
            A = make_planes(act[ia], nw, c2.lout, c2.cout, split_out);
            AFG_CUDA(ctx, split_gn(ctx, bp.c2, raw, nw, res, 1, A, st));
            AFG_LAUNCH_CHECK(ctx, "residual block (split)");
        }
        {
            KScope ks(ctx, st, KK_HEAD, 2.0 * nw * P.l_last * P.c_last, 4.0 * nw * (double)P.l_last * P.c_last);
            AFG_CUDA(ctx, launch_pdl(k_head_split, dim3(nw), dim3(256), 0, st, A, P.l_last, P.c_last, (const float *)P.fc_w,
                                     (const float *)P.fc_b, logits, w0));
        }
        AFG_LAUNCH_CHECK(ctx, "k_head_split");
    }
    return AFG_OK;
}
