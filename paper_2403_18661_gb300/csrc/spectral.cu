// Welch PSD and FFT-domain whitening (the filter build is in filter.cu)
// (Sec. IV, "Noise sampling" paragraph: PSD from 8 s, frequency-domain whitening,
// 0.5 s crop at each edge; Sec. VI: PSD from the first 64 s of state).
//
// Kernels
//   k_periodogram     one Hann-windowed segment per CTA: FP32 real FFT in
//                     shared memory (radix-16 passes, fft16.cuh), the window
//                     applied to the spectrum (a three-bin convolution),
//                     |X_k|^2 formed in FP32 after an exact power-of-two
//                     scaling of the segment's spectrum, stored as FP32 with
//                     the segment's exponent
//   k_psd_mean        sum over the K segments of each epoch in pairs of floats
//                     (FP64 where segments are too far apart in power), a run of
//                     epochs per thread
//   k_psd_mean64      the same in FP64, for many segments or a short step
//   k_whiten          one 8192-output overlap-save block per CTA: FP32 real
//                     FFT of 8192 + F - 1 samples (zero padded to NFFT),
//                     multiply by the epoch's gains, inverse FFT, keep the
//                     outputs whose support lies inside the block.  The
//                     forward transform's last pass, the split, the gains,
//                     the inverse split and the inverse transform's first
//                     pass are one fused shared-memory pass.
#include <math.h>
#include <stdio.h>

#include <mutex>

#include "afg_internal.cuh"
#include "fft16.cuh"

namespace {

// The FP32 transforms' twiddle table (layout in fft16.cuh): entry i = exp(-i pi a_i), a_i an exact
// binary fraction, evaluated in FP64 and rounded to FP32.
__global__ void k_tw32() {
    using namespace r16;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= TW_TOTAL) return;
    double a;
    if (i < TW16_END) {
        const int ns = i < tw16_off(16) ? 2 : i < tw16_off(32) ? 16 : i < tw16_off(256) ? 32 : i < tw16_off(512) ? 256 : 512;
        const int loc = i - tw16_off(ns), m = loc / ns, k = loc % ns;  // m = 0, 1, 2: w1, w4, w8
        a = (double)((m == 0 ? 1 : m == 1 ? 4 : 8) * k) / (double)(8 * ns);
    } else if (i < TW_SPLIT) {
        const int loc = i - TW16_END;  // Ns - 2 <= loc < 2 Ns - 2
        int ns = 2;
        while (loc >= 2 * ns - 2) ns *= 2;
        a = (double)(loc - (ns - 2)) / (double)(2 * ns);
    } else {
        a = (double)(i - TW_SPLIT) / 8192.0;
    }
    double s, c;
    sincospi(a, &s, &c);
    g_tw[i] = make_float2((float)c, (float)-s);
}

// Forward radix-2 pass (Ns = 4096) and real-FFT split for task j of the
// Welch kernel, 1 <= j <= 2048: the butterflies j and 4096 - j give Z at
// j, j + 4096, 4096 - j and 8192 - j, i.e. the split pairs (j, NC - j) and
// (j + 4096, 4096 - j).  The four spectrum values U at bins j, 8192 - j, j + 4096
// and 4096 - j replace the four Z values they came from (the same slots: tasks
// touch disjoint slot sets).  (At j = 2048 the two butterflies coincide and only
// the first pair is written.)
__device__ __forceinline__ void welch_mid_task(float2 *d, int j) {
    using namespace r16;
    const float2 a = d[pad(j)], b = d[pad(j + 4096)], c = d[pad(4096 - j)], e = d[pad(8192 - j)];
    const float2 w = tw_split<-1>(j);      // W^j
    const float2 u = tw_split<-1>(2 * j);  // radix-2 twiddle of butterfly j
    const float2 u2 = make_float2(-u.x, u.y);      // of butterfly 4096 - j: -conj(u)
    const float2 ub = cmul(u, b), ue = cmul(u2, e);
    const float2 zj = cadd(a, ub), zj4 = csub(a, ub), zc = cadd(c, ue), zc4 = csub(c, ue);
    float2 x1, x1n, x2, x2n;
    split_fwd(zj, zc4, w, x1, x1n);             // bins j, 8192 - j
    split_fwd(zj4, zc, mul_i<-1>(w), x2, x2n);  // bins j + 4096, 4096 - j (W^{j+4096} = -i W^j)
    d[pad(j)] = x1;
    d[pad(8192 - j)] = x1n;
    if (j < 2048) {
        d[pad(j + 4096)] = x2;
        d[pad(4096 - j)] = x2n;
    }
}

// grid (n_seg, n_det), r16::NT threads; segment g of detector d covers x[d][g*hop, g*hop + NFFT).
// The periodic Hann window is applied in the frequency domain: its DFT has three non-zero bins,
// so the windowed spectrum is X_k = U_k / 2 - (U_{k-1} + U_{k+1}) / 4 with U the spectrum of the
// unwindowed segment (U_{-1} = conj U_1, U_{NC+1} = conj U_{NC-1} for a real segment).
// Row of a segment: P[k] for k <= NC, to be read as P[k] 2^e with e an integer in slot PER_EXP.
// (PER_ZERO: a segment of zeros.)
constexpr int PER_EXP = NBIN, PER_ROW = NBIN + 3, PER_ZERO = -(1 << 30);

__global__ void __launch_bounds__(r16::NT, 2) k_periodogram(const float *__restrict__ x, int64_t x_stride, int hop,
                                                             float *__restrict__ P, int64_t n_seg,
                                                             const float *const *__restrict__ rows, float scale) {
    using namespace r16;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *d = reinterpret_cast<float2 *>(smem_raw);
    float2 *u_nyq = d + SLOTS;  // U_NC (real)
    pdl_trigger();  // (launched plainly: what it reads is complete)
    const int64_t g = blockIdx.x;
    const int det = blockIdx.y;
    const int t = threadIdx.x;
    // row det starts at x + det * x_stride, or at rows[det] (rows of unrelated buffers)
    const float *src = (rows ? rows[det] : x + det * x_stride) + g * (int64_t)hop;
    // z_n = x_2n + i x_2n+1, n = t + 512 r (the first pass's inputs)
    float2 v[16];
    if ((reinterpret_cast<uintptr_t>(src) & 7) == 0) {  // 8-byte loads of (x_2n, x_2n+1)
        const float2 *s2 = reinterpret_cast<const float2 *>(src);
#pragma unroll
        for (int r = 0; r < 16; ++r) v[r] = s2[t + NT * r];
    } else {
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const int i0 = 2 * (t + NT * r);
            v[r] = make_float2(src[i0], src[i0 + 1]);
        }
    }
    forward_r16(d, v);
    // the unwindowed spectrum U_0 .. U_NC into the transform's slots
    if (t == 0) {
        // butterfly 0: Z_0, Z_4096; bins 0, NC (from the self-pair k = 0) and 4096
        const float2 a = d[pad(0)], b = d[pad(4096)];
        float2 x0, xn, x4, x4d;
        split_fwd(cadd(a, b), cadd(a, b), make_float2(1.0f, 0.0f), x0, xn);
        split_fwd(csub(a, b), csub(a, b), make_float2(0.0f, -1.0f), x4, x4d);
        d[pad(0)] = x0;
        *u_nyq = xn;
        d[pad(4096)] = x4;
    } else {
        welch_mid_task(d, t);
    }
#pragma unroll
    for (int m = 1; m < 4; ++m) welch_mid_task(d, t + NT * m);
    if (t == NT - 1) welch_mid_task(d, 2048);
    __syncthreads();
    // windowed bins k = 16 t .. 16 t + 15 (and NC) in registers, each spectrum value read once (18 reads a thread; bins
    // t + 512 m read each value three times, and shared memory is the busiest pipe of this kernel), and the
    // largest component magnitude of the block
    float *out = P + ((int64_t)det * n_seg + g) * PER_ROW;
    float2 U[18];  // U_{16 t - 1} .. U_{16 t + 16}
    {
        const float2 *p = d + pad(16 * t);  // = d + 17 t
#pragma unroll
        for (int m = 0; m < 16; ++m) U[m + 1] = p[m];
        U[0] = t ? p[-2] : conj(U[2]);
        U[17] = t < NT - 1 ? p[17] : *u_nyq;
    }
    float2 X[16];
    float mx = 0.f;
#pragma unroll
    for (int m = 0; m < 16; ++m) {
        X[m] = make_float2(0.5f * U[m + 1].x - 0.25f * (U[m].x + U[m + 2].x), 0.5f * U[m + 1].y - 0.25f * (U[m].y + U[m + 2].y));
        mx = fmaxf(mx, fmaxf(fabsf(X[m].x), fabsf(X[m].y)));
    }
    float2 Xn = make_float2(0.f, 0.f);
    if (t == NT - 1) {  // bin NC: U_NC + 1 = conj U_NC - 1
        const float2 r = conj(U[16]);
        Xn = make_float2(0.5f * U[17].x - 0.25f * (U[16].x + r.x), 0.5f * U[17].y - 0.25f * (U[16].y + r.y));
        mx = fmaxf(mx, fmaxf(fabsf(Xn.x), fabsf(Xn.y)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float *wmax = reinterpret_cast<float *>(u_nyq + 1);  // [NT / 32]
    if ((t & 31) == 0) wmax[t >> 5] = mx;
    __syncthreads();
    mx = 0.f;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) mx = fmaxf(mx, wmax[w]);
    // |X_k|^2 = 2^-2s ((2^s X.re)^2 + (2^s X.im)^2): the power-of-two scale is exact and brings the largest
    // component near 2^40, so the FP32 squares neither overflow nor underflow (strain spectra sit near
    // 1e-19, whose squares are below FP32's range); the sum is rounded once in FP32 (relative 1.2e-7, far
    // below the FP32 transform's own error) and stored as it is, with the exponent -2s in the row: half the
    // bytes of the double it stands for.  NaN and infinity pass through.
    int e = 0;
    frexpf(mx, &e);
    const int sc = min(40 - e, 120);
    const float s2 = __int_as_float((127 + sc) << 23);  // 2^sc (sc >= -88)
    // c_k scale |X_k|^2 (the density scale and one-sided doubling of the mean, applied here so that the mean
    // over segments is a plain sum)
    auto p2 = [&](float2 q, float f) {
        const float a = q.x * s2, b = q.y * s2, u = fmaf(b, b, a * a) * f;
        return u < 0x1p-126f ? 0.f : u;  // zero (or below 2^-126 of the scaled range); NaN stays
    };
    const float f2 = 2.0f * scale;
    float4 *o4 = reinterpret_cast<float4 *>(out + 16 * t);  // (rows are 16-byte aligned)
#pragma unroll
    for (int m = 0; m < 4; ++m)
        o4[m] = make_float4(p2(X[4 * m], (t | m) ? f2 : scale), p2(X[4 * m + 1], f2), p2(X[4 * m + 2], f2), p2(X[4 * m + 3], f2));
    if (t == NT - 1) {
        out[NC] = p2(Xn, scale);
        out[PER_EXP] = __int_as_float(mx == 0.f ? PER_ZERO : -2 * sc);
    }
}

// The double u 2^e, bit by bit (no FP64 instruction); u zero, normal, infinite or NaN.
__device__ __forceinline__ double scaled_double(float v, int e) {
    const uint32_t u = __float_as_uint(v) & 0x7FFFFFFFu;
    uint32_t hi = (u >> 3) + ((uint32_t)(896 + e) << 20), lo = u << 29;
    if (u >= 0x7F800000u) hi = 0x7FF00000u | (u & 0x7FFFFFu ? 0x80000u : 0u), lo = 0u;
    if (u < 0x00800000u) hi = lo = 0u;
    return __hiloint2double((int)hi, (int)lo);
}

// Two sums of non-negative floats (two bins) as h + l (l a few roundings of h at most), in packed instructions
struct Pair2 {
    float2 h, l;
};
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ Pair2 padd(Pair2 a, Pair2 b) {
    const float2 s = __fadd2_rn(a.h, b.h), t = sub2(s, a.h);
    const float2 e = __fadd2_rn(sub2(a.h, sub2(s, t)), sub2(b.h, t));
    return {s, __fadd2_rn(__fadd2_rn(a.l, b.l), e)};
}
__device__ __forceinline__ Pair2 padd(Pair2 a, float2 b) {
    const float2 s = __fadd2_rn(a.h, b), t = sub2(s, a.h);
    return {s, __fadd2_rn(a.l, __fadd2_rn(sub2(a.h, sub2(s, t)), sub2(b, t)))};
}
__device__ __forceinline__ Pair2 psum(float2 a, float2 b) {
    const float2 s = __fadd2_rn(a, b), t = sub2(s, a);
    return {s, __fadd2_rn(sub2(a, sub2(s, t)), sub2(b, t))};
}
// The double (h + l) 2^e from its bits: the low part as an integer of the high part's last double place.  (A sum with
// an infinity in it: the high part is infinite, the low one NaN from inf - inf.)
__device__ __forceinline__ double pair_double(float ah, float al, int e) {
    const float h = __fadd_rn(ah, al), l = __fsub_rn(al, __fsub_rn(h, ah));
    const uint32_t u = __float_as_uint(h), E = u >> 23;
    if (E - 1u >= 253u) return scaled_double(isinf(ah) ? ah : h, e);  // zero, (nearly) infinite or NaN
    const int li = __float2int_rn(l * __uint_as_float((254 - E) << 23) * 0x1p52f);  // |l| <= half a place of h: < 2^28
    // mantissa 2^52 (1.m) + li in two words
    uint32_t lo = (u << 29) + (uint32_t)li;
    uint32_t hi = ((u & 0x7FFFFFu) >> 3) + (uint32_t)(li >> 31) + (lo < (u << 29) ? 1u : 0u);  // (below the leading one)
    int ed = (int)E + 896 + e;
    if (hi >> 31) {  // h a power of two and l < 0: one binade down
        hi = (((hi + 0x100000u) << 1) | (lo >> 31)) - 0x100000u;
        lo <<= 1;
        --ed;
    }
    return __hiloint2double((int)(((uint32_t)ed << 20) + hi), (int)lo);
}

// The epochs [0, n_e) of one bin in FP64: column src of a run's rows (the row's exponent is src[exp]) into dst.
// The sum slides: the segments that enter are added and those that leave subtracted.  An error stays in the sum at the
// size of the largest it has been, so where it has fallen by 2^8 (a much louder segment left) or is no longer finite it
// is formed afresh.  Bound by FP64 additions (16 clk a warp and SM, 63 clk from one to the next) where the runs are many, by
// the latency of the loads where they are few: those of B terms are in flight together, one bin a thread and blocks of
// 64 (two bins a thread, a term at a time: 258 us for one PSD of 439 segments, 592 for 40 at step 8; so 47 and 97).
constexpr int PSD_CANCEL = 8 << 20;  // 2^8 in the high word of a double

// K terms from row src on, in order
__device__ __noinline__ double psd_sum64(const float *src, int exp, int K) {
    constexpr int B = 16;
    double a = 0.0;
    for (int q = 0; q < K; q += B, src += B * PER_ROW) {
        float v[B];
        int e[B];
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const float *r = src + min(i, K - 1 - q) * PER_ROW;
            v[i] = r[0];
            e[i] = __float_as_int(r[exp]);
        }
#pragma unroll
        for (int i = 0; i < B; ++i)
            if (q + i < K) a += scaled_double(v[i], e[i]);
    }
    return a;
}

__device__ __forceinline__ void psd_run64(const float *src, int exp, int seg_step, int K, double *dst, int n_e) {
    constexpr int B = 8;
    if (seg_step >= K) {  // no segment is shared
        for (int i = 0; i < n_e; ++i) dst[(int64_t)i * NBIN] = psd_sum64(src + (int64_t)i * seg_step * PER_ROW, exp, K);
        return;
    }
    double acc = psd_sum64(src, exp, K);
    *dst = acc;
    int top = __double2hiint(acc);  // of the largest sum since the last fresh one (non-negative doubles order as ints)
    const int n = (n_e - 1) * seg_step;  // slides by one segment; epoch i is reached after i seg_step
    const int64_t ahead = (int64_t)K * PER_ROW;
    int left = seg_step;
    for (int j = 0; j < n; j += B, src += B * PER_ROW) {
        float in[B], out[B];
        int ei[B], eo[B];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const float *r = src + min(b, n - 1 - j) * PER_ROW;
            out[b] = r[0];
            eo[b] = __float_as_int(r[exp]);
            in[b] = r[ahead];
            ei[b] = __float_as_int(r[ahead + exp]);
        }
#pragma unroll
        for (int b = 0; b < B; ++b) {
            if (j + b >= n) return;
            acc += scaled_double(in[b], ei[b]) - scaled_double(out[b], eo[b]);
            const int hi = __double2hiint(acc);
            top = max(top, hi);
            if (--left == 0) {
                left = seg_step;
                dst += NBIN;
                if (hi < top - PSD_CANCEL || hi >= 0x7FF00000) {
                    acc = psd_sum64(src + (b + 1) * PER_ROW, exp, K);
                    top = __double2hiint(acc);
                }
                *dst = acc;
            }
        }
    }
}

constexpr int PSD_SEGS = 512;  // segments of a run the pair sums hold scales for

// Sums in pairs of floats (else in FP64): up to 16 segments, whose run's scales fit, and fewer than 8 times the step
// (else the slide's few FP64 additions are less than K pair additions an epoch, as 113 us against 88 for 500 epochs of
// 15 segments at step 1 and 158 for either at 16 and 2).
inline bool psd_pairs(int64_t n_psd, int64_t seg_step, int64_t K) {
    return K <= 16 && (n_psd == 1 || K < 8 * seg_step) && (std::min<int64_t>(PSD_EPT, n_psd) - 1) * seg_step + K <= PSD_SEGS;
}

// grid (ceil(NBIN / PSD_T64), ceil(n_psd / PSD_EPT), n_det): epochs as FP64 sums
constexpr int PSD_T64 = 64;

__global__ void __launch_bounds__(PSD_T64) k_psd_mean64(const float *P, int64_t n_seg, int seg_step, int K, double *psd,
                                                        int64_t n_psd) {
    const int k = blockIdx.x * PSD_T64 + threadIdx.x;
    const int64_t e0 = (int64_t)blockIdx.y * PSD_EPT;
    pdl_trigger();  // (launched plainly)
    if (k >= NBIN) return;
    psd_run64(P + ((int64_t)blockIdx.z * n_seg + e0 * seg_step) * PER_ROW + k, PER_EXP - k, seg_step, K,
              psd + ((int64_t)blockIdx.z * n_psd + e0) * NBIN + k, (int)min((int64_t)PSD_EPT, n_psd - e0));
}

// grid (ceil(NBIN / 2 PSD_T), ceil(n_psd / PSD_EPT), n_det): the bins of epochs [e0, e0 + PSD_EPT) as sums of the
// periodograms (already scaled by the density factor; epoch e sums segments [e seg_step, e seg_step + K)).
// The sums are pairs of floats over the run's largest exponent (about 46 bits; the terms have 24 and an FP32
// transform's error) and only the result is a double: this GPU retires 2 FP64 adds a clock and SM, and the FP64
// prefix sums of the 64 s PSDs kept that pipe 81 % busy.  For those (step 2, 15 segments) an epoch is a tree
// over shared partial sums: with A_i = P_2i + P_2i+1, B_i = A_i + A_i+1, C_i = B_i + B_i+2, epoch e is
// C_e + B_e+4 + A_e+6 + P_2e+14, six pair additions.  Other short sums (psd_pairs) are formed directly; runs
// whose exponents differ by more than 80 (a segment 2^40 times another) in FP64.
// A thread takes bins k and k + PSD_T as the halves of packed additions (the loads and stores of both coalesce).
constexpr int PSD_T = 128;

__global__ void __launch_bounds__(PSD_T) k_psd_mean(const float *P, int64_t n_seg, int seg_step, int K,
                                                    double *__restrict__ psd, int64_t n_psd) {
    __shared__ float sf[PSD_SEGS];  // 2^(e_s - e_max) of the run's segments
    __shared__ int elo, ehi;
    const int tid = threadIdx.x, k = blockIdx.x * 2 * PSD_T + tid;
    const int64_t e0 = (int64_t)blockIdx.y * PSD_EPT;
    const int n_e = (int)min((int64_t)PSD_EPT, n_psd - e0);
    const float *src = P + ((int64_t)blockIdx.z * n_seg + e0 * seg_step) * PER_ROW;
    double *dst = psd + ((int64_t)blockIdx.z * n_psd + e0) * NBIN + k;
    const int64_t ns = (int64_t)(n_e - 1) * seg_step + K;
    pdl_wait();
    pdl_trigger();
    bool pairs;
    {
        if (tid == 0) {
            elo = 1 << 20;
            ehi = -(1 << 20);
        }
        __syncthreads();
        for (int s = tid; s < ns; s += PSD_T) {
            const int e = __float_as_int(src[(int64_t)s * PER_ROW + PER_EXP]);
            if (e == PER_ZERO) continue;
            atomicMin(&elo, e);
            atomicMax(&ehi, e);
        }
        __syncthreads();
        pairs = ehi - elo <= 80;
        if (pairs)
            for (int s = tid; s < ns; s += PSD_T) {
                const int e = __float_as_int(src[(int64_t)s * PER_ROW + PER_EXP]);
                sf[s] = e == PER_ZERO ? 0.f : __int_as_float((127 + e - ehi) << 23);
            }
        __syncthreads();
    }
    const bool second = k + PSD_T < NBIN;  // (else the second half repeats the first)
    if (k >= NBIN) return;
    const int k2 = second ? PSD_T : 0;
    src += k;
    auto put = [&](int i, Pair2 a) {
        dst[(int64_t)i * NBIN] = pair_double(a.h.x, a.l.x, ehi);
        if (second) dst[(int64_t)i * NBIN + PSD_T] = pair_double(a.h.y, a.l.y, ehi);
    };
    const float2 zero = make_float2(0.f, 0.f);
    if (pairs && seg_step == 2 && K == 15) {
        constexpr int ST = 6;  // steps whose loads are in flight together
        Pair2 a1 = {zero, zero}, b1 = a1, b2 = a1, c1 = a1, c2 = a1, c3 = a1;  // A_i-1, B_i-2 .., C_i-4 ..
        float2 p = make_float2(src[0] * sf[0], src[k2] * sf[0]);
        const float *row = src + PER_ROW;
        for (int i0 = 0; i0 < n_e + 6; i0 += ST, row += 2 * ST * PER_ROW) {
            float2 q[2 * ST];
            if (2 * (i0 + ST) < ns) {
#pragma unroll
                for (int j = 0; j < 2 * ST; ++j) {
                    const float f = sf[2 * i0 + 1 + j];
                    q[j] = make_float2(row[j * PER_ROW] * f, row[j * PER_ROW + k2] * f);
                }
            } else {
#pragma unroll
                for (int j = 0; j < 2 * ST; ++j) {
                    const bool in = 2 * i0 + 1 + j < ns;
                    const float f = in ? sf[2 * i0 + 1 + j] : 0.f;
                    q[j] = in ? make_float2(row[j * PER_ROW] * f, row[j * PER_ROW + k2] * f) : zero;
                }
            }
#pragma unroll
            for (int j = 0; j < ST; ++j) {
                const int i = i0 + j;
                const Pair2 a = psum(p, q[2 * j]);
                p = q[2 * j + 1];
                // the newest A is a = A_i: B_i-1, C_i-3, epoch i - 6
                const Pair2 b = padd(a1, a), c = padd(b2, b);
                if (i >= 6 && i < n_e + 6) put(i - 6, padd(padd(padd(c3, b1), a), p));
                a1 = a;
                b2 = b1;
                b1 = b;
                c3 = c2;
                c2 = c1;
                c1 = c;
            }
        }
        return;
    }
    if (pairs) {
        for (int i = 0; i < n_e; ++i) {
            Pair2 a = {zero, zero};
#pragma unroll 5
            for (int q = 0; q < K; ++q) {
                const int s = i * seg_step + q;
                const float *r = src + (int64_t)s * PER_ROW;
                a = padd(a, make_float2(r[0] * sf[s], r[k2] * sf[s]));
            }
            put(i, a);
        }
        return;
    }
    // (psd_run64's code beside the pair sums takes them from 71 registers to 96 and a fifth of their rate)
#pragma unroll 1
    for (int i = 0; i < n_e * (second ? 2 : 1); ++i) {
        const int e = second ? i >> 1 : i, kk = second && (i & 1) ? PSD_T : 0;
        const float *r = src + (int64_t)e * seg_step * PER_ROW;
        double a = 0.0;
#pragma unroll 4
        for (int q = 0; q < K; ++q, r += PER_ROW) a += scaled_double(r[kk], __float_as_int(r[PER_EXP - k]));
        dst[(int64_t)e * NBIN + kk] = a;
    }
}

// 4-byte asynchronous copy global -> shared (completes at cp_async_wait_all)
__device__ __forceinline__ void cp_async4(float *dst, const float *src) {
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
}

// Fused mid pass of the whitening kernel for task j, 1 <= j <= NCX / 4, of a
// transform of NCX complex points (H = NCX / 2): the forward radix-2 butterflies j
// and H - j (Ns = H) give Z at j, j + H, H - j, NCX - j; the split pairs (j, NCX - j)
// and (j + H, H - j) are multiplied by the gains g (on the transform's own grid) and
// split back; the inverse radix-2 butterflies j and H - j (Ns = 1) produce o[0..1]
// for d[2j], d[2j + 1] and o[2..3] for d[2(H - j)], d[2(H - j) + 1].
template <int NCX>
__device__ __forceinline__ void whiten_mid_task(const float2 *d, const float *g, int j, float2 (&o)[4]) {
    using namespace r16;
    constexpr int H = NCX / 2;
    const float2 a = d[pad(j)], b = d[pad(j + H)], c = d[pad(H - j)], e = d[pad(NCX - j)];
    static_assert(8192 % NCX == 0, "split table step");
    constexpr int SP = 8192 / NCX;
    const float2 w = tw_split<-1>(SP * j);      // W^j, W = exp(-2 pi i / 2 NCX)
    const float2 u = tw_split<-1>(2 * SP * j);  // radix-2 twiddle of butterfly j
    const float2 u2 = make_float2(-u.x, u.y);               // of butterfly H - j
    const float2 ub = cmul(u, b), ue = cmul(u2, e);
    const float2 zj = cadd(a, ub), zj4 = csub(a, ub), zc = cadd(c, ue), zc4 = csub(c, ue);
    const float2 w4 = mul_i<-1>(w);                         // W^{j + H}
    float2 x1, x1n, x2, x2n, p1, p1n, p2, p2n;
    split_fwd(zj, zc4, w, x1, x1n);
    split_fwd(zj4, zc, w4, x2, x2n);
    split_inv(cscale(x1, g[j]), cscale(x1n, g[NCX - j]), w, p1, p1n);     // Z'_j, Z'_{NCX-j}
    split_inv(cscale(x2, g[j + H]), cscale(x2n, g[H - j]), w4, p2, p2n);  // Z'_{j+H}, Z'_{H-j}
    o[0] = cadd(p1, p2);
    o[1] = csub(p1, p2);
    o[2] = cadd(p2n, p1n);
    o[3] = csub(p2n, p1n);
}

// Task 0 of the mid pass: butterfly 0 gives Z_0 and Z_H, each its own split partner
// (bin 0 with the Nyquist bin NCX, and bin H); o[0..1] go to d[0], d[1].
template <int NCX>
__device__ __forceinline__ void whiten_mid_task0(const float2 *d, const float *g, float2 (&o)[4]) {
    using namespace r16;
    constexpr int H = NCX / 2;
    const float2 a = d[pad(0)], b = d[pad(H)];
    const float2 z0 = cadd(a, b), z4 = csub(a, b);
    const float2 one = make_float2(1.0f, 0.0f), mi = make_float2(0.0f, -1.0f);  // W^0, W^H
    float2 x0, xn, x4, x4d, p0, pn, p4, p4d;
    split_fwd(z0, z0, one, x0, xn);
    split_inv(cscale(x0, g[0]), cscale(xn, g[NCX]), one, p0, pn);
    split_fwd(z4, z4, mi, x4, x4d);
    split_inv(cscale(x4, g[H]), cscale(x4d, g[H]), mi, p4, p4d);
    o[0] = cadd(p0, p4);
    o[1] = csub(p0, p4);
    o[2] = o[0];
    o[3] = o[1];
}

constexpr int WHITEN_SMEM = r16::SLOTS * (int)sizeof(float2) + NBIN * (int)sizeof(float);
// density factor of the mean of K periodograms (periodic Hann: sum w^2 = 3 NFFT / 8), applied per segment
inline float psd_scale(int64_t K, int fs) { return (float)(1.0 / ((double)K * (double)fs * (3.0 * NFFT / 8.0))); }

constexpr int WELCH_SMEM = (r16::SLOTS + 1) * (int)sizeof(float2) + (r16::NT / 32) * (int)sizeof(float);

// One overlap-save block: the FIR of src[0 .. cnt + F - 1) (cnt <= 16385 - F; samples past
// `avail` read as zero) -> outputs q in [0, cnt) written as out(q, value), or straight to lin[q]
// when the caller's destination is the linear row lin (nullptr: always through out).
// smem: r16::SLOTS float2 for the transform, then NBIN floats for the gains gk,
// which are copied in asynchronously while the forward transform runs.
// EARLY: the samples are complete before the launch, the gains only after pdl_wait(), which comes after the forward
// transform.
template <bool EARLY = false, typename Out>
__device__ __forceinline__ void whiten_block(unsigned char *smem, const float *__restrict__ src, int64_t avail,
                                             const float *__restrict__ gk, int F, int64_t cnt, Out out,
                                             float *__restrict__ lin = nullptr) {
    using namespace r16;
    float2 *d = reinterpret_cast<float2 *>(smem);
    float *gs = reinterpret_cast<float *>(smem + SLOTS * sizeof(float2));
    const int t = threadIdx.x;
    if (!EARLY)
        for (int k = t; k < NBIN; k += NT) cp_async4(gs + k, gk + k);
    const int half = F / 2;
    // samples that reach a kept output (cnt + F - 1 <= 16384: indices within the block are ints)
    const int need = (int)cnt + F - 1;
    const int lim = avail <= 0 ? 0 : avail < (int64_t)need ? (int)avail : need;
    float2 v[16];
    if (avail >= 2 * NC && (reinterpret_cast<uintptr_t>(src) & 7) == 0) {  // whole block in memory: 8-byte loads
        const float2 *s2 = reinterpret_cast<const float2 *>(src);
#pragma unroll
        for (int r = 0; r < 16; ++r) v[r] = s2[t + NT * r];
        if (2 * (t + NT * 15) + 1 >= lim) {  // this thread holds samples past `need`: they read as zero
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const int i0 = 2 * (t + NT * r);
                if (i0 >= lim) v[r].x = 0.0f;
                if (i0 + 1 >= lim) v[r].y = 0.0f;
            }
        }
    } else {
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const int i0 = 2 * (t + NT * r);
            v[r] = make_float2(i0 < lim ? src[i0] : 0.0f, i0 + 1 < lim ? src[i0 + 1] : 0.0f);
        }
    }
    forward_r16(d, v);
    if (EARLY) {
        pdl_wait();
        pdl_trigger();
        for (int k = t; k < NBIN; k += NT) cp_async4(gs + k, gk + k);
    }
    cp_async_wait_all();
    __syncthreads();
    float2 o[4][4], ox[4];
    if (t == 0) whiten_mid_task0<NC>(d, gs, o[0]);
    else whiten_mid_task<NC>(d, gs, t, o[0]);
#pragma unroll
    for (int m = 1; m < 4; ++m) whiten_mid_task<NC>(d, gs, t + NT * m, o[m]);
    if (t == NT - 1) whiten_mid_task<NC>(d, gs, 2048, ox);
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        const int j = t + NT * m, jc = 4096 - j;
        d[pad(2 * j)] = o[m][0];
        d[pad(2 * j + 1)] = o[m][1];
        if (j != 0) {
            d[pad(2 * jc)] = o[m][2];
            d[pad(2 * jc + 1)] = o[m][3];
        }
    }
    if (t == NT - 1) {
        d[pad(4096)] = ox[0];
        d[pad(4097)] = ox[1];
    }
    __syncthreads();
    inverse_r16(d, v);
    // complex sample c = t + 512 q holds real samples 2c, 2c + 1; output q0 = 2c - F/2
    const int cnt32 = (int)cnt;
    // outputs (q0, q0 + 1) as one 8-byte store where the destination is linear and q0 lands 8-byte aligned
    const bool pairs = lin != nullptr && (half & 1) == 0 && (reinterpret_cast<uintptr_t>(lin) & 7) == 0;
#pragma unroll
    for (int q = 0; q < 16; ++q) {
        const float2 y = v[out16(q)];
        const int q0 = 2 * (t + NT * q) - half;
        if (pairs && q0 >= 0 && q0 + 1 < cnt32) {
            *reinterpret_cast<float2 *>(lin + q0) = y;
        } else {
            if (q0 >= 0 && q0 < cnt32) out(q0, y.x);
            if (q0 + 1 >= 0 && q0 + 1 < cnt32) out(q0 + 1, y.y);
        }
    }
}

template <typename Out>
__device__ __forceinline__ void whiten_block_s(unsigned char *smem, const float *__restrict__ src, int64_t avail,
                                               const float *__restrict__ stg, int64_t i_new,
                                               const float *__restrict__ gk, int F, int64_t cnt, Out out);

// Block layout of one whitening launch.  Every filter epoch (the whole span when epoch_len is 0) is covered by
// blocks of bl = 16385 - F outputs (rounded down to 64) on the 16384-point transform, the most its circular
// convolution keeps, and the epoch's remainder by one more block: on the 4096-point transform where it fits
// (4097 - F outputs; 2048 of a 16384-sample epoch with F = 2048), else on the 16384-point one.  An 8192-output
// block instead would keep half of every 16384-point transform.
struct WhitenLayout {
    int64_t span, bl, n_full, rem, bpe, n_blocks;
    bool small_rem;
};
__host__ __device__ inline WhitenLayout whiten_layout(int64_t out_len, int64_t epoch_len, int F) {
    WhitenLayout w;
    w.span = epoch_len > 0 ? epoch_len : out_len;
    w.bl = ((int64_t)(2 * r16::NT * 16 + 1 - F) / 64) * 64;
    w.n_full = w.span / w.bl;
    w.rem = w.span - w.n_full * w.bl;
    w.bpe = w.n_full + (w.rem > 0 ? 1 : 0);
    w.small_rem = w.rem > 0 && w.rem <= (int64_t)(2 * r16::NC_S + 1 - F);
    const int64_t n_ep = epoch_len > 0 ? (out_len + epoch_len - 1) / epoch_len : 1;
    w.n_blocks = out_len > 0 ? n_ep * w.bpe : 0;
    return w;
}

// Block (e, i) of a whitening launch: y[d][e span + i bl, + cnt) with the gains of epoch e (cnt <= 0: none)
struct WhitenBlock {
    int64_t o, cnt, ep;
};
__device__ __forceinline__ WhitenBlock whiten_block_at(const WhitenLayout &L, int64_t e, int64_t i, int64_t out_len,
                                                       int64_t epoch_len, int64_t n_psd) {
    WhitenBlock b;
    b.o = e * L.span + i * L.bl;
    b.cnt = i < L.n_full ? L.bl : L.rem;
    if (b.cnt > out_len - b.o) b.cnt = out_len - b.o;
    b.ep = epoch_len > 0 ? e : 0;
    if (b.ep > n_psd - 1) b.ep = n_psd - 1;
    return b;
}

// grid (n_ep * n16, n_det): the blocks on the 16384-point transform, n16 per epoch (bpe, or n_full where the
// remainder goes to k_whiten_rem); block (e, i) = (blockIdx.x / n16, blockIdx.x % n16).
// EARLY (one wave of blocks, which find room beside the few CTAs of a short filter build): a programmatic dependent of
// the build, which triggers once what came before it is complete, so the forward transforms run during the build.
// Else the gains come in during the forward transform.
template <bool EARLY>
__global__ void __launch_bounds__(r16::NT, 2) k_whiten(const float *__restrict__ x, int64_t n, int64_t x_stride,
                                                        const float *gains, int64_t n_psd,
                                                        int64_t out_first, int64_t out_len, int64_t epoch_len, int F,
                                                        float *__restrict__ y, int64_t y_stride) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const WhitenLayout L = whiten_layout(out_len, epoch_len, F);
    const int64_t n16 = L.small_rem ? L.n_full : L.bpe;
    const int64_t e = (int64_t)blockIdx.x / n16;
    const WhitenBlock b = whiten_block_at(L, e, (int64_t)blockIdx.x - e * n16, out_len, epoch_len, n_psd);
    if (b.cnt <= 0) return;
    const int det = blockIdx.y;
    const int64_t s0 = out_first + b.o - F / 2;  // raw index of block sample 0
    float *dst = y + det * y_stride + b.o;
    whiten_block<EARLY>(smem_raw, x + det * x_stride + s0, n - s0, gains + ((int64_t)det * n_psd + b.ep) * NBIN, F, b.cnt,
                        [dst](int64_t q, float v) { dst[q] = v; }, dst);
}

// grid (n_ep, n_det): each epoch's remainder block on the 4096-point transform (whiten_layout().small_rem).
// A launch of its own: its 26 KB of shared memory lets several CTAs share an SM, which the short transform's
// barrier-bound passes need.
__global__ void __launch_bounds__(r16::NT_S) k_whiten_rem(const float *__restrict__ x, int64_t n, int64_t x_stride,
                                                         const float *__restrict__ gains, int64_t n_psd,
                                                         int64_t out_first, int64_t out_len, int64_t epoch_len, int F,
                                                         float *__restrict__ y, int64_t y_stride) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_trigger();  // (launched plainly)
    const WhitenLayout L = whiten_layout(out_len, epoch_len, F);
    const WhitenBlock b = whiten_block_at(L, blockIdx.x, L.n_full, out_len, epoch_len, n_psd);
    if (b.cnt <= 0) return;
    const int det = blockIdx.y;
    const int64_t s0 = out_first + b.o - F / 2;
    float *dst = y + det * y_stride + b.o;
    whiten_block_s(smem_raw, x + det * x_stride + s0, n - s0, nullptr, 0, gains + ((int64_t)det * n_psd + b.ep) * NBIN,
                   F, b.cnt, [dst](int64_t q, float v) { dst[q] = v; });
}

// Whitening pieces of many streams in one launch: grid (n_desc, 2).  Piece i
// whitens raw samples src(d) = desc.x + d * x_stride + [0, cnt + F - 1) with
// gains desc.gains + d * NBIN into the mirrored ring desc.y (row stride
// y_stride, ring length y_ring): output q goes to ring slots
// (y_pos + q) mod y_ring and that + y_ring.
// (Launched as a programmatic dependent of the scatter or gains refresh before it.)
__global__ void __launch_bounds__(r16::NT, 2) k_whiten_multi(const WhitenPiece *__restrict__ pieces, int F) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_trigger();
    const WhitenPiece pc = pieces[blockIdx.x];
    pdl_wait();  // raw rings (scatter) and gains (refresh) come from the kernels before
    const int det = blockIdx.y;
    float *yr = pc.y + det * pc.y_stride;
    const int64_t ring = pc.y_ring, pos = pc.y_pos;
    whiten_block(smem_raw, pc.x + det * pc.x_stride, pc.cnt + F - 1, pc.gains + det * NBIN, F, pc.cnt,
                 [yr, ring, pos](int64_t q, float v) {
                     int64_t m = pos + q;
                     if (m >= ring) m -= ring;
                     yr[m] = v;
                     yr[m + ring] = v;
                 });
}

constexpr int WHITEN_SMEM_S = r16::SLOTS_S * (int)sizeof(float2) + (r16::NC_S + 1) * (int)sizeof(float);

// Largest piece of the 4096-point block for a filter of F taps (0 if F leaves too few).
int whiten_piece_max_s(int F) {
    const int m = 2 * r16::NC_S - F + 1;
    return m >= 512 ? m : 0;
}

// One overlap-save block of the 4096-point transform: the FIR of src[0 .. cnt + F - 1)
// (cnt <= 4097 - F, samples past `avail` read as zero) -> outputs q in [0, cnt) written as
// out(q, value).  The taps span fewer than 4096 lags, so the gains of this grid are those
// of the 16384-point grid at every 4th bin; they are rescaled by 4 for the shorter
// transform's 1 / 2048 normalisation (exact in FP32).
// stg (may be null): input i >= i_new comes from stg[i - i_new] instead of src[i].
template <typename Out>
__device__ __forceinline__ void whiten_block_s(unsigned char *smem, const float *__restrict__ src, int64_t avail,
                                               const float *__restrict__ stg, int64_t i_new,
                                               const float *__restrict__ gk, int F, int64_t cnt, Out out) {
    using namespace r16;
    constexpr int GS = NC / NC_S;  // bins of the 16384-point grid per bin of this one
    float2 *d = reinterpret_cast<float2 *>(smem);
    float *gs = reinterpret_cast<float *>(smem + SLOTS_S * sizeof(float2));
    const int t = threadIdx.x;
    for (int k = t; k <= NC_S; k += NT_S) cp_async4(gs + k, gk + GS * k);
    const int half = F / 2;
    const int64_t need = cnt + F - 1;
    const int64_t lim = need < avail ? need : avail;
    auto sample = [&](int64_t i) -> float {
        if (i >= lim) return 0.0f;
        return (stg && i >= i_new) ? stg[i - i_new] : src[i];
    };
    float2 v[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int64_t i0 = 2 * (int64_t)(t + NT_S * r);
        v[r] = make_float2(sample(i0), sample(i0 + 1));
    }
    forward_s(d, v);
    cp_async_wait_all();
    __syncthreads();
    for (int k = t; k <= NC_S; k += NT_S) gs[k] *= (float)GS;
    __syncthreads();
    // one task per thread (tasks 0 .. NC_S / 4 - 1), the last thread also task NC_S / 4
    static_assert(NT_S == NC_S / 4, "one mid-pass task per thread");
    float2 o[4], ox[4];
    if (t == 0) whiten_mid_task0<NC_S>(d, gs, o);
    else whiten_mid_task<NC_S>(d, gs, t, o);
    if (t == NT_S - 1) whiten_mid_task<NC_S>(d, gs, NC_S / 4, ox);
    __syncthreads();
    {
        const int j = t, jc = NC_S / 2 - j;
        d[pad(2 * j)] = o[0];
        d[pad(2 * j + 1)] = o[1];
        if (j != 0) {
            d[pad(2 * jc)] = o[2];
            d[pad(2 * jc + 1)] = o[3];
        }
    }
    if (t == NT_S - 1) {
        d[pad(NC_S / 2)] = ox[0];
        d[pad(NC_S / 2 + 1)] = ox[1];
    }
    __syncthreads();
    float2 y[4];
    inverse_s(d, y);
    // complex sample c = t + 512 r holds real samples 2c, 2c + 1; output q0 = 2c - F/2
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int64_t q0 = 2 * (int64_t)(t + NT_S * r) - half;
        if (q0 >= 0 && q0 < cnt) out(q0, y[r].x);
        if (q0 + 1 >= 0 && q0 + 1 < cnt) out(q0 + 1, y[r].y);
    }
}

// k_whiten_multi with the 4096-point block (512 threads): pieces of at most 4097 - F outputs.
__global__ void __launch_bounds__(r16::NT_S) k_whiten_multi_s(const WhitenPiece *__restrict__ pieces, int F) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    pdl_trigger();
    const WhitenPiece pc = pieces[blockIdx.x];
    pdl_wait();  // raw rings (scatter) and gains (refresh) come from the kernels before
    const int det = blockIdx.y;
    const float *stg = pc.stg ? pc.stg + det * pc.stg_stride : nullptr;
    if (pc.sc_ring) {  // the stream's new samples into its mirrored raw ring (read by later steps)
        float *row = pc.sc_ring + det * 2 * pc.sc_R;
        for (int64_t k = threadIdx.x; k < pc.sc_n; k += r16::NT_S) {
            int64_t m = pc.sc_pos + k;
            if (m >= pc.sc_R) m -= pc.sc_R;
            const float v = stg[k];
            row[m] = v;
            row[m + pc.sc_R] = v;
        }
    }
    float *yr = pc.y + det * pc.y_stride;
    const int64_t ring = pc.y_ring, pos = pc.y_pos;
    whiten_block_s(smem_raw, pc.x + det * pc.x_stride, pc.cnt + F - 1, stg, pc.i_new, pc.gains + det * NBIN, F,
                   pc.cnt,
                   [yr, ring, pos](int64_t q, float v) {
                       int64_t m = pos + q;
                       if (m >= ring) m -= ring;
                       yr[m] = v;
                       yr[m + ring] = v;
                   });
}

int set_attrs(afg_ctx *ctx) {
    AFG_CUDA(ctx, allow_smem(k_periodogram, WELCH_SMEM));
    AFG_CUDA(ctx, allow_smem(k_whiten<false>, WHITEN_SMEM));
    AFG_CUDA(ctx, allow_smem(k_whiten<true>, WHITEN_SMEM));
    AFG_CUDA(ctx, allow_smem(k_whiten_multi, WHITEN_SMEM));
    AFG_CUDA(ctx, allow_smem(k_whiten_multi_s, WHITEN_SMEM_S));
    return AFG_OK;
}

}  // namespace

// Fill the FP32 twiddle table of the current device once per process (it is a per-module device variable;
// every context on the device and the context-free Welch entry point share it).  Synchronous: the table is
// complete when this returns, before any transform can be launched on the device.
static cudaError_t ensure_tw32() {
    static std::mutex mu;
    static bool done[256] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 256) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(mu);
    if (done[dev]) return cudaSuccess;
    cudaStream_t st;
    if ((e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking)) != cudaSuccess) return e;
    k_tw32<<<(r16::TW_TOTAL + 255) / 256, 256, 0, st>>>();
    e = cudaGetLastError();
    const cudaError_t e2 = cudaStreamSynchronize(st);
    cudaStreamDestroy(st);
    if (e == cudaSuccess) e = e2;
    if (e == cudaSuccess) done[dev] = true;
    return e;
}

int afg_make_twiddles(afg_ctx *ctx) {
    if (ensure_tw32() != cudaSuccess) return AFG_ERR_CUDA;
    return set_attrs(ctx);
}

// the mean over the epochs of n_rows rows of periodograms, a programmatic dependent of their launch
static cudaError_t launch_psd_mean(const float *P, int64_t n_seg, int seg_step, int K, double *psd, int64_t n_psd, int n_rows,
                                   cudaStream_t st) {
    if (!psd_pairs(n_psd, seg_step, K)) {
        // (launched plainly: early blocks crowd the first SMs that fall free, and those SMs' FP64 pipes: one PSD of 439
        // segments 102 us, 47 so)
        k_psd_mean64<<<dim3((NBIN + PSD_T64 - 1) / PSD_T64, (unsigned)((n_psd + PSD_EPT - 1) / PSD_EPT), n_rows), PSD_T64, 0, st>>>(
            P, n_seg, seg_step, K, psd, n_psd);
        return cudaGetLastError();
    }
    return launch_pdl(k_psd_mean, dim3((NBIN + 2 * PSD_T - 1) / (2 * PSD_T), (unsigned)((n_psd + PSD_EPT - 1) / PSD_EPT), n_rows),
                      dim3(PSD_T), 0, st, P, n_seg, seg_step, K, psd, n_psd);
}

int launch_psd(afg_ctx *ctx, const float *x, int64_t n, int n_det, int64_t n_psd, int64_t psd_step,
               int64_t psd_span, double *psd, cudaStream_t st, int64_t x_stride) {
    if (x_stride <= 0) x_stride = n;
    const int hop = ctx->cfg.hop;
    const int64_t K = (psd_span - NFFT) / hop + 1;
    const int64_t seg_step = n_psd > 1 ? psd_step / hop : 0;
    const int64_t n_seg = (n_psd - 1) * seg_step + K;
    float *P = nullptr;
    int rc = afg_ws_reserve(ctx, WS_PERIODOGRAM, periodogram_bytes(n_det * n_seg), (void **)&P);
    if (rc) return rc;
    if (n_seg > 0x7fffffff) return afg_fail(ctx, AFG_ERR_ARG, "psd_estimate: too many segments");
    {
        // one read of every segment, one periodogram written per segment
        KScope ks(ctx, st, KK_PERIODOGRAM, 0.0, (double)n_det * n_seg * (NFFT * 4.0 + NBIN * 4.0));
        k_periodogram<<<dim3((unsigned)n_seg, n_det), r16::NT, WELCH_SMEM, st>>>(x, x_stride, hop, P, n_seg, nullptr,
                                                                                 psd_scale(K, ctx->cfg.fs));
    }
    AFG_LAUNCH_CHECK(ctx, "k_periodogram");
    {
        KScope ks(ctx, st, KK_PSD_MEAN, 0.0, (double)n_det * (n_seg * 4.0 + n_psd * 8.0) * NBIN);
        AFG_CUDA(ctx, launch_psd_mean(P, n_seg, (int)seg_step, (int)K, psd, n_psd, n_det, st));
    }
    AFG_LAUNCH_CHECK(ctx, "k_psd_mean");
    return AFG_OK;
}

int launch_whiten(afg_ctx *ctx, const float *x, int64_t n, int n_det, const double *psd, int64_t n_psd,
                  int64_t out_first, int64_t out_len, int64_t epoch_len, float *y, int64_t y_stride,
                  cudaStream_t st, int64_t x_stride) {
    if (x_stride <= 0) x_stride = n;
    float *gains = nullptr;
    int rc = afg_ws_reserve(ctx, WS_FILTER, (size_t)n_det * n_psd * NBIN * sizeof(float), (void **)&gains);
    if (rc) return rc;
    rc = launch_filter(ctx, psd, n_det, n_psd, gains, st);
    if (rc) return rc;
    if (out_len <= 0) return AFG_OK;
    const WhitenLayout wl = whiten_layout(out_len, epoch_len, ctx->cfg.fir_len);
    const int64_t n_ep = wl.bpe > 0 ? wl.n_blocks / wl.bpe : 0;
    const int64_t nb = n_ep * (wl.small_rem ? wl.n_full : wl.bpe);
    if (nb > 0x7fffffff) return afg_fail(ctx, AFG_ERR_ARG, "whiten: too many blocks");
    // one wave of blocks after a build of few filters: the forward transforms run beside it (64 s span: 98 -> 86 us with
    // the network's set-up overlapped the same way); a dependent launch of many blocks only took slots (1.38 -> 1.44 ms)
    const bool early = nb * n_det <= 2 * 152 && (int64_t)n_det * n_psd <= 152;
    {
        // algorithmic: read the cropped span once, write the output once, read the gains
        const double F = ctx->cfg.fir_len;
        KScope ks(ctx, st, KK_WHITEN, 0.0, (double)n_det * ((2.0 * out_len + F - 1.0) * 4.0 + n_psd * NBIN * 4.0));
        if (nb > 0 && early)
            AFG_CUDA(ctx, launch_pdl(k_whiten<true>, dim3((unsigned)nb, n_det), dim3(r16::NT), WHITEN_SMEM, st, x, n, x_stride,
                                     (const float *)gains, n_psd, out_first, out_len, epoch_len, (int)ctx->cfg.fir_len, y,
                                     y_stride));
        else if (nb > 0)
            k_whiten<false><<<dim3((unsigned)nb, n_det), r16::NT, WHITEN_SMEM, st>>>(x, n, x_stride, gains, n_psd, out_first,
                                                                                     out_len, epoch_len, ctx->cfg.fir_len,
                                                                                     y, y_stride);
    }
    AFG_LAUNCH_CHECK(ctx, "k_whiten");
    if (wl.small_rem && n_ep > 0) {
        KScope ks(ctx, st, KK_WHITEN, 0.0, 0.0);  // (the bytes are counted with the launch above)
        k_whiten_rem<<<dim3((unsigned)n_ep, n_det), r16::NT_S, WHITEN_SMEM_S, st>>>(
            x, n, x_stride, gains, n_psd, out_first, out_len, epoch_len, ctx->cfg.fir_len, y, y_stride);
    }
    AFG_LAUNCH_CHECK(ctx, "k_whiten_rem");
    return AFG_OK;
}

bool whiten_multi_takes_staging(const afg_ctx *ctx) { return whiten_piece_max_s(ctx->cfg.fir_len) != 0; }

// Most outputs one piece of launch_whiten_multi may hold.
int whiten_multi_piece_max(const afg_ctx *ctx) {
    const int m = whiten_piece_max_s(ctx->cfg.fir_len);
    return m ? m : WB;
}

// One PSD per row of psd_span samples, row r starting at rows_dev[r] (device array of n_rows
// pointers): the Welch periodograms of all rows in one launch and their means in another, into
// psd [n_rows][NBIN].  The same kernels and arithmetic as launch_psd with n_psd = 1.
int launch_psd_rows(afg_ctx *ctx, const float *const *rows_dev, int n_rows, int64_t psd_span, double *psd,
                    cudaStream_t st) {
    if (n_rows <= 0) return AFG_OK;
    const int hop = ctx->cfg.hop;
    const int64_t K = (psd_span - NFFT) / hop + 1;
    float *P = nullptr;
    int rc = afg_ws_reserve(ctx, WS_PERIODOGRAM, periodogram_bytes(n_rows * K), (void **)&P);
    if (rc) return rc;
    {
        KScope ks(ctx, st, KK_PERIODOGRAM, 0.0, (double)n_rows * K * (NFFT * 4.0 + NBIN * 4.0));
        k_periodogram<<<dim3((unsigned)K, (unsigned)n_rows), r16::NT, WELCH_SMEM, st>>>(nullptr, 0, hop, P, K,
                                                                                        rows_dev, psd_scale(K, ctx->cfg.fs));
    }
    AFG_LAUNCH_CHECK(ctx, "k_periodogram");
    {
        KScope ks(ctx, st, KK_PSD_MEAN, 0.0, (double)n_rows * (K * 4.0 + 8.0) * NBIN);
        AFG_CUDA(ctx, launch_psd_mean(P, K, 0, (int)K, psd, 1, n_rows, st));
    }
    AFG_LAUNCH_CHECK(ctx, "k_psd_mean");
    return AFG_OK;
}

// grid (n_rows): row r of src [n_rows][len] to dst_dev[r] (device array of n_rows pointers)
__global__ void k_scatter_rows(const float *__restrict__ src, float *const *__restrict__ dst, int len) {
    const float *s = src + (int64_t)blockIdx.x * len;
    float *d = dst[blockIdx.x];
    for (int i = threadIdx.x; i < len; i += blockDim.x) d[i] = s[i];
}

int launch_scatter_rows(afg_ctx *ctx, const float *src, float *const *dst_dev, int n_rows, int len, cudaStream_t st) {
    if (n_rows <= 0) return AFG_OK;
    k_scatter_rows<<<n_rows, 256, 0, st>>>(src, dst_dev, len);
    AFG_LAUNCH_CHECK(ctx, "k_scatter_rows");
    return AFG_OK;
}

int launch_whiten_multi(afg_ctx *ctx, const WhitenPiece *pieces_dev, int n_pieces, int64_t total_out,
                        cudaStream_t st) {
    if (n_pieces <= 0) return AFG_OK;
    const double F = ctx->cfg.fir_len;
    KScope ks(ctx, st, KK_WHITEN, 0.0, 2.0 * ((2.0 * total_out + n_pieces * (F - 1.0)) * 4.0 + n_pieces * NBIN * 4.0));
    if (whiten_piece_max_s(ctx->cfg.fir_len))  // pieces were cut to the 4096-point block
        AFG_CUDA(ctx, launch_pdl(k_whiten_multi_s, dim3((unsigned)n_pieces, 2), dim3(r16::NT_S), WHITEN_SMEM_S, st,
                                 pieces_dev, ctx->cfg.fir_len));
    else
        AFG_CUDA(ctx, launch_pdl(k_whiten_multi, dim3((unsigned)n_pieces, 2), dim3(r16::NT), WHITEN_SMEM, st,
                                 pieces_dev, ctx->cfg.fir_len));
    return AFG_OK;
}

// The Welch kernels on caller-provided scratch and twiddles (no workspace,
// no context, no accounting).  P must hold periodogram_bytes(n_det * n_seg).
cudaError_t launch_psd_on(const float *x, int64_t n, int n_det, int64_t n_psd, int64_t psd_step, int64_t psd_span,
                          int hop, int fs, float *P, double *psd, cudaStream_t st) {
    const int64_t K = (psd_span - NFFT) / hop + 1;
    const int64_t seg_step = n_psd > 1 ? psd_step / hop : 0;
    const int64_t n_seg = (n_psd - 1) * seg_step + K;
    k_periodogram<<<dim3((unsigned)n_seg, n_det), r16::NT, WELCH_SMEM, st>>>(x, n, hop, P, n_seg, nullptr,
                                                                             psd_scale(K, fs));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_psd_mean(P, n_seg, (int)seg_step, (int)K, psd, n_psd, n_det, st);
}

// Fill the twiddle table and opt the periodogram kernel into its 68 KiB of dynamic shared memory on the
// current device.
cudaError_t prepare_psd_kernels() {
    const cudaError_t e = ensure_tw32();
    if (e != cudaSuccess) return e;
    return allow_smem(k_periodogram, WELCH_SMEM);
}
