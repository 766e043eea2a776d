// Whitening-filter build (Sec. IV, "Noise sampling" paragraph: the filter whose magnitude is the inverse
// ASD, made FIR by a taper): gains of each PSD's filter on the 16384-point transform of the whitening.
//
//   amplitude  A_k = psd_k^-1/2 at and above the highpass, else 0
//   taps       h_m = (1/N) sum_k A_k e^{+2 pi i k m / N},  g_m = sqrt(2/fs) taper(m) h_m,  |m| <= F/2
//   gains      G_k = sum_m g_m e^{-2 pi i k m / N}, real (g is even), stored as FP32 divided by NC
//
// k_filter_pair, k_filter_one (F <= 2048): the whole build on chip, in pairs of floats (high + low
// part, about 46 bits; the sums and products are the error-free transformations of Dekker and Knuth).  An error is
// 2^-46 of the filter's largest amplitude, below the FP32 rounding of a gain down to 2^-22 of the largest.  What that
// leaves at smaller gains is out of reach of the outputs: the whitening's FP32 transform has 2^-24 of the strain's largest
// amplitude at every bin.  (Whitened strain of PSDs from flat to f^-20, highpass 0, 10 and 32 Hz, gains over up to 15
// decades: the error against 64 bits is that of FP64 filters to four digits.)  This GPU retires 2 FP64 FMAs a clock and SM
// against 128 FP32 ones, and a pair operation takes 8 FP32 instructions: three FP64 kernels with their
// intermediate transforms in memory took 5.0 ms for 5402 filters (FP64 pipe 85 % busy) and 41 us for two; this
// takes 0.95 ms and 22 us, and the whitened strain differs by 7e-10 of its norm (its error is 1.2e-6).
// k_filter_build (longer filters): one CTA per filter, FP64.
#include <math.h>

#include <mutex>

#include "afg_internal.cuh"
#include "fft.cuh"

namespace {

constexpr int NT64 = 1024;  // threads of the FP64 filter kernel

__global__ void k_twiddles(double2 *tw64) {
    int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= NFFT) return;
    double s, c;
    sincospi(2.0 * (double)k / (double)NFFT, &s, &c);
    tw64[k] = make_double2(c, -s);
}

// grid (n_psd, n_det); builds the whitening gains of one (detector, epoch)
__global__ void __launch_bounds__(NT64) k_filter_build(const double *__restrict__ psd, int64_t n_psd, double fs,
                                                        double f_hp, int F, const double2 *__restrict__ tw,
                                                        float *__restrict__ gains) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2 *d = reinterpret_cast<double2 *>(smem_raw);
    pdl_trigger();  // (launched plainly)
    const int64_t e = blockIdx.x;
    const int det = blockIdx.y;
    const double *p = psd + ((int64_t)det * n_psd + e) * NBIN;
    // amplitude response: psd^-1/2 at and above the highpass, zero below
    for (int k = threadIdx.x; k < NBIN; k += NT64) {
        double f = (double)k * fs / (double)NFFT;
        double pk = p[k];
        double a = (f >= f_hp && pk > 0.0) ? rsqrt(pk) : 0.0;
        d[k] = make_double2(a, 0.0);
    }
    __syncthreads();
    // zero-phase impulse response h = IDFT_NFFT(A) / NFFT (real, even)
    real_split_inverse<double2, NT64>(d, tw);
    fft_nc<double2, +1, NT64>(d, tw);
    // taper to F taps about m = 0 and rescale; zero every other sample.
    // Sample i of the circular buffer is lag m = i (i < NFFT/2) or i - NFFT.
    const double norm = sqrt(2.0 / fs) / (double)NC;
    double *t = reinterpret_cast<double *>(d);
    const int half = F / 2;
    for (int i = threadIdx.x; i < NFFT; i += NT64) {
        int m = i < NFFT / 2 ? i : i - NFFT;
        double v = 0.0;
        if (m >= -half && m < half) {
            double taper = 0.5 - 0.5 * cospi(2.0 * (double)(m + half) / (double)F);
            v = t[i] * norm * taper;
        }
        t[i] = v;
    }
    __syncthreads();
    // gains G_k = DFT_NFFT(g)_k (real for the even g); stored divided by NC,
    // the factor the inverse half-length transform of k_whiten leaves over
    fft_nc<double2, -1, NT64>(d, tw);
    real_split_forward<double2, NT64>(d, tw);
    float *out = gains + ((int64_t)det * n_psd + e) * NBIN;
    for (int k = threadIdx.x; k < NBIN; k += NT64) out[k] = (float)(d[k].x / (double)NC);
}

// ---------------------------------------------------------------- pairs of floats
// A real number as h + l; dc: a complex one, (re, im) in each float2, stored as a float4.  l stays within a few
// roundings of h (no renormalisation inside a butterfly).  Every operation is an intrinsic: no contraction.
struct dd {
    float h, l;
};
struct dc {
    float2 h, l;
};
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

__device__ __forceinline__ dc cadd(dc a, dc b) {  // two-sum of the high parts, the low parts and its error added
    const float2 s = add2(a.h, b.h), t = sub2(s, a.h);
    const float2 e = add2(sub2(a.h, sub2(s, t)), sub2(b.h, t));
    return {s, add2(add2(a.l, b.l), e)};
}
__device__ __forceinline__ dc csub(dc a, dc b) {
    const float2 s = sub2(a.h, b.h), t = sub2(s, a.h);
    const float2 e = sub2(sub2(a.h, sub2(s, t)), add2(b.h, t));
    return {s, add2(sub2(a.l, b.l), e)};
}
__device__ __forceinline__ dc norm(dc a) {
    const float2 s = add2(a.h, a.l);
    return {s, sub2(a.l, sub2(s, a.h))};
}
__device__ __forceinline__ dc mul_ni(dc a) { return {make_float2(a.h.y, -a.h.x), make_float2(a.l.y, -a.l.x)}; }  // -i a
// both parts times a real pair (c + cl): product, its error and the cross terms
__device__ __forceinline__ dc scale(dc a, float c, float cl) {
    const float2 C = make_float2(c, c), p = __fmul2_rn(a.h, C);
    const float2 e = __ffma2_rn(a.h, C, make_float2(-p.x, -p.y));
    return {p, __ffma2_rn(a.l, C, __ffma2_rn(a.h, make_float2(cl, cl), e))};
}
__device__ __forceinline__ dd add(dd a, dd b) {
    const float s = __fadd_rn(a.h, b.h), t = __fsub_rn(s, a.h);
    const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, t)), __fsub_rn(b.h, t));
    return {s, __fadd_rn(__fadd_rn(a.l, b.l), e)};
}
__device__ __forceinline__ dd mul(dd a, dd b) {
    const float p = __fmul_rn(a.h, b.h);
    return {p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p)))};
}
__device__ __forceinline__ dd neg(dd a) { return {-a.h, -a.l}; }
__device__ __forceinline__ dd re(dc a) { return {a.h.x, a.l.x}; }
__device__ __forceinline__ dd im(dc a) { return {a.h.y, a.l.y}; }
__device__ __forceinline__ dc cmk(dd a, dd b) { return {make_float2(a.h, b.h), make_float2(a.l, b.l)}; }
// a w = (a.re, a.re) (w.re, w.im) + (a.im, a.im) (-w.im, w.re), both products and their sum packed
__device__ __forceinline__ dc cmul(dc a, dc w) {
    const float2 A = make_float2(a.h.x, a.h.x), B = make_float2(a.h.y, a.h.y);
    const float2 Al = make_float2(a.l.x, a.l.x), Bl = make_float2(a.l.y, a.l.y);
    const float2 V = make_float2(-w.h.y, w.h.x), Vl = make_float2(-w.l.y, w.l.x);
    const float2 p = __fmul2_rn(A, w.h), q = __fmul2_rn(B, V);
    float2 e = __ffma2_rn(A, w.h, make_float2(-p.x, -p.y));
    e = __ffma2_rn(Al, w.h, __ffma2_rn(A, w.l, e));
    float2 f = __ffma2_rn(B, V, make_float2(-q.x, -q.y));
    f = __ffma2_rn(Bl, V, __ffma2_rn(B, Vl, f));
    return cadd(dc{p, e}, dc{q, f});
}
__device__ __forceinline__ float4 pk(dc a) { return make_float4(a.h.x, a.h.y, a.l.x, a.l.y); }
__device__ __forceinline__ dc up(float4 v) { return {make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__host__ __device__ constexpr float hi_of(double v) { return (float)v; }
__host__ __device__ constexpr float lo_of(double v) { return (float)(v - (double)(float)v); }

// DFTs with the kernel e^{-2 pi i / n}
__device__ __forceinline__ void dft4(dc &a, dc &b, dc &c, dc &d) {
    const dc e0 = cadd(a, c), e1 = csub(a, c), o0 = cadd(b, d), o1 = mul_ni(csub(b, d));
    a = cadd(e0, o0);
    c = csub(e0, o0);
    b = cadd(e1, o1);
    d = csub(e1, o1);
}
constexpr double R_HALF = 0.70710678118654752440084436210485;  // cos(pi / 4)
constexpr double C_PI8 = 0.92387953251128675612818318939679;   // cos(pi / 8)
constexpr double S_PI8 = 0.38268343236508977172845998403040;   // sin(pi / 8)
// a e^{-i pi q / 8}, q = 1, 2, 3, 6, 9 (the turns a radix-16 or radix-8 butterfly needs)
template <int Q>
__device__ __forceinline__ dc turn(dc a) {
    if (Q == 2) return scale(cadd(a, mul_ni(a)), hi_of(R_HALF), lo_of(R_HALF));
    if (Q == 6) return scale(csub(mul_ni(a), a), hi_of(R_HALF), lo_of(R_HALF));
    constexpr double c = Q == 1 ? C_PI8 : Q == 3 ? S_PI8 : -C_PI8;
    constexpr double s = Q == 1 ? S_PI8 : Q == 3 ? C_PI8 : -S_PI8;
    return cmul(a, dc{make_float2(hi_of(c), -hi_of(s)), make_float2(lo_of(c), -lo_of(s))});
}
// 16-point DFT as 4 x 4; output m = k1 + 4 k2 is left in v[4 k1 + k2]
__device__ __forceinline__ void dft16(dc (&v)[16]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) dft4(v[c], v[c + 4], v[c + 8], v[c + 12]);
    v[5] = turn<1>(v[5]);
    v[6] = turn<2>(v[6]);
    v[7] = turn<3>(v[7]);
    v[9] = turn<2>(v[9]);
    v[10] = mul_ni(v[10]);
    v[11] = turn<6>(v[11]);
    v[13] = turn<3>(v[13]);
    v[14] = turn<6>(v[14]);
    v[15] = turn<9>(v[15]);
#pragma unroll
    for (int k = 0; k < 4; ++k) dft4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
}
// 8-point DFT of v[0..8) in natural order
__device__ __forceinline__ void dft8(dc *v) {
    dft4(v[0], v[2], v[4], v[6]);
    dft4(v[1], v[3], v[5], v[7]);
    const dc o0 = v[1], o1 = turn<2>(v[3]), o2 = mul_ni(v[5]), o3 = turn<6>(v[7]);
    const dc e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
    v[1] = cadd(e1, o1); v[5] = csub(e1, o1);
    v[2] = cadd(e2, o2); v[6] = csub(e2, o2);
    v[3] = cadd(e3, o3); v[7] = csub(e3, o3);
}

// ---------------------------------------------------------------- tables (per device, filled once)
constexpr int FL = 2048;  // points of a sub-transform
constexpr int FP = 8;     // residues
// twiddles e^{-2 pi i n / 2048}; then the residue turns W[kind][n] of lag m = n or n - 2048 (w_r = e^{-2 pi i r m / N}):
// w_0 + i w_4, w_1 + i w_2, w_3
__device__ float4 g_ftab[4 * FL];
// taper with its constant factors, sqrt(2 / fs) taper(m) / (N NC), m in [0, 1024); per context

__global__ void k_filter_tables() {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 4 * FL) return;
    const int kind = i / FL, n = i % FL;
    double re, im;
    if (kind == 0) {
        sincospi(2.0 * n / FL, &im, &re);
        im = -im;
    } else {
        const int m = n < FL / 2 ? n : n - FL;
        auto w = [&](int r, double &c, double &s) {
            sincospi(2.0 * r * m / NFFT, &s, &c);
            s = -s;
        };
        double c2 = 0.0, s2 = 0.0;
        w(kind == 1 ? 0 : kind == 2 ? 1 : 3, re, im);
        if (kind < 3) w(kind == 1 ? 4 : 2, c2, s2);
        re -= s2;
        im += c2;
    }
    g_ftab[i] = make_float4((float)re, (float)im, (float)(re - (double)(float)re), (float)(im - (double)(float)im));
}
__global__ void k_filter_taper(float2 *tap, double fs, int F) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= FL / 2) return;
    const int half = F / 2;
    const double v = m < half ? sqrt(2.0 / fs) * (0.5 - 0.5 * cospi(2.0 * (double)(m + half) / (double)F)) /
                                    ((double)NFFT * (double)NC)
                              : 0.0;
    tap[m] = make_float2((float)v, (float)(v - (double)(float)v));
}

// ---------------------------------------------------------------- the build
__device__ __forceinline__ int fpad(int i) { return i + (i >> 4); }
constexpr int FSLOTS = FL + FL / 16;
constexpr int FGT = 128;  // threads of a sub-transform: 16 points each

__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(FGT) : "memory"); }

// 2048-point transform of a group of 128 threads: in, v[r] = x[t + 128 r]; out, v[8 q + r] = X[t + 128 q + 256 r].
// Radix 16, 16, 8 (Stockham); one pad slot in 17 makes every 16-byte access conflict-free.
__device__ __forceinline__ void fft2048(dc (&v)[16], float4 *d, int t, int g) {
    auto tw = [&](int i) { return up(__ldg(&g_ftab[i])); };
    dft16(v);
#pragma unroll
    for (int m = 0; m < 16; ++m) d[fpad(t * 16 + m)] = pk(norm(v[4 * (m & 3) + (m >> 2)]));
    group_sync(g);
    const int k = t & 15;
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = up(d[fpad(t + FGT * r)]);
#pragma unroll
    for (int r = 1; r < 16; ++r) v[r] = cmul(v[r], tw(8 * r * k));
    dft16(v);
    group_sync(g);
#pragma unroll
    for (int m = 0; m < 16; ++m) d[fpad((t - k) * 16 + k + 16 * m)] = pk(norm(v[4 * (m & 3) + (m >> 2)]));
    group_sync(g);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int j = t + FGT * q;
#pragma unroll
        for (int r = 0; r < 8; ++r) v[8 * q + r] = up(d[fpad(j + 256 * r)]);
#pragma unroll
        for (int r = 1; r < 8; ++r) v[8 * q + r] = cmul(v[8 * q + r], tw(r * j));
        dft8(v + 8 * q);
    }
}

// psd^-1/2 of a positive finite double 1.f x 2^(e - 1023), times 2^s with 2 s <= e - 1023: mantissa in a pair, one
// Newton step of the reciprocal square root in pairs.
__device__ __forceinline__ int exp_of(long long b) {  // e; subnormals count on below 1
    const int e = (int)(b >> 52);
    return e ? e : 12 - __clzll(b);
}
__device__ __forceinline__ dd amplitude(long long b, int s) {
    int e = (int)(b >> 52);
    if (!e) {  // subnormal: shift the leading bit into place
        const int z = __clzll(b) - 11;
        b <<= z;
        e = 1 - z;
    }
    int E = e - 1023 - 2 * s;  // >= 0
    float mh = __int_as_float(0x3F800000 | (int)((b >> 29) & 0x7FFFFF));
    float ml = (float)(int)(b & 0x1FFFFFFF) * 0x1p-52f;
    if (E & 1) {
        mh += mh;
        ml += ml;
        --E;
    }
    E >>= 1;
    if (E > 126) return {0.f, 0.f};  // 2^-126 of the filter's largest amplitude
    const float y = rsqrtf(mh), p = __fmul_rn(y, y), pe = __fmaf_rn(y, y, -p);
    const float q = __fmul_rn(mh, p), qe = __fmaf_rn(mh, p, -q);
    float r = __fsub_rn(__fsub_rn(1.f, q), qe);  // 1 - m y^2
    r = __fmaf_rn(-mh, pe, r);
    r = __fmaf_rn(-ml, p, r);
    const float c = __fmul_rn(__fmul_rn(y, r), __fmaf_rn(0.375f, r, 0.5f));
    const float h = __fadd_rn(y, c), f = __int_as_float((127 - E) << 23);
    return {h * f, __fsub_rn(c, __fsub_rn(h, y)) * f};
}

// N splits into P = 8 sub-transforms of L = 2048 points by residue r = k mod 8 (frequency decimation), which is
// all the |m| < 1024 lags need: with w_r(m) = e^{-2 pi i r m / N} and Z_r = sum_j A_{8 j + r} e^{+2 pi i j m / L},
//   N h_m = sum_r conj(w_r) Z_r,      G_{8 j + r} = sum_m g_m w_r(m) e^{-2 pi i j m / L}.
// A and G are real and even, so residue 8 - r is residue r reversed and r = 0 .. 4 are enough (1, 2, 3 count
// twice), and a complex transform carries two real sequences: C of A_r1 + i A_r2 adds, with
// f(n) = Re(C[n] conj(w_r1 + i w_r2)), f(m) + f(-m) = 2 Re(conj(w_r1) Z_r1 + conj(w_r2) Z_r2) to h_m; the transform of
// g (w_r1 + i w_r2) is G_{8 j + r1} + i G_{8 j + r2}.  The pairs are (0, 4) and (1, 2) of a filter, and residue 3 of two
// filters (f: the real and the imaginary part of C conj(w_3)).
//
// The inverse transform is conj(FFT(conj x)): the second residue enters negated and the result is read as its
// conjugate.  Amplitudes are scaled by the power of two that brings the largest near 1 (strain PSDs are near 1e-46),
// undone in the gains.
constexpr int ARS = 1026, GRS = 1028;  // rows of the amplitudes (float2) and gains by residue: no bank conflicts

// bits of a PSD value that has an amplitude, else 0 (below the highpass; infinity: amplitude 0; NaN; not positive)
__device__ __forceinline__ long long psd_bits(long long b, int k, int k_hp) {
    return k < k_hp || b >= 0x7FF0000000000000LL || b < 0 ? 0LL : b;
}
// the gains' scale 2^-s in two exact steps (past the floats' range: 0 or infinity, as the FP64 gain would round)
struct Unscale {
    float p1, p2;
    __device__ __forceinline__ Unscale(int emin) {
        const int s = emin < (1 << 20) ? (emin - 1023) >> 1 : 0;
        const int e1 = max(-126, min(127, -s)), e2 = max(-126, min(127, -s - e1));
        p1 = __int_as_float((127 + e1) << 23);
        p2 = __int_as_float((127 + e2) << 23);
    }
    __device__ __forceinline__ float operator()(float g) const { return g * p1 * p2; }
};

// f(n) of conj C and the turn w: Re(C conj w) and Im(C conj w)
__device__ __forceinline__ dd f_re(dc c, dc w) { return add(mul(re(c), re(w)), neg(mul(im(c), im(w)))); }
__device__ __forceinline__ dd f_im(dc c, dc w) { return neg(add(mul(im(c), re(w)), mul(re(c), im(w)))); }

// Many filters: one CTA builds two with five transforms side by side, 128 threads each; amplitudes, taps and gains
// stay in shared memory, so a filter costs one read of its PSD and one write of its gains.
// Bound by the instructions of the pair arithmetic (20 warps of 96 registers, 48 % of the issue slots).
constexpr int F2_NG = 5, F2_T = F2_NG * FGT;
constexpr int F2_REGION = F2_NG * FSLOTS * 16;  // amplitudes, transforms and gains, one after the other; then the taps
constexpr int F2_BYTES = F2_REGION + 2 * 1024 * 8;
static_assert(2 * FP * ARS * 8 <= F2_REGION && 2 * FP * GRS * 4 <= F2_REGION, "overlaid stages");

__global__ void __launch_bounds__(F2_T, 1) k_filter_pair(const double *__restrict__ psd, int64_t nf, int k_hp,
                                                         const float2 *__restrict__ tap, float *__restrict__ gains) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int emin[2];
    float2 *amp = reinterpret_cast<float2 *>(smem_raw);  // [2][FP][ARS]: A_{8 i + rho}
    float2 *taps = reinterpret_cast<float2 *>(smem_raw + F2_REGION);
    float *gst = reinterpret_cast<float *>(smem_raw);    // [2][FP][GRS]
    const int tid = threadIdx.x, g = tid / FGT, t = tid % FGT;
    const int64_t f0 = (int64_t)blockIdx.x * 2;
    const int n_here = (int)min((int64_t)2, nf - f0);
    float4 *d = reinterpret_cast<float4 *>(smem_raw) + g * FSLOTS;

    // ---- amplitudes: every PSD value is loaded once, all loads in flight together
    {
        constexpr int PER = (2 * NBIN + F2_T - 1) / F2_T;
        if (tid < 2) emin[tid] = 1 << 20;
        long long b[PER];
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int x = tid + i * F2_T;
            b[i] = x < n_here * NBIN ? __ldg(reinterpret_cast<const long long *>(psd) + f0 * NBIN + x) : 0LL;
            b[i] = psd_bits(b[i], x < NBIN ? x : x - NBIN, k_hp);
        }
        __syncthreads();
        int e0 = 1 << 20, e1 = 1 << 20;
#pragma unroll
        for (int i = 0; i < PER; ++i)
            if (b[i]) {
                const int x = exp_of(b[i]);
                if (tid + i * F2_T < NBIN) e0 = min(e0, x);
                else e1 = min(e1, x);
            }
        e0 = __reduce_min_sync(0xffffffffu, e0);
        e1 = __reduce_min_sync(0xffffffffu, e1);
        if ((tid & 31) == 0) {
            atomicMin(&emin[0], e0);
            atomicMin(&emin[1], e1);
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int x = tid + i * F2_T, f = x < NBIN ? 0 : 1, k = x - f * NBIN;
            if (x >= 2 * NBIN) break;
            dd a = {0.f, 0.f};
            if (b[i]) a = amplitude(b[i], (emin[f] - 1023) >> 1);
            amp[(f * FP + (k & 7)) * ARS + (k >> 3)] = make_float2(a.h, a.l);
        }
        __syncthreads();
    }

    // ---- inverse transforms: this group's kind (0: residues 0 and 4, 1: 1 and 2, 2: 3 of both filters) and filter
    const int kind = g == 4 ? 2 : g & 1, fa = g == 4 ? 0 : g >> 1;
    const int r1 = kind == 0 ? 0 : kind == 1 ? 1 : 3, r2 = kind == 0 ? 4 : kind == 1 ? 2 : 3;
    auto amp_at = [&](int f, int r, int j) {  // A_{8 j + r}, j in [0, 2048): bins past N/2 are mirrored
        if (j < 1024) return amp[(f * FP + r) * ARS + j];
        return r == 0 ? amp[f * FP * ARS + 2048 - j] : amp[(f * FP + 8 - r) * ARS + 2047 - j];
    };
    dc v[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int j = t + FGT * r;
        const float2 a = amp_at(fa, r1, j), b = amp_at(kind < 2 ? fa : 1, r2, j);
        v[r] = {make_float2(a.x, -b.x), make_float2(a.y, -b.y)};
    }
    __syncthreads();  // the amplitudes are read: the transforms overwrite them
    fft2048(v, d, t, g);
    group_sync(g);
    const float4 *wt = g_ftab + (1 + kind) * FL;
    float2 *fs = reinterpret_cast<float2 *>(d);  // f(n) [2048], and of the second filter behind it
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int n = t + FGT * q + 256 * r;
            const dc c = v[8 * q + r], w = up(__ldg(&wt[n]));
            const dd a = f_re(c, w);
            fs[n] = make_float2(a.h, a.l);
            if (kind == 2) {
                const dd b = f_im(c, w);
                fs[FL + n] = make_float2(b.h, b.l);
            }
        }
    __syncthreads();

    // ---- taps g_m, m in [0, 1024)
    for (int i = tid; i < 2 * 1024; i += F2_T) {
        const int f = i >> 10, m = i & 1023, mm = (FL - m) & (FL - 1);
        const float2 *s04 = reinterpret_cast<const float2 *>(smem_raw + (size_t)(2 * f) * FSLOTS * 16);
        const float2 *s12 = reinterpret_cast<const float2 *>(smem_raw + (size_t)(2 * f + 1) * FSLOTS * 16);
        const float2 *s3 = reinterpret_cast<const float2 *>(smem_raw + (size_t)4 * FSLOTS * 16) + f * FL;
        auto pair = [&](const float2 *s) { return add(dd{s[m].x, s[m].y}, dd{s[mm].x, s[mm].y}); };
        const dd z = pair(s04);
        const float2 tp = __ldg(&tap[m]);
        const dd h = mul(add(add(dd{0.5f * z.h, 0.5f * z.l}, pair(s12)), pair(s3)), dd{tp.x, tp.y});
        taps[i] = make_float2(h.h, h.l);
    }
    __syncthreads();

    // ---- forward transforms
#pragma unroll
    for (int r = 0; r < 16; ++r) {
        const int n = t + FGT * r, m = n <= 1024 ? n : FL - n;
        const dc w = up(__ldg(&wt[n]));
        auto tp = [&](int f) {
            const float2 a = m < 1024 ? taps[f * 1024 + m] : make_float2(0.f, 0.f);
            return dd{a.x, a.y};
        };
        const dd a = tp(fa);
        v[r] = kind == 2 ? cmul(cmk(a, tp(1)), w) : cmk(mul(a, re(w)), mul(a, im(w)));  // (g_a + i g_b) w_3
    }
    fft2048(v, d, t, g);
    __syncthreads();  // every transform has left shared memory: the gains overlay it
    auto put = [&](int f, int r, int j, float x) {
        int k = 8 * j + r;
        if (k > NFFT / 2) {
            if (r == 0 || r == 4) return;  // its own mirror
            k = NFFT - k;
        }
        gst[(f * FP + (k & 7)) * GRS + (k >> 3)] = x;
    };
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int j = t + FGT * q + 256 * r;
            const dc c = v[8 * q + r];
            put(fa, r1, j, __fadd_rn(c.h.x, c.l.x));
            put(kind < 2 ? fa : 1, r2, j, __fadd_rn(c.h.y, c.l.y));
        }
    __syncthreads();
    for (int f = 0; f < n_here; ++f) {
        const Unscale un(emin[f]);
        float *out = gains + (f0 + f) * NBIN;
        for (int k = tid; k < NBIN; k += F2_T) out[k] = un(gst[(f * FP + (k & 7)) * GRS + (k >> 3)]);
    }
}

// Few filters (an epoch refresh, one span): one filter per cluster of three CTAs, a transform each, so that one
// filter's chain of pair operations runs on three SMs (two filters: about 31 us as one CTA of 384 threads each,
// 22 us now).  Each CTA scans the whole PSD for the scale, forms the amplitudes of its own residues, and sends its
// part of the taps to the other two through distributed shared memory.
constexpr int F1_REGION = FSLOTS * 16;
constexpr int F1_BYTES = F1_REGION + 4 * 1024 * 8;  // then the three parts of the taps, and the taps
static_assert(4 * ARS * 8 <= F1_REGION, "overlaid stages");

__device__ __forceinline__ void st_cluster(float2 *local, int rank, float2 v) {  // the same variable of CTA `rank`
    uint32_t p;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(p) : "r"((uint32_t)__cvta_generic_to_shared(local)), "r"(rank));
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(p), "f"(v.x), "f"(v.y) : "memory");
}

__global__ void __launch_bounds__(FGT) k_filter_one(const double *psd, int k_hp,
                                                                             const float2 *__restrict__ tap,
                                                                             float *__restrict__ gains) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int emin;
    float2 *amp = reinterpret_cast<float2 *>(smem_raw);  // rows of the residues (r1, 8 - r1, r2, 8 - r2), or (r1, r2)
    float2 *parts = reinterpret_cast<float2 *>(smem_raw + F1_REGION), *taps = parts + 3 * 1024;
    float4 *d = reinterpret_cast<float4 *>(smem_raw);
    const int t = threadIdx.x, kind = blockIdx.x % 3;
    const int64_t f = blockIdx.x / 3;
    const long long *p = reinterpret_cast<const long long *>(psd) + f * NBIN;
    const int r1 = kind == 0 ? 0 : kind == 1 ? 1 : 3, r2 = kind == 0 ? 4 : kind == 1 ? 2 : -1;
    asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");  // (waited for before the first remote store)
    if (t == 0) emin = 1 << 20;
    __syncthreads();
    pdl_wait();     // the PSD
    pdl_trigger();  // (not before: a dependent may rely on what came before this launch)
    constexpr int BATCH = 33;  // 2 x 33 x 128 >= NBIN
    int e = 1 << 20;
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        long long b[BATCH];
#pragma unroll
        for (int i = 0; i < BATCH; ++i) {
            const int k = t + FGT * (BATCH * h + i);
            b[i] = k < NBIN ? psd_bits(p[k], k, k_hp) : 0LL;
        }
#pragma unroll
        for (int i = 0; i < BATCH; ++i)
            if (b[i]) e = min(e, exp_of(b[i]));
    }
    e = __reduce_min_sync(0xffffffffu, e);
    if ((t & 31) == 0) atomicMin(&emin, e);
    __syncthreads();
    // amplitudes A_{8 i + rho} of this CTA's residues: row 0 rho = r1, 1: 8 - r1, 2: r2, 3: 8 - r2 (kind 0: 0 and 4 are
    // their own mirrors, rows 0 and 2)
    const int s = (emin - 1023) >> 1;
    for (int row = 0; row < (r2 < 0 ? 2 : 4); ++row) {
        if (kind == 0 && (row & 1)) continue;
        const int rho = row == 0 ? r1 : row == 1 ? 8 - r1 : row == 2 ? r2 : 8 - r2;
#pragma unroll 8
        for (int i = t; i < 1024 + (rho == 0); i += FGT) {
            const int k = 8 * i + rho;
            const long long b = psd_bits(p[k], k, k_hp);
            dd a = {0.f, 0.f};
            if (b) a = amplitude(b, s);
            amp[row * ARS + i] = make_float2(a.h, a.l);
        }
    }
    __syncthreads();
    auto amp_at = [&](int row, int r, int j) {  // A_{8 j + r}, j in [0, 2048): bins past N/2 are mirrored
        if (j < 1024) return amp[row * ARS + j];
        return r == 0 ? amp[row * ARS + 2048 - j] : amp[(row + (kind != 0)) * ARS + 2047 - j];
    };
    const float4 *wt = g_ftab + (1 + kind) * FL;
    dc v[16];
    // the transform's code exists once, in a loop over the two stages
#pragma unroll 1
    for (int stage = 0; stage < 2; ++stage) {
        if (stage == 0) {
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const int j = t + FGT * r;
                const float2 a = amp_at(0, r1, j), b = r2 < 0 ? make_float2(0.f, 0.f) : amp_at(2, r2, j);
                v[r] = {make_float2(a.x, -b.x), make_float2(a.y, -b.y)};
            }
            __syncthreads();  // the amplitudes are read: the transform overwrites them
        } else {
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                const int n = t + FGT * r, m = n <= 1024 ? n : FL - n;
                const dc w = up(__ldg(&wt[n]));
                const float2 a = m < 1024 ? taps[m] : make_float2(0.f, 0.f);
                v[r] = cmk(mul(dd{a.x, a.y}, re(w)), mul(dd{a.x, a.y}, im(w)));
            }
        }
        fft2048(v, d, t, 0);
        if (stage == 1) break;
        __syncthreads();
        float2 *fs = reinterpret_cast<float2 *>(d);
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int n = t + FGT * q + 256 * r;
                const dd a = f_re(v[8 * q + r], up(__ldg(&wt[n])));
                fs[n] = make_float2(a.h, a.l);
            }
        __syncthreads();
        asm volatile("barrier.cluster.wait;" ::: "memory");  // every CTA of the cluster has started
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int m = t + FGT * i, mm = (FL - m) & (FL - 1);
            const dd z = add(dd{fs[m].x, fs[m].y}, dd{fs[mm].x, fs[mm].y});
            const float c = kind == 0 ? 0.5f : 1.f;
            for (int o = 0; o < 3; ++o) st_cluster(parts + kind * 1024 + m, o, make_float2(c * z.h, c * z.l));
        }
        asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int m = t + FGT * i;
            auto part = [&](int o) { return dd{parts[o * 1024 + m].x, parts[o * 1024 + m].y}; };
            const float2 tp = __ldg(&tap[m]);
            const dd h = mul(add(add(part(0), part(1)), part(2)), dd{tp.x, tp.y});
            taps[m] = make_float2(h.h, h.l);
        }
        __syncthreads();
    }
    const Unscale un(emin);
    float *out = gains + f * NBIN;
    auto put = [&](int r, int j, float x) {
        const int k = 8 * j + r;
        if (k <= NFFT / 2) out[k] = un(x);
        else if (r != 0 && r != 4) out[NFFT - k] = un(x);
    };
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int j = t + FGT * q + 256 * r;
            const dc c = v[8 * q + r];
            put(r1, j, __fadd_rn(c.h.x, c.l.x));
            if (r2 >= 0) put(r2, j, __fadd_rn(c.h.y, c.l.y));
        }
}

// Fill the tables of the current device once per process (complete when this returns).
cudaError_t ensure_filter_tables() {
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
    k_filter_tables<<<4 * FL / 256, 256, 0, st>>>();
    e = cudaGetLastError();
    const cudaError_t e2 = cudaStreamSynchronize(st);
    cudaStreamDestroy(st);
    if (e == cudaSuccess) e = e2;
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_filter_one, cudaFuncAttributeMaxDynamicSharedMemorySize, F1_BYTES);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_filter_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, F2_BYTES);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_filter_build, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)((NC + 1) * sizeof(double2)));
    if (e == cudaSuccess) done[dev] = true;
    return e;
}

}  // namespace

// First bin k in [0, N/2] with k fs / N >= f_hp (N/2 + 1: none; also for NaN)
static int first_bin(double f_hp, int fs) {
    if (f_hp != f_hp) return NFFT / 2 + 1;
    int lo = 0, hi = NFFT / 2 + 1;  // the test is monotonic in k
    while (lo < hi) {
        const int mid = (lo + hi) / 2;
        if ((double)mid * (double)fs / (double)NFFT >= f_hp) hi = mid;
        else lo = mid + 1;
    }
    return lo;
}

// The context's filter tables: the taper in pairs for F <= 2048, the FP64 twiddles for longer filters.
int filter_prepare(afg_ctx *ctx) {
    if (ensure_filter_tables() != cudaSuccess) return AFG_ERR_CUDA;
    const bool pairs = ctx->cfg.fir_len <= FILTER_LAGS;
    const size_t bytes = pairs ? (FL / 2) * sizeof(float2) : NFFT * sizeof(double2);
    if (cudaMalloc(&ctx->filter_tab, bytes) != cudaSuccess) {
        cudaGetLastError();
        return AFG_ERR_OOM;
    }
    ctx->bytes_held += (int64_t)bytes;
    KScope ks(ctx, 0, KK_TWIDDLES, 0.0, (double)bytes);
    if (pairs)
        k_filter_taper<<<FL / 2 / 256, 256>>>(static_cast<float2 *>(ctx->filter_tab), (double)ctx->cfg.fs, ctx->cfg.fir_len);
    else
        k_twiddles<<<NFFT / 256, 256>>>(static_cast<double2 *>(ctx->filter_tab));
    AFG_LAUNCH_CHECK(ctx, "filter tables");
    return AFG_OK;
}

// gains [n_det][n_psd][NBIN] from psd [n_det][n_psd][NBIN]
int launch_filter(afg_ctx *ctx, const double *psd, int n_det, int64_t n_psd, float *gains, cudaStream_t st) {
    const int64_t nf = (int64_t)n_det * n_psd;
    if (nf <= 0) return AFG_OK;
    if (nf > 0x7fffffff) return afg_fail(ctx, AFG_ERR_ARG, "filter build: too many filters");
    // algorithmic work of one filter: an inverse and a forward transform of a real, even sequence of NFFT points,
    // 1.25 N log2 N flops each (half of a real FFT's 2.5 N log2 N); its PSD read and its gains written
    static_assert(NFFT == 1 << 14, "flop count assumes log2(NFFT) = 14");
    KScope ks(ctx, st, KK_FILTER, (double)nf * 2.0 * 1.25 * NFFT * 14.0, (double)nf * NBIN * (8.0 + 4.0));
    if (ctx->cfg.fir_len <= FILTER_LAGS) {
        const int k_hp = first_bin(ctx->cfg.f_highpass, ctx->cfg.fs);
        const float2 *tap = static_cast<const float2 *>(ctx->filter_tab);
        if (nf <= 152)  // fewer pairs than half of the SMs: three CTAs a filter
            AFG_CUDA(ctx, launch_pdl_cluster(k_filter_one, dim3((unsigned)(3 * nf)), dim3(FGT), F1_BYTES, st, 3, psd, k_hp, tap,
                                             gains));
        else
            k_filter_pair<<<(unsigned)((nf + 1) / 2), F2_T, F2_BYTES, st>>>(psd, nf, k_hp, tap, gains);
    } else {
        k_filter_build<<<dim3((unsigned)n_psd, n_det), NT64, (NC + 1) * sizeof(double2), st>>>(
            psd, n_psd, (double)ctx->cfg.fs, ctx->cfg.f_highpass, ctx->cfg.fir_len,
            static_cast<const double2 *>(ctx->filter_tab), gains);
    }
    AFG_LAUNCH_CHECK(ctx, "filter build");
    return AFG_OK;
}
