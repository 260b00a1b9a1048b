// Batched tone DFT of tone counts with small prime factors (2, 3, 5, 7): a
// mixed-radix fast Fourier transform in FP32 (Cooley and Tukey 1965; the
// self-sorting order of Stockham, so no digit reversal pass).
//
// Pass with radix r after the radices before it multiplied to m:  butterfly
// j < N/r takes x[j + q N/r], q < r, turns them by exp(-j 2 pi q k/(m r)),
// k = j mod m, transforms them and writes y[(j/m) m r + k + q m].  The first
// pass reads P and the last one writes T (both runs of consecutive values);
// the passes between go through two buffers in shared memory, one value of
// padding after 16 so that strides of 2, 4, 8 and 16 spread over the banks.
// The twiddles of a pass lie in the order its threads read them (N less the
// first radix in all, from FP64): through L1, or (CHAIN) from shared memory,
// where they arrive with the first pass's values.
//
// Two precisions.  The CUDA-core mode works in FP32.  The tensor-core modes are
// to be no less accurate than the contraction.  Its rms error grows with N (split
// BF16 0.55e-7 at N = 20, 1.08e-7 at 256, 1.72e-7 at 1024; split TF32 1.2 to
// 2.0e-7), that of FP32 butterflies hardly (0.66e-7, 0.92e-7, 1.07e-7): from
// kFftSingleN tones on FP32 is the more accurate in every measure (rms, mean,
// worst channel, worst tone) at every count that comes here, of noise and of
// pulses; closest at N = 500 against split BF16, 1.13e-7 and 1.22e-7 rms (at 486
// tones the worst channel was not).  Below it, and
// wherever a delay follows (a batch's finalize), they carry double-float values
// through each pass and round to FP32 between passes (0.35 to 0.5e-7): with FP32
// alone the delay of a strong comb of 1024 tones moved by 1.07e-3 of its sigma.
//
// Why not the dense contraction of dft_tc.cu here: that does 8 N^2 operations a
// channel, this one 5 N log2 N, and its sums are log2 N long instead of N.
// C 4096, N 1024, 67 MB: FP32 direct sum 2930 us, split-TF32 contraction 176 us,
// this kernel 25 us a call in FP32 (20 in a graph that finds its data in L2; bound
// by latency and issue slots, index arithmetic and shared-memory exchanges beside
// the butterflies; HBM alone would take 10 us) and 50 us with double-float passes
// (the FP32 pipes: about 300 operations a value).  N 256, C 4096, double-float:
// 33 -> 12.5 us.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <vector>

namespace pcal_fft {

constexpr int kFftMaxPasses = 12;
constexpr int kFftSingleN = 500;  // tensor-core modes: FP32 inside passes from here on

struct FftPlan {
    int N, passes;             // passes == 0: N has a prime factor above 7 (or is 1)
    int radix[kFftMaxPasses];  // their product is N
    bool wide;                 // double-float inside a pass
    void* tw;                  // twiddles of the passes after the first, [q - 1][k] each
    uint32_t by_nb[kFftMaxPasses], by_m[kFftMaxPasses];  // division by N / radix and by m (over)
};

constexpr int kThreads = 128;
constexpr int kSms = 152;  // of a GB300
constexpr int kTileValues = 2048;  // values a CTA holds, where N allows (35 KB in two buffers)
// FP32 transforms whose calls of few channels are one chain of latencies: their
// kernel stages the twiddles and divides by multiplication, as a load of
// twiddles behind each pass's barrier and two divisions a butterfly were links of
// it.  300 channels, a call in a graph, without / with: N 32 2.55 / 2.38 us, N 50 3.00 /
// 2.74, N 96 3.17 / 2.83, N 128 3.70 / 2.75 (the direct sum 1.8, 2.3, 3.0, 4.3; 4096 channels
// 4.9, 10, 21, 41 and the FFT 2.8, 4.8, 5.3, 4.1).  With more tones the butterflies
// outweigh both (and N 512 got slower: 4096 channels 11.2 / 12.9).
constexpr int kChainMinN = 32, kChainMaxN = 128;

__host__ __device__ constexpr int pad(int i) { return i + (i >> 4); }

// A constant or twiddle as the nearest float and the float nearest the rest.
struct Const {
    float h, l;
};
#define PCAL_FFT_CONST(x) Const{(float)(x), (float)((x) - (double)(float)(x))}

// ---- FP32 values ---------------------------------------------------------------

struct Single {
    using Twiddle = float2;  // cos, sin
    float x, y;
    __device__ static __forceinline__ Single load(float2 v) { return {v.x, v.y}; }
    __device__ __forceinline__ float2 round() const { return make_float2(x, y); }
};
__device__ __forceinline__ Single operator+(Single a, Single b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ Single operator-(Single a, Single b) { return {a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ Single mul_mj(Single a) { return {a.y, -a.x}; }  // times -j
__device__ __forceinline__ Single scale(Single a, Const c) { return {a.x * c.h, a.y * c.h}; }
__device__ __forceinline__ Single mul_add(Single a, Const c, Single s) {
    return {fmaf(a.x, c.h, s.x), fmaf(a.y, c.h, s.y)};
}
__device__ __forceinline__ Single mul(Single a, Const c, Const s) {  // times c + j s
    return {fmaf(a.x, c.h, -(a.y * s.h)), fmaf(a.x, s.h, a.y * c.h)};
}
__device__ __forceinline__ Single turn(Single a, float2 w) { return mul(a, Const{w.x, 0.f}, Const{w.y, 0.f}); }

// ---- double-float values (inside a pass; rounded to FP32 between passes) ----------

struct Real2 {
    float h, l;
};
// (two_sum; products are formed with __fmul_rn so that none is contracted into a sum)
__device__ __forceinline__ Real2 radd(Real2 a, Real2 b) {
    const float s = a.h + b.h, t = s - a.h;
    return {s, ((a.h - (s - t)) + (b.h - t)) + (a.l + b.l)};
}
__device__ __forceinline__ Real2 rneg(Real2 a) { return {-a.h, -a.l}; }
__device__ __forceinline__ Real2 rscale(Real2 a, Const c) {
    const float p = __fmul_rn(a.h, c.h);
    return {p, fmaf(a.h, c.l, fmaf(a.l, c.h, fmaf(a.h, c.h, -p)))};
}

struct Double {
    using Twiddle = float4;  // cos (h, l), sin (h, l)
    Real2 x, y;
    __device__ static __forceinline__ Double load(float2 v) { return {{v.x, 0.f}, {v.y, 0.f}}; }
    __device__ __forceinline__ float2 round() const { return make_float2(x.h + x.l, y.h + y.l); }
};
__device__ __forceinline__ Double operator+(Double a, Double b) { return {radd(a.x, b.x), radd(a.y, b.y)}; }
__device__ __forceinline__ Double operator-(Double a, Double b) {
    return {radd(a.x, rneg(b.x)), radd(a.y, rneg(b.y))};
}
__device__ __forceinline__ Double mul_mj(Double a) { return {a.y, rneg(a.x)}; }
__device__ __forceinline__ Double scale(Double a, Const c) { return {rscale(a.x, c), rscale(a.y, c)}; }
__device__ __forceinline__ Double mul_add(Double a, Const c, Double s) { return s + scale(a, c); }
__device__ __forceinline__ Double mul(Double a, Const c, Const s) {
    return {radd(rscale(a.x, c), rneg(rscale(a.y, s))), radd(rscale(a.x, s), rscale(a.y, c))};
}
__device__ __forceinline__ Double turn(Double a, float4 w) { return mul(a, Const{w.x, w.y}, Const{w.z, w.w}); }

// ---- in-place DFTs of R values, natural order in and out -----------------------------

template <class V>
__device__ __forceinline__ void dft4(V& a, V& b, V& c, V& d) {
    const V s = a + c, t = a - c, u = b + d, v = mul_mj(b - d);
    a = s + u;
    b = t + v;
    c = s - u;
    d = t - v;
}

// cos and sin of 2 pi i / R for the odd radices.
template <int R>
__device__ __forceinline__ Const odd_cos(int i) {
    constexpr Const c3[] = {PCAL_FFT_CONST(1.0), PCAL_FFT_CONST(-0.5), PCAL_FFT_CONST(-0.5)};
    constexpr Const c5[] = {PCAL_FFT_CONST(1.0), PCAL_FFT_CONST(0.30901699437494742410),
                            PCAL_FFT_CONST(-0.80901699437494742410), PCAL_FFT_CONST(-0.80901699437494742410),
                            PCAL_FFT_CONST(0.30901699437494742410)};
    constexpr Const c7[] = {PCAL_FFT_CONST(1.0), PCAL_FFT_CONST(0.62348980185873353053),
                            PCAL_FFT_CONST(-0.22252093395631440429), PCAL_FFT_CONST(-0.90096886790241912624),
                            PCAL_FFT_CONST(-0.90096886790241912624), PCAL_FFT_CONST(-0.22252093395631440429),
                            PCAL_FFT_CONST(0.62348980185873353053)};
    return R == 3 ? c3[i % 3] : R == 5 ? c5[i % 5] : c7[i % 7];
}
template <int R>
__device__ __forceinline__ Const odd_sin(int i) {
    constexpr Const s3[] = {PCAL_FFT_CONST(0.0), PCAL_FFT_CONST(0.86602540378443864676),
                            PCAL_FFT_CONST(-0.86602540378443864676)};
    constexpr Const s5[] = {PCAL_FFT_CONST(0.0), PCAL_FFT_CONST(0.95105651629515357212),
                            PCAL_FFT_CONST(0.58778525229247312917), PCAL_FFT_CONST(-0.58778525229247312917),
                            PCAL_FFT_CONST(-0.95105651629515357212)};
    constexpr Const s7[] = {PCAL_FFT_CONST(0.0), PCAL_FFT_CONST(0.78183148246802980871),
                            PCAL_FFT_CONST(0.97492791218182360702), PCAL_FFT_CONST(0.43388373911755812048),
                            PCAL_FFT_CONST(-0.43388373911755812048), PCAL_FFT_CONST(-0.97492791218182360702),
                            PCAL_FFT_CONST(-0.78183148246802980871)};
    return R == 3 ? s3[i % 3] : R == 5 ? s5[i % 5] : s7[i % 7];
}

// Odd radices: the sums and differences of x_m and x_{R-m} against cos and
// sin of 2 pi k m / R; X_k and X_{R-k} together.
template <int R, class V>
__device__ __forceinline__ void dft_odd(V (&v)[R]) {
    constexpr int H = (R - 1) / 2;
    V s[H], d[H];
    V sum = v[0];
    const V v0 = v[0];
#pragma unroll
    for (int m = 1; m <= H; ++m) {
        s[m - 1] = v[m] + v[R - m];
        d[m - 1] = v[m] - v[R - m];
        sum = sum + s[m - 1];
    }
#pragma unroll
    for (int k = 1; k <= H; ++k) {
        V a = mul_add(s[0], odd_cos<R>(k), v0), b = scale(d[0], odd_sin<R>(k));
#pragma unroll
        for (int m = 2; m <= H; ++m) {
            a = mul_add(s[m - 1], odd_cos<R>(k * m), a);
            b = mul_add(d[m - 1], odd_sin<R>(k * m), b);
        }
        const V jb = mul_mj(b);
        v[k] = a + jb;
        v[R - k] = a - jb;
    }
    v[0] = sum;
}

template <int R, class V>
__device__ __forceinline__ void dft_small(V (&v)[R]) {
    constexpr Const kH = PCAL_FFT_CONST(0.70710678118654752440);                                         // cos pi/4
    constexpr Const kC = PCAL_FFT_CONST(0.92387953251128675613), kS = PCAL_FFT_CONST(0.38268343236508977173);  // pi/8
    constexpr Const nC{-kC.h, -kC.l}, nS{-kS.h, -kS.l};
    // times exp(-j pi/4) and exp(-j 3 pi/4): (a -+ j a) scaled
    auto eighth = [&](V a) { return scale(a + mul_mj(a), kH); };
    auto three_eighths = [&](V a) { return scale(mul_mj(a) - a, kH); };
    if constexpr (R == 2) {
        const V t = v[0] - v[1];
        v[0] = v[0] + v[1];
        v[1] = t;
    } else if constexpr (R == 4) {
        dft4(v[0], v[1], v[2], v[3]);
    } else if constexpr (R == 8) {
        dft4(v[0], v[2], v[4], v[6]);
        dft4(v[1], v[3], v[5], v[7]);
        v[3] = eighth(v[3]);
        v[5] = mul_mj(v[5]);
        v[7] = three_eighths(v[7]);
        const V a[4] = {v[0], v[2], v[4], v[6]}, b[4] = {v[1], v[3], v[5], v[7]};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            v[k] = a[k] + b[k];
            v[k + 4] = a[k] - b[k];
        }
    } else if constexpr (R == 16) {
#pragma unroll
        for (int n = 0; n < 4; ++n) dft4(v[n], v[n + 4], v[n + 8], v[n + 12]);
        // A[n][k] sits in v[n + 4k]; times exp(-j 2 pi n k / 16)
        v[5] = mul(v[5], kC, nS);
        v[6] = eighth(v[6]);
        v[7] = mul(v[7], kS, nC);
        v[9] = eighth(v[9]);
        v[10] = mul_mj(v[10]);
        v[11] = three_eighths(v[11]);
        v[13] = mul(v[13], kS, nC);
        v[14] = three_eighths(v[14]);
        v[15] = mul(v[15], nC, kS);
#pragma unroll
        for (int k = 0; k < 4; ++k) dft4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
        // X[k + 4 k2] sits in v[4k + k2]
#pragma unroll
        for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int k2 = k + 1; k2 < 4; ++k2) {
                const V t = v[4 * k + k2];
                v[4 * k + k2] = v[4 * k2 + k];
                v[4 * k2 + k] = t;
            }
    } else {
        dft_odd<R>(v);
    }
}

// x / d as the high word of x * over(d), for d > 1 and x d < 2^32.
inline uint32_t over(int d) { return d > 1 ? (uint32_t)((1ull << 32) / (uint64_t)d + 1) : 0; }

struct FftArgs {
    FftPlan p;
    const float2* P;
    float2* T;
    int64_t C;
    int G;  // channels per CTA
    uint32_t tw_at;  // staged twiddles: bytes into shared memory
};

// One pass over the CTA's channels: radix R, m = product of the radices
// before; from and to are a shared buffer, or null for P and T.
template <int R, class V, bool CHAIN>
__device__ __forceinline__ void fft_pass(const FftArgs& a, int s, int m, const typename V::Twiddle* tw, const float2* from,
                                         float2* to, int64_t c0, int channels) {
    const int N = a.p.N, nb = N / R, pitch = pad(N) + 1;
    const int total = channels * nb;
    for (int b = threadIdx.x; b < total; b += kThreads) {
        int c, hi;
        if constexpr (CHAIN) {
            c = (int)__umulhi((uint32_t)b, a.p.by_nb[s]);
            hi = m > 1 ? (int)__umulhi((uint32_t)(b - c * nb), a.p.by_m[s]) : b - c * nb;
        } else {
            c = b / nb;
            hi = (b - c * nb) / m;
        }
        const int j = b - c * nb, k = j - hi * m;
        V v[R];
        if (from) {
            const float2* x = from + c * pitch;
#pragma unroll
            for (int q = 0; q < R; ++q) v[q] = V::load(x[pad(j + q * nb)]);
        } else {
            const float2* x = a.P + (c0 + c) * N + j;
#pragma unroll
            for (int q = 0; q < R; ++q) v[q] = V::load(__ldcs(x + q * nb));
        }
        if (m > 1) {
#pragma unroll
            for (int q = 1; q < R; ++q) {
                const typename V::Twiddle* w = tw + (q - 1) * m + k;
                v[q] = turn(v[q], CHAIN ? *w : __ldg(w));
            }
        }
        dft_small<R>(v);
        const int o = hi * m * R + k;
        if (to) {
            float2* y = to + c * pitch;
#pragma unroll
            for (int q = 0; q < R; ++q) y[pad(o + q * m)] = v[q].round();
        } else {
            float2* y = a.T + (c0 + c) * N + o;
#pragma unroll
            for (int q = 0; q < R; ++q) __stcs(y + q * m, v[q].round());
        }
    }
}

template <class V, bool CHAIN>
__global__ void __launch_bounds__(kThreads) fft_kernel(const __grid_constant__ FftArgs a) {
    extern __shared__ __align__(16) float2 fft_smem[];
    const int64_t c0 = (int64_t)blockIdx.x * a.G;
    const int channels = a.C - c0 < a.G ? (int)(a.C - c0) : a.G;
    float2* buf0 = fft_smem;
    float2* buf1 = fft_smem + (size_t)a.G * (pad(a.p.N) + 1);
    int m = 1;
    const typename V::Twiddle* tw = static_cast<const typename V::Twiddle*>(a.p.tw);
    if constexpr (CHAIN) {
        // (behind the buffers; in place at the first pass's barrier)
        auto* staged = reinterpret_cast<typename V::Twiddle*>(reinterpret_cast<uint8_t*>(fft_smem) + a.tw_at);
        for (int i = threadIdx.x; i < a.p.N - a.p.radix[0]; i += kThreads) staged[i] = __ldg(tw + i);
        tw = staged;
    }
    for (int s = 0; s < a.p.passes; ++s) {
        const int r = a.p.radix[s];
        const float2* from = s == 0 ? nullptr : s & 1 ? buf0 : buf1;
        float2* to = s == a.p.passes - 1 ? nullptr : s & 1 ? buf1 : buf0;
        switch (r) {
            case 2: fft_pass<2, V, CHAIN>(a, s, m, tw, from, to, c0, channels); break;
            case 3: fft_pass<3, V, CHAIN>(a, s, m, tw, from, to, c0, channels); break;
            case 4: fft_pass<4, V, CHAIN>(a, s, m, tw, from, to, c0, channels); break;
            case 5: fft_pass<5, V, CHAIN>(a, s, m, tw, from, to, c0, channels); break;
            case 7: fft_pass<7, V, CHAIN>(a, s, m, tw, from, to, c0, channels); break;
            case 8: fft_pass<8, V, CHAIN>(a, s, m, tw, from, to, c0, channels); break;
            default: fft_pass<16, V, CHAIN>(a, s, m, tw, from, to, c0, channels); break;
        }
        if (m > 1) tw += (r - 1) * m;
        m *= r;
        __syncthreads();
    }
}

inline size_t tile_bytes(const FftPlan& p, int G) {
    return (size_t)(p.passes > 2 ? 2 : p.passes - 1) * G * (pad(p.N) + 1) * sizeof(float2);
}

// Channels per CTA: kTileValues values, but fewer where that leaves SMs idle.
inline int tile_channels(const FftPlan& p, int64_t C) {
    int64_t G = kTileValues / p.N > 0 ? kTileValues / p.N : 1;
    const int64_t even = (C + kSms - 1) / kSms;
    if (G > even) G = even;
    return (int)G;
}

// Radices of N: its power of two in factors of at most 16 as equal as they come
// (the first and the last pass then read and write runs of at least 4 values),
// and its 3s, 5s and 7s between them.
inline bool fft_factors(int N, FftPlan* p) {
    *p = FftPlan{};
    p->N = N;
    if (N < 2) return false;
    int twos = 0, rest = N;
    while (rest % 2 == 0) {
        rest /= 2;
        ++twos;
    }
    const int parts = (twos + 3) / 4;
    int out[kFftMaxPasses], n = 0;
    for (int i = 0; i < parts; ++i) out[n++] = 1 << ((twos * (i + 1)) / parts - (twos * i) / parts);
    if (twos == 4 && rest == 1) {
        out[0] = out[1] = 4;
        n = 2;
    }
    const int odd[3] = {3, 5, 7};
    int k = 0, odds[kFftMaxPasses];
    for (int f : odd)
        while (rest % f == 0) {
            rest /= f;
            odds[k++] = f;
        }
    if (rest != 1 || n + k > kFftMaxPasses) return false;
    p->passes = n + k;
    int at = 0;
    if (n > 0) p->radix[at++] = out[0];
    for (int i = 0; i < k; ++i) p->radix[at++] = odds[i];
    for (int i = 1; i < n; ++i) p->radix[at++] = out[i];
    return true;
}

// Plan and device tables (allocates).  wide: double-float values inside a pass,
// else FP32.
inline cudaError_t fft_create(int N, bool wide, FftPlan* p) {
    if (!fft_factors(N, p)) return cudaErrorInvalidValue;
    p->wide = wide;
    for (int s = 0, product = 1; s < p->passes; product *= p->radix[s++]) {
        p->by_nb[s] = over(N / p->radix[s]);
        p->by_m[s] = over(product);
    }
    std::vector<float> tw;
    auto put = [&](double x) {
        tw.push_back((float)x);
        if (wide) tw.push_back((float)(x - (double)(float)x));
    };
    int m = p->radix[0];
    for (int s = 1; s < p->passes; ++s) {
        const int r = p->radix[s];
        for (int q = 1; q < r; ++q)
            for (int k = 0; k < m; ++k) {
                const double th = -2.0 * M_PI * (double)(q * k) / (double)(m * r);
                put(cos(th));
                put(sin(th));
            }
        m *= r;
    }
    cudaError_t e = cudaMalloc(&p->tw, tw.size() * sizeof(float) + 16);
    if (e == cudaSuccess && !tw.empty())
        e = cudaMemcpy(p->tw, tw.data(), tw.size() * sizeof(float), cudaMemcpyHostToDevice);
    return e;
}

inline void fft_destroy(FftPlan* p) {
    cudaFree(p->tw);
    p->tw = nullptr;
}

// T[c] = the N-point DFT of P[c], c < C (C >= 1).
inline cudaError_t launch_fft(const FftPlan& p, const float2* P, int64_t C, float2* T, cudaStream_t s) {
    FftArgs a{};
    a.p = p;
    a.P = P;
    a.T = T;
    a.C = C;
    a.G = tile_channels(p, C);
    const unsigned grid = (unsigned)((C + a.G - 1) / a.G);
    const bool chain = !p.wide && p.N >= kChainMinN && p.N <= kChainMaxN;  // (more than one pass)
    size_t smem = tile_bytes(p, a.G);
    if (chain) {
        a.tw_at = (uint32_t)((smem + 15) / 16 * 16);
        smem = a.tw_at + (size_t)(p.N - p.radix[0]) * sizeof(float2);
    }
    auto* k = p.wide ? fft_kernel<Double, false> : chain ? fft_kernel<Single, true> : fft_kernel<Single, false>;
    k<<<grid, kThreads, smem, s>>>(a);
    return cudaGetLastError();
}

#undef PCAL_FFT_CONST

}  // namespace pcal_fft
