// Long-period plans (pcal_rotplan_*): offsets whose combined period L is too
// long to fold (prime offsets; L above 2^20) or that are not whole hertz.
//
// There is no short period to fold over, so the sums of the paper's own route
// are formed: every sample rotated by exp(-j*w_o*n) (Eq. 3) and added into bin
// n mod N (Eq. 2).  The rotation is factored so that no rotator is advanced
// per sample.  A call's samples are cut into stripes of S samples (S a
// multiple of N); with n = n_cta + (j*K + k)*S + p,
//
//   exp(-j w n) = G(n_cta) * E[j] * W[k] * F[p]:
//
// W[k], the turn of k stripes, is the same for every position p, so a thread
// that owns fixed positions p multiplies each of its samples by a table entry
// that the whole block shares; the sum of a block of K stripes takes one
// complex multiplication by E[j], and the CTA's total one by F[p] and by G.
// W, E and F depend on the plan alone (FP64 sincospi of exactly reduced
// phases, tabulated once); G is one FP64 phasor per CTA.  All sums beyond a
// block are double-float.  Inside a block:
//   float32, 2-bit  x * W[k] as an exact product (FMA residual) in a
//                   compensated FP32 sum (two_sum; 11 FP32 operations per
//                   component); a 2-bit code picks its product level * W[k]
//                   from a table in shared memory
//   int8            W in fixed point, six balanced base-256 digits (2^-46):
//                   each digit's sum is exact in int32 with __dp4a over four
//                   stripes at a time
// Bound: 2-bit the issue slots (85 % of them, 180 us for 256M samples).  int8 and
// float32 no pipe: 3 IDP4A (half rate) and half a PRMT a sample are 44 of int8's 64 us
// for 256M samples (4.0 TB/s; issue slots 59 %, the FMA pipe 37 %, throttled between),
// 22 FP32 operations a sample 9 of float32's 22 us for 16M (3.0 TB/s; issue slots 66 %, the
// FMA pipe 54 % while the SMs are busy, which is four fifths of the time); with 13 to 15
// warps an SM the rest is latency, and the start and the merge of CTAs of 26 and
// 6 stages.  A double-float rotator advanced by one complex
// multiplication per sample (about 120 dependent FP32 operations) took 1152
// and 90 us.  Also measured on int8: three CTAs per SM with 16 KB stages 68 us
// (the fixed cost per CTA outweighs the warps), four stages of 16 KB 74 us.
//
// Movement: a CTA's stripes are contiguous, so one thread streams them through
// a ring of 32 KB shared-memory stages with 1-D bulk copies (evict-first
// in L2).  The samples before the first 16-byte boundary and after the last
// one (at most 30 bytes) are rotated one by one in an extra CTA.
#include <math.h>
#include <string.h>

#include <new>

#include "df64.cuh"
#include "internal.cuh"
#include "ptx.cuh"

namespace {

using pcal_df::df;
using namespace pcal_ptx;

constexpr int kStages = 3;
constexpr int kStageTarget = 32 * 1024;  // bytes of a stage, where whole stripes allow
constexpr int kBlocks = 256;             // blocks of K stripes a CTA can fold in one launch (entries of E)
constexpr int kDigits = 6;               // base-256 digits of a fixed-point weight
constexpr int kFracBits = 46;            // its resolution: |W| <= 1 is at most 64 in the leading digit
constexpr int kNarrow = 256;             // threads up to which kShare CTAs share an SM
constexpr int kShare = 2;
constexpr int kEdgeMax = 2 * 15 * 4;     // samples in two runs of at most 15 bytes
constexpr int kRotMaxSmem = 226 * 1024;  // (and 1 KB of static shared memory at most)

// How a plan's samples are cut: fixed when it is created.
struct RotGeom {
    int N, S, T;       // stripe: S samples, T = S / 4 threads of four positions
    int K;             // stripes per block
    int ks;            // stripes per stage (K is a multiple)
    int threads;       // T rounded up to whole warps
    int stage_bytes;   // of samples; a multiple of 16
    int ctas;          // most CTAs of a launch
    int digits;        // int8 with digit weights
    size_t smem;
};

struct RotArgs {
    RotGeom g;
    const uint8_t* x;       // 16-byte aligned first sample of the stripes
    int64_t n0;             // its absolute index
    int64_t n;              // samples in whole 16-byte words
    int64_t units;          // stages of samples, the last one possibly short
    int ctas;               // CTAs that fold stripes; one more takes the edges if there are any
    const uint8_t* edge_x;  // the call's samples; edges: [0, head) and [tail_at, tail_at + tail)
    int64_t edge_n0, tail_at;
    int head, tail;
    double r_hi, r_lo;      // f_offset / fs as a double-double
    df lev[4];              // 2-bit code values
    const float4* W;        // [K] re (hi, lo), im (hi, lo)
    const uint4* Wd;        // [K / 4][3]: digit words of four stripes, re 0..5 then im 0..5
    const float4* E;        // [kBlocks]
    const float4* F;        // [S]
    float4* acc;            // [ctas + 1][N]: re (hi, lo), im (hi, lo); the last row takes the edges
    unsigned int* err;
};

// frac(n * (r_hi + r_lo)) for 0 <= n < 2^52, about 1e-16 absolute: n is split
// into two exactly representable parts, each product into its rounded value
// and its exact error (fma), and only fractional parts are added.
__device__ __forceinline__ double frac_mul(int64_t n, double r_hi, double r_lo) {
    const double nh = (double)(n >> 26) * 67108864.0;
    const double nl = (double)(n & 0x3FFFFFF);
    const double p = nh * r_hi, e = fma(nh, r_hi, -p);
    const double q = nl * r_hi, g = fma(nl, r_hi, -q);
    double f = (p - floor(p)) + (q - floor(q));
    f += e + g + (double)n * r_lo;
    return f - floor(f);
}

// exp(-j*2*pi*c) as a double-float complex: re (hi, lo), im (hi, lo).
__device__ __forceinline__ float4 phasor_df(double c) {
    double s, co;
    sincospi(2.0 * c, &s, &co);
    s = -s;
    const float ch = (float)co, sh = (float)s;
    return make_float4(ch, (float)(co - (double)ch), sh, (float)(s - (double)sh));
}

__device__ __forceinline__ float4 cadd(float4 a, float4 b) {
    const df r = pcal_df::add(df{a.x, a.y}, df{b.x, b.y}), i = pcal_df::add(df{a.z, a.w}, df{b.z, b.w});
    return make_float4(r.hi, r.lo, i.hi, i.lo);
}

__device__ __forceinline__ float4 cmul(float4 a, float4 b) {
    const df ar{a.x, a.y}, ai{a.z, a.w}, br{b.x, b.y}, bi{b.z, b.w};
    const df r = pcal_df::sub(pcal_df::mul(ar, br), pcal_df::mul(ai, bi));
    const df i = pcal_df::add(pcal_df::mul(ar, bi), pcal_df::mul(ai, br));
    return make_float4(r.hi, r.lo, i.hi, i.lo);
}

__device__ __forceinline__ void bulk_load_hint(void* dst, const void* src, uint32_t bytes, uint64_t* bar,
                                               uint64_t policy) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::
            "r"(smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar)), "l"(policy)
        : "memory");
}

// s + c += p + e with p + e the exact (or double-float) addend: two_sum and
// one compensation term.
__device__ __forceinline__ void comp_add(float& s, float& c, float p, float e) {
    const df t = pcal_df::two_sum(s, p);
    s = t.hi;
    c += t.lo + e;
}

// x * (wh + wl) into (s, c).
__device__ __forceinline__ void comp_fma(float& s, float& c, float x, float wh, float wl) {
    const float p = __fmul_rn(x, wh);  // (not contracted into the sum)
    comp_add(s, c, p, fmaf(x, wl, fmaf(x, wh, -p)));
}

// sum_i d[i] * 256^(5-i) * 2^-kFracBits as a double-float, |d[i]| <= 2^23: the
// digit sums are exact as floats, the leading and the trailing three add
// exactly in a double-float.  (64-bit conversions instead ran on the FP64 pipe:
// 12 % of a 256M-sample call.)
__device__ __forceinline__ df digits_df(const int* d) {
    constexpr float kHi = 1.0f / (float)(1ll << (kFracBits - 24)), kLo = 1.0f / (float)(1ll << kFracBits);
    const df h = pcal_df::add_f(pcal_df::two_sum((float)d[0] * 65536.f, (float)d[1] * 256.f), (float)d[2]);
    const df l = pcal_df::add_f(pcal_df::two_sum((float)d[3] * 65536.f, (float)d[4] * 256.f), (float)d[5]);
    return pcal_df::add(df{h.hi * kHi, h.lo * kHi}, df{l.hi * kLo, l.lo * kLo});
}

__device__ __forceinline__ df sample_df(int fmt, const RotArgs& a, int64_t i) {
    if (fmt == PCAL_I8) return df{(float)reinterpret_cast<const int8_t*>(a.edge_x)[i], 0.f};
    if (fmt == PCAL_F32) return df{reinterpret_cast<const float*>(a.edge_x)[i], 0.f};
    return a.lev[(a.edge_x[i >> 2] >> (2 * (int)(i & 3))) & 3];
}

// The samples outside the 16-byte words, rotated one by one: thread e takes
// sample e, then the bins add theirs in sample order.
template <int FMT>
__device__ void fold_edges(const RotArgs& a, float4* val, int* col) {
    const int count = a.head + a.tail, N = a.g.N;
    for (int e = threadIdx.x; e < count; e += blockDim.x) {
        const int64_t i = e < a.head ? e : a.tail_at + (e - a.head);
        const float4 w = phasor_df(frac_mul(a.edge_n0 + i, a.r_hi, a.r_lo));
        const df x = sample_df(FMT, a, i);
        const df re = pcal_df::mul(x, df{w.x, w.y}), im = pcal_df::mul(x, df{w.z, w.w});
        val[e] = make_float4(re.hi, re.lo, im.hi, im.lo);
        col[e] = (int)((a.edge_n0 + i) % N);
    }
    __syncthreads();
    float4* acc = a.acc + (size_t)a.g.ctas * N;
    for (int b = threadIdx.x; b < N; b += blockDim.x) {
        bool any = false;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int e = 0; e < count; ++e)
            if (col[e] == b) {
                s = cadd(s, val[e]);
                any = true;
            }
        if (any) acc[b] = cadd(acc[b], s);
    }
}

// Shared memory: kStages stages of samples (afterwards S float4 of the merge),
// the block's weights (float32, int8: float4 [K]; 2-bit: float4 [K][4];
// digits: uint4 [K / 4][3]).
__host__ __device__ inline size_t weight_bytes(int fmt, int digits, int K) {
    return digits ? (size_t)K / 4 * 48 : (size_t)K * (fmt == PCAL_2BIT ? 64 : 16);
}
__host__ __device__ inline size_t ring_bytes(const RotGeom& g) {
    const size_t r = (size_t)kStages * g.stage_bytes, m = (size_t)g.S * 16;
    return ((r > m ? r : m) + 15) / 16 * 16;
}

template <int FMT, bool DIGITS, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) rotplan_fold_kernel(const __grid_constant__ RotArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    __shared__ __align__(8) uint64_t full[kStages];
    __shared__ float4 s_G;
    __shared__ int s_fail;
    const RotGeom& g = a.g;
    const int tid = threadIdx.x;
    if ((int)blockIdx.x >= a.ctas) {
        fold_edges<FMT>(a, reinterpret_cast<float4*>(smem), reinterpret_cast<int*>(smem + 16 * kEdgeMax));
        return;
    }
    const int64_t u0 = a.units * blockIdx.x / a.ctas;
    const int nu = (int)(a.units * (blockIdx.x + 1) / a.ctas - u0);
    const int64_t stage_samples = (int64_t)g.ks * g.S;
    const uint8_t* src = a.x + u0 * g.stage_bytes;
    uint8_t* weights = smem + ring_bytes(g);
    const uint64_t policy = tid == 0 ? l2_policy_evict_first() : 0ull;
    // samples of unit u of this CTA
    auto valid_of = [&](int u) -> int64_t {
        const int64_t left = a.n - (u0 + u) * stage_samples;
        return left < stage_samples ? left : stage_samples;
    };
    auto issue = [&](int u) {
        const int64_t v = valid_of(u);
        const uint32_t bytes = (uint32_t)(FMT == PCAL_F32 ? 4 * v : FMT == PCAL_I8 ? v : v / 4);
        mbar_arrive_expect_tx(&full[u % kStages], bytes);
        bulk_load_hint(smem + (size_t)(u % kStages) * g.stage_bytes, src + (size_t)u * g.stage_bytes, bytes,
                       &full[u % kStages], policy);
    };
    if (tid == 0) {
        for (int s = 0; s < kStages; ++s) mbar_init(&full[s], 1);
        s_fail = 0;
        fence_barrier_init();
        for (int u = 0; u < kStages && u < nu; ++u) issue(u);
    }
    // the last warp takes the CTA's own phasor (a chain of FP64 operations)
    if (tid / 32 == (int)blockDim.x / 32 - 1) {
        const float4 G = phasor_df(frac_mul(a.n0 + u0 * stage_samples, a.r_hi, a.r_lo));
        if (tid % 32 == 0) s_G = G;
    }
    if constexpr (DIGITS) {
        for (int i = tid; i < g.K / 4 * 3; i += blockDim.x) reinterpret_cast<uint4*>(weights)[i] = a.Wd[i];
    } else if constexpr (FMT == PCAL_2BIT) {
        for (int i = tid; i < g.K * 4; i += blockDim.x) {
            const float4 w = a.W[i / 4];
            const df l = a.lev[i % 4];
            const df re = pcal_df::mul(l, df{w.x, w.y}), im = pcal_df::mul(l, df{w.z, w.w});
            reinterpret_cast<float4*>(weights)[i] = make_float4(re.hi, re.lo, im.hi, im.lo);
        }
    } else {
        for (int i = tid; i < g.K; i += blockDim.x) reinterpret_cast<float4*>(weights)[i] = a.W[i];
    }
    __syncthreads();

    const bool own = tid < g.T;
    const int KU = g.K / g.ks;  // units per block
    float sr[4], cr[4], si[4], ci[4];
    int d[4][2 * kDigits];
    float4 tot[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        tot[v] = make_float4(0.f, 0.f, 0.f, 0.f);
        sr[v] = cr[v] = si[v] = ci[v] = 0.f;
#pragma unroll
        for (int q = 0; q < 2 * kDigits; ++q) d[v][q] = 0;
    }
    int ku = 0, block = 0, u = 0, st = 0;
    uint32_t phase = 0;
    for (; u < nu; ++u) {
        uint8_t* stage = smem + st * g.stage_bytes;
        if (!mbar_wait(&full[st], phase)) {
            atomicOr(a.err, PCAL_DERR_FULL_WAIT);
            s_fail = 1;
        }
        int stripes = g.ks;
        const int64_t valid = u == nu - 1 ? valid_of(u) : stage_samples;
        if (valid < stage_samples) {
            // the call's last, short unit: zeros (which add nothing) behind its
            // float32 or int8 samples; a 2-bit zero is a code, so there each
            // thread stops after its own last whole byte (valid is a multiple of 4)
            if (FMT == PCAL_2BIT) {
                const int64_t mine = valid - 4 * tid;
                stripes = mine > 0 ? (int)((mine + g.S - 1) / g.S) : 0;
            } else {
                const int from = (int)(FMT == PCAL_F32 ? 4 * valid : valid);
                for (int o = from + 4 * tid; o < g.stage_bytes; o += 4 * blockDim.x)
                    *reinterpret_cast<uint32_t*>(stage + o) = 0u;
                __syncthreads();
            }
        }
        if (own) {
            if constexpr (DIGITS) {
                const uint8_t* p = stage + 4 * tid;
                const uint4* wq = reinterpret_cast<const uint4*>(weights) + (size_t)ku * g.ks / 4 * 3;
#pragma unroll 2
                for (int k = 0; k < stripes; k += 4, p += 4 * g.S, wq += 3) {
                    const uint32_t w0 = *reinterpret_cast<const uint32_t*>(p);
                    const uint32_t w1 = *reinterpret_cast<const uint32_t*>(p + g.S);
                    const uint32_t w2 = *reinterpret_cast<const uint32_t*>(p + 2 * g.S);
                    const uint32_t w3 = *reinterpret_cast<const uint32_t*>(p + 3 * g.S);
                    // four stripes x four positions of bytes, transposed
                    const uint32_t t0 = __byte_perm(w0, w1, 0x5140), t1 = __byte_perm(w2, w3, 0x5140);
                    const uint32_t t2 = __byte_perm(w0, w1, 0x7362), t3 = __byte_perm(w2, w3, 0x7362);
                    const uint32_t x[4] = {__byte_perm(t0, t1, 0x5410), __byte_perm(t0, t1, 0x7632),
                                           __byte_perm(t2, t3, 0x5410), __byte_perm(t2, t3, 0x7632)};
                    const uint4 q0 = wq[0], q1 = wq[1], q2 = wq[2];
                    const uint32_t q[12] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w, q2.x, q2.y, q2.z, q2.w};
#pragma unroll
                    for (int v = 0; v < 4; ++v)
#pragma unroll
                        for (int m = 0; m < 12; ++m) d[v][m] = __dp4a((int)x[v], (int)q[m], d[v][m]);
                }
            } else if constexpr (FMT == PCAL_2BIT) {
                const uint8_t* p = stage + tid;
                const float4* wq = reinterpret_cast<const float4*>(weights) + (size_t)ku * g.ks * 4;
#pragma unroll 4
                for (int k = 0; k < stripes; ++k, p += g.S / 4, wq += 4) {
                    const uint32_t c = *p;
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const float4 w = wq[(c >> (2 * v)) & 3u];
                        comp_add(sr[v], cr[v], w.x, w.y);
                        comp_add(si[v], ci[v], w.z, w.w);
                    }
                }
            } else {
                const uint8_t* p = stage + (FMT == PCAL_F32 ? 16 : 4) * tid;
                const float4* wq = reinterpret_cast<const float4*>(weights) + (size_t)ku * g.ks;
                const int pitch = FMT == PCAL_F32 ? 4 * g.S : g.S;
#pragma unroll 4
                for (int k = 0; k < stripes; ++k, p += pitch, ++wq) {
                    float x[4];
                    if (FMT == PCAL_F32) {
                        const float4 f = *reinterpret_cast<const float4*>(p);
                        x[0] = f.x;
                        x[1] = f.y;
                        x[2] = f.z;
                        x[3] = f.w;
                    } else {
                        const char4 c = *reinterpret_cast<const char4*>(p);
                        x[0] = (float)c.x;
                        x[1] = (float)c.y;
                        x[2] = (float)c.z;
                        x[3] = (float)c.w;
                    }
                    const float4 w = *wq;
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        comp_fma(sr[v], cr[v], x[v], w.x, w.y);
                        comp_fma(si[v], ci[v], x[v], w.z, w.w);
                    }
                }
            }
            if (++ku == KU || u == nu - 1) {
                // end of a block: its sums, turned by E[block] (E[0] = 1), into the totals
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    df re, im;
                    if constexpr (DIGITS) {
                        re = digits_df(d[v]);
                        im = digits_df(d[v] + kDigits);
#pragma unroll
                        for (int m = 0; m < 2 * kDigits; ++m) d[v][m] = 0;
                    } else {
                        re = pcal_df::two_sum(sr[v], cr[v]);
                        im = pcal_df::two_sum(si[v], ci[v]);
                        sr[v] = cr[v] = si[v] = ci[v] = 0.f;
                    }
                    const float4 z = make_float4(re.hi, re.lo, im.hi, im.lo);
                    tot[v] = block == 0 ? z : cadd(tot[v], cmul(z, a.E[block]));
                }
                ku = 0;
                ++block;
            }
        }
        __syncthreads();
        if (*reinterpret_cast<volatile int*>(&s_fail)) break;
        if (tid == 0 && u + kStages < nu) issue(u + kStages);
        if (++st == kStages) {
            st = 0;
            phase ^= 1u;
        }
    }
    // the finalize may launch (it waits for this kernel before it reads a row)
    allow_dependents();
    if (s_fail) {
        // copies in flight (of units u .. u + kStages - 1) land before the
        // CTA's shared memory is reused
        if (tid == 0)
            for (int v = u; v < u + kStages && v < nu; ++v)
                if (!mbar_wait(&full[v % kStages], (uint32_t)(v / kStages) & 1)) atomicOr(a.err, PCAL_DERR_DRAIN_WAIT);
        return;
    }
    // the totals turned by F, the S / N positions of each bin added, and the
    // bin's sum, turned by G, added to this CTA's row
    float4* m = reinterpret_cast<float4*>(smem);
    if (own) {
#pragma unroll
        for (int v = 0; v < 4; ++v) m[4 * tid + v] = cmul(tot[v], a.F[4 * tid + v]);
    }
    // (halving: 64 positions in turn took 3 us where N is 16)
    int rows = g.S / g.N;
    for (;;) {
        __syncthreads();
        if (rows == 1) break;
        const int half = (rows + 1) / 2;
        for (int p = tid; p < (rows - half) * g.N; p += blockDim.x) m[p] = cadd(m[p], m[p + half * g.N]);
        rows = half;
    }
    float4* acc = a.acc + (size_t)blockIdx.x * g.N;
    const int first = (int)(a.n0 % g.N);  // every CTA starts at a multiple of N behind n0
    for (int b = tid; b < g.N; b += blockDim.x) {
        const int c = first + b < g.N ? first + b : first + b - g.N;
        acc[c] = cadd(acc[c], cmul(m[b], s_G));
    }
}

// The plan's tables: W (or its digits), E and F.
__global__ void rotplan_tables_kernel(RotGeom g, double r_hi, double r_lo, float4* W, uint4* Wd, float4* E, float4* F) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < g.S) F[i] = phasor_df(frac_mul(i, r_hi, r_lo));
    if (i < kBlocks) E[i] = phasor_df(frac_mul((int64_t)i * g.K * g.S, r_hi, r_lo));
    if (i >= g.K) return;
    const double c = frac_mul((int64_t)i * g.S, r_hi, r_lo);
    if (!g.digits) {
        W[i] = phasor_df(c);
        return;
    }
    double s, co;
    sincospi(2.0 * c, &s, &co);
    // balanced base-256 digits, least significant first
    int8_t* out = reinterpret_cast<int8_t*>(Wd) + (size_t)(i / 4) * 48 + i % 4;
    for (int part = 0; part < 2; ++part) {
        long long v = llrint((part ? -s : co) * (double)(1ll << kFracBits));
        for (int q = kDigits - 1; q >= 0; --q) {
            const int dgt = (int)(int8_t)(v & 0xff);
            out[4 * (part * kDigits + q)] = (int8_t)dgt;
            v = (v - dgt) >> 8;
        }
    }
}

__global__ void rotplan_twiddles_kernel(float2* twN, int N) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= N) return;
    double s, c;
    sincospi(2.0 * (double)m / (double)N, &s, &c);
    twN[m] = make_float2((float)c, (float)-s);
}

int gcd_int(int a, int b) { return b ? gcd_int(b, a % b) : a; }

// Stripes of at most 1024 samples where N allows (so that a bin's positions fill a CTA's
// threads whatever N is): a whole number of bins and of the threads' four
// positions.  Tones that are no multiple of four can need up to 4N = 4092.
RotGeom rot_geom(int N, int fmt, int sms) {
    RotGeom g{};
    const int base = N / gcd_int(N, 4) * 4;
    const int mult = base < 1024 ? 1024 / base : 1;
    g.N = N;
    g.S = base * mult;
    g.T = g.S / 4;
    g.threads = (g.T + 31) / 32 * 32;
    const bool narrow = g.threads <= kNarrow;
    // digit weights need 48 counters a thread: not for the widest CTAs
    g.digits = fmt == PCAL_I8 && narrow;
    g.K = g.digits ? 512 : 128;
    const int stripe = fmt == PCAL_F32 ? 4 * g.S : fmt == PCAL_I8 ? g.S : g.S / 4;
    // whole 16-byte words per stage, whole groups of four stripes
    g.ks = fmt == PCAL_2BIT ? 16 : 4;
    while (2 * g.ks * stripe <= kStageTarget && 2 * g.ks <= 128) g.ks *= 2;
    if (fmt == PCAL_F32)
        while (g.ks > 1 && g.ks * stripe > kStageTarget) g.ks /= 2;
    g.stage_bytes = g.ks * stripe;
    g.ctas = narrow ? kShare * sms : sms;
    g.smem = ring_bytes(g) + weight_bytes(fmt, g.digits, g.K);
    if (g.smem < 20 * kEdgeMax) g.smem = 20 * kEdgeMax;
    return g;
}

using RotKernel = void (*)(RotArgs);

RotKernel rot_kernel(const RotGeom& g, int fmt) {
    const bool narrow = g.threads <= kNarrow;
    if (fmt == PCAL_I8)
        return g.digits ? rotplan_fold_kernel<PCAL_I8, true, kNarrow, kShare>
                        : rotplan_fold_kernel<PCAL_I8, false, 1024, 1>;
    if (fmt == PCAL_F32)
        return narrow ? rotplan_fold_kernel<PCAL_F32, false, kNarrow, kShare>
                      : rotplan_fold_kernel<PCAL_F32, false, 1024, 1>;
    return narrow ? rotplan_fold_kernel<PCAL_2BIT, false, kNarrow, kShare>
                  : rotplan_fold_kernel<PCAL_2BIT, false, 1024, 1>;
}

}  // namespace

struct pcal_rotplan {
    int64_t fs, fc;
    double fo;
    int N, fmt;
    RotGeom g;
    double r_hi, r_lo;
    double levels[4];
    int64_t n_abs, period_start;
    float4* d_acc;        // [g.ctas + 1][N] partial sums of the period
    float4* d_W;          // weights of a block: float4 [K], or the digit words
    float4* d_E;          // [kBlocks]
    float4* d_F;          // [S]
    unsigned int* d_err;
    float2* d_twN;
    // 5N+3 results, N+2 post-processing values, the error bits: pinned memory that
    // the finalize writes through its device address (a copy behind it cost the
    // host's wait 5 us)
    double* h_res;
    double* d_res;
    cudaStream_t last_stream;
    bool results_valid;
};

extern "C" int pcal_rotplan_create(double fs, double f_comb, double f_offset, int N, int sample_format,
                                   pcal_rotplan** out) {
    if (!out) return PCAL_EINVAL;
    *out = nullptr;
    if (!(fs > 0) || !(f_comb > 0) || fs != floor(fs) || f_comb != floor(f_comb) || fs > 9.0e15 ||
        !(f_offset >= 0.0) || !(f_offset < f_comb) || (sample_format != PCAL_F32 && sample_format != PCAL_I8 &&
                                                        sample_format != PCAL_2BIT))
        return PCAL_EINVAL;
    const int64_t ifs = (int64_t)fs, ifc = (int64_t)f_comb;
    if (ifs % ifc != 0 || N != ifs / ifc) return PCAL_EINVAL;
    if (N > PCAL_BATCH_MAX_N) return PCAL_ETOOLARGE;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) !=
                                                  cudaSuccess) {
        (void)cudaGetLastError();
        return PCAL_ECUDA;
    }
    pcal_rotplan* r = new (std::nothrow) pcal_rotplan();
    if (!r) return PCAL_ENOMEM;
    r->fs = ifs;
    r->fc = ifc;
    r->fo = f_offset;
    r->N = N;
    r->fmt = sample_format;
    r->g = rot_geom(N, sample_format, sms);
    r->r_hi = f_offset / fs;
    r->r_lo = fma(-r->r_hi, fs, f_offset) / fs;
    const double lv[4] = {-3.3359, -1.0, 1.0, 3.3359};
    memcpy(r->levels, lv, sizeof(lv));
    r->n_abs = r->period_start = 0;
    r->last_stream = nullptr;
    r->results_valid = false;
    const size_t acc_bytes = sizeof(float4) * (size_t)N * (r->g.ctas + 1);
    cudaError_t e = cudaMalloc(&r->d_acc, acc_bytes);
    if (e == cudaSuccess) e = cudaMemset(r->d_acc, 0, acc_bytes);
    if (e == cudaSuccess) e = cudaMalloc(&r->d_W, sizeof(float4) * r->g.K);
    if (e == cudaSuccess) e = cudaMalloc(&r->d_E, sizeof(float4) * kBlocks);
    if (e == cudaSuccess) e = cudaMalloc(&r->d_F, sizeof(float4) * r->g.S);
    if (e == cudaSuccess) e = prepare_rot_finalize();
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(rot_kernel(r->g, sample_format), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kRotMaxSmem);
    if (e == cudaSuccess) e = cudaMalloc(&r->d_twN, sizeof(float2) * N);
    if (e == cudaSuccess) e = cudaMalloc(&r->d_err, sizeof(unsigned int));
    if (e == cudaSuccess) e = cudaMemset(r->d_err, 0, sizeof(unsigned int));
    if (e == cudaSuccess)
        e = cudaHostAlloc(reinterpret_cast<void**>(&r->h_res), sizeof(double) * (6 * (size_t)N + 6), cudaHostAllocMapped);
    if (e == cudaSuccess) {
        memset(static_cast<void*>(r->h_res), 0, sizeof(double) * (6 * (size_t)N + 6));
        e = cudaHostGetDevicePointer(reinterpret_cast<void**>(&r->d_res), r->h_res, 0);
    }
    if (e == cudaSuccess) {
        rotplan_twiddles_kernel<<<(N + 255) / 256, 256>>>(r->d_twN, N);
        const int most = r->g.S > r->g.K ? r->g.S : r->g.K;
        rotplan_tables_kernel<<<(most + 127) / 128, 128>>>(r->g, r->r_hi, r->r_lo, r->d_W,
                                                           reinterpret_cast<uint4*>(r->d_W), r->d_E, r->d_F);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        pcal_rotplan_destroy(r);
        return e == cudaErrorMemoryAllocation ? PCAL_ENOMEM : PCAL_ECUDA;
    }
    *out = r;
    return PCAL_OK;
}

extern "C" int pcal_rotplan_destroy(pcal_rotplan* r) {
    if (!r) return PCAL_OK;
    if (r->last_stream) cudaStreamSynchronize(r->last_stream);
    cudaFree(r->d_acc);
    cudaFree(r->d_W);
    cudaFree(r->d_E);
    cudaFree(r->d_F);
    cudaFree(r->d_twN);
    cudaFree(r->d_err);
    if (r->h_res) cudaFreeHost(r->h_res);
    (void)cudaGetLastError();
    delete r;
    return PCAL_OK;
}

extern "C" int pcal_rotplan_set_levels(pcal_rotplan* r, const double levels[4]) {
    if (!r || !levels) return PCAL_EINVAL;
    memcpy(r->levels, levels, sizeof(r->levels));
    return PCAL_OK;
}

extern "C" int pcal_rotplan_accumulate(pcal_rotplan* r, const void* samples, int64_t n, void* stream) {
    if (!r || n < 0 || (n > 0 && !samples)) return PCAL_EINVAL;
    if (r->fmt == PCAL_2BIT && n % 4 != 0) return PCAL_EINVAL;
    if (r->n_abs + n >= (1LL << 52)) return PCAL_ETOOLARGE;
    if (n == 0) return PCAL_OK;
    const uint8_t* x = static_cast<const uint8_t*>(samples);
    const int fmt = r->fmt;
    if (fmt == PCAL_F32 && reinterpret_cast<uintptr_t>(x) % 4 != 0) return PCAL_EINVAL;
    auto bytes_of = [&](int64_t m) { return fmt == PCAL_F32 ? 4 * m : fmt == PCAL_I8 ? m : m / 4; };
    auto samples_in = [&](int64_t b) { return fmt == PCAL_F32 ? b / 4 : fmt == PCAL_I8 ? b : 4 * b; };
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const RotGeom& g = r->g;
    // at most kBlocks blocks per CTA in one launch (8 to 80 billion samples)
    const int64_t most = (int64_t)g.ctas * (kBlocks - 1) * g.K * g.S;
    while (n > 0) {
        const int64_t m = n < most ? n : most;  // (a multiple of 4: S is)
        RotArgs a{};
        a.g = g;
        const int64_t bytes = bytes_of(m);
        int64_t head = (int64_t)((16 - reinterpret_cast<uintptr_t>(x) % 16) % 16);
        if (head > bytes) head = bytes;
        const int64_t body = (bytes - head) / 16 * 16;
        a.x = x + head;
        a.head = (int)samples_in(head);
        a.n0 = r->n_abs + a.head;
        a.n = samples_in(body);
        a.tail_at = a.head + a.n;
        a.tail = (int)(m - a.tail_at);
        a.edge_x = x;
        a.edge_n0 = r->n_abs;
        const int64_t stage_samples = (int64_t)g.ks * g.S;
        a.units = (a.n + stage_samples - 1) / stage_samples;
        a.ctas = (int)(a.units < g.ctas ? a.units : g.ctas);
        a.r_hi = r->r_hi;
        a.r_lo = r->r_lo;
        for (int c = 0; c < 4; ++c) {
            a.lev[c].hi = (float)r->levels[c];
            a.lev[c].lo = (float)(r->levels[c] - (double)a.lev[c].hi);
        }
        a.W = r->d_W;
        a.Wd = reinterpret_cast<const uint4*>(r->d_W);
        a.E = r->d_E;
        a.F = r->d_F;
        a.acc = r->d_acc;
        a.err = r->d_err;
        const int grid = a.ctas + (a.head + a.tail > 0 ? 1 : 0);
        rot_kernel(g, fmt)<<<grid, g.threads, g.smem, s>>>(a);
        if (cudaGetLastError() != cudaSuccess) return PCAL_ECUDA;
        r->n_abs += m;
        r->last_stream = s;
        x += bytes;
        n -= m;
    }
    return PCAL_OK;
}

extern "C" int pcal_rotplan_finalize_device(pcal_rotplan* r, void* stream) {
    if (!r) return PCAL_EINVAL;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int64_t M = r->n_abs - r->period_start;
    // adds the rows of partial sums and clears them for the next period
    const cudaError_t e = launch_rot_finalize(r->d_acc, r->g.ctas + 1, r->N, (double)r->fs, (double)r->fc, M,
                                              r->d_twN, r->d_res, r->d_err, s);
    if (e != cudaSuccess) return PCAL_ECUDA;
    r->period_start = r->n_abs;
    r->last_stream = s;
    r->results_valid = true;
    return PCAL_OK;
}

extern "C" int pcal_rotplan_read_results(pcal_rotplan* r, double* phasors, double* amp, double* phase,
                                         double* unwrapped, double* td, double* sigma, double* td_peak,
                                         double* bandpass_phase) {
    if (!r) return PCAL_EINVAL;
    if (!r->results_valid) return PCAL_EBUSY;
    const int64_t N = r->N;
    if (cudaStreamSynchronize(r->last_stream) != cudaSuccess) return PCAL_ECUDA;
    const double* h = r->h_res;
    unsigned int err;
    memcpy(&err, h + 6 * N + 5, sizeof(err));
    if (err) return PCAL_ETIMEOUT;
    if (phasors) memcpy(phasors, h, sizeof(double) * 2 * N);
    if (amp) memcpy(amp, h + 2 * N, sizeof(double) * N);
    if (phase) memcpy(phase, h + 3 * N, sizeof(double) * N);
    if (unwrapped) memcpy(unwrapped, h + 4 * N, sizeof(double) * N);
    if (td) *td = h[5 * N];
    if (sigma) *sigma = h[5 * N + 1];
    if (td_peak) *td_peak = h[5 * N + 3];
    if (bandpass_phase) memcpy(bandpass_phase, h + 5 * N + 5, sizeof(double) * N);
    return PCAL_OK;
}
