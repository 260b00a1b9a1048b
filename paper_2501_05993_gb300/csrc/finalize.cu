// Finalize kernels of libpcal: from the L accumulated bins to N tone phasors
// and the delay (paper Sec. 2).
//
//   decode   S[k] from the exact bins (2-bit: the level table applied to the
//            per-code counts; int8/float32: the sums)
//   rotate   R[k] = S[k] * exp(-j*2*pi*f_offset*k/fs)        (Eq. 3)
//   fold     P[b] = sum_m R[b + m*N]                          (Eq. 2)
//            integer bins: exact sums of integer x fixed-point rotator per
//            thread (residue_int), float32 bins FP64 per thread; then
//            double-float (df) across threads
//   DFT      T_i = sum_b P[b] exp(-j*2*pi*i*b/N)   (DFT(P), Sec. 2)   FP32
//   products amp_i = 2|T_i|/M and phase arg(T_i)+pi/2 (sin model of Eq. 1)
//            in FP32; the phase unwrapped along the comb and the delay as
//            the |T|^2-weighted least-squares slope of phase versus tone
//            frequency (phi_i = 2*pi*f_i*t_d, Eq. 1) in df.
//
// The rotator phase is reduced exactly in integers, (f_offset/g * k) mod L,
// and looked up in the plan's table of exp(-j*2*pi*m/L) (the precomputed
// rotator of Sec. 2 after Eq. 4, built once per plan: FP64, or fixed point of
// 54 fractional bits where the decode is in integers).  GB300 runs FP64 at
// about 1/64 of its FP32 rate, so FP64 stops after the per-bin rotation at
// the latest; every sum over many terms after that uses df (see df64.cuh),
// which keeps about 48 bits with FP32 instructions.
//
// Work split.  One thread-block cluster does everything where it can: each
// CTA folds a slice of the bins into a partial P, the partials meet in
// distributed shared memory, and CTA 0 runs the DFT from shared memory and the
// products, so no result makes a round trip through global memory and the
// launch runs beside the next fold on the SMs that it leaves free.  That takes
// every integer plan of N <= 1024, and float32 plans of N <= 256 and L <= 32768
// or of more tones at such periods or without pending partials (large_plan).
// Otherwise the fold kernel gives each CTA whole
// residues b (no two CTAs add into the same P[b]); the last CTA to finish (an
// atomic ticket, no waiting) runs the DFT for small N and the products.  For
// large N a second kernel spreads the DFT over CTAs and its last CTA runs the
// products.  What bounds a cluster is its chain of dependent steps, the
// instructions of each fetched from L2 once; alone 9 to 11 us at 64 tones and
// L 6400, 29 us at 256 tones and L 256,000 beside a fold.
#include <cooperative_groups.h>
#include <math.h>

#include <mutex>

#include "df64.cuh"
#include "internal.cuh"

namespace {

using pcal_df::df;

constexpr int kDftInFoldMaxN = 256;
constexpr int kDftTonesPerCta = 32;
enum { kFew, kMany, kLarge, kAny };  // kinds of cluster finalize (cluster_finalize)
constexpr int kFewN = 64;
constexpr int kFmtRotated = 16;  // cluster finalize of bins that are rotated already

struct FinArgs {
    int fmt;
    int spilled;  // 2-bit: 1 the wide arrays hold counts of this period too, 2 they alone do
    int bc;   // residues b per fold CTA
    int tpb;  // threads per residue (power of two)
    int64_t L, N, so;
    unsigned long long rcp_L;  // floor((2^64 - 1) / L)
    int64_t q, rem, a0;  // samples in bin k: q + ((k - a0) mod L < rem)
    double lev0, c_l, c_h, c_hl;
    int exact;             // integer bins small enough for residue_int
    df k_a, k_b, k_c, k_h; // 2-bit: weights of residue_int's sums
    double M;
    float two_over_m;
    df two_pi_fc;  // 2*pi*f_comb in df
    unsigned long long* acc2;
    unsigned long long* wide2;
    long long* acc8;
    float2* accf;  // float32 bins in df (hi, lo)
    // float32: fold partials not yet added into accf (slot e: [pf_rg[e]][pf_cols], column 0 = bin pf_ka[e])
    const float2* pf[kPartSlots];
    int64_t pf_rg[kPartSlots];
    int64_t pf_ka[kPartSlots];
    int n_pf;
    int64_t pf_cols;
    const long long* counts4;  // no-allocation entry: the caller's counts [L][4]
    double lev[4];             // no-allocation entry: the code levels
    const double2* tw;     // exp(-j 2 pi m/L), or
    const int4* twi;       // (integer kLarge plans, batches) the same in fixed point (rotator_fixed)
    const float2* twN;
    float4* P;     // P[b] as df re (x, y), df im (z, w)
    float2* T;     // FP32 tone phasors
    double* res;
    double* extra;  // post-processing, N+2 doubles (or null): peak delay, peak position, corrected bandpass phase
    float2* Pout;   // cluster finalize: if set, store P here and stop before the DFT
    float4* rows;   // kFmtRotated: [L / N][N] rotated sums in df
    double fs_hz;
    unsigned int* ticket;
};

// x mod L for 0 <= x < 2^40 (a 64-bit remainder is a subroutine of a hundred
// instructions, and a finalize of few bins waited for three of them).
__host__ __device__ inline unsigned long long reciprocal(int64_t L) { return ~0ull / (unsigned long long)L; }
__device__ __forceinline__ int mod_L(const FinArgs& a, int64_t x) {
    const unsigned int L = (unsigned int)a.L;
    const unsigned int q = (unsigned int)__umul64hi((unsigned long long)x, a.rcp_L);  // the quotient or one less
    const unsigned int r = (unsigned int)x - q * L;
    return (int)(r >= L ? r - L : r);
}

// Decode bin k to its real value S[k] (FP64).  NoAlloc: the caller's
// per-(bin, code) counts.
template <bool NoAlloc, int FMT = -1>
__device__ __forceinline__ double read_bin(const FinArgs& a, int64_t k) {
    const int fmt = FMT < 0 ? a.fmt : FMT;
    if constexpr (NoAlloc) {
        const long long* c = a.counts4 + 4 * k;
        return a.lev[0] * (double)c[0] + a.lev[1] * (double)c[1] + a.lev[2] * (double)c[2] + a.lev[3] * (double)c[3];
    }
    if (fmt == PCAL_2BIT) {
        const unsigned long long v = a.spilled == 2 ? 0ull : a.acc2[k];
        unsigned long long sl = v & PCAL_F21_MASK, sh = (v >> 21) & PCAL_F21_MASK, shl = (v >> 42) & PCAL_F21_MASK;
        if (a.spilled) {
            sl += a.wide2[k];
            sh += a.wide2[a.L + k];
            shl += a.wide2[2 * a.L + k];
        }
        int64_t r = k - a.a0;
        if (r < 0) r += a.L;
        const double cnt = (double)(a.q + (r < a.rem ? 1 : 0));
        // S = sum_c level[c]*count[c] with count[3] = shl, count[2] = sh - shl,
        // count[1] = sl - shl, count[0] = cnt - sl - sh + shl.
        return a.lev0 * cnt + a.c_l * (double)sl + a.c_h * (double)sh + a.c_hl * (double)shl;
    }
    if (fmt == PCAL_I8) return (double)a.acc8[k];
    const float2 v = a.accf[k];
    if (a.n_pf == 0) return (double)v.x + (double)v.y;
    // the pending fold partials of this bin, slot by slot, row group by row
    // group, in double-float (a fixed order: the result does not depend on
    // timing).  Inline: out of line (a call per bin) the C1 step took
    // 1.5 us longer.
    df s{v.x, v.y};
    for (int e = 0; e < a.n_pf; ++e) {
        const int64_t R = a.pf_rg[e], stride = a.pf_cols;
        for (int64_t c = k >= a.pf_ka[e] ? k - a.pf_ka[e] : k - a.pf_ka[e] + a.L; c < a.pf_cols; c += a.L) {
            const float2* col = a.pf[e] + c;
            int64_t rg = 0;
            // eight loads in flight, then their additions in row-group order
            for (; rg + 8 <= R; rg += 8) {
                float2 w[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) w[u] = col[(rg + u) * stride];
#pragma unroll
                for (int u = 0; u < 8; ++u) s = pcal_df::add(s, pcal_df::two_sum(w[u].x, w[u].y));
            }
            for (; rg < R; ++rg) {
                const float2 w = col[rg * stride];
                s = pcal_df::add(s, pcal_df::two_sum(w.x, w.y));
            }
        }
    }
    return (double)s.hi + (double)s.lo;
}

// The rotator table of integer bins: each component as W = round(x * 2^54) in
// two halves, W = hi * 2^27 + lo with 0 <= lo < 2^27: within 2^-55 of the FP64
// sincospi, which itself rounds at 2^-54 above one half and finer below (the
// sums that it enters are rounded to about 48 bits at their end, and P to FP32).
constexpr int kRotBits = 54, kRotHalf = 27;

__device__ __forceinline__ int2 rotator_fixed(double x) {
    const long long W = llrint(x * (double)(1ll << kRotBits));
    return make_int2((int)(W >> kRotHalf), (int)(W & ((1ll << kRotHalf) - 1)));
}

// exp(-j*2*pi*m/L): the plan's table, FP64 or (FIXED) fixed point; NoAlloc
// evaluates it here.
template <bool NoAlloc, bool FIXED = false>
__device__ __forceinline__ double2 rotator(const FinArgs& a, int64_t m) {
    if constexpr (NoAlloc) {
        double sn, cs;
        sincospi(2.0 * (double)m / (double)a.L, &sn, &cs);
        return make_double2(cs, -sn);
    }
    if constexpr (FIXED) {
        const int4 w = a.twi[m];
        constexpr double kHi = 1.0 / (double)(1ll << (kRotBits - kRotHalf)), kLo = 1.0 / (double)(1ll << kRotBits);
        return make_double2(fma((double)w.x, kHi, (double)w.y * kLo), fma((double)w.z, kHi, (double)w.w * kLo));
    }
    return a.tw[m];
}

// Clear bin k for the next integration period.
// FMT: the plan's sample format where the kernel is specialised for one
// (its other formats' code is left out), or -1 for the run-time a.fmt.
template <int FMT = -1>
__device__ __forceinline__ void clear_bin(const FinArgs& a, int64_t k) {
    const int fmt = FMT < 0 ? a.fmt : FMT;
    if (fmt == PCAL_2BIT) {
        if (a.spilled != 2) a.acc2[k] = 0;
        if (a.spilled) {
            a.wide2[k] = 0;
            a.wide2[a.L + k] = 0;
            a.wide2[2 * a.L + k] = 0;
        }
    } else if (fmt == PCAL_I8) {
        a.acc8[k] = 0;
    } else {
        a.accf[k] = make_float2(0.f, 0.f);
    }
}

// Programmatic dependent launch: wait for the preceding kernel's results;
// allow the following kernel to start launching.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void allow_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Completion ticket: a release-acquire increment, so the arriving CTA's
// stores are visible to the CTA that draws the last ticket.
__device__ __forceinline__ unsigned int ticket_acq_rel(unsigned int* t) {
    unsigned int old;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(t) : "memory");
    return old;
}

__device__ __forceinline__ df df_of(double x) {
    const float hi = (float)x;
    return df{hi, (float)(x - (double)hi)};
}

__device__ __forceinline__ df shfl_xor_df(df v, int o) {
    return df{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}

// K block-wide df sums (fixed order: warp butterflies, then the totals of
// the first nw warps in warp order -- the other warps hold zeros); every
// thread receives them.  blockDim.x: a multiple of 32; sm: 32*K float2.
template <int K>
__device__ void block_sums_df(df (&v)[K], float2* sm, int nw) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int j = 0; j < K; ++j)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[j] = pcal_df::add(v[j], shfl_xor_df(v[j], o));
    if (nw == 1) {
        __syncthreads();  // keep the barrier count equal for every nw
        return;
    }
    if (lane == 0 && warp < nw)
#pragma unroll
        for (int j = 0; j < K; ++j) sm[warp * K + j] = make_float2(v[j].hi, v[j].lo);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < K; ++j) {
        df s{0.f, 0.f};
        for (int w = 0; w < nw; ++w) s = pcal_df::add(s, df{sm[w * K + j].x, sm[w * K + j].y});
        v[j] = s;
    }
    __syncthreads();
}

// Exclusive block-wide df prefix sum (fixed order).
__device__ df block_exclusive_scan_df(df v, float2* sm) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    df inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const df u{__shfl_up_sync(0xffffffffu, inc.hi, o), __shfl_up_sync(0xffffffffu, inc.lo, o)};
        if (lane >= o) inc = pcal_df::add(inc, u);
    }
    if (lane == 31) sm[warp] = make_float2(inc.hi, inc.lo);
    __syncthreads();
    df before{0.f, 0.f};
    for (int w = 0; w < warp; ++w) before = pcal_df::add(before, df{sm[w].x, sm[w].y});
    __syncthreads();
    return pcal_df::sub(pcal_df::add(before, inc), v);
}

__device__ __forceinline__ float wrap_pi_f(float x) {
    // into [-pi, pi)
    return x - 6.283185307179586f * floorf((x + 3.141592653589793f) * 0.15915494309189535f);
}

// Tones [i0, i1) of the N-point DFT of P, in FP32, written to global T and,
// when sT is given, to shared memory.  P (hi + lo) and the twiddles are
// staged in shared memory first.  Groups of g threads (a power of two <= 32)
// share a tone and combine their partial sums with a fixed butterfly.
template <bool NoAlloc>
__device__ void dft_tones(const FinArgs& a, int64_t i0, int64_t i1, float2* sP, float2* sTw, float2* sT) {
    const int64_t N = a.N;
    for (int64_t b = threadIdx.x; b < N; b += blockDim.x) {
        const float4 v = __ldcg(&a.P[b]);
        sP[b] = make_float2(v.x + v.y, v.z + v.w);
        if constexpr (NoAlloc) {
            float sn, cs;
            sincospif(2.0f * (float)b / (float)N, &sn, &cs);
            sTw[b] = make_float2(cs, -sn);
        } else {
            sTw[b] = a.twN[b];
        }
    }
    __syncthreads();
    const int64_t ntone = i1 - i0;
    int g = 1;
    while (g < 32 && (int64_t)(g * 2) * ntone <= (int64_t)blockDim.x) g *= 2;
    const int groups = blockDim.x / g;
    const int sub = threadIdx.x % g;
    for (int64_t base = 0; base < ntone; base += groups) {
        const int64_t i = i0 + base + threadIdx.x / g;
        float re = 0.f, im = 0.f;
        if (i < i1) {
            int idx = (int)((i * sub) % N);
            const int step = (int)((i * g) % N);
            const int n = (int)N;
            for (int b = sub; b < n; b += g) {
                const float2 p = sP[b];
                const float2 w = sTw[idx];
                re = fmaf(p.x, w.x, fmaf(-p.y, w.y, re));
                im = fmaf(p.x, w.y, fmaf(p.y, w.x, im));
                idx += step;
                if (idx >= n) idx -= n;
            }
        }
        for (int o = g / 2; o > 0; o >>= 1) {
            re += __shfl_xor_sync(0xffffffffu, re, o);
            im += __shfl_xor_sync(0xffffffffu, im, o);
        }
        if (i < i1 && sub == 0) {
            a.T[i] = make_float2(re, im);
            if (sT) sT[i] = make_float2(re, im);
        }
    }
    __syncthreads();
}

// Shared memory of the products: T[N] float2, psi[N] float, un[N] float2,
// then reduction scratch (96 float2) and the two df results.
struct ProductsSmem {
    float2* T;
    float* psi;
    float2* un;
    float2* red;
    float2* out;  // [0] td (df), [1] sigma (df)
};

__host__ __device__ inline size_t products_bytes(int64_t N) {
    return (size_t)N * 8 + (size_t)((N * 4 + 15) / 16) * 16 + (size_t)N * 8 + 98 * 8;
}

__device__ inline ProductsSmem products_layout(uint8_t* base, int64_t N) {
    ProductsSmem m;
    m.T = reinterpret_cast<float2*>(base);
    m.psi = reinterpret_cast<float*>(base + N * 8);
    m.un = reinterpret_cast<float2*>(base + N * 8 + ((N * 4 + 15) / 16) * 16);
    m.red = m.un + N;
    m.out = m.red + 96;
    return m;
}

// Post-processing (Sec. 2, Sec. 3): the delay from the time-domain pulse --
// the largest |P[b]| and the vertex of the parabola through it and its two
// neighbours; a delay t_d puts the pulse at b = -t_d*fs (mod N) -- into
// extra[0] (seconds, wrapped into one comb period) and extra[1] (the peak
// position in bins).  One warp; P is read from `P` (float2, re/im).
__device__ void peak_delay_warp(const FinArgs& a, const float2* P) {
    const int N = (int)a.N;
    const int lane = threadIdx.x & 31;
    float best = -1.f;
    int bi = 0;
#pragma unroll 1
    for (int b = lane; b < N; b += 32) {
        const float2 z = P[b];
        const float v = z.x * z.x + z.y * z.y;
        if (v > best) {
            best = v;
            bi = b;
        }
    }
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > best || (ov == best && oi < bi)) {
            best = ov;
            bi = oi;
        }
    }
    if (lane == 0) {
        // FP32 throughout (a position to ~1e-5 bin): scalar FP64 square roots
        // and divisions are long dependent chains on GB300's FP64 pipe
        const float2 zm = P[(bi + N - 1) % N], zp = P[(bi + 1) % N];
        const float ym = sqrtf(zm.x * zm.x + zm.y * zm.y), y0 = sqrtf(best);
        const float yp = sqrtf(zp.x * zp.x + zp.y * zp.y);
        const float den = ym - 2.f * y0 + yp;
        const float pos = (float)bi + (den != 0.f ? 0.5f * (ym - yp) / den : 0.f);
        // -pos wrapped into [-N/2, N/2) bins, then seconds
        float q = -pos;
        q -= (float)N * floorf((q + 0.5f * (float)N) / (float)N);
        a.extra[0] = best > 0.f ? (double)(q / (float)a.fs_hz) : __longlong_as_double(0x7ff8000000000000ll);
        a.extra[1] = (double)pos;
    }
}

// Amplitude, phase, unwrapped phase and the weighted LS delay fit over all N
// tones, from T in shared memory; one CTA.  The first nt threads (whole
// warps, about 8 tones each) do the arithmetic; all threads then write the
// FP64 results.
__device__ void tone_products(const FinArgs& a, const ProductsSmem& m) {
    const int64_t N = a.N;
    const int t = threadIdx.x;
    int nt = (int)((N + 7) / 8 + 31) / 32 * 32;
    if (nt > (int)blockDim.x) nt = blockDim.x;
    const int nw = nt / 32;  // warps holding tones
    const int64_t chunk = (N + nt - 1) / nt;
    const int64_t c0 = t < nt ? (t * chunk < N ? t * chunk : N) : N;
    const int64_t c1 = c0 + chunk < N ? c0 + chunk : N;
    // 1. phase per tone, FP32
    for (int64_t i = c0; i < c1; ++i) {
        const float2 z = m.T[i];
        m.psi[i] = wrap_pi_f(atan2f(z.y, z.x) + 1.5707963267948966f);
    }
    __syncthreads();
    // 2. unwrap: u_i = psi_0 + sum_{j=1..i} wrap(psi_j - psi_{j-1}), df sums
    df local{0.f, 0.f};
    for (int64_t i = c0; i < c1; ++i)
        if (i > 0) local = pcal_df::add_f(local, wrap_pi_f(m.psi[i] - m.psi[i - 1]));
    df run = pcal_df::add_f(block_exclusive_scan_df(local, m.red), m.psi[0]);
    for (int64_t i = c0; i < c1; ++i) {
        if (i > 0) run = pcal_df::add_f(run, wrap_pi_f(m.psi[i] - m.psi[i - 1]));
        m.un[i] = make_float2(run.hi, run.lo);
    }
    // 3. weighted least squares of u_i against the tone index x_i = i (the
    //    frequency is f_i = f_comb*i + f_offset), weights w_i = |T_i|^2
    df s3[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    for (int64_t i = c0; i < c1; ++i) {
        const float2 z = m.T[i];
        const float w = z.x * z.x + z.y * z.y;
        s3[0] = pcal_df::add_f(s3[0], w);
        s3[1] = pcal_df::add(s3[1], pcal_df::two_prod(w, (float)i));
        s3[2] = pcal_df::add(s3[2], pcal_df::mul_f(df{m.un[i].x, m.un[i].y}, w));
    }
    block_sums_df<3>(s3, m.red, nw);
    const df W = s3[0];
    df td{__int_as_float(0x7fc00000), 0.f}, sig{__int_as_float(0x7fc00000), 0.f};  // NaN until fitted
    df xbar{0.f, 0.f}, ubar{0.f, 0.f}, slope{0.f, 0.f};
    bool fitted = false;
    if (N >= 2 && W.hi > 0.f) {
        xbar = pcal_df::div(s3[1], W);
        ubar = pcal_df::div(s3[2], W);
        // centred sums; the residual sum follows from Syy - slope*Sxu
        df s2[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
        for (int64_t i = c0; i < c1; ++i) {
            const float2 z = m.T[i];
            const float w = z.x * z.x + z.y * z.y;
            const df dx = pcal_df::sub(df{(float)i, 0.f}, xbar);
            const df du = pcal_df::sub(df{m.un[i].x, m.un[i].y}, ubar);
            const df wdx = pcal_df::mul_f(dx, w);
            s2[0] = pcal_df::add(s2[0], pcal_df::mul(wdx, dx));
            s2[1] = pcal_df::add(s2[1], pcal_df::mul(wdx, du));
            s2[2] = pcal_df::add(s2[2], pcal_df::mul_f(pcal_df::mul(du, du), w));
        }
        block_sums_df<3>(s2, m.red, nw);
        if (s2[0].hi > 0.f) {
            slope = pcal_df::div(s2[1], s2[0]);  // rad per tone index
            fitted = true;
            td = pcal_df::div(slope, a.two_pi_fc);
            if (N > 2) {
                df ssr = pcal_df::sub(s2[2], pcal_df::mul(slope, s2[1]));
                if (ssr.hi < 0.f) ssr = df{0.f, 0.f};
                sig = pcal_df::div(pcal_df::sqrt_df(pcal_df::div(ssr, pcal_df::mul_f(s2[0], (float)(N - 2)))),
                                   a.two_pi_fc);
            }
        }
    }
    if (t == 0) {
        m.out[0] = make_float2(td.hi, td.lo);
        m.out[1] = make_float2(sig.hi, sig.lo);
    }
    if (a.extra)  // bandpass phase with the fitted delay removed
        for (int64_t i = c0; i < c1; ++i) {
            const df r = pcal_df::sub(pcal_df::sub(df{m.un[i].x, m.un[i].y}, ubar),
                                      pcal_df::mul(slope, pcal_df::sub(df{(float)i, 0.f}, xbar)));
            a.extra[2 + i] = fitted ? (double)r.hi + (double)r.lo : __longlong_as_double(0x7ff8000000000000ll);
        }
    __syncthreads();
    // 4. FP64 results, written by all threads
    double* amp = a.res + 2 * N;
    double* ph = a.res + 3 * N;
    double* unw = a.res + 4 * N;
    for (int64_t i = t; i < N; i += blockDim.x) {
        const float2 z = m.T[i];
        a.res[2 * i] = (double)z.x;
        a.res[2 * i + 1] = (double)z.y;
        amp[i] = (double)(sqrtf(z.x * z.x + z.y * z.y) * a.two_over_m);
        ph[i] = (double)m.psi[i];
        unw[i] = (double)m.un[i].x + (double)m.un[i].y;
    }
    if (t == 0) {
        a.res[5 * N] = (double)m.out[0].x + (double)m.out[0].y;
        a.res[5 * N + 1] = (double)m.out[1].x + (double)m.out[1].y;
        a.res[5 * N + 2] = a.M;
    }
}

// Decode + FP64 rotation + fold of whole residues; the last CTA continues.
// Thread t works on residue b = blockIdx.x*bc + t/tpb and bins b + m*N for
// m = t%tpb, t%tpb + tpb, ...; the tpb threads of a residue are contiguous
// (tpb a power of two) and combine with shuffles, then across warps.
template <bool NoAlloc>
__global__ void fin_fold_kernel(FinArgs a) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ bool is_last;
    grid_dependency_wait();  // the bins of the preceding fold
    allow_dependents();
    const int tpb = a.tpb;
    const int bl = threadIdx.x / tpb, sub = threadIdx.x % tpb;
    const int64_t b = (int64_t)blockIdx.x * a.bc + bl;
    const bool active = bl < a.bc && b < a.N;
    const int64_t per = a.L / a.N;
    double re = 0.0, im = 0.0;
    if (active) {
        for (int64_t m = sub; m < per; m += tpb) {
            const int64_t k = b + m * a.N;
            const double S = read_bin<NoAlloc>(a, k);
            const double2 w = rotator<NoAlloc>(a, (a.so * k) % a.L);
            re = fma(S, w.x, re);
            im = fma(S, w.y, im);
        }
    }
    df dre = df_of(re), dim = df_of(im);
    const int width = tpb < 32 ? tpb : 32;
    for (int o = width / 2; o > 0; o >>= 1) {
        dre = pcal_df::add(dre, shfl_xor_df(dre, o));
        dim = pcal_df::add(dim, shfl_xor_df(dim, o));
    }
    if (tpb <= 32) {
        if (active && sub == 0) a.P[b] = make_float4(dre.hi, dre.lo, dim.hi, dim.lo);
    } else {
        float4* wsum = reinterpret_cast<float4*>(smem);
        if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = make_float4(dre.hi, dre.lo, dim.hi, dim.lo);
        __syncthreads();
        if (active && sub == 0) {
            df sr{0.f, 0.f}, si{0.f, 0.f};
            const int w0 = threadIdx.x >> 5;
            for (int w = 0; w < tpb / 32; ++w) {
                const float4 v = wsum[w0 + w];
                sr = pcal_df::add(sr, df{v.x, v.y});
                si = pcal_df::add(si, df{v.z, v.w});
            }
            a.P[b] = make_float4(sr.hi, sr.lo, si.hi, si.lo);
        }
    }
    __threadfence();  // the P stores of this CTA's writers
    __syncthreads();
    if (threadIdx.x == 0) is_last = ticket_acq_rel(&a.ticket[0]) == gridDim.x - 1;
    // clear this CTA's bins for the next period; the fence above did not
    // have to wait for these stores
    if (!NoAlloc && active)
        for (int64_t m = sub; m < per; m += tpb) clear_bin(a, b + m * a.N);
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    if (threadIdx.x == 0) a.ticket[0] = 0;
    if (a.N <= kDftInFoldMaxN) {
        // shared memory: products area, then P and the twiddles for the DFT
        const ProductsSmem m = products_layout(smem, a.N);
        float2* sP = reinterpret_cast<float2*>(smem + products_bytes(a.N));
        dft_tones<NoAlloc>(a, 0, a.N, sP, sP + a.N, m.T);
        tone_products(a, m);
        if (a.extra && threadIdx.x < 32) peak_delay_warp(a, sP);
    }
}

// ---- one-cluster finalize (N <= kClusterMaxN) ------------------------------

constexpr int kClusterMaxN = 256;       // single plans: the cluster path up to here
constexpr int kClusterBigN = 1024;      // batches and kLarge plans: the cluster path up to here (DFT spread over the cluster)
constexpr int kClusterThreads = 256;
// kLarge plans decode up to thousands of bins a CTA: twice the warps hide the
// loads (the DFT and the products keep the order of 256 threads).
constexpr int kLargeThreads = 512;
constexpr size_t kClusterPadSmem = 24 * 1024;
constexpr int64_t kClusterMaxL = 32768;

// Exclusive df prefix sum across the 32 lanes of a warp (fixed order).
__device__ __forceinline__ df warp_exclusive_scan_df(df v) {
    const int lane = threadIdx.x & 31;
    df inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const df u{__shfl_up_sync(0xffffffffu, inc.hi, o), __shfl_up_sync(0xffffffffu, inc.lo, o)};
        if (lane >= o) inc = pcal_df::add(inc, u);
    }
    const df prev{__shfl_up_sync(0xffffffffu, inc.hi, 1), __shfl_up_sync(0xffffffffu, inc.lo, 1)};
    return lane == 0 ? df{0.f, 0.f} : prev;
}

// Threads per block sum of the products: the order of every sum over tones is
// set by the lanes' contiguous chunks.  WARP order (short periods, batches,
// long-period plans): 32 lanes; BLOCK order (LARGE plans): about 8 tones a lane.
__host__ __device__ inline int product_lanes(int N, bool block_order) {
    if (!block_order) return 32;
    const int nt = ((N + 7) / 8 + 31) / 32 * 32;
    return nt < kClusterThreads / 2 ? nt : kClusterThreads / 2;
}

// Per-tone arrays of the products are kept by (place in the chunk, lane), one
// word of padding a row: lanes that walk their chunks together and threads
// that take consecutive tones both spread over the banks.  (Lanes 32 tones
// apart in plain arrays met in one bank: 57 us for 1024 tones.)
struct ToneIndex {
    int chunk, pitch;
    __device__ __forceinline__ int operator()(int i) const {
        const int l = i / chunk;
        return (i - l * chunk) * pitch + l;
    }
};
__host__ __device__ inline int tone_slots(int N) { return N + N / 32 + 144; }  // at least chunk * (lanes + 1)

// Dynamic shared memory of the cluster finalize for N tones.  The partials and
// the DFT's twiddles share their memory with the products that follow.
struct ClusterSmem {
    float2* sP;   // [N] P
    float2* sT;   // [N] tone phasors
    float4* Pr;   // [N] this CTA's partial P (df re, df im)
    float2* sTw;  // [N rounded up to 16] DFT twiddles, swizzled (tw_slot)
};

// ... and of the products in the place of Pr and sTw.
struct ProductsArea {
    float2* un;    // [4][tone_slots]: unwrapped phase (df), then three arrays of terms of sums over tones (df)
    float* psi;    // [tone_slots]
    float* w;      // [tone_slots]
    float2* red;   // [8 warps][3] partial sums
    int slots;
    __device__ __forceinline__ float2* term(int j) const { return un + (j + 1) * slots; }
};

__host__ __device__ inline size_t cluster_smem_bytes(int64_t N) {
    const size_t both = (size_t)N * 16, parts = (size_t)N * 16 + (size_t)(N + 15) / 16 * 16 * 8,
                 prod = (size_t)tone_slots((int)N) * 40 + 8 * 26;
    return both + (parts > prod ? parts : prod) + 16;
}

__device__ inline ClusterSmem cluster_layout(uint8_t* base, int64_t N) {
    ClusterSmem m;
    m.sP = reinterpret_cast<float2*>(base);
    m.sT = m.sP + N;
    uint8_t* q = base + 16 * N;
    m.Pr = reinterpret_cast<float4*>(q);
    m.sTw = reinterpret_cast<float2*>(q + 16 * N);
    return m;
}

__device__ inline ProductsArea products_area(uint8_t* base, int N) {
    ProductsArea m;
    m.slots = tone_slots(N);
    m.un = reinterpret_cast<float2*>(base + 16 * (size_t)N);
    m.psi = reinterpret_cast<float*>(m.un + 4 * m.slots);
    m.w = m.psi + m.slots;
    m.red = reinterpret_cast<float2*>(m.w + m.slots);
    return m;
}

// K df sums over the 32 lanes by a fixed butterfly; every lane gets them.
// The steps are a loop, not unrolled: this code runs once per finalize, so
// its size (instruction fetch) costs more than its loop overhead.
template <int K>
__device__ __forceinline__ void warp_sums_df(df (&v)[K]) {
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int j = 0; j < K; ++j) v[j] = pcal_df::add(v[j], shfl_xor_df(v[j], o));
}

// The products of tone_products, by one warp with no block barrier: lane l
// takes the contiguous tones [l*c, l*c + c), c = ceil(N/32).  Loops over a
// lane's tones are not unrolled, for the reason given at warp_sums_df.
__device__ __noinline__ void tone_products_warp(const FinArgs& a, const float2* __restrict__ sT,
                                                float* __restrict__ psi, float* __restrict__ wt,
                                                float2* __restrict__ un, float2* __restrict__ out) {
    double* const extra = a.extra;
    const int N = (int)a.N;
    const int lane = threadIdx.x & 31;
    const int c = (N + 31) / 32;
    const int i0 = lane * c < N ? lane * c : N;
    const int i1 = i0 + c < N ? i0 + c : N;
    // 1. phase and weight per tone, FP32
#pragma unroll 1
    for (int i = i0; i < i1; ++i) {
        const float2 z = sT[i];
        psi[i] = wrap_pi_f(atan2f(z.y, z.x) + 1.5707963267948966f);
        wt[i] = z.x * z.x + z.y * z.y;
    }
    __syncwarp();
    // 2. unwrap: u_i = psi_0 + sum_{j=1..i} wrap(psi_j - psi_{j-1}), df sums
    const int j0 = i0 > 1 ? i0 : 1;
    df local{0.f, 0.f};
#pragma unroll 1
    for (int i = j0; i < i1; ++i) local = pcal_df::add_f(local, wrap_pi_f(psi[i] - psi[i - 1]));
    df run = pcal_df::add_f(warp_exclusive_scan_df(local), psi[0]);
#pragma unroll 1
    for (int i = i0; i < i1; ++i) {
        if (i > 0) run = pcal_df::add_f(run, wrap_pi_f(psi[i] - psi[i - 1]));
        un[i] = make_float2(run.hi, run.lo);
    }
    // 3. weighted least squares of u_i against the tone index x_i = i (the
    //    frequency is f_i = f_comb*i + f_offset), weights w_i = |T_i|^2
    df s3[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
#pragma unroll 1
    for (int i = i0; i < i1; ++i) {
        const float w = wt[i];
        s3[0] = pcal_df::add_f(s3[0], w);
        s3[1] = pcal_df::add(s3[1], pcal_df::two_prod(w, (float)i));
        s3[2] = pcal_df::add(s3[2], pcal_df::mul_f(df{un[i].x, un[i].y}, w));
    }
    warp_sums_df<3>(s3);
    const df W = s3[0];
    df td{__int_as_float(0x7fc00000), 0.f}, sig{__int_as_float(0x7fc00000), 0.f};  // NaN until fitted
    df xbar{0.f, 0.f}, ubar{0.f, 0.f}, slope{0.f, 0.f};
    bool fitted = false;
    if (N >= 2 && W.hi > 0.f) {
        xbar = pcal_df::div(s3[1], W);
        ubar = pcal_df::div(s3[2], W);
        // centred sums; the residual sum follows from Syy - slope*Sxu
        df s2[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
#pragma unroll 1
        for (int i = i0; i < i1; ++i) {
            const float w = wt[i];
            const df dx = pcal_df::sub(df{(float)i, 0.f}, xbar);
            const df du = pcal_df::sub(df{un[i].x, un[i].y}, ubar);
            const df wdx = pcal_df::mul_f(dx, w);
            s2[0] = pcal_df::add(s2[0], pcal_df::mul(wdx, dx));
            s2[1] = pcal_df::add(s2[1], pcal_df::mul(wdx, du));
            s2[2] = pcal_df::add(s2[2], pcal_df::mul_f(pcal_df::mul(du, du), w));
        }
        warp_sums_df<3>(s2);
        if (s2[0].hi > 0.f) {
            slope = pcal_df::div(s2[1], s2[0]);  // rad per tone index
            fitted = true;
            td = pcal_df::div(slope, a.two_pi_fc);
            if (N > 2) {
                df ssr = pcal_df::sub(s2[2], pcal_df::mul(slope, s2[1]));
                if (ssr.hi < 0.f) ssr = df{0.f, 0.f};
                sig = pcal_df::div(pcal_df::sqrt_df(pcal_df::div(ssr, pcal_df::mul_f(s2[0], (float)(N - 2)))),
                                   a.two_pi_fc);
            }
        }
    }
    if (lane == 0) {
        out[0] = make_float2(td.hi, td.lo);
        out[1] = make_float2(sig.hi, sig.lo);
    }
    if (extra) {
        // bandpass phase with the fitted delay removed: u_i - ubar - slope*(i - xbar)
#pragma unroll 1
        for (int i = i0; i < i1; ++i) {
            const df r = pcal_df::sub(pcal_df::sub(df{un[i].x, un[i].y}, ubar),
                                      pcal_df::mul(slope, pcal_df::sub(df{(float)i, 0.f}, xbar)));
            extra[2 + i] = fitted ? (double)r.hi + (double)r.lo : __longlong_as_double(0x7ff8000000000000ll);
        }
    }
}

// The FP64 result vector from the products in shared memory, by the block.
__device__ void write_results_block(const FinArgs& a, const float2* sT, const ProductsArea& m) {
    const int N = (int)a.N;
    double* amp = a.res + 2 * N;
    double* ph = a.res + 3 * N;
    double* unw = a.res + 4 * N;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const float2 z = sT[i];
        a.res[2 * i] = (double)z.x;
        a.res[2 * i + 1] = (double)z.y;
        amp[i] = (double)(sqrtf(m.w[i]) * a.two_over_m);
        ph[i] = (double)m.psi[i];
        unw[i] = (double)m.un[i].x + (double)m.un[i].y;
    }
    if (threadIdx.x == 0) {
        a.res[5 * N] = (double)m.red[0].x + (double)m.red[0].y;
        a.res[5 * N + 1] = (double)m.red[1].x + (double)m.red[1].y;
        a.res[5 * N + 2] = a.M;
    }
}

// Amplitude, phase, unwrapped phase, the weighted LS delay fit over all N
// tones, the post-processing and the FP64 result vector, by one block of
// kClusterThreads from T and P in shared memory.  Everything that belongs to
// one tone is done by all threads; only the sums over tones run lane by lane in
// their fixed order (add_f and add chains of ceil(N/lanes) steps and a
// butterfly), the three sums of a fit side by side in different warps.  For
// more than kWarpProductsN tones: with fewer its barriers and its size cost
// more than the one-warp form takes (64 tones: 6.3 against 4 us).
constexpr int kWarpProductsN = 128;

template <bool BLOCK_ORDER>
__device__ __noinline__ void tone_products_all(const FinArgs& a, uint8_t* base) {
    const int N = (int)a.N, t = threadIdx.x, T = (int)blockDim.x;
    const float2* sP = reinterpret_cast<const float2*>(base);
    const float2* sT = sP + N;
    const ProductsArea m = products_area(base, N);
    const int nt = product_lanes(N, BLOCK_ORDER), nw = BLOCK_ORDER ? nt / 32 : 1;
    const int chunk = (N + nt - 1) / nt;
    const ToneIndex ix{chunk, nt + 1};
    const int grp = t / nt, lt = t - grp * nt, G = T / nt;  // groups of nt threads
    const int lane = t & 31, gw = lt >> 5;
    const int n_mine = lt * chunk < N ? (N - lt * chunk < chunk ? N - lt * chunk : chunk) : 0;  // tones of this lane
    // 1. phase and weight per tone, FP32
#pragma unroll 1
    for (int i = t; i < N; i += T) {
        const float2 z = sT[i];
        const int q = ix(i);
        m.psi[q] = wrap_pi_f(atan2f(z.y, z.x) + 1.5707963267948966f);
        m.w[q] = z.x * z.x + z.y * z.y;
    }
    __syncthreads();
    float* step = reinterpret_cast<float*>(m.term(0));  // wrapped phase steps
#pragma unroll 1
    for (int i = t; i < N; i += T) step[ix(i)] = i > 0 ? wrap_pi_f(m.psi[ix(i)] - m.psi[ix(i - 1)]) : 0.f;
    __syncthreads();
    // 2. unwrap: u_i = psi_0 + sum_{j=1..i} wrap(psi_j - psi_{j-1}), df sums
    df local{0.f, 0.f};
    const int skip = lt == 0 ? 1 : 0;  // tone 0 has no step
    if (grp == 0) {
#pragma unroll 4
        for (int j = skip; j < n_mine; ++j) local = pcal_df::add_f(local, step[j * ix.pitch + lt]);
    } else if (t >= T - 32) {
        if (a.extra) peak_delay_warp(a, sP);
    }
    df before;
    if constexpr (BLOCK_ORDER) {
        df inc = local;
#pragma unroll 1
        for (int o = 1; o < 32; o <<= 1) {
            const df u{__shfl_up_sync(0xffffffffu, inc.hi, o), __shfl_up_sync(0xffffffffu, inc.lo, o)};
            if (lane >= o) inc = pcal_df::add(inc, u);
        }
        if (grp == 0 && lane == 31) m.red[gw] = make_float2(inc.hi, inc.lo);
        __syncthreads();
        before = df{0.f, 0.f};
        for (int w = 0; w < gw; ++w) before = pcal_df::add(before, df{m.red[w].x, m.red[w].y});
        before = pcal_df::sub(pcal_df::add(before, inc), local);
    } else {
        before = warp_exclusive_scan_df(local);
    }
    if (grp == 0) {
        df run = pcal_df::add_f(before, m.psi[0]);
#pragma unroll 4
        for (int j = 0; j < n_mine; ++j) {
            if (j >= skip) run = pcal_df::add_f(run, step[j * ix.pitch + lt]);
            m.un[j * ix.pitch + lt] = make_float2(run.hi, run.lo);
        }
    }
    __syncthreads();
    // Sum `j` of three by group j % G: red[warp * 3 + j], then everybody adds the warps in order.
    auto three_sums = [&](auto&& chain, df (&out)[3]) {
#pragma unroll 1
        for (int j = grp; j < 3; j += G) {
            df v = chain(j);
#pragma unroll 1
            for (int o = 16; o > 0; o >>= 1) v = pcal_df::add(v, shfl_xor_df(v, o));
            if (lane == 0) m.red[gw * 3 + j] = make_float2(v.hi, v.lo);
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            if (nw == 1) {
                out[j] = df{m.red[j].x, m.red[j].y};
            } else {
                df v{0.f, 0.f};
                for (int w = 0; w < nw; ++w) v = pcal_df::add(v, df{m.red[w * 3 + j].x, m.red[w * 3 + j].y});
                out[j] = v;
            }
        }
        __syncthreads();
    };
    // 3. weighted least squares of u_i against the tone index x_i = i (the
    //    frequency is f_i = f_comb*i + f_offset), weights w_i = |T_i|^2
#pragma unroll 1
    for (int i = t; i < N; i += T) {
        const int q = ix(i);
        const df v = pcal_df::mul_f(df{m.un[q].x, m.un[q].y}, m.w[q]);
        m.term(2)[q] = make_float2(v.hi, v.lo);
    }
    __syncthreads();
    df s3[3], s2[3];
    three_sums(
        [&](int j) {
            df v{0.f, 0.f};
            if (j == 0) {
#pragma unroll 4
                for (int k = 0; k < n_mine; ++k) v = pcal_df::add_f(v, m.w[k * ix.pitch + lt]);
            } else if (j == 1) {
#pragma unroll 4
                for (int k = 0; k < n_mine; ++k)
                    v = pcal_df::add(v, pcal_df::two_prod(m.w[k * ix.pitch + lt], (float)(lt * chunk + k)));
            } else {
#pragma unroll 4
                for (int k = 0; k < n_mine; ++k) {
                    const float2 u = m.term(2)[k * ix.pitch + lt];
                    v = pcal_df::add(v, df{u.x, u.y});
                }
            }
            return v;
        },
        s3);
    const df W = s3[0];
    df td{__int_as_float(0x7fc00000), 0.f}, sig{__int_as_float(0x7fc00000), 0.f};  // NaN until fitted
    df xbar{0.f, 0.f}, ubar{0.f, 0.f}, slope{0.f, 0.f};
    bool fitted = false;
    if (N >= 2 && W.hi > 0.f) {
        xbar = pcal_df::div(s3[1], W);
        ubar = pcal_df::div(s3[2], W);
        // centred sums; the residual sum follows from Syy - slope*Sxu
#pragma unroll 1
        for (int i = t; i < N; i += T) {
            const int q = ix(i);
            const float w = m.w[q];
            const df dx = pcal_df::sub(df{(float)i, 0.f}, xbar);
            const df du = pcal_df::sub(df{m.un[q].x, m.un[q].y}, ubar);
            const df wdx = pcal_df::mul_f(dx, w);
            const df xx = pcal_df::mul(wdx, dx), xu = pcal_df::mul(wdx, du),
                     uu = pcal_df::mul_f(pcal_df::mul(du, du), w);
            m.term(0)[q] = make_float2(xx.hi, xx.lo);
            m.term(1)[q] = make_float2(xu.hi, xu.lo);
            m.term(2)[q] = make_float2(uu.hi, uu.lo);
        }
        __syncthreads();
        three_sums(
            [&](int j) {
                df v{0.f, 0.f};
#pragma unroll 4
                for (int k = 0; k < n_mine; ++k) {
                    const float2 u = m.term(j)[k * ix.pitch + lt];
                    v = pcal_df::add(v, df{u.x, u.y});
                }
                return v;
            },
            s2);
        if (s2[0].hi > 0.f) {
            slope = pcal_df::div(s2[1], s2[0]);  // rad per tone index
            fitted = true;
            td = pcal_df::div(slope, a.two_pi_fc);
            if (N > 2) {
                df ssr = pcal_df::sub(s2[2], pcal_df::mul(slope, s2[1]));
                if (ssr.hi < 0.f) ssr = df{0.f, 0.f};
                sig = pcal_df::div(pcal_df::sqrt_df(pcal_df::div(ssr, pcal_df::mul_f(s2[0], (float)(N - 2)))),
                                   a.two_pi_fc);
            }
        }
    }
    // 4. FP64 results and the bandpass phase with the fitted delay removed,
    //    u_i - ubar - slope*(i - xbar)
#pragma unroll 1
    for (int i = t; i < N; i += T) {
        const int q = ix(i);
        const float2 z = sT[i], u = m.un[q];
        a.res[2 * i] = (double)z.x;
        a.res[2 * i + 1] = (double)z.y;
        a.res[2 * N + i] = (double)(sqrtf(m.w[q]) * a.two_over_m);
        a.res[3 * N + i] = (double)m.psi[q];
        a.res[4 * N + i] = (double)u.x + (double)u.y;
        if (a.extra) {
            const df r = pcal_df::sub(pcal_df::sub(df{u.x, u.y}, ubar),
                                      pcal_df::mul(slope, pcal_df::sub(df{(float)i, 0.f}, xbar)));
            a.extra[2 + i] = fitted ? (double)r.hi + (double)r.lo : __longlong_as_double(0x7ff8000000000000ll);
        }
    }
    if (t == 0) {
        a.res[5 * N] = (double)td.hi + (double)td.lo;
        a.res[5 * N + 1] = (double)sig.hi + (double)sig.lo;
        a.res[5 * N + 2] = a.M;
    }
}

// Decode, rotate (FP64, Eq. 3) and fold residue b over m = m, m + step, ...
// below m_end (bins k = b + m*N), clearing each bin; returns the FP64 sum.
// FIXED: the rotators are the fixed-point table (a test of it in the loop cost
// float32 plans of 128 tones and L 25,600 2 us of 25).
template <int FMT, bool FIXED>
__device__ __forceinline__ double2 fold_residue(const FinArgs& a, int b, int m, int step, int m_end) {
    double re = 0.0, im = 0.0;
    if (m >= m_end) return make_double2(0.0, 0.0);
    const int L = (int)a.L, N = (int)a.N;
    int k = b + m * N;
    int idx = mod_L(a, a.so * k);  // rotator index (f_offset/g * k) mod L
    const int kstep = step * N;
    const int istep = mod_L(a, a.so * kstep);
    if (FMT == PCAL_2BIT && !FIXED && !a.spilled) {
        // S = lev0*cnt + c_l*sum(l) + c_h*sum(h) + c_hl*sum(h AND l),
        // cnt = q or q + 1; the fields are below 2^21
        const double s_q = a.lev0 * (double)a.q, s_q1 = a.lev0 * (double)(a.q + 1);
        const int a0 = (int)a.a0, rem = (int)a.rem;
#pragma unroll 2
        for (; m < m_end; m += step) {
            const unsigned long long v = a.acc2[k];
            const double2 w = a.tw[idx];
            a.acc2[k] = 0;
            int rr = k - a0;
            if (rr < 0) rr += L;
            const double S = fma(a.c_hl, (double)(int)((v >> 42) & PCAL_F21_MASK),
                                 fma(a.c_h, (double)(int)((v >> 21) & PCAL_F21_MASK),
                                     fma(a.c_l, (double)(int)(v & PCAL_F21_MASK), rr < rem ? s_q1 : s_q)));
            re = fma(S, w.x, re);
            im = fma(S, w.y, im);
            k += kstep;
            idx += istep;
            if (idx >= L) idx -= L;
        }
    } else {
#pragma unroll 1
        for (; m < m_end; m += step) {
            const double S = read_bin<false, FMT>(a, k);
            const double2 w = rotator<false, FIXED>(a, idx);
            re = fma(S, w.x, re);
            im = fma(S, w.y, im);
            clear_bin<FMT>(a, k);
            k += kstep;
            idx += istep;
            if (idx >= L) idx -= L;
        }
    }
    return make_double2(re, im);
}

// Sum of s * W over bins, exact in 64 bits: high and low halves of W apart.
struct IntSum {
    long long rh = 0, rl = 0, ih = 0, il = 0;
    __device__ __forceinline__ void add(int s, const int4& w) {
        rh += (long long)s * w.x;
        rl += (long long)s * w.y;
        ih += (long long)s * w.z;
        il += (long long)s * w.w;
    }
};

// (hi * 2^27 + lo) * 2^-54 as a double-float; |hi|, |lo| < 2^62.
__device__ __forceinline__ df int_df(long long hi, long long lo) {
    hi += lo >> kRotHalf;
    lo &= (1ll << kRotHalf) - 1;
    // hi in pieces of 25, 24 and 14 bits: exact floats
    const float h = (float)(int)(hi >> 38) * 2048.f;
    const float m = (float)(int)((hi >> 14) & 0xFFFFFF) * (1.f / 8192.f);
    const float l = (float)(int)(hi & 0x3FFF) * (1.f / 134217728.f);
    df r = pcal_df::quick_two_sum(h, m);
    r = pcal_df::add_f(r, l);
    return pcal_df::add_f(r, (float)(int)lo * (1.f / 18014398509481984.f));
}

__device__ __forceinline__ void add_scaled(df& re, df& im, const IntSum& s, df k) {
    re = pcal_df::add(re, pcal_df::mul(int_df(s.rh, s.rl), k));
    im = pcal_df::add(im, pcal_df::mul(int_df(s.ih, s.il), k));
}

// Residue b over m = m, m + step, ... below m_end of integer bins, in integers:
// the decode and rotation of Eq. 3 with no FP64 instruction (GB300 issues two
// FP64 operations per SM and clock; about 14 of them a 2-bit bin, conversions
// included, bounded every finalize).  With the sums sl, sh and shl of a bin's l,
// h and (h AND l) bits over cnt samples, A = sl + sh - cnt and B = sh - sl, the
// levels v0..v3 give
//   S = A ((v1 + v2)/2 - v0) + B (v2 - v1)/2 + cnt (v1 + v2)/2
//       + shl (v3 - v2 - v1 + v0),
// so the usual antisymmetric levels need two exact sums of (integer x fixed-point
// rotator) per component, int8 bins one.  a.exact: every factor is below 2^26, so
// 512 terms stay below 2^62.  The bins are cleared.  Measured: 64 live channels
// (L up to 102,400) batch finalize 145 -> 108 us, L 12,800 int8 plan finalize
// 14.5 -> 13.1 us; wide plans (LARGE below) 35 us in two kernels over all SMs
// after the fold -> one cluster beside the next fold (1024 tones: 91 -> 79 us a
// step).
// SRC: 0 packed 2-bit words (or int8 sums), 1 packed and spilled, 2 the wide
// arrays alone.  U: bins whose loads are in flight together (from clamped
// addresses past the end: a load behind a branch waited for the one before it,
// 3.5 us for eight).
template <int FMT, int SRC, int U>
__device__ __forceinline__ float4 residue_int(const FinArgs& a, int b, int m, int step, int m_end) {
    df re{0.f, 0.f}, im{0.f, 0.f};
    if (m >= m_end) return make_float4(0.f, 0.f, 0.f, 0.f);
    const int L = (int)a.L, N = (int)a.N;
    // bin k = b + m N turns by so k mod L: by so N m here, which the lanes of a
    // warp mostly share (their loads of the table are one), and by so b at the end
    int k = b + m * N;
    const int kstep = step * N;
    const int4* __restrict__ twi = a.twi;
    int idx = mod_L(a, a.so * ((int64_t)m * N));
    const int istep = mod_L(a, a.so * kstep);
    const int q = (int)a.q, a0 = (int)a.a0, rem = (int)a.rem;
    const bool use_c = a.k_c.hi != 0.f, use_h = a.k_h.hi != 0.f;
    while (m < m_end) {
        const int end = (m_end - m) / step >= 512 ? m + 512 * step : m_end;  // (512: a multiple of U)
        IntSum A, B, Cn, H;
#pragma unroll 1
        while (m < end) {
            int4 w[U];
            unsigned long long v[U], wl[U], wh[U], wb[U];
            int at[U];
            bool in[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                in[u] = m + u * step < end;
                at[u] = in[u] ? k + u * kstep : k;
                w[u] = __ldg(twi + idx);
                if (FMT == PCAL_I8) v[u] = (unsigned long long)a.acc8[at[u]];
                if (FMT == PCAL_2BIT && SRC != 2) v[u] = a.acc2[at[u]];
                if (FMT == PCAL_2BIT && SRC != 0) {
                    wl[u] = a.wide2[at[u]];
                    wh[u] = a.wide2[L + at[u]];
                    wb[u] = use_h ? a.wide2[2 * L + at[u]] : 0ull;
                }
                idx += istep;
                if (idx >= L) idx -= L;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (in[u])
                    clear_bin<FMT>(a, at[u]);
                else
                    w[u] = make_int4(0, 0, 0, 0);
                if (FMT == PCAL_2BIT) {
                    int x = 0, y = 0, z = 0;
                    if (SRC != 2) {
                        x = (int)(v[u] & PCAL_F21_MASK);
                        y = (int)((v[u] >> 21) & PCAL_F21_MASK);
                        z = (int)((v[u] >> 42) & PCAL_F21_MASK);
                    }
                    if (SRC != 0) {
                        x += (int)wl[u];
                        y += (int)wh[u];
                        z += (int)wb[u];
                    }
                    int rr = at[u] - a0;
                    if (rr < 0) rr += L;
                    const int cnt = q + (rr < rem ? 1 : 0);
                    A.add(x + y - cnt, w[u]);
                    B.add(y - x, w[u]);
                    if (use_c) Cn.add(cnt, w[u]);
                    if (use_h) H.add(z, w[u]);
                } else {
                    A.add((int)v[u], w[u]);
                }
            }
            k += U * kstep;
            m += U * step;
        }
        if (FMT == PCAL_2BIT) {
            add_scaled(re, im, A, a.k_a);
            add_scaled(re, im, B, a.k_b);
            if (use_c) add_scaled(re, im, Cn, a.k_c);
            if (use_h) add_scaled(re, im, H, a.k_h);
        } else {
            re = pcal_df::add(re, int_df(A.rh, A.rl));
            im = pcal_df::add(im, int_df(A.ih, A.il));
        }
    }
    const int4 w = __ldg(twi + mod_L(a, a.so * b));
    const df wr = int_df(w.x, w.y), wi = int_df(w.z, w.w);
    const df r = pcal_df::sub(pcal_df::mul(re, wr), pcal_df::mul(im, wi));
    const df i = pcal_df::add(pcal_df::mul(re, wi), pcal_df::mul(im, wr));
    return make_float4(r.hi, r.lo, i.hi, i.lo);
}

// Whether a period's integer bins fit residue_int: samples per bin below 2^26
// (2-bit; no level beyond the floats of a double-float) or 2^19 (int8, up to
// 128 each).
__host__ __device__ inline int exact_bins(int fmt, int64_t q, double k_a, double k_b, double k_c, double k_h) {
    if (fmt == PCAL_I8) return q + 1 < (1ll << 19);
    if (fmt != PCAL_2BIT || q + 1 >= (1ll << 26)) return 0;
    const double k[4] = {k_a, k_b, k_c, k_h};
    double most = 0.0;
    for (double v : k) {
        const double w = v < 0.0 ? -v : v;
        if (w > most) most = w;
    }
    return most < 1e25 && most > 1e-20;
}

__host__ __device__ inline df split_df(double x) {
    const float hi = (float)x;
    return df{hi, (float)(x - (double)hi)};
}

// Residue b over m = m, m + step, ... below m_end as double-float (re hi, re
// lo, im hi, im lo).  kFmtRotated: the bins are rotated complex sums already
// (the rows of a long-period plan), added in row order.
template <int FMT, int KIND>
__device__ __forceinline__ float4 residue_df(const FinArgs& a, int b, int m, int step, int m_end) {
    if constexpr (FMT == kFmtRotated) {
        df re{0.f, 0.f}, im{0.f, 0.f};
        const int N = (int)a.N;
#pragma unroll 4
        for (; m < m_end; m += step) {
            const float4 v = a.rows[(int64_t)m * N + b];
            a.rows[(int64_t)m * N + b] = make_float4(0.f, 0.f, 0.f, 0.f);
            re = pcal_df::add(re, df{v.x, v.y});
            im = pcal_df::add(im, df{v.z, v.w});
        }
        return make_float4(re.hi, re.lo, im.hi, im.lo);
    } else {
        if constexpr (FMT < 0) {  // (two CTAs share an SM: fewer registers)
            if (a.exact)
                return a.fmt == PCAL_2BIT ? residue_int<PCAL_2BIT, 2, 4>(a, b, m, step, m_end)
                                          : residue_int<PCAL_I8, 0, 8>(a, b, m, step, m_end);
        } else if constexpr (FMT != PCAL_F32 && KIND == kLarge) {
            if (a.exact)
                return a.spilled ? residue_int<FMT, 1, 2>(a, b, m, step, m_end)
                                 : residue_int<FMT, 0, 4>(a, b, m, step, m_end);
        }
        constexpr bool kFixed = FMT < 0 || (FMT != PCAL_F32 && KIND == kLarge);
        const double2 z = fold_residue<FMT, kFixed>(a, b, m, step, m_end);
        const df dre = df_of(z.x), dim = df_of(z.y);
        return make_float4(dre.hi, dre.lo, dim.hi, dim.lo);
    }
}

// Slot of DFT twiddle ix in shared memory: the low four bits of its index are
// mixed with the next eight, so that the strides i of tone i (powers of two
// among them) spread over the banks.
__device__ __forceinline__ int tw_slot(int ix) { return ix ^ ((ix >> 4) & 15) ^ ((ix >> 8) & 15); }

// Threads per tone of a DFT that `share` tones split a block for (a power of
// two, at most 32): they set the order of a tone's FP32 sum (thread gs takes
// b = gs, gs + g, ...; then a fixed butterfly).
__host__ __device__ inline int dft_threads(int share) {
    int g = 1;
    while (g < 32 && g * 2 * share <= kClusterThreads) g *= 2;
    return g;
}

// Tones [i0, i1) of the N-point DFT of sP in FP32, g threads each, written to
// dst[i] (shared memory of this CTA or, through the cluster, of another).
// PAIRS: i in [i0, i1) of 1 .. N/2, each with the tone N - i, whose twiddles
// are the conjugates: one lookup serves both.  (Tone 0 goes apart: with it in
// the list, 256 tones took 129 threads, and the fifth warp shared a scheduler
// with the first for the whole sum.)  Four steps at a time, their twiddle
// indices from the first one's.
template <bool PAIRS>
__device__ __forceinline__ void dft_tones_smem(const float2* sP, const float2* sTw, int N, int i0, int i1, float2* dst,
                                               int g) {
    const int t = threadIdx.x;
    const int n = i1 - i0;
    const int groups = blockDim.x / g;
    const int gs = t % g;
#pragma unroll 1
    for (int base = 0; base < n; base += groups) {
        const int i = i0 + base + t / g;
        float sre = 0.f, sim = 0.f, cre = 0.f, cim = 0.f;
        auto add = [&](float2 p, float2 w) {
            sre = fmaf(p.x, w.x, fmaf(-p.y, w.y, sre));
            sim = fmaf(p.x, w.y, fmaf(p.y, w.x, sim));
            if (PAIRS) {
                cre = fmaf(p.x, w.x, fmaf(p.y, w.y, cre));
                cim = fmaf(p.x, -w.y, fmaf(p.y, w.x, cim));
            }
        };
        if (i < i1) {
            const unsigned int un = (unsigned int)N;
            unsigned int ix = (unsigned int)(i * gs) % un;  // i, g below 2^11
            const unsigned int step = (unsigned int)(i * g) % un;
            int bb = gs;
            if (bb + 3 * g < N) {
                unsigned int off[4];  // k steps on
                off[0] = 0;
#pragma unroll
                for (int k = 1; k < 4; ++k) {
                    off[k] = off[k - 1] + step;
                    off[k] = min(off[k], off[k] - un);
                }
                unsigned int four = off[3] + step;
                four = min(four, four - un);
#pragma unroll 1
                for (; bb + 3 * g < N; bb += 4 * g) {
                    float2 p[4], w[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        unsigned int x = ix + off[k];
                        x = min(x, x - un);
                        p[k] = sP[bb + k * g];
                        w[k] = sTw[tw_slot((int)x)];
                    }
#pragma unroll
                    for (int k = 0; k < 4; ++k) add(p[k], w[k]);
                    ix += four;
                    ix = min(ix, ix - un);
                }
            }
#pragma unroll 1
            for (; bb < N; bb += g) {
                add(sP[bb], sTw[tw_slot((int)ix)]);
                ix += step;
                ix = min(ix, ix - un);
            }
        }
#pragma unroll 1
        for (int o = g / 2; o > 0; o >>= 1) {
            sre += __shfl_xor_sync(0xffffffffu, sre, o);
            sim += __shfl_xor_sync(0xffffffffu, sim, o);
            if (PAIRS) {
                cre += __shfl_xor_sync(0xffffffffu, cre, o);
                cim += __shfl_xor_sync(0xffffffffu, cim, o);
            }
        }
        if (i < i1 && gs == 0) {
            dst[i] = make_float2(sre, sim);
            if (PAIRS && 2 * i != N) dst[N - i] = make_float2(cre, cim);
        }
    }
}

// Tone 0 the same way (every twiddle is the first one), by the g threads from
// t0 on (within one warp).
__device__ __forceinline__ void dft_zero(const float2* sP, float2 w, int N, float2* dst, int g, int t0) {
    const int gs = (int)threadIdx.x - t0;
    if (((int)threadIdx.x >> 5) != (t0 >> 5)) return;  // (whole warps)
    float sre = 0.f, sim = 0.f;
    if (gs >= 0 && gs < g) {
#pragma unroll 4
        for (int bb = gs; bb < N; bb += g) {
            const float2 p = sP[bb];
            sre = fmaf(p.x, w.x, fmaf(-p.y, w.y, sre));
            sim = fmaf(p.x, w.y, fmaf(p.y, w.x, sim));
        }
    }
#pragma unroll 1
    for (int o = g / 2; o > 0; o >>= 1) {
        sre += __shfl_xor_sync(0xffffffffu, sre, o);
        sim += __shfl_xor_sync(0xffffffffu, sim, o);
    }
    if (gs == 0) dst[0] = make_float2(sre, sim);
}

// All tones of a DFT of at most kFewN: the same sums in a loop that is short
// as code (16 steps at most), from twiddles in their plain order.
__device__ __forceinline__ void dft_few(const float2* sP, const float2* sTw, int N, float2* dst, int g) {
    const int t = threadIdx.x, gs = t % g, i = t / g;
    float sre = 0.f, sim = 0.f;
    if (i < N) {
        const unsigned int un = (unsigned int)N;
        unsigned int ix = (unsigned int)(i * gs) % un;
        const unsigned int step = (unsigned int)(i * g) % un;
#pragma unroll 4
        for (int bb = gs; bb < N; bb += g) {
            const float2 p = sP[bb];
            const float2 w = sTw[ix];
            sre = fmaf(p.x, w.x, fmaf(-p.y, w.y, sre));
            sim = fmaf(p.x, w.y, fmaf(p.y, w.x, sim));
            ix += step;
            ix = min(ix, ix - un);
        }
    }
#pragma unroll 1
    for (int o = g / 2; o > 0; o >>= 1) {
        sre += __shfl_xor_sync(0xffffffffu, sre, o);
        sim += __shfl_xor_sync(0xffffffffu, sim, o);
    }
    if (i < N && gs == 0) dst[i] = make_float2(sre, sim);
}

// The whole finalize in one cluster of C CTAs.  Thread t of every CTA takes
// residue b = t % N and every (blockDim/N)-th index m of its CTA's slice
// [per*r/C, per*(r+1)/C) of m = 0..per-1 (per = L/N), i.e. bins k = b + m*N:
// consecutive threads read consecutive bins.  Per bin: decode and rotation
// in FP64 (Eq. 3), then the bin is cleared for the next period.  The lanes of
// a residue are added in df in shared memory (fixed order).  CTA 0 then adds
// the C partials of every residue (rank order) read through distributed
// shared memory, spread over all its threads, and runs the DFT and the
// products.
// Runs in every CTA of the cluster; returns true in the CTA that wrote the
// results (rank 0), after it wrote them.
// KIND: what the kernel has to hold.  A finalize runs once per step and its
// instructions come from L2, slowly beside a streaming fold, so each kernel
// leaves out what its plans never use (an integer decode and the wide paths
// in the one kernel: C2 decode 4.7 -> 11.8 us beside the next fold).
//   kFew, kMany  plans of at most kFewN, kClusterMaxN tones and short periods:
//                FP64 decode (1 to 8 bins a thread), one-warp products up to
//                kWarpProductsN tones
//   kLarge       the other integer plans: integer decode; their DFT and products
//                keep the order of fin_dft_kernel and fin_fold_kernel: tones in
//                groups of kDftTonesPerCta, products in BLOCK order
//   kAny         batches (integer decode) and long-period plans
template <int FMT, int KIND>
__device__ __forceinline__ bool cluster_finalize(const FinArgs& a) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    // per (lane, residue) df partials: re hi, re lo, im hi, im lo
    __shared__ float4 part[KIND == kLarge ? kLargeThreads : kClusterThreads];
    extern __shared__ __align__(16) uint8_t dsm[];
    const int C = (int)cluster.num_blocks(), r = (int)cluster.block_rank();
    const int N = (int)a.N;
    const ClusterSmem sm = cluster_layout(dsm, N);
    float4* Pr = sm.Pr;
    float2 *sP = sm.sP, *sTw = sm.sTw, *sT = sm.sT;
    const int t = threadIdx.x;
    // N > kClusterThreads: one lane per residue, the residues in turns
    constexpr bool LARGE = KIND == kLarge;
    const bool big = KIND >= kLarge && N > kClusterThreads;
    const int lanes = big ? 1 : (int)blockDim.x / N;
    if (r == 0 || N > kClusterMaxN)
        for (int i = t; i < N; i += blockDim.x) sTw[KIND == kFew ? i : tw_slot(i)] = a.twN[i];
    // L <= PCAL_MAX_L: bin and rotator indices fit 32 bits (so*k does not)
    const int L = (int)a.L;
    const int per = L / N;
    const int m1 = per * (r + 1) / C;
    if (!big) {
        // thread t: residue t % N, every lanes-th m of this CTA's slice
        const int b = t % N, ml = t / N;
        if (ml < lanes) {
            part[t] = residue_df<FMT, KIND>(a, b, per * r / C + ml, lanes, m1);
        }
        __syncthreads();
        if (t < N) {
            df sr{0.f, 0.f}, si{0.f, 0.f};
#pragma unroll 1
            for (int l = 0; l < lanes; ++l) {
                const float4 v = part[l * N + t];
                sr = pcal_df::add(sr, df{v.x, v.y});
                si = pcal_df::add(si, df{v.z, v.w});
            }
            Pr[t] = make_float4(sr.hi, sr.lo, si.hi, si.lo);
        }
    } else {
        // one thread per residue, the residues in turns
#pragma unroll 1
        for (int b = t; b < N; b += blockDim.x) Pr[b] = residue_df<FMT, KIND>(a, b, per * r / C, 1, m1);
    }
    cluster.sync();  // every CTA's partial P is complete
    if (big) {
        // every CTA adds its share of the residues (the C partials in rank order,
        // loads issued in fours) and hands the sums to all of them
        for (int i = N * r / C + t; i < N * (r + 1) / C; i += blockDim.x) {
            df sr{0.f, 0.f}, si{0.f, 0.f};
#pragma unroll 1
            for (int q0 = 0; q0 < C; q0 += 4) {
                float4 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    v[u] = q0 + u < C ? *cluster.map_shared_rank(&Pr[i], q0 + u) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    sr = pcal_df::add(sr, df{v[u].x, v[u].y});
                    si = pcal_df::add(si, df{v[u].z, v[u].w});
                }
            }
            const float2 p = make_float2(sr.hi + sr.lo, si.hi + si.lo);
            for (int q = 0; q < C; ++q) cluster.map_shared_rank(sP, q)[i] = p;
        }
    } else if (r == 0) {
        // residue i: the C partials in rank order, loads issued in fours;
        // G threads share a residue when N is small
        const int G = lanes < C ? lanes : C;
        const int g = t / N;
        if (g < G) {
            const int i = t % N;
            df sr{0.f, 0.f}, si{0.f, 0.f};
#pragma unroll 1
            for (int q0 = g; q0 < C; q0 += 4 * G) {
                float4 v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int q = q0 + u * G;
                    v[u] = q < C ? *cluster.map_shared_rank(&Pr[i], q) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    sr = pcal_df::add(sr, df{v[u].x, v[u].y});
                    si = pcal_df::add(si, df{v[u].z, v[u].w});
                }
            }
            part[t] = make_float4(sr.hi, sr.lo, si.hi, si.lo);
        }
        __syncthreads();
        if (t < N) {
            df sr{0.f, 0.f}, si{0.f, 0.f};
#pragma unroll 1
            for (int gg = 0; gg < G; ++gg) {
                const float4 v = part[gg * N + t];
                sr = pcal_df::add(sr, df{v.x, v.y});
                si = pcal_df::add(si, df{v.z, v.w});
            }
            sP[t] = make_float2(sr.hi + sr.lo, si.hi + si.lo);
        }
    }
    cluster.sync();  // P is complete (in CTA 0; big: in all); the other CTAs' Pr is no longer read
    if (KIND == kAny && a.Pout) {
        // the DFT runs elsewhere (the batched tensor-core DFT)
        if (r == 0)
            for (int i = t; i < N; i += blockDim.x) a.Pout[i] = sP[i];
        return false;
    }
    if (!big) {
        if (r != 0) return false;
        if (KIND == kFew)
            dft_few(sP, sTw, N, sT, dft_threads(N));
        else {
            const int g = dft_threads(N);
            dft_tones_smem<true>(sP, sTw, N, 1, N / 2 + 1, sT, g);
            dft_zero(sP, sTw[0], N, sT, g, kClusterThreads / 2);
        }
    } else {
        // every CTA: its share of the tones, into CTA 0's sT
        float2* dst = cluster.map_shared_rank(sT, 0);
        // threads per tone: of LARGE groups of kDftTonesPerCta tones, of equal
        // shares of the tones, or (long-period plans) of one CTA with all of them;
        // where the last or the larger shares have another count, tone by tone
        const int least = LARGE ? (N % kDftTonesPerCta ? N % kDftTonesPerCta : kDftTonesPerCta)
                                : (FMT == kFmtRotated ? N : N / C);
        const int most = LARGE ? kDftTonesPerCta : (FMT == kFmtRotated ? N : (N + C - 1) / C);
        if (dft_threads(least) == dft_threads(most)) {
            const int H = N / 2, g = dft_threads(most);
            dft_tones_smem<true>(sP, sTw, N, 1 + H * r / C, 1 + H * (r + 1) / C, dst, g);
            if (r == C - 1) dft_zero(sP, sTw[0], N, dst, g, kClusterThreads / 2);
        } else if constexpr (LARGE) {
            for (int i0 = r * kDftTonesPerCta; i0 < N; i0 += C * kDftTonesPerCta) {
                const int n = N - i0 < kDftTonesPerCta ? N - i0 : kDftTonesPerCta;
                dft_tones_smem<false>(sP, sTw, N, i0, i0 + n, dst, dft_threads(n));
            }
        } else {
            const int i0 = N * r / C, i1 = N * (r + 1) / C;
            dft_tones_smem<false>(sP, sTw, N, i0, i1, dst, dft_threads(i1 - i0));
        }
        cluster.sync();  // CTA 0 holds every tone
        if (r != 0) return false;
    }
    __syncthreads();
    if (LARGE || (KIND != kFew && N > kWarpProductsN)) {
        tone_products_all<LARGE>(a, dsm);
    } else {
        const ProductsArea pm = products_area(dsm, N);
        if (t < 32) tone_products_warp(a, sT, pm.psi, pm.w, pm.un, pm.red);
        else if (t < 64 && a.extra) peak_delay_warp(a, sP);
        __syncthreads();
        write_results_block(a, sT, pm);
    }
    return true;
}

// One instantiation per sample format: the finalize runs once per step and its
// instructions come from L2 (slow beside a streaming fold), so each plan's
// kernel holds only its own format's decode.
template <int FMT, int KIND>
__global__ void __launch_bounds__(KIND == kLarge ? kLargeThreads : kClusterThreads, 1) fin_cluster_kernel(FinArgs a) {
    // The next fold may launch at once: it adds into the other set of bins
    // and waits for this kernel before its first atomic.
    allow_dependents();
    grid_dependency_wait();  // the bins of the preceding fold
    cluster_finalize<FMT, KIND>(a);
}

// Finalize arguments of one batched channel from its device state.
__device__ inline FinArgs batch_fin_args(const BatchChan& bc) {
    const int64_t n_tot = bc.n_abs - bc.period_start;
    FinArgs a{};
    a.fmt = bc.fmt;
    a.spilled = 2;  // 2-bit sums live in the wide arrays
    a.L = bc.L;
    a.rcp_L = bc.rcp_L;
    a.N = bc.N;
    a.so = bc.so;
    a.q = n_tot / bc.L;
    a.rem = n_tot % bc.L;
    a.a0 = bc.period_start % bc.L;
    a.lev0 = bc.lev0;
    a.c_l = bc.c_l;
    a.c_h = bc.c_h;
    a.c_hl = bc.c_hl;
    a.M = (double)n_tot;
    a.two_over_m = n_tot > 0 ? (float)(2.0 / (double)n_tot) : 0.0f;
    a.two_pi_fc.hi = (float)bc.two_pi_fc;
    a.two_pi_fc.lo = (float)(bc.two_pi_fc - (double)a.two_pi_fc.hi);
    a.exact = exact_bins(bc.fmt, a.q, bc.k_a, bc.k_b, bc.k_c, bc.c_hl);
    a.k_a = split_df(bc.k_a);
    a.k_b = split_df(bc.k_b);
    a.k_c = split_df(bc.k_c);
    a.k_h = split_df(bc.c_hl);
    a.wide2 = bc.wide2;
    a.acc8 = bc.acc8;
    a.twi = bc.twi;
    a.twN = bc.twN;
    a.res = bc.res;
    a.extra = bc.res + 5 * bc.N + 3;
    a.fs_hz = bc.fs;
    return a;
}

// Batch finalize: cluster c finalizes channel c of the batch from the
// channel's device state, then starts the channel's next period.  split:
// stop after P (stored in the channel's P slot) for the batched DFT; the
// products kernel finishes the channel.  A programmatic dependent of the
// fold: it waits for the fold's bins and indices before reading any state.
__global__ void __launch_bounds__(kClusterThreads, 2) batch_fin_kernel(BatchChan* ch, const int* list, int split) {
    namespace cg = cooperative_groups;
    allow_dependents();
    grid_dependency_wait();
    const int i = (int)(blockIdx.x / cg::this_cluster().num_blocks());
    const int c = list ? list[i] : i;
    BatchChan& bc = ch[c];
    // The arguments live in shared memory: a per-thread copy passed by
    // reference to the out-of-line products went to each thread's stack, and
    // those stores (376 B x 256 threads x 16 CTAs per channel, ~88 MB for 64
    // channels) left dirty L2 lines that the next fold had to write back
    // (+50 us per C3 step).
    __shared__ FinArgs a;
    if (threadIdx.x == 0) {
        a = batch_fin_args(bc);
        if (split) a.Pout = bc.Pslot;
    }
    __syncthreads();
    // every CTA has read the state above before the first cluster barrier
    // inside, and rank 0 returns after the last one
    if (cluster_finalize<-1, kAny>(a) && threadIdx.x == 0) bc.period_start = bc.n_abs;
}

// After the batched DFT: block c runs channel c's products and
// post-processing from its tone and P slots and starts its next period.
__global__ void __launch_bounds__(kClusterThreads, 1) batch_products_kernel(BatchChan* ch) {
    BatchChan& bc = ch[blockIdx.x];
    __shared__ FinArgs a;  // in shared memory, not on every thread's stack
    if (threadIdx.x == 0) a = batch_fin_args(bc);
    __syncthreads();
    extern __shared__ __align__(16) uint8_t dsm[];
    const ClusterSmem sm = cluster_layout(dsm, bc.N);
    const int t = threadIdx.x;
    for (int i = t; i < bc.N; i += blockDim.x) {
        sm.sT[i] = bc.Tslot[i];
        sm.sP[i] = bc.Pslot[i];
    }
    __syncthreads();
    if (bc.N > kWarpProductsN) {
        tone_products_all<false>(a, dsm);
    } else {
        const ProductsArea pm = products_area(dsm, bc.N);
        if (t < 32) tone_products_warp(a, sm.sT, pm.psi, pm.w, pm.un, pm.red);
        else if (t < 64 && a.extra) peak_delay_warp(a, sm.sP);
        __syncthreads();
        write_results_block(a, sm.sT, pm);
    }
    __syncthreads();
    if (t == 0) bc.period_start = bc.n_abs;
}

// Spread DFT for large N; the last CTA runs the products.
template <bool NoAlloc>
__global__ void fin_dft_kernel(FinArgs a) {
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ bool is_last;
    grid_dependency_wait();  // P of the fold kernel
    allow_dependents();
    const int64_t i0 = (int64_t)blockIdx.x * kDftTonesPerCta;
    const int64_t i1 = i0 + kDftTonesPerCta < a.N ? i0 + kDftTonesPerCta : a.N;
    float2* sP = reinterpret_cast<float2*>(smem);
    dft_tones<NoAlloc>(a, i0, i1, sP, sP + a.N, nullptr);
    __threadfence();  // the T stores of this CTA
    __syncthreads();
    if (threadIdx.x == 0) is_last = ticket_acq_rel(&a.ticket[1]) == gridDim.x - 1;
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    if (threadIdx.x == 0) a.ticket[1] = 0;
    const ProductsSmem m = products_layout(smem, a.N);
    for (int64_t i = threadIdx.x; i < a.N; i += blockDim.x) m.T[i] = __ldcg(&a.T[i]);
    __syncthreads();
    tone_products(a, m);
    if (a.extra) {
        // P again, into the shared memory the products no longer need
        __syncthreads();
        float2* sP = reinterpret_cast<float2*>(smem);
        for (int64_t b = threadIdx.x; b < a.N; b += blockDim.x) {
            const float4 v = __ldcg(&a.P[b]);
            sP[b] = make_float2(v.x + v.y, v.z + v.w);
        }
        __syncthreads();
        if (threadIdx.x < 32) peak_delay_warp(a, sP);
    }
}

// exactly one of tw (float32 bins) and twi (integer bins) is given
__global__ void init_twiddles_kernel(double2* tw, int4* twi, int64_t L, float2* twN, int64_t N, int64_t sc) {
    for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < L; m += (int64_t)gridDim.x * blockDim.x) {
        double s, c;
        sincospi(2.0 * (double)m / (double)L, &s, &c);
        if (twi) {
            const int2 re = rotator_fixed(c), im = rotator_fixed(-s);
            twi[m] = make_int4(re.x, re.y, im.x, im.y);
        } else {
            tw[m] = make_double2(c, -s);
        }
        if (m % sc == 0 && m / sc < N) twN[m / sc] = make_float2((float)c, (float)-s);
    }
}

// Launch as a programmatic dependent of the preceding kernel in the stream.
template <typename... Args>
cudaError_t launch_pdl(void (*k)(Args...), int grid, int block, size_t smem, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, args...);
}

}  // namespace

cudaError_t launch_rotators(bool fixed, void* tw, int64_t L, float2* twN, int64_t N, int64_t step_comb,
                            cudaStream_t s) {
    int64_t g = (L + 255) / 256;
    if (g > 1024) g = 1024;
    init_twiddles_kernel<<<(unsigned)g, 256, 0, s>>>(fixed ? nullptr : static_cast<double2*>(tw),
                                                     fixed ? static_cast<int4*>(tw) : nullptr, L, twN, N, step_comb);
    return cudaGetLastError();
}

// Plans that the short-period clusters do not take, up to kClusterBigN tones:
// one cluster too, integer bins with the integer decode; float32 bins (an FP64
// rotation, two operations per SM and clock) of more than 256 tones, which
// would need a second kernel for their DFT, at shorter periods, and, where no
// partials wait to be added (f32_cluster), up to kLargeF32L.  The others spread
// over the SMs.  float32 finalizes with a short call, spread / cluster: 256 tones and
// fewer L 50,000 17.6 / 19.4 us, L 64,000 17.7 / 20.4, L 100,000 19.5 / 24.9, L 128,000 (128 tones)
// 20.4 / 27.5; N 512 L 51,200 30 / 26, L 102,400 32 / 29; N 1024 L 102,400 50 / 39; N 700 L 140,000
// 39 / 41.  Behind bulk folds (one a finalize, 256 MB): N 300 L 30,000 52 / 44, N 700 L 35,000 64 / 66,
// N 1000 L 100,000 76 / 81.
constexpr int64_t kLargeF32L = 131072;
static bool large_plan(const pcal_geometry& g) {
    return g.N <= kClusterBigN && (g.N > kClusterMaxN || g.L > kClusterMaxL) &&
           (g.format != PCAL_F32 || (g.N > kClusterMaxN && g.L <= kLargeF32L));
}
static bool f32_cluster(const pcal_plan* p) { return p->g.L <= kClusterMaxL || p->n_pending == 0; }

namespace {

// Launch the finalize kernels for filled-in arguments (everything but the
// work split, which is chosen here).
template <bool NoAlloc>
cudaError_t launch_finalize_args(FinArgs a, int num_sms, cudaStream_t s, int* launches) {
    const int64_t N = a.N;
    int G = (int)(N < num_sms ? N : num_sms);
    a.bc = (int)((N + G - 1) / G);
    G = (int)((N + a.bc - 1) / a.bc);
    // tpb = the largest power of two with bc*tpb <= 256; the block is a
    // multiple of 32 threads (the shuffles and the DFT need whole warps)
    a.tpb = 1;
    while (a.bc * a.tpb * 2 <= 256) a.tpb *= 2;
    const int threads = (a.bc * a.tpb + 31) / 32 * 32;
    size_t smem = (size_t)threads * 16;
    if (N <= kDftInFoldMaxN) {
        const size_t need = products_bytes(N) + (size_t)N * 16;  // products + P + twiddles
        if (need > smem) smem = need;
    }
    cudaError_t e = cudaSuccess;
    static size_t fold_smem_set = 0;
    if (smem > 48 * 1024 && smem > fold_smem_set) {
        e = cudaFuncSetAttribute(fin_fold_kernel<NoAlloc>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        fold_smem_set = smem;
    }
    e = launch_pdl(fin_fold_kernel<NoAlloc>, G, threads, smem, s, a);
    *launches += 1;
    if (e != cudaSuccess || N <= kDftInFoldMaxN) return e;
    const int threads2 = 256;
    const size_t smem2 = (size_t)N * 16 > products_bytes(N) ? (size_t)N * 16 : products_bytes(N);
    static size_t dft_smem_set = 0;
    if (smem2 > 48 * 1024 && smem2 > dft_smem_set) {
        e = cudaFuncSetAttribute(fin_dft_kernel<NoAlloc>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem2);
        if (e != cudaSuccess) return e;
        dft_smem_set = smem2;
    }
    e = launch_pdl(fin_dft_kernel<NoAlloc>, (int)((N + kDftTonesPerCta - 1) / kDftTonesPerCta), threads2, smem2, s, a);
    *launches += 1;
    return e;
}

// Cluster size for fin_cluster_kernel on the current device: 16 CTAs where
// the device can co-schedule them (a non-portable size), else the portable
// 8; 0 when no cluster fits.  Evaluated once per device.
int cluster_size_for_device() {
    static std::mutex mu;
    static int cached[64];
    static bool known[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> lock(mu);
    if (known[dev]) return cached[dev];
    int best = 0;
    for (auto k : {fin_cluster_kernel<PCAL_2BIT, kFew>, fin_cluster_kernel<PCAL_I8, kFew>,
                   fin_cluster_kernel<PCAL_F32, kFew>, fin_cluster_kernel<PCAL_2BIT, kMany>,
                   fin_cluster_kernel<PCAL_I8, kMany>, fin_cluster_kernel<PCAL_F32, kMany>,
                   fin_cluster_kernel<PCAL_2BIT, kLarge>, fin_cluster_kernel<PCAL_I8, kLarge>,
                   fin_cluster_kernel<PCAL_F32, kLarge>}) {
        if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
            (void)cudaGetLastError();
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(cluster_smem_bytes(kClusterBigN) + kClusterPadSmem)) != cudaSuccess)
            (void)cudaGetLastError();
    }
    for (int c : {16, 8}) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(c);
        cfg.blockDim = dim3(kClusterThreads);
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = c;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, fin_cluster_kernel<PCAL_2BIT, kFew>, &cfg) == cudaSuccess && n > 0) {
            best = c;
            break;
        }
        (void)cudaGetLastError();
    }
    cached[dev] = best;
    known[dev] = true;
    return best;
}

}  // namespace

cudaError_t launch_init_twiddles(pcal_plan* p, cudaStream_t s) {
    p->stats.kernel_launches += 1;
    // (fixed point for the plans whose finalize is the cluster's integer decode)
    p->fixed_tw = p->g.format != PCAL_F32 && large_plan(p->g) && cluster_size_for_device() > 0;
    return launch_rotators(p->fixed_tw, p->d_tw, p->g.L, p->d_twN, p->g.N, p->g.step_comb, s);
}

namespace {

// One cluster of C CTAs as a programmatic dependent of the preceding kernel.
// The CTAs ask for kClusterPadSmem more shared memory than they use, so that
// none of them fits on an SM beside a CTA of the fold that overlaps it (about
// 205 KB each): sharing an SM with a fold CTA slowed the finalize 2-3x.  The
// fold leaves kFinalizeReserveSms SMs for it.
cudaError_t launch_cluster_finalize(const FinArgs& a, int C, int kind, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(kind == kLarge ? kLargeThreads : kClusterThreads);
    cfg.dynamicSmemBytes = cluster_smem_bytes(a.N) + kClusterPadSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = C;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    switch ((kind << 2) | a.fmt) {
        case (kLarge << 2) | PCAL_2BIT: return cudaLaunchKernelEx(&cfg, fin_cluster_kernel<PCAL_2BIT, kLarge>, a);
        case (kLarge << 2) | PCAL_I8: return cudaLaunchKernelEx(&cfg, fin_cluster_kernel<PCAL_I8, kLarge>, a);
        case (kLarge << 2) | PCAL_F32: return cudaLaunchKernelEx(&cfg, fin_cluster_kernel<PCAL_F32, kLarge>, a);
        case (kMany << 2) | PCAL_2BIT: return cudaLaunchKernelEx(&cfg, fin_cluster_kernel<PCAL_2BIT, kMany>, a);
        case (kMany << 2) | PCAL_I8: return cudaLaunchKernelEx(&cfg, fin_cluster_kernel<PCAL_I8, kMany>, a);
        case (kMany << 2) | PCAL_F32: return cudaLaunchKernelEx(&cfg, fin_cluster_kernel<PCAL_F32, kMany>, a);
        case (kFew << 2) | PCAL_2BIT: return cudaLaunchKernelEx(&cfg, fin_cluster_kernel<PCAL_2BIT, kFew>, a);
        case (kFew << 2) | PCAL_I8: return cudaLaunchKernelEx(&cfg, fin_cluster_kernel<PCAL_I8, kFew>, a);
        case (kFew << 2) | PCAL_F32: return cudaLaunchKernelEx(&cfg, fin_cluster_kernel<PCAL_F32, kFew>, a);
        default: return cudaErrorInvalidValue;
    }
}

// Finalize of a long-period plan: its rows of partial sums are added (and
// cleared) by one cluster, then the DFT, the products and the post-processing
// of the folded path.  (One CTA that added 9,728 rows of 16 bins took 115 us.)
__global__ void __launch_bounds__(kClusterThreads, 1) rot_finalize_kernel(FinArgs a, const unsigned int* err) {
    grid_dependency_wait();  // the rows of the preceding fold
    if (cluster_finalize<kFmtRotated, kAny>(a) && threadIdx.x == 0)
        *reinterpret_cast<unsigned int*>(a.res + 6 * a.N + 5) = *err;
}

}  // namespace

cudaError_t launch_rot_finalize(float4* rows, int n_rows, int N, double fs, double fc, int64_t M,
                                const float2* twN, double* res, const unsigned int* err, cudaStream_t s) {
    FinArgs a{};
    a.N = N;
    a.L = (int64_t)N * n_rows;
    a.rows = rows;
    a.fs_hz = fs;
    a.M = (double)M;
    a.two_over_m = M > 0 ? (float)(2.0 / (double)M) : 0.0f;
    const double tpf = 6.283185307179586476925 * fc;
    a.two_pi_fc.hi = (float)tpf;
    a.two_pi_fc.lo = (float)(tpf - (double)a.two_pi_fc.hi);
    a.twN = twN;
    a.res = res;
    a.extra = res + 5 * (int64_t)N + 3;
    // (one CTA where no larger cluster fits: slower, and all that a part of a GPU may have)
    const int fits = cluster_size_for_device(), C = fits > 0 ? fits : 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(kClusterThreads);
    cfg.dynamicSmemBytes = cluster_smem_bytes(N);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, rot_finalize_kernel, a, err);
}

cudaError_t prepare_rot_finalize() {
    const int C = cluster_size_for_device();
    cudaError_t e = cudaFuncSetAttribute(rot_finalize_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)cluster_smem_bytes(kClusterBigN));
    if (e == cudaSuccess && C > 8)
        e = cudaFuncSetAttribute(rot_finalize_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

cudaError_t prepare_batch_finalize() {
    const int C = cluster_size_for_device();
    if (C == 0) return cudaErrorNotSupported;
    cudaError_t e = cudaFuncSetAttribute(batch_fin_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)cluster_smem_bytes(kClusterBigN));
    if (e == cudaSuccess && C > 8)
        e = cudaFuncSetAttribute(batch_fin_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(batch_products_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)cluster_smem_bytes(kClusterBigN));
    return e;
}

cudaError_t launch_batch_products(BatchChan* d_ch, int n_ch, int max_n, cudaStream_t s) {
    if (max_n > kClusterBigN) return cudaErrorInvalidValue;
    batch_products_kernel<<<n_ch, kClusterThreads, cluster_smem_bytes(max_n), s>>>(d_ch);
    return cudaGetLastError();
}

// prepare_batch_finalize() must have succeeded on this device (it makes the
// CUDA calls that a stream capture does not allow).  max_n: the largest N of
// the batch's channels.
cudaError_t launch_batch_finalize(BatchChan* d_ch, int n_ch, int max_n, const int* d_list, cudaStream_t s, int split) {
    // 8-CTA clusters: with one cluster per channel the launch is several waves
    // of CTAs, and fewer, longer clusters finish sooner (64 channels of up to
    // L 25600: 16 CTAs 53 us, 8 CTAs 43 us, 4 CTAs 57 us; same phasors)
    int C = cluster_size_for_device();
    if (C > 8) C = 8;
    if (C == 0) return cudaErrorNotSupported;
    if (max_n > kClusterBigN) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(n_ch * C);
    cfg.blockDim = dim3(kClusterThreads);
    cfg.dynamicSmemBytes = cluster_smem_bytes(max_n);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, batch_fin_kernel, d_ch, d_list, split);
}

namespace {


void set_common(FinArgs& a, const pcal_geometry& g, int64_t n_tot) {
    a.fs_hz = (double)g.fs;
    a.L = g.L;
    a.rcp_L = reciprocal(g.L);
    a.N = g.N;
    a.so = g.step_offset;
    a.M = (double)n_tot;
    a.two_over_m = n_tot > 0 ? (float)(2.0 / (double)n_tot) : 0.0f;
    const double tpf = 6.283185307179586476925 * (double)g.f_comb;
    a.two_pi_fc.hi = (float)tpf;
    a.two_pi_fc.lo = (float)(tpf - (double)a.two_pi_fc.hi);
}

}  // namespace

cudaError_t launch_finalize(pcal_plan* p, cudaStream_t s) {
    const pcal_geometry& g = p->g;
    const bool f32 = g.format == PCAL_F32;
    const bool small = g.N <= kClusterMaxN && g.L <= kClusterMaxL;
    const bool large = large_plan(g) && (f32 ? f32_cluster(p) : p->fixed_tw);
    // float32 bins of a long period, several folds' partials: added by all SMs
    // first (a cluster's 16 CTAs add them bin by bin).  Three folds of 16 MB and a
    // finalize, with / without: L 6,400 28.6 / 28.6 us, L 10,000 29 / 33, L 25,600 38 / 45, L 32,000
    // 28 / 39.  One fold's stay for the decode, which then starts beside the next
    // fold: 64 MB L 6,400 16.9 / 15.7, L 16,000 19.2 / 17.7, 256 MB L 25,600 42.9 / 40.3.
    if (f32 && (small || large) && g.L >= kLongPeriodL && p->n_pending > 1) {
        const cudaError_t e = flush_partials(p, s);
        if (e != cudaSuccess) return e;
    }
    FinArgs a{};
    const int64_t n_tot = p->n_abs - p->period_start;
    set_common(a, g, n_tot);
    a.fmt = g.format;
    a.spilled = p->spilled ? 1 : 0;
    a.q = n_tot / g.L;
    a.rem = n_tot % g.L;
    a.a0 = p->period_start % g.L;
    const double* lv = p->levels;
    a.lev0 = lv[0];
    a.c_l = lv[1] - lv[0];
    a.c_h = lv[2] - lv[0];
    a.c_hl = lv[3] - lv[2] - lv[1] + lv[0];
    const double k_c = 0.5 * (lv[1] + lv[2]), k_a = k_c - lv[0], k_b = 0.5 * (lv[2] - lv[1]);
    a.exact = exact_bins(g.format, a.q, k_a, k_b, k_c, a.c_hl);
    a.k_a = split_df(k_a);
    a.k_b = split_df(k_b);
    a.k_c = split_df(k_c);
    a.k_h = split_df(a.c_hl);
    a.acc2 = cur_acc2(p);
    a.wide2 = cur_wide2(p);
    a.acc8 = cur_acc8(p);
    a.accf = cur_accf(p);
    if (g.format == PCAL_F32) {
        for (int e = 0; e < p->n_pending; ++e) {
            a.pf[e] = p->pending[e].base;
            a.pf_rg[e] = p->pending[e].row_groups;
            a.pf_ka[e] = p->pending[e].k_a;
        }
        a.n_pf = p->n_pending;
        a.pf_cols = g.row_samples / g.samples_per_byte_x4;
    }
    if (p->fixed_tw)
        a.twi = static_cast<const int4*>(p->d_tw);
    else
        a.tw = static_cast<const double2*>(p->d_tw);
    a.twN = p->d_twN;
    a.P = reinterpret_cast<float4*>(p->d_P);
    a.T = reinterpret_cast<float2*>(p->d_T);
    a.res = p->d_res;
    a.extra = p->d_res + 5 * g.N + 3;
    a.ticket = p->d_ticket;
    cudaError_t e = cudaErrorUnknown;
    bool done = false;
    if (small || large) {
        const int C = cluster_size_for_device();
        if (C > 0) {
            p->stats.kernel_launches += 1;
            e = launch_cluster_finalize(a, C, !small ? kLarge : g.N <= kFewN ? kFew : kMany, s);
            done = true;
        }
    }
    if (!done) {
        if (p->fixed_tw) return cudaErrorNotSupported;  // (its clusters fit when it was created)
        int launches = 0;
        e = launch_finalize_args<false>(a, p->num_sms, s, &launches);
        p->stats.kernel_launches += launches;
    }
    if (e == cudaSuccess) p->n_pending = 0;  // the finalize added them (and clears the bins)
    return e;
}

// ---- finalize without any allocation -------------------------------------------
//
// Some callers cannot allocate GPU memory at all: code running inside a
// pre-sized memory pool or arena, a process whose device memory budget is
// fixed at start-up, or a stream that is being captured into a CUDA graph,
// where a cudaMalloc is not allowed.  For them pcal_tones_from_counts_noalloc
// runs the finalize kernels with their scratch (the folded bins P, the tone
// phasors T and the completion tickets) in the file-scope array below, which
// every GPU that loads this library holds until the process exits; the
// rotator and DFT twiddles are evaluated on the fly instead of read from a
// plan's tables.  Everything else comes from the caller.

namespace {

constexpr int kNoAllocMaxN = 1024;

struct NoAllocScratch {
    float4 P[kNoAllocMaxN];
    float2 T[kNoAllocMaxN];
    unsigned int ticket[4];
};

// ~24.6 KB per device.
static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(NoAllocScratch)];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
NoAllocScratch* g_noalloc_ptr[kMaxDevices];  // device address of the array, per device
int g_noalloc_sms[kMaxDevices];

// Device address of the scratch array on the current device.  In host code
// the array's name is only a host-side stand-in, so the address must come
// from cudaGetSymbolAddress, once per device, with that device current.
cudaError_t noalloc_scratch(NoAllocScratch** out, int* num_sms) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_ptr[dev]) {
        void* ptr = nullptr;
        e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        e = cudaDeviceGetAttribute(&g_noalloc_sms[dev], cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        g_noalloc_ptr[dev] = static_cast<NoAllocScratch*>(ptr);
    }
    *out = g_noalloc_ptr[dev];
    *num_sms = g_noalloc_sms[dev];
    return cudaSuccess;
}

}  // namespace

extern "C" int pcal_tones_from_counts_noalloc(double fs, double f_comb, double f_offset, int N,
                                              const int64_t* d_counts, int64_t n_samples, const double levels[4],
                                              double* d_results, void* stream) {
    pcal_geometry g;
    int rc = pcal_plan_geometry(fs, f_comb, f_offset, N, PCAL_2BIT, &g);
    if (rc != PCAL_OK) return rc;
    if (g.N > kNoAllocMaxN) return PCAL_ETOOLARGE;
    if (!d_counts || !d_results || !levels || n_samples < 0) return PCAL_EINVAL;
    for (int i = 0; i < 4; ++i)
        if (!(levels[i] == levels[i]) || levels[i] > 1e300 || levels[i] < -1e300) return PCAL_EINVAL;
    NoAllocScratch* sc = nullptr;
    int num_sms = 0;
    cudaError_t e = noalloc_scratch(&sc, &num_sms);
    if (e != cudaSuccess) return e == cudaErrorMemoryAllocation ? PCAL_ENOMEM : PCAL_ECUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // the completion tickets must start at zero (the array keeps whatever the
    // previous call, possibly an interrupted one, left there)
    e = cudaMemsetAsync(sc->ticket, 0, sizeof(sc->ticket), s);
    if (e != cudaSuccess) return PCAL_ECUDA;
    FinArgs a{};
    set_common(a, g, n_samples);
    a.fmt = PCAL_2BIT;
    a.counts4 = reinterpret_cast<const long long*>(d_counts);
    for (int i = 0; i < 4; ++i) a.lev[i] = levels[i];
    a.tw = nullptr;   // rotator evaluated per bin (no plan table)
    a.twN = nullptr;  // DFT twiddles evaluated per CTA
    a.P = sc->P;
    a.T = sc->T;
    a.ticket = sc->ticket;
    a.res = d_results;
    int launches = 0;
    e = launch_finalize_args<true>(a, num_sms, s, &launches);
    return e == cudaSuccess ? PCAL_OK : PCAL_ECUDA;
}
