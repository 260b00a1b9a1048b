// Ragged-edge and short fold kernels of libpcal and the small bookkeeping kernels.
//
// The ragged kernels fold any run of samples at any alignment straight into
// the plan's bins (Eq. 2 with the period L of Eq. 4).  They handle the head
// before the first 16-byte boundary, the tail after the last whole bulk row,
// and runs with next to nothing to add up before their atomics or stores
// (api.cu: few_samples); the short folds below take what else is too short for
// the bulk kernel.  2-bit and int8 bins are exact integers, so atomic order does
// not matter; float32 bins are summed by one thread per bin in sample order, so
// they are deterministic.
//
// Every kernel that touches the bins here is launched as a programmatic
// dependent of the kernel before it: it lets its own successor start
// launching at once, then waits for its predecessor (whose adds, or the
// finalize's clearing, come first) before it touches the bins.  The stream's
// kernels therefore still complete in launch order, while their launches
// overlap.
#include "df64.cuh"
#include "fold_direct.cuh"
#include "internal.cuh"
#include "ptx.cuh"

namespace {

__device__ __forceinline__ void chain_in() {
    pcal_ptx::allow_dependents();
    pcal_ptx::grid_dependency_wait();
}

__global__ void ragged_2bit_kernel(const uint8_t* __restrict__ bytes, int64_t n_bytes, int64_t k0, int64_t L,
                                   unsigned long long* __restrict__ acc) {
    chain_in();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_bytes;
         i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t b = bytes[i];
        if (b == 0) continue;
        int64_t k = (k0 + 4 * i) % L;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t c = (b >> (2 * j)) & 3u;
            if (c) {
                unsigned long long l = c & 1u, h = c >> 1;
                atomicAdd(&acc[k], l | (h << 21) | ((l & h) << 42));
            }
            if (++k == L) k = 0;
        }
    }
}

__global__ void ragged_i8_kernel(const int8_t* __restrict__ x, int64_t n, int64_t k0, int64_t L,
                                 long long* __restrict__ acc) {
    chain_in();
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        int v = x[i];
        if (v) atomicAdd(reinterpret_cast<unsigned long long*>(&acc[(k0 + i) % L]), (unsigned long long)(long long)v);
    }
}

// One thread per bin k: sums the samples of two runs (before and behind a bulk
// launch's rows) that fall into bin k, in order, in double-float, and adds the
// sum to the plan's double-float bin.
struct FloatRun {
    const float* x;
    int64_t n, k0;  // samples, phase of the first one
};

__global__ void ragged_f32_kernel(FloatRun r0, FloatRun r1, int64_t L, float2* __restrict__ acc) {
    chain_in();
    const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (k >= L) return;
    pcal_df::df s{0.f, 0.f};
    bool any = false;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const FloatRun& r = e ? r1 : r0;
        int64_t t = k >= r.k0 ? k - r.k0 : k - r.k0 + L;  // first sample of the run in bin k
        any = any || t < r.n;
        for (; t < r.n; t += L) s = pcal_df::add_f(s, r.x[t]);
    }
    if (!any) return;
    const float2 a = acc[k];
    s = pcal_df::add(pcal_df::df{a.x, a.y}, s);
    acc[k] = make_float2(s.hi, s.lo);
}

// ---- short folds -------------------------------------------------------------
//
// Inputs too short for the bulk kernel, 10 ms of a recorder for instance.  One
// sample per thread and atomic (2-bit, int8) or one thread per bin (float32)
// took 6 and 8 us for 160 and 640 KB (steps of 19.5 us, and 7.3 us a chunk of a
// live period); here the rows (a period L each, widened as the bulk kernel's)
// are folded by small CTAs, one column block of a chunk of rows each, and what
// is no whole 16-byte word at either end sample by sample in one more CTA: 3.8
// and 3.3 us (12.3 us a step, 3.2 us a chunk, which is the host's call).

struct ShortBlock {
    const uint32_t* base;
    int row_words, cols;
};

struct ShortArgs {
    ShortBlock rows, part;   // whole rows, and the words behind the last one
    int n_rows, blocks, chunk_rows, tasks;  // tasks: column blocks x chunks of rows
    int part_blocks;
    const uint8_t* edge[2];  // the bytes before and behind
    int edge_n[2];           // samples of each
    int64_t k_rows, k_part, k_edge[2];  // phases of their first samples
    int64_t L;
    unsigned long long* acc2;
    long long* acc8;
};

template <int FMT>
__global__ void __launch_bounds__(pcal_direct::kDirectThreads) short_fold_kernel(const __grid_constant__ ShortArgs a) {
    using namespace pcal_direct;
    extern __shared__ __align__(1024) uint8_t smem[];
    chain_in();
    const uint32_t L = (uint32_t)a.L;
    if ((int)blockIdx.x >= a.tasks + a.part_blocks) {
        for (int e = 0; e < 2; ++e)
            for (int i = threadIdx.x; i < a.edge_n[e]; i += blockDim.x) {
                const uint32_t k = (uint32_t)((a.k_edge[e] + i) % a.L);
                if (FMT == PCAL_2BIT) {
                    const uint32_t c = (a.edge[e][i >> 2] >> (2 * (i & 3))) & 3u;
                    const unsigned long long l = c & 1u, h = c >> 1;
                    if (c) atomicAdd(&a.acc2[k], l | (h << 21) | ((l & h) << 42));
                } else {
                    const int v = (int8_t)a.edge[e][i];
                    if (v) atomicAdd(reinterpret_cast<unsigned long long*>(&a.acc8[k]), (unsigned long long)(long long)v);
                }
            }
        return;
    }
    const bool part = (int)blockIdx.x >= a.tasks;
    const int task = part ? (int)blockIdx.x - a.tasks : (int)blockIdx.x;
    const int blocks = part ? a.part_blocks : a.blocks;
    const int chunk = task / blocks, col = (task - chunk * blocks) * direct_cols(FMT);
    const ShortBlock D = part ? a.part : a.rows;
    const int r0 = part ? 0 : chunk * a.chunk_rows;
    const int r1 = part ? 1 : (r0 + a.chunk_rows < a.n_rows ? r0 + a.chunk_rows : a.n_rows);
    constexpr int kSpw = FMT == PCAL_2BIT ? 16 : 4;
    const uint32_t base = (uint32_t)(((part ? a.k_part : a.k_rows) + (int64_t)col * kSpw) % a.L);
    const uint64_t policy = l2_policy_evict_first();
    if constexpr (FMT == PCAL_2BIT)
        direct_count_2bit(D, r0, r1, col, smem, policy, [&](int t, uint32_t sl, uint32_t sh, uint32_t shl) {
            if (sl | sh)
                atomicAdd(&a.acc2[wrap_bin(base, (uint32_t)t, L)], (unsigned long long)sl |
                                                                       ((unsigned long long)sh << 21) |
                                                                       ((unsigned long long)shl << 42));
        });
    else
        direct_count_i8(D, r0, r1, col, smem, policy, [&](int t, int v) {
            if (v)
                atomicAdd(reinterpret_cast<unsigned long long*>(&a.acc8[wrap_bin(base, (uint32_t)t, L)]),
                          (unsigned long long)(long long)v);
        });
}

// float32: blockDim.y groups of warps, 32 bins each; a group's warps take the
// periods in turn (eight loads in flight each), sum in double-float, and the
// warps' sums are added in order to the bins.  Deterministic: nothing depends
// on timing.
__global__ void __launch_bounds__(1024) short_f32_kernel(const float* __restrict__ x, int64_t n, int64_t k0, int64_t L,
                                                         float2* __restrict__ acc) {
    __shared__ float2 s_sum[32][32];
    chain_in();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    float2(*const sums)[32] = s_sum + threadIdx.y * warps;
    const int64_t c = ((int64_t)blockIdx.x * blockDim.y + threadIdx.y) * 32 + lane;  // place within a period of the run
    pcal_df::df s{0.f, 0.f};
    if (c < L) {
        const int64_t step = (int64_t)warps * L;
        int64_t t = c + warp * L;
        for (; t + 7 * step < n; t += 8 * step) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = __ldcs(x + t + u * step);
#pragma unroll
            for (int u = 0; u < 8; ++u) s = pcal_df::add_f(s, v[u]);
        }
        float v[8];
#pragma unroll
        for (int u = 0; u < 7; ++u) v[u] = t + u * step < n ? __ldcs(x + t + u * step) : 0.f;
#pragma unroll
        for (int u = 0; u < 7; ++u)
            if (t + u * step < n) s = pcal_df::add_f(s, v[u]);
    }
    sums[warp][lane] = make_float2(s.hi, s.lo);
    __syncthreads();
    if (warp == 0 && c < L && c < n) {
        const int64_t k = k0 + c < L ? k0 + c : k0 + c - L;
        const float2 a = acc[k];
        for (int w = 1; w < warps; ++w) s = pcal_df::add(s, pcal_df::df{sums[w][lane].x, sums[w][lane].y});
        s = pcal_df::add(pcal_df::df{a.x, a.y}, s);
        acc[k] = make_float2(s.hi, s.lo);
    }
}

// Move the packed 21-bit fields into the wide 64-bit arrays and clear them.
__global__ void spill2_kernel(unsigned long long* __restrict__ acc, unsigned long long* __restrict__ wide,
                              int64_t L) {
    chain_in();
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < L; k += (int64_t)gridDim.x * blockDim.x) {
        unsigned long long v = acc[k];
        if (v) {
            wide[k] += v & PCAL_F21_MASK;
            wide[L + k] += (v >> 21) & PCAL_F21_MASK;
            wide[2 * L + k] += (v >> 42) & PCAL_F21_MASK;
            acc[k] = 0;
        }
    }
}

// Exact per-(bin, code) counts of the current period: [L][4] int64.
__global__ void export2_kernel(const unsigned long long* __restrict__ acc, const unsigned long long* __restrict__ wide,
                               int64_t L, int64_t q, int64_t rem, int64_t a0, long long* __restrict__ out) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < L; k += (int64_t)gridDim.x * blockDim.x) {
        unsigned long long v = acc[k];
        long long sl = (long long)((v & PCAL_F21_MASK) + wide[k]);
        long long sh = (long long)(((v >> 21) & PCAL_F21_MASK) + wide[L + k]);
        long long shl = (long long)(((v >> 42) & PCAL_F21_MASK) + wide[2 * L + k]);
        int64_t r = (k - a0 + L) % L;
        long long cnt = q + (r < rem ? 1 : 0);
        out[4 * k + 3] = shl;
        out[4 * k + 2] = sh - shl;
        out[4 * k + 1] = sl - shl;
        out[4 * k + 0] = cnt - sl - sh + shl;
    }
}

// Failure detection without a fault: every thread of one block waits on an
// mbarrier phase that nothing completes, with the bounded wait of the fold
// kernels and a short limit; each thread that gives up sets a bit, and the
// block then returns normally.
__global__ void wait_timeout_kernel(uint64_t limit_ns, unsigned int* flags) {
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        pcal_ptx::mbar_init(&bar, (1u << 20) - 1);  // the largest count: more arrivals than will come
        pcal_ptx::fence_barrier_init();
    }
    __syncthreads();
    if (!pcal_ptx::mbar_wait(&bar, 0, limit_ns)) atomicOr(flags, PCAL_DERR_FULL_WAIT);
    __syncthreads();
}

// Launch with programmatic stream serialization (see chain_in).
template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*k)(KArgs...), int grid, dim3 block, cudaStream_t s, size_t smem, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, static_cast<Args&&>(args)...);
}

inline int grid_for(int64_t work, int threads, int num_sms) {
    int64_t g = (work + threads - 1) / threads;
    int64_t cap = (int64_t)num_sms * 8;
    if (g > cap) g = cap;
    return g < 1 ? 1 : (int)g;
}

}  // namespace

cudaError_t launch_ragged_f32(pcal_plan* p, const uint8_t* d0, int64_t n0, int64_t k0, const uint8_t* d1, int64_t n1,
                              int64_t k1, cudaStream_t s) {
    const int64_t L = p->g.L;
    const FloatRun r0{reinterpret_cast<const float*>(d0), n0, k0 % L}, r1{reinterpret_cast<const float*>(d1), n1, k1 % L};
    p->stats.kernel_launches += 1;
    p->folds.ragged += 1;
    return launch_chained(ragged_f32_kernel, (int)((L + 255) / 256), 256, s, 0, r0, r1, L, cur_accf(p));
}

cudaError_t launch_ragged(pcal_plan* p, const uint8_t* d_bytes, int64_t n, int64_t k0, cudaStream_t s) {
    const int64_t L = p->g.L;
    if (n <= 0) return cudaSuccess;
    cudaError_t e;
    switch (p->g.format) {
        case PCAL_2BIT: {
            const int64_t nb = n / 4;
            e = launch_chained(ragged_2bit_kernel, grid_for(nb, 256, p->num_sms), 256, s, 0, d_bytes, nb, k0, L,
                               cur_acc2(p));
            break;
        }
        case PCAL_I8:
            e = launch_chained(ragged_i8_kernel, grid_for(n, 256, p->num_sms), 256, s, 0,
                               reinterpret_cast<const int8_t*>(d_bytes), n, k0, L, cur_acc8(p));
            break;
        default: return launch_ragged_f32(p, d_bytes, n, k0, nullptr, 0, 0, s);
    }
    p->stats.kernel_launches += 1;
    p->folds.ragged += 1;
    return e;
}

cudaError_t launch_short(pcal_plan* p, const uint8_t* d, int64_t n, int64_t k0, cudaStream_t s) {
    using namespace pcal_direct;
    const int64_t L = p->g.L;
    p->folds.short_folds += 1;
    if (p->g.format == PCAL_F32) {
        // a warp per eight periods (its loads in flight together), at most eight,
        // or 32 where each would still take many
        const int64_t periods = (n + L - 1) / L;
        const int warps = periods > 512 ? 32 : periods > 56 ? 8 : (int)((periods + 7) / 8);
        // CTAs of up to eight warps, for the bins that the run reaches (a CTA of one
        // warp for every 32 bins of the period: 32 us for 1 of its 1,000,000 bins' periods)
        const int groups = warps < 8 ? 8 / warps : 1;
        const int64_t places = n < L ? n : L, per_cta = 32 * groups;
        p->stats.kernel_launches += 1;
        return launch_chained(short_f32_kernel, (int)((places + per_cta - 1) / per_cta), dim3(32 * warps, groups), s, 0,
                              reinterpret_cast<const float*>(d), n, k0, L, cur_accf(p));
    }
    const int spb = p->g.format == PCAL_2BIT ? 4 : 1;  // samples per byte
    const int64_t bytes = n / spb, row_bytes = p->g.row_samples / spb;
    int64_t head = (int64_t)((16 - reinterpret_cast<uintptr_t>(d) % 16) % 16);
    if (head > bytes) head = bytes;
    const int64_t rows = (bytes - head) / row_bytes, at = head + rows * row_bytes;
    const int64_t part = (bytes - at) / 16 * 16;
    const int cols = direct_cols(p->g.format);
    ShortArgs a{};
    a.rows = ShortBlock{reinterpret_cast<const uint32_t*>(d + head), (int)(row_bytes / 4), (int)(row_bytes / 4)};
    a.part = ShortBlock{reinterpret_cast<const uint32_t*>(d + at), 0, (int)(part / 4)};
    a.n_rows = (int)rows;
    a.blocks = (int)((row_bytes / 4 + cols - 1) / cols);
    // chunks of at least 128 2-bit or 64 int8 rows (below that the atomic adds
    // of 512 bins cost as much as the loads), of about eight per resident CTA
    int64_t least = p->g.format == PCAL_2BIT ? 128 : 64;
    const int64_t even = bytes / (8 * kDirectCtas * p->num_sms) / (4 * cols);
    if (least < even) least = even < kDirectRows / 2 ? even : kDirectRows / 2;
    const int64_t chunks = rows / least > 0 ? rows / least : 1;
    a.chunk_rows = (int)((rows + chunks - 1) / chunks);
    if (a.chunk_rows < 1) a.chunk_rows = 1;
    a.tasks = rows > 0 ? a.blocks * (int)((rows + a.chunk_rows - 1) / a.chunk_rows) : 0;
    a.part_blocks = (int)((part / 4 + cols - 1) / cols);
    a.edge[0] = d;
    a.edge_n[0] = (int)(head * spb);
    a.edge[1] = d + at + part;
    a.edge_n[1] = (int)((bytes - at - part) * spb);
    a.L = L;
    a.k_edge[0] = k0;
    a.k_rows = (k0 + head * spb) % L;
    a.k_part = a.k_rows;  // rows are whole periods
    a.k_edge[1] = (k0 + (at + part) * spb) % L;
    a.acc2 = cur_acc2(p);
    a.acc8 = cur_acc8(p);
    const int grid = a.tasks + a.part_blocks + (a.edge_n[0] + a.edge_n[1] > 0 ? 1 : 0);
    p->stats.kernel_launches += 1;
    return p->g.format == PCAL_2BIT ? launch_chained(short_fold_kernel<PCAL_2BIT>, grid, kDirectThreads, s, kDirectSmem, a)
                                    : launch_chained(short_fold_kernel<PCAL_I8>, grid, kDirectThreads, s, kDirectSmem, a);
}

cudaError_t prepare_short() {
    cudaError_t e = cudaFuncSetAttribute(short_fold_kernel<PCAL_2BIT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         pcal_direct::kDirectSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(short_fold_kernel<PCAL_I8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 pcal_direct::kDirectSmem);
    return e;
}

cudaError_t launch_spill2(pcal_plan* p, cudaStream_t s) {
    const cudaError_t e =
        launch_chained(spill2_kernel, grid_for(p->g.L, 256, p->num_sms), 256, s, 0, cur_acc2(p), cur_wide2(p),
                       p->g.L);
    p->stats.kernel_launches += 1;
    return e;
}

cudaError_t launch_export_bins(pcal_plan* p, void* d_out, cudaStream_t s) {
    const int64_t L = p->g.L;
    const int64_t n_tot = p->n_abs - p->period_start;
    export2_kernel<<<grid_for(L, 256, p->num_sms), 256, 0, s>>>(cur_acc2(p), cur_wide2(p), L, n_tot / L, n_tot % L,
                                                                  p->period_start % L,
                                                                  reinterpret_cast<long long*>(d_out));
    p->stats.kernel_launches += 1;
    return cudaGetLastError();
}

extern "C" int pcal_selftest_wait_timeout(double limit_s, unsigned int* flags_out) {
    if (!flags_out || !(limit_s > 0.0) || limit_s > 2.0) return PCAL_EINVAL;
    unsigned int* d = nullptr;
    cudaError_t e = cudaMalloc(&d, sizeof(unsigned int));
    if (e == cudaSuccess) e = cudaMemset(d, 0, sizeof(unsigned int));
    if (e == cudaSuccess) {
        wait_timeout_kernel<<<1, 64>>>((uint64_t)(limit_s * 1e9), d);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e == cudaSuccess) e = cudaMemcpy(flags_out, d, sizeof(unsigned int), cudaMemcpyDeviceToHost);
    cudaFree(d);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        return PCAL_ECUDA;
    }
    return *flags_out ? PCAL_ETIMEOUT : PCAL_OK;
}
