// Fold of a block of rows by a small CTA: four warps take batches of rows in
// turn, each through its own three-batch ring in shared memory (cp.async, 16
// bytes a lane), and every lane counts its own words (int8 four, 2-bit one a
// row) in registers; the four warps' counts are added and handed out sample by
// sample.  A block (`Block`): base, the first word of row 0 (16-byte aligned);
// row_words between rows; cols, the words of a row that count (a multiple of 4).
// Used by the batched fold (batch.cu) and the short folds of single plans
// (fold_ragged.cu).
#pragma once

#include <stdint.h>

#include "bitplane.cuh"
#include "pcal.h"
#include "ptx.cuh"

namespace pcal_direct {

using namespace pcal_ptx;

constexpr int kDirectWarps = 4;
constexpr int kDirectThreads = 32 * kDirectWarps;
constexpr int kDirectCtas = 4;                     // per SM (48 KB of shared memory each)
constexpr int kDirectU = 7;                        // upper bit planes: at most 4095 rows per warp
constexpr int kDirectRows = 4064 * kDirectWarps;   // rows of a task, at most
constexpr int kDirectBatch = 4096;                 // bytes of a batch: 8 int8 rows or 32 2-bit rows of a warp
constexpr int kDirectRing = 3;
constexpr int kDirectSmem = kDirectWarps * kDirectRing * kDirectBatch;

__host__ __device__ constexpr int direct_cols(int fmt) { return fmt == PCAL_2BIT ? 32 : 128; }

// 16 bytes of this lane from global to shared memory; zeros where !have.
__device__ __forceinline__ void copy_async(uint32_t dst, const void* src, bool have, uint64_t policy) {
    asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2, %3;" ::"r"(dst), "l"(src),
                 "r"(have ? 16 : 0), "l"(policy)
                 : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}

// Bin of sample `off` behind bin `base` (both below 2^21).
__device__ __forceinline__ uint32_t wrap_bin(uint32_t base, uint32_t off, uint32_t L) {
    uint32_t b = base + off;
    if (b >= L) b -= L;
    if (b >= L) b %= L;
    return b;
}

// The batches of rows [r0, r1) that warp `warp` takes: 4 KB each, ROWS rows of
// 4096 / ROWS bytes, every kDirectWarps-th.  count(p) folds a batch that lies
// at p row after row.
template <int ROWS, class Block, class Count>
__device__ __forceinline__ void direct_batches(const Block& D, long long r0, long long r1, int col, int warp,
                                               uint8_t* ring, uint64_t policy, Count count) {
    constexpr int kLanes = kDirectBatch / ROWS / 16;  // lanes that copy one row
    constexpr int kStep = 32 / kLanes;                // rows of one copy of the warp
    const int lane = threadIdx.x & 31, row_in = lane / kLanes, piece = lane % kLanes;
    const int n = (int)(r1 - r0), all = (n + ROWS - 1) / ROWS;
    const int mine = all > warp ? (all - warp + kDirectWarps - 1) / kDirectWarps : 0;
    const bool active = col + 4 * piece < D.cols;
    // (a lane without columns copies nothing, from an address of the block all the same)
    const uint32_t* src0 = D.base + r0 * D.row_words + (active ? col + 4 * piece : 0);
    const uint32_t dst0 = smem_addr(ring) + lane * 16;
    auto issue = [&](int k) {
        if (k < mine) {
            const int row = (warp + k * kDirectWarps) * ROWS + row_in;
            const uint32_t dst = dst0 + (k % kDirectRing) * kDirectBatch;
            if (row + ROWS - kStep < n) {  // a whole batch
                const uint32_t* src = src0 + (long long)row * D.row_words;
#pragma unroll
                for (int i = 0; i < ROWS / kStep; ++i, src += kStep * (long long)D.row_words)
                    copy_async(dst + i * 512, src, active, policy);
            } else {
                for (int i = 0; i < ROWS / kStep; ++i) {
                    const int r = row + i * kStep;
                    copy_async(dst + i * 512, src0 + (long long)(r < n ? r : 0) * D.row_words, active && r < n, policy);
                }
            }
        }
        copy_commit();
    };
    issue(0);
    issue(1);
    for (int k = 0; k < mine; ++k) {
        issue(k + 2);
        copy_wait<2>();
        __syncwarp();  // the other lanes' copies too
        count(ring + (k % kDirectRing) * kDirectBatch);
        __syncwarp();  // before the slot is filled again
    }
    copy_wait<0>();
}

// 2-bit: counts of the CTA's rows as the packed words of transpose16x2 in
// every warp's scratch, added over the warps, then flush(t, sl, sh, shl) for
// the sums of the l, h and (h AND l) bits of its 512 (or fewer) consecutive
// samples.
template <class Block, class Flush>
__device__ __forceinline__ void direct_count_2bit(const Block& D, long long r0, long long r1, int col, uint8_t* smem,
                                                  uint64_t policy, Flush flush) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t w1 = 0, w2 = 0, w4 = 0, w8 = 0, w16 = 0, wu[kDirectU], d1 = 0, d2 = 0, d4 = 0, d8 = 0, du[kDirectU];
#pragma unroll
    for (int u = 0; u < kDirectU; ++u) wu[u] = du[u] = 0;
    uint8_t* ring = smem + warp * kDirectRing * kDirectBatch;
    direct_batches<32>(D, r0, r1, col, warp, ring, policy, [&](const uint8_t* p) {
        uint32_t x[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) x[i] = *reinterpret_cast<const uint32_t*>(p + i * 128 + 4 * lane);
        pcal_bits::add32<kDirectU>(x, w1, w2, w4, w8, w16, wu, d1, d2, d4, d8, du);
    });
    // positions 2j (l) and 2j + 1 (h) of sample j: word position % 16, half
    // position / 16; words 0..15 the l and h sums, 16..31 the (h AND l) sums
    uint32_t* sm = reinterpret_cast<uint32_t*>(ring);
    uint32_t A[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) A[i] = 0;
    A[0] = w1;
    A[1] = w2;
    A[2] = w4;
    A[3] = w8;
    A[4] = w16;
#pragma unroll
    for (int u = 0; u < kDirectU; ++u) A[5 + u] = wu[u];
    pcal_bits::transpose16x2(A);
#pragma unroll
    for (int i = 0; i < 16; ++i) sm[i * 33 + lane] = A[i];
#pragma unroll
    for (int i = 0; i < 16; ++i) A[i] = 0;
    A[0] = d1;
    A[1] = d2;
    A[2] = d4;
    A[3] = d8;
#pragma unroll
    for (int u = 0; u < kDirectU; ++u) A[4 + u] = du[u];
    pcal_bits::transpose16x2(A);
#pragma unroll
    for (int i = 0; i < 16; ++i) sm[(16 + i) * 33 + lane] = A[i];
    __syncthreads();
    // (at most 16,256 rows: no half of a sum overflows)
    uint32_t* s0 = reinterpret_cast<uint32_t*>(smem);
    constexpr int kPitch = kDirectRing * kDirectBatch / 4;
#pragma unroll
    for (int i = threadIdx.x; i < 1024; i += kDirectThreads) {
        uint32_t* q = s0 + (i >> 5) * 33 + (i & 31);
        uint32_t v = 0;
#pragma unroll
        for (int w = 0; w < kDirectWarps; ++w) v += q[w * kPitch];
        q[0] = v;
    }
    __syncthreads();
    const int tasks = (D.cols - col < 32 ? D.cols - col : 32) * 16;
#pragma unroll 2
    for (int t = threadIdx.x; t < tasks; t += kDirectThreads) {
        const int cl = t >> 4, j = t & 15;
        const int pl = 2 * j, ph = 2 * j + 1;
        const uint32_t sl = (s0[(pl & 15) * 33 + cl] >> (16 * (pl >> 4))) & 0xFFFFu;
        const uint32_t sh = (s0[(ph & 15) * 33 + cl] >> (16 * (ph >> 4))) & 0xFFFFu;
        const uint32_t shl = ((s0[(16 + (pl & 15)) * 33 + cl] >> (16 * (pl >> 4))) & 0xFFFFu) +
                             ((s0[(16 + (ph & 15)) * 33 + cl] >> (16 * (ph >> 4))) & 0xFFFFu);
        flush(t, sl, sh, shl);
    }
}

// int8: flush(t, v) for the sums of the 512 (or fewer) consecutive samples of
// the block's columns.
template <class Block, class Flush>
__device__ __forceinline__ void direct_count_i8(const Block& D, long long r0, long long r1, int col, uint8_t* smem,
                                                uint64_t policy, Flush flush) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int s[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) s[i] = 0;
    uint8_t* ring = smem + warp * kDirectRing * kDirectBatch;
    direct_batches<8>(D, r0, r1, col, warp, ring, policy, [&](const uint8_t* p) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint4 v = *reinterpret_cast<const uint4*>(p + i * 512 + 16 * lane);
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                s[4 * q] = __dp4a((int)w[q], 0x00000001, s[4 * q]);
                s[4 * q + 1] = __dp4a((int)w[q], 0x00000100, s[4 * q + 1]);
                s[4 * q + 2] = __dp4a((int)w[q], 0x00010000, s[4 * q + 2]);
                s[4 * q + 3] = __dp4a((int)w[q], 0x01000000, s[4 * q + 3]);
            }
        }
    });
    int* sm = reinterpret_cast<int*>(ring);
#pragma unroll
    for (int i = 0; i < 16; ++i) sm[lane * 17 + i] = s[i];
    __syncthreads();
    const int left = (D.cols - col) * 4;
    const int tasks = left < 512 ? left : 512;
    const int* s0 = reinterpret_cast<const int*>(smem);
    constexpr int kPitch = kDirectRing * kDirectBatch / 4;
#pragma unroll 4
    for (int t = threadIdx.x; t < tasks; t += kDirectThreads) {
        const int* q = s0 + (t >> 4) * 17 + (t & 15);
        int v = 0;
#pragma unroll
        for (int w = 0; w < kDirectWarps; ++w) v += q[w * kPitch];
        flush(t, v);
    }
}

}  // namespace pcal_direct
