// Mixed-radix FFT of the batched tone DFT (dft_fft.cu): host declarations.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

constexpr int kFftMaxPasses = 12;

struct FftPlan {
    int N, passes;             // passes == 0: N has a prime factor above 7 (or is 1)
    int radix[kFftMaxPasses];  // their product is N
    bool wide;                 // double-float inside a pass
    void* tw;                  // twiddles of the passes after the first, [q - 1][k] each
};

// The radices of N; false where the FFT does not take it.
bool fft_factors(int N, FftPlan* p);
// Plan and device tables (allocates).  wide: double-float values inside a pass, else FP32.
cudaError_t fft_create(int N, bool wide, FftPlan* p);
void fft_destroy(FftPlan* p);
// T[c] = the N-point DFT of P[c], c < C (C >= 1).
cudaError_t launch_fft(const FftPlan& p, const float2* P, int64_t C, float2* T, cudaStream_t s);
