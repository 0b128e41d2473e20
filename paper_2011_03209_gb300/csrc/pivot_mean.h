// Mean of the pivots, column by column, the same bit for bit from the kernel and
// on the host (a cloud in host memory has its pivots gathered there): kMeanParts
// FP32 sums of every kMeanParts-th pivot, added up in order, over K.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define MGB_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define MGB_HOST_DEVICE inline
#endif

namespace mgb {

constexpr int kMeanParts = 8;

MGB_HOST_DEVICE float pivot_part(const float* Pv, int K, int dp, int column, int part)
{
    float s = 0.f;
#ifdef __CUDACC__
#pragma unroll 16
#endif
    for (int i = part; i < K; i += kMeanParts) s += Pv[(int64_t)i * dp + column];
    return s;
}

// part[w * pitch]: the parts of one column
MGB_HOST_DEVICE float mean_of_parts(const float* part, int pitch, int K)
{
    float s = part[0];
    for (int w = 1; w < kMeanParts; ++w) s += part[w * pitch];
    return s / (float)K;
}

inline void pivot_mean_host(const float* Pv, int K, int dp, float* c)
{
    for (int k = 0; k < dp; ++k) {
        float part[kMeanParts];
        for (int w = 0; w < kMeanParts; ++w) part[w] = pivot_part(Pv, K, dp, k, w);
        c[k] = mean_of_parts(part, 1, K);
    }
}

}  // namespace mgb
