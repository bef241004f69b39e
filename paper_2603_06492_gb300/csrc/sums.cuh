// Fixed-order sums of partial results, shared by the last launch of a call and
// the grouped GEMM launch.
#pragma once

#include "common.cuh"

namespace noble {

// Fixed-order sums of partial results: out_j[i] = sum_z part_j[z * stride_j + i]
// (z ascending) for up to eight outputs in one launch.
struct SplitJobs {
    const float *part[8];
    float *out[8];
    int64_t n[8], stride[8], begin[9];  // stride: elements between consecutive partials
    int nparts;
    int jparts[8];  // partials of job j when non-zero, else nparts (sum_warp and sum_block)
    int njobs;
};
// One warp over 32 consecutive outputs: the partials of an output in eight
// ranges [w P/8, (w+1) P/8), each added in ascending order (side by side: eight
// or sixteen loads in flight), then the eight sums in order -- deterministic.
__device__ __forceinline__ void sum_warp(const SplitJobs &J, int64_t block, int lane)
{
    const int64_t idx = block * 32 + lane;
    if (idx >= J.begin[J.njobs]) return;
    int j = 0;
    while (idx >= J.begin[j + 1]) ++j;
    const int64_t i = idx - J.begin[j], st = J.stride[j];
    const int np = J.jparts[j] ? J.jparts[j] : J.nparts;
    const int per = (np + 7) / 8;
    const float *pp = J.part[j] + i;
    float s[8];
#pragma unroll
    for (int w = 0; w < 8; ++w) s[w] = 0.f;
#pragma unroll 2
    for (int z = 0; z < per; ++z) {
        float v[8];
#pragma unroll
        for (int w = 0; w < 8; ++w) v[w] = w * per + z < np ? pp[(int64_t)(w * per + z) * st] : 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) s[w] += v[w];
    }
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += s[w];
    J.out[j][i] = t;
}

// The same sums by eight warps of a block, one range each.
__device__ __forceinline__ void sum_block(const SplitJobs &J, int64_t block)
{
    __shared__ float sm[8][33];
    const int lane = threadIdx.x % 32, w = threadIdx.x / 32;
    const int64_t idx = block * 32 + lane;
    const bool in = idx < J.begin[J.njobs];
    int j = 0;
    if (in)
        while (idx >= J.begin[j + 1]) ++j;
    const int64_t i = in ? idx - J.begin[j] : 0;
    const int np = J.jparts[j] ? J.jparts[j] : J.nparts;
    const int per = (np + 7) / 8;
    const int zb = w * per, ze = min(np, zb + per);
    float s = 0.f;
    if (in) {
        // eight loads in flight, then added in ascending z
        const float *pp = J.part[j] + i;
        const int64_t st = J.stride[j];
        int z = zb;
        for (; z + 8 <= ze; z += 8) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = pp[(int64_t)(z + u) * st];
#pragma unroll
            for (int u = 0; u < 8; ++u) s += v[u];
        }
        for (; z < ze; ++z) s += pp[(int64_t)z * st];
    }
    sm[w][lane] = s;
    __syncthreads();
    if (w == 0 && in) {
        float t = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) t += sm[k][lane];
        J.out[j][i] = t;
    }
}

}  // namespace noble
