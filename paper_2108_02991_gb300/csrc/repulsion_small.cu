// Repulsion sums of few samples: R_i = sum_j (k_i - k_j)/|k_i - k_j| (paper eq.
// Fr_grad with H' = 1; in energy mode sum_j |k_i - k_j|), directed.
//
// The symmetric kernel (repulsion_sym.cu) works on pairs of 1024-sample tiles,
// one CTA of four warps a pair: 1024 samples are one item and leave 151 SMs
// idle, 8192 are 36 items.  Here a warp takes 64 targets (two a lane) against
// a slice of the sources, and the slices are as short as it takes to give
// every SM sixteen warps.  Twice the arithmetic, but on the whole GPU.
// Totals are fixed-point integers as there (exact, order-free).
//
// Bound: latency up to ~4000 samples, FP32 issue (11.5 instructions a directed
// pair) above.  Measured (gradient; the call's scope, uniform samples): 1024
// samples 8.2 us against 78 with the symmetric kernel, 4096 16 against 77, 8192
// 43 against 78, 11000 71 against 88, 12288 87 against 78, 16384 128 against 78;
// the rule of the dispatch (api.cu) follows from these.
#include <cuda_runtime.h>
#include <cstdint>

#include "kernels.h"
#include "ptx.cuh"

namespace sparkling {

namespace {

constexpr int kSmallThreads = 128;
constexpr int kSmallTargets = 64;          // targets of a warp
constexpr int kSmallMinSlice = 16;         // sources of a slice at least
constexpr int kSmallWarpsPerSm = 16;

template <bool ENERGY>
__global__ void __launch_bounds__(kSmallThreads) repulsion_small_kernel(
    const float4 *__restrict__ pos, int N, int groups, int slices, float eps2,
    unsigned long long *acc)
{
    constexpr int NV = ENERGY ? 1 : 3;
    const int lane = threadIdx.x & 31;
    const int w = (int)(blockIdx.x * (kSmallThreads / 32) + (threadIdx.x >> 5));
    if (w >= groups * slices) return;
    const int g = w % groups, s = w / groups;
    const int j0 = (int)((int64_t)N * s / slices), j1 = (int)((int64_t)N * (s + 1) / slices);
    float tx[2], ty[2], tz[2], f[2][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const int i = g * kSmallTargets + t * 32 + lane;
        const float4 p = pos[i < N ? i : N - 1];
        tx[t] = p.x; ty[t] = p.y; tz[t] = p.z;
    }
#pragma unroll 8
    for (int j = j0; j < j1; ++j) {
        const float4 q = __ldg(pos + j);
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const float dx = tx[t] - q.x, dy = ty[t] - q.y, dz = tz[t] - q.z;
            const float r2 = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, eps2)));
            const float ri = rsqrt_sfu(r2);
            if (ENERGY) {
                f[t][0] = fmaf(r2, ri, f[t][0]);
            } else {
                f[t][0] = fmaf(dx, ri, f[t][0]);
                f[t][1] = fmaf(dy, ri, f[t][1]);
                f[t][2] = fmaf(dz, ri, f[t][2]);
            }
        }
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const int i = g * kSmallTargets + t * 32 + lane;
        if (i < N)
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                const long long x = __float2ll_rn(f[t][v] * 4294967296.0f);
                if (x) atomicAdd(acc + (int64_t)i * NV + v, (unsigned long long)x);
            }
    }
}

} // namespace

cudaError_t launch_repulsion_small(const float4 *pos, int64_t N, float eps2, bool energy,
                                   unsigned long long *acc, int sms, cudaStream_t st)
{
    const int n = (int)N, groups = (n + kSmallTargets - 1) / kSmallTargets;
    int slices = (sms * kSmallWarpsPerSm + groups - 1) / groups;
    const int most = (n + kSmallMinSlice - 1) / kSmallMinSlice;
    if (slices > most) slices = most;
    // FP32 sums of at most 1024 terms, as in the symmetric kernel
    const int least = (n + kTile - 1) / kTile;
    if (slices < least) slices = least;
    const int64_t warps = (int64_t)groups * slices;
    const unsigned grid = (unsigned)((warps + kSmallThreads / 32 - 1) / (kSmallThreads / 32));
    if (energy)
        repulsion_small_kernel<true><<<grid, kSmallThreads, 0, st>>>(pos, n, groups, slices, eps2, acc);
    else
        repulsion_small_kernel<false><<<grid, kSmallThreads, 0, st>>>(pos, n, groups, slices, eps2, acc);
    return cudaGetLastError();
}

} // namespace sparkling
