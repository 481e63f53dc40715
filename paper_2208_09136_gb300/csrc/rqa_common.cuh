// Device helpers shared by the cell kernels: distances on the fly and the
// persistent work loop.
#pragma once
#include <cstdint>
#include "rqa_internal.h"

namespace rqa {

constexpr unsigned FULL = 0xffffffffu;

// Record the first device-side error; later ones are dropped.
__device__ __forceinline__ void set_status(int *status, int code)
{
    atomicCAS(status, 0, code);
}

// Add 1 to the shared word at shared-space address a when x <= y
// (unsigned), as one compare and one predicated reduction: no branch, so a
// warp whose lanes disagree does not split, and no predicate turned into an
// integer and back.  a is not touched when x > y; a caller folds a further
// condition into x (x = ~0u when it fails, with y < ~0u).
__device__ __forceinline__ void red_shared_if_le(uint32_t a, uint32_t x, uint32_t y)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.le.u32 q, %1, %2;\n\t@q red.shared.add.u32 [%0], 1;\n\t}"
                 :: "r"(a), "r"(x), "r"(y) : "memory");
}

// Add 1 to the shared word at shared-space address a: one reduction, no
// predicate.  A cell that counts nowhere adds to a per-lane scratch word
// instead, so no branch region is needed around the reduction.
__device__ __forceinline__ void red_shared(uint32_t a)
{
    asm volatile("red.shared.add.u32 [%0], 1;" :: "r"(a) : "memory");
}

// max(a, b, c) in one instruction (three-input FP32 max of sm_100 and later);
// exact, like two two-input maxima.
__device__ __forceinline__ float fmax3(float a, float b, float c)
{
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Maximum norm of the M per-coordinate differences a[q] - b[q] (Sect. 2):
// absolute values folded into the maxima, three at a time.
template <int M>
__device__ __forceinline__ float maxnorm(const float (&diff)[M])
{
    float d = fabsf(diff[0]);
    int q = 1;
#pragma unroll
    for (; q + 1 < M; q += 2) d = fmax3(d, fabsf(diff[q]), fabsf(diff[q + 1]));
#pragma unroll
    for (; q < M; ++q) d = fmaxf(d, fabsf(diff[q]));
    return d;
}

// Distance of cell (i, i + dl), any embedding, read through L1.
__device__ __forceinline__ float cell_dist(const float *__restrict__ ys, int i, int dl, int tau, int m)
{
    const int j = i + dl;
    float d = fabsf(__ldg(ys + i) - __ldg(ys + j));
    for (int q = 1; q < m; ++q)
        d = fmaxf(d, fabsf(__ldg(ys + i + q * tau) - __ldg(ys + j + q * tau)));
    return d;
}

// Embedding variants with their own kernel instantiation.
enum Embed : int { E_GENERIC = 0, E_M2 = 2, E_M3 = 3, E_M4 = 4,
                   E_M1T1 = 11, E_M3T1 = 31, E_M3T3 = 33 };

// Host: allow `kern` its dynamic shared memory.  The limit belongs to the
// kernel, not to the call, so every launch sets the largest size that any call
// needs (`most`): host threads with calls of different sizes would otherwise
// lower it between each other's set and launch.
template <class Kern>
inline cudaError_t allow_smem(Kern kern, int most)
{
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

// Host: CTAs of `kern` (THREADS threads, `smem` dynamic bytes) resident per
// SM, and the SM count of the current device; both cached per host thread (the
// last 64 sizes asked for, as a call's sizes vary with its targets and thresholds).
inline int resident_per_sm(const void *kern, int smem, int threads = THREADS)
{
    struct Entry { const void *k; int dev, s, v; };
    static thread_local Entry cache[64];
    static thread_local unsigned n = 0;
    int dev = 0;
    cudaGetDevice(&dev);
    for (unsigned i = 0; i < (n < 64 ? n : 64); ++i)
        if (cache[i].k == kern && cache[i].s == smem && cache[i].dev == dev) return cache[i].v;
    int v = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kern, threads, smem) != cudaSuccess) {
        cudaGetLastError();
        v = 1;
    }
    v = v < 1 ? 1 : v;
    cache[n % 64] = Entry{kern, dev, smem, v};
    n = n + 1 < 128 ? n + 1 : 64;
    return v;
}

inline int sm_count_current()
{
    static thread_local int cache[64] = {};
    int d = 0;
    cudaGetDevice(&d);
    if (d >= 0 && d < 64 && cache[d]) return cache[d];
    int v = 0;
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, d);
    if (d >= 0 && d < 64) cache[d] = v;
    return v;
}

// A persistent grid: at most the CTAs that can be resident at once.
inline int persistent_cap(const void *kern, int smem, int grid, int threads = THREADS)
{
    const int cap = sm_count_current() * resident_per_sm(kern, smem, threads);
    return grid < cap ? grid : (cap > 0 ? cap : 1);
}

}  // namespace rqa
