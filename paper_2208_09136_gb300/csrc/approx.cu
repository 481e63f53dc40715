// The paper's approximate threshold search (given in its source as a
// comment, Sect. 2): each series mapped onto [0, 1], RR evaluated at a fixed
// grid of thresholds, and for each target the grid threshold whose RR is the
// closest.  Kept for comparison with the exact selection of select.cu.
//
// Grid, in the series' own units and FP32 with correctly rounded operations
// so that any implementation reproduces it: thr_i = i * ((max - min) / n),
// i = 1..n.  A cell is recurrent at thr_i iff d <= thr_i (upper triangle).
#include <cstdint>
#include "dense.cuh"

namespace rqa {

constexpr int GT = 256;  // threads of the grid kernels

// Per series: min and max of the values, then the grid.
__global__ void __launch_bounds__(GT)
k_grid_thr(const float *__restrict__ y, const SeriesDev *__restrict__ series, int n_thr, float *thr)
{
    __shared__ float smin[GT / 32], smax[GT / 32];
    const int s = blockIdx.x;
    const SeriesDev sd = series[s];
    float lo = 3.4e38f, hi = -3.4e38f;
    for (uint32_t i = threadIdx.x; i < (uint32_t)sd.n; i += GT) {  // n + GT may pass 2^31
        const float v = y[sd.off + i];
        lo = fminf(lo, v);
        hi = fmaxf(hi, v);
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(FULL, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(FULL, hi, o));
    }
    if ((threadIdx.x & 31) == 0) {
        smin[threadIdx.x >> 5] = lo;
        smax[threadIdx.x >> 5] = hi;
    }
    __syncthreads();
    lo = smin[0];
    hi = smax[0];
    for (int w = 1; w < GT / 32; ++w) {
        lo = fminf(lo, smin[w]);
        hi = fmaxf(hi, smax[w]);
    }
    const float scale = __fdiv_rn(__fsub_rn(hi, lo), (float)n_thr);
    for (int i = threadIdx.x; i < n_thr; i += GT)
        thr[(int64_t)s * n_thr + i] = __fmul_rn((float)(i + 1), scale);
}

// Counting pass: for every cell the number of grid thresholds below its
// distance, r = #{i : thr_i < d} in 0..n, histogrammed per series: bin r holds
// the cells first recurrent at thr_{r+1}.
//
// The grid is uniform, so r follows from one multiplication: with rho the
// integer nearest to d / scale, every thr_i with i < rho lies below d and every
// one with i > rho above it (the rounding of 1 / scale, of the product and of
// thr_i moves d / scale by less than n 2^-22, far from one half), so
// r = rho - 1 + [thr_rho < d] (0 for rho = 0): one multiply-add into the
// integers of [2^23, 2^24), one DPX clamp, one lookup, one compare and one
// shared reduction per cell.  A binary search took log2(n) dependent lookups
// (400 thresholds, 4e7 cells: 5.5 ms of counting).  Grids whose step or its
// reciprocal could be subnormal or overflow are searched, all lanes in step;
// so are constant series and those whose step rounds to zero.
template <class Src>
__global__ void __launch_bounds__(GT)
k_count_grid(CellArgs a, const float *__restrict__ thr, int n_thr, uint64_t *hist)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ Unit unit;
    __shared__ int next_part, unit_rows;
    __shared__ uint32_t sink[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *win = reinterpret_cast<uint32_t *>(smem) + warp * Src::WORDS;
    uint32_t *h = reinterpret_cast<uint32_t *>(smem) + (GT / 32) * Src::WORDS;  // bin r + 1; bin 0 belongs to r = 0
    uint32_t *tk = h + n_thr + 2;  // keys of thr_0 = 0, thr_1, .., thr_n
    for (int x = threadIdx.x; x < n_thr + 2; x += GT) h[x] = 0;
    int cur = -1;
    uint64_t acc = 0;
    float inv = 0.f;
    bool uni = false;
    auto flush = [&]() {
        if (cur < 0) return;
        __syncthreads();
        unsigned long long *gh = reinterpret_cast<unsigned long long *>(hist + (int64_t)cur * (n_thr + 1));
        for (int x = threadIdx.x; x < n_thr + 2; x += GT)
            if (h[x]) {
                atomicAdd(gh + (x ? x - 1 : 0), (unsigned long long)h[x]);
                h[x] = 0;
            }
        acc = 0;
        __syncthreads();
    };
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned t = atomicAdd(a.queue, 1u);
            if ((int64_t)t < a.n_units) {
                unit = unit_of<false>(a, (int64_t)t);
                next_part = 0;
                unit_rows = part_rows(unit, GT / 32);
            } else {
                unit.s = -1;
            }
        }
        __syncthreads();
        const Unit w = unit;
        if (w.s < 0) break;
        const SeriesDev sd = a.series[w.s];
        if (w.s != cur) {
            flush();
            cur = w.s;
            const float *tg = thr + (int64_t)cur * n_thr;
            for (int x = threadIdx.x; x <= n_thr; x += GT) tk[x] = x ? __float_as_uint(tg[x - 1]) : 0u;
            const float scale = tg[0];  // 1 * ((max - min) / n)
            uni = scale >= 0x1p-100f && scale <= 0x1p100f;
            inv = uni ? 1.f / scale : 0.f;
            __syncthreads();
        }
        const uint64_t cells = (uint64_t)(w.b_hi - w.b_lo) * DB * (uint64_t)(w.r_hi - w.r_lo);
        if (acc + cells > 0xffffffffull) flush();
        acc += cells;
        const uint32_t sink_a = static_cast<uint32_t>(__cvta_generic_to_shared(&sink[lane]));
        const uint32_t h_a = static_cast<uint32_t>(__cvta_generic_to_shared(h));
        Src src;
        src.init(a.y + sd.off, sd, lane, win);
        auto bands = [&](auto &&f) {
            each_part(unit, unit_rows, &next_part, lane,
                      [&](int d0, int r_lo, int r_hi) { walk_keys(src, sd.ne, d0, r_lo, r_hi, lane, f); });
        };
        auto count = [&](auto &&bin) {  // bin(key): r + 1
            bands([&](const float (&d)[4][DPL], auto valid) {
                uint32_t r1[4][DPL];
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int j = 0; j < DPL; ++j) r1[r][j] = bin(__float_as_uint(d[r][j]));
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int j = 0; j < DPL; ++j) red_shared(valid(r, j) ? h_a + (r1[r][j] << 2) : sink_a);
            });
        };
        if (uni) {
            count([&](uint32_t key) -> uint32_t {
                const float f = fmaf(__uint_as_float(key), inv, 8388608.f);
                const int rho = __viaddmin_s32_relu((int)__float_as_uint(f), -0x4B000000, n_thr);
                return (uint32_t)rho + (tk[rho] < key ? 1u : 0u);
            });
        } else {
            count([&](uint32_t key) -> uint32_t {
                int lo = 0;  // grid keys below key (ascending); n_thr <= 1024
#pragma unroll 1
                for (int step = 1024; step; step >>= 1) {
                    const int c = lo + step;
                    lo = (tk[min(c, n_thr)] < key) & (c <= n_thr) ? c : lo;
                }
                return (uint32_t)lo + 1u;
            });
        }
    }
    flush();
}

// Per series: grid counts C_j = #{d <= thr_j} (prefix sums of the bins) and,
// for each target, the first j minimising |C_j den - rr_num P| (exact).  One
// warp scans the bins, then a warp per target searches.
__global__ void __launch_bounds__(GT)
k_select_grid(const uint64_t *hist, const float *thr, const SeriesDev *series, int n_thr,
              const int32_t *rr_num, int rr_den, int K, float *eps_out, double *rr_out,
              uint64_t *count_out)
{
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *c = reinterpret_cast<uint64_t *>(smem);  // n_thr prefix counts
    const int s = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t *h = hist + (int64_t)s * (n_thr + 1);
    for (int x = threadIdx.x; x < n_thr; x += GT) c[x] = h[x];
    __syncthreads();
    if (warp == 0) {
        uint64_t base = 0;
        for (int x0 = 0; x0 < n_thr; x0 += 32) {
            uint64_t v = x0 + lane < n_thr ? c[x0 + lane] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint64_t u = __shfl_up_sync(FULL, v, o);
                if (lane >= o) v += u;
            }
            v += base;
            if (x0 + lane < n_thr) c[x0 + lane] = v;
            base = __shfl_sync(FULL, v, 31);
        }
    }
    __syncthreads();
    const uint64_t P = series[s].P;
    for (int k = warp; k < K; k += GT / 32) {
        const unsigned __int128 target = (unsigned __int128)(uint64_t)rr_num[k] * P;
        int best = 0x7fffffff;
        unsigned __int128 best_err = ~(unsigned __int128)0;
        for (int j = lane; j < n_thr; j += 32) {
            const unsigned __int128 v = (unsigned __int128)c[j] * (unsigned)rr_den;
            const unsigned __int128 err = v > target ? v - target : target - v;
            if (err < best_err) {
                best_err = err;
                best = j;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {  // the smallest error, then the smallest j
            const uint64_t hi = __shfl_xor_sync(FULL, (uint64_t)(best_err >> 64), o);
            const uint64_t lo = __shfl_xor_sync(FULL, (uint64_t)best_err, o);
            const int bj = __shfl_xor_sync(FULL, best, o);
            const unsigned __int128 err = ((unsigned __int128)hi << 64) | lo;
            if (err < best_err || (err == best_err && bj < best)) {
                best_err = err;
                best = bj;
            }
        }
        if (lane == 0) {
            const int64_t o = (int64_t)s * K + k;
            eps_out[o] = thr[(int64_t)s * n_thr + best];
            if (rr_out) rr_out[o] = (double)c[best] / (double)P;
            if (count_out) count_out[o] = c[best];
        }
    }
}

cudaError_t launch_grid_select(const CellArgs &a, int S, int n_thr, float *thr, uint64_t *hist,
                               const int32_t *rr_num_dev, int rr_den, int K, float *eps_out,
                               double *rr_out, uint64_t *count_out, int grid, int embed,
                               cudaStream_t st)
{
    if (!a.y || !a.series || !a.order || !a.uprefix || !a.queue || a.n_units < 1 || a.n_pos < 1 ||
        a.m_max < 1 || a.nb < 1 || a.rc < RB || a.rc % RB || S < 1 || n_thr < 1 || n_thr > 1024 || !thr || !hist || !rr_num_dev || K < 1 || K > KMAX || !eps_out ||
        grid < 1)
        return cudaErrorInvalidValue;
    k_grid_thr<<<S, GT, 0, st>>>(a.y, a.series, n_thr, thr);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    void (*kern)(CellArgs, const float *, int, uint64_t *);
    int words = WIN_WORDS;
    switch (embed) {
    case E_M1T1: kern = k_count_grid<DiagSrc<1, 1>>; break;
    case E_M3T1: kern = k_count_grid<DiagSrc<3, 1>>; break;
    case E_M3T3: kern = k_count_grid<DiagSrc<3, 3>>; break;
    default:
        kern = a.m_max <= WinSrc::MAXM ? k_count_grid<WinSrc> : k_count_grid<GenSrc>;
        words = a.m_max <= WinSrc::MAXM ? WinSrc::WORDS : GenSrc::WORDS;
    }
    auto smem_of = [&](int n) { return ((GT / 32) * words + 2 * n + 3) * 4; };
    const int smem = smem_of(n_thr);
    if ((e = allow_smem(kern, smem_of(1024))) != cudaSuccess) return e;
    grid = persistent_cap(reinterpret_cast<const void *>(kern), smem, grid, GT);
    kern<<<grid, GT, smem, st>>>(a, thr, n_thr, hist);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    k_select_grid<<<S, GT, n_thr * 8, st>>>(hist, thr, a.series, n_thr, rr_num_dev, rr_den, K, eps_out,
                                            rr_out, count_out);
    return cudaGetLastError();
}

}  // namespace rqa
