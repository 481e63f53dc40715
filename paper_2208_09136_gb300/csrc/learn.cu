// The learned threshold bracket: distance sketch, a small FP32 network with
// its forward and backward passes, the pinball loss, Adam, and the step that
// turns predicted intervals into the coarse buckets the first counting round
// splits at once.  None of it affects a result, only how many counting
// passes the exact selection needs.
//
// The network is three dense layers on at most a few thousand rows, so the
// contractions are hand-tiled FP32 FFMA (32 x 32 output tiles, 4 x 4 per
// thread); at this size the tensor cores would not change the step time.
#include <cstdint>
#include "rqa_common.cuh"
#include <algorithm>
#include "rqa_learn_internal.h"

namespace rqa {

// ------------------------------------------------------------ SplitMix64
__device__ __forceinline__ uint64_t sm64_mix(uint64_t z)
{
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
constexpr uint64_t SM64_GAMMA = 0x9E3779B97F4A7C15ull;
constexpr uint64_t SERIES_MULT = 0xD1B54A32D192ED03ull;

// ------------------------------------------------------------ sketch
// One CTA per series: 4096 random pairs, their distances sorted in shared
// memory (bitonic network on the bit patterns), 128 quantiles, their logs.
// Bound by the latency of the network's 78 steps: 1024 threads take two
// exchanges each per step, and steps of stride <= 32 stay inside a warp's 64
// keys, so 28 of them end in a barrier of the CTA instead of all.
constexpr int SKETCH_T = 1024;
static_assert(SKETCH_PAIRS % (2 * SKETCH_T) == 0, "whole warps exchange in every step");
__global__ void __launch_bounds__(SKETCH_T)
k_sketch(const float *__restrict__ y, const SeriesDev *series, int s_base, uint64_t seed,
         float *feats, float *centre, float *qdist)
{
    __shared__ uint32_t keys[SKETCH_PAIRS];
    __shared__ float fl[SKETCH_BINS];
    const int s = s_base + blockIdx.x;
    const SeriesDev sd = series[s];
    const float *ys = y + sd.off;
    const uint64_t ks = sm64_mix(seed ^ ((uint64_t)(s + 1) * SERIES_MULT));
    for (int p = threadIdx.x; p < SKETCH_PAIRS; p += SKETCH_T) {
        const uint64_t a = sm64_mix(ks + (uint64_t)(2 * p + 1) * SM64_GAMMA);
        const uint64_t b = sm64_mix(ks + (uint64_t)(2 * p + 2) * SM64_GAMMA);
        const int i = (int)(a % (uint64_t)sd.ne);
        int j = (int)(b % (uint64_t)(sd.ne - 1));
        if (j >= i) ++j;
        float d = fabsf(ys[i] - ys[j]);
        for (int q = 1; q < sd.m; ++q)
            d = fmaxf(d, fabsf(ys[i + q * sd.tau] - ys[j + q * sd.tau]));
        keys[p] = __float_as_uint(d);
    }
    __syncthreads();
    // bitonic sort, ascending
    for (int size = 2; size <= SKETCH_PAIRS; size <<= 1) {
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
#pragma unroll
            for (int t = threadIdx.x; t < SKETCH_PAIRS / 2; t += SKETCH_T) {
                const int lo = 2 * t - (t & (stride - 1));
                const int hi = lo + stride;
                const bool up = (lo & size) == 0;
                const uint32_t x = keys[lo], z = keys[hi];
                if ((x > z) == up) {
                    keys[lo] = z;
                    keys[hi] = x;
                }
            }
            // the next step's stride: half of this one, or the next size's first
            if (stride > 32 || (stride > 1 ? stride >> 1 : size) > 32) __syncthreads();
            else __syncwarp();
        }
    }
    const int t = threadIdx.x;
    if (t < SKETCH_BINS) {
        const float q = __uint_as_float(keys[32 * t + 16]);
        if (qdist) qdist[(int64_t)s * SKETCH_BINS + t] = q;
        fl[t] = logf(fmaxf(q, 1.17549435e-38f));  // ln(max(q, 2^-126))
    }
    __syncthreads();
    const float c = fl[SKETCH_BINS / 2];
    float *f = feats + (int64_t)s * FEATURES;
    if (t < SKETCH_BINS) f[t] = fl[t] - c;
    if (t == 0) {
        f[128] = log10f((float)sd.n);
        f[129] = (float)sd.m;
        f[130] = (float)sd.tau;
        if (centre) centre[s] = c;
    }
}

cudaError_t launch_sketch(const float *y, const SeriesDev *series, int s_base, int S,
                          uint64_t seed, float *feats, float *centre, float *qdist, cudaStream_t st)
{
    if (!y || !series || !feats || S < 1) return cudaErrorInvalidValue;
    k_sketch<<<S, SKETCH_T, 0, st>>>(y, series, s_base, seed, feats, centre, qdist);
    return cudaGetLastError();
}

// ------------------------------------------------------------ GEMM
// C[M x N] = op(A) op(B) (+ bias[N]) (ReLU) (* [mask > 0]), row-major.
// op(A) is A [M x K] or, TA, A stored [K x M]; op(B) is B [K x N] or, TB,
// B stored [N x K].  rowsum (optional): the sums over K of op(A)'s rows (a
// bias gradient, whose operand the weight gradient reads anyway).
//
// The layers are far too small to fill the chip (256 x 256 x 256 is 0.5 us at
// the FP32 rate), so a GEMM is bound by the latency of its chain of loads: a
// 32 x 32 tile per CTA (64 CTAs at 256 x 256), panels of 128 values of K with
// all their loads in flight at once, and the K of a panel divided among four
// groups of 64 threads whose partial tiles are added at the end.  At 256 rows
// the eight GEMMs of a training step take 8 to 17 us each (cold caches), where
// 64 x 64 tiles with sixteen values of K per step took 12 to 48 us and the
// bias gradients three more launches of 16 us.
constexpr int GT = 32, GK = 128, GG = 4;  // tile, panel of K, groups of threads along K
static_assert(MLP_ROWS == 65535 * GT, "row tiles of a launch");

template <bool TA, bool TB>
__global__ void __launch_bounds__(256)
k_gemm(const float *__restrict__ A, const float *__restrict__ B, float *__restrict__ C, int M,
       int N, int K, const float *__restrict__ bias, bool relu, const float *__restrict__ mask,
       float *__restrict__ rowsum)
{
    __shared__ float As[GK][GT + 1];
    __shared__ float Bs[GK][GT + 1];
    const int t = threadIdx.x, g = t >> 6, tx = t & 7, ty = (t >> 3) & 7;
    const int m0 = blockIdx.y * GT, n0 = blockIdx.x * GT;
    float acc[4][4] = {}, rs[4] = {};
    for (int k0 = 0; k0 < K; k0 += GK) {
        float va[GK * GT / 256], vb[GK * GT / 256];
#pragma unroll
        for (int i = 0; i < GK * GT / 256; ++i) {
            const int e = t + 256 * i;
            // consecutive threads along the operand's contiguous direction
            const int ka = TA ? e / GT : e % GK, ma = TA ? e % GT : e / GK;
            const int kb = TB ? e % GK : e / GT, nb = TB ? e / GK : e % GT;
            va[i] = m0 + ma < M && k0 + ka < K
                        ? __ldg(A + (TA ? (int64_t)(k0 + ka) * M + m0 + ma : (int64_t)(m0 + ma) * K + k0 + ka)) : 0.f;
            vb[i] = n0 + nb < N && k0 + kb < K
                        ? __ldg(B + (TB ? (int64_t)(n0 + nb) * K + k0 + kb : (int64_t)(k0 + kb) * N + n0 + nb)) : 0.f;
        }
        __syncthreads();  // the panel before is used up
#pragma unroll
        for (int i = 0; i < GK * GT / 256; ++i) {
            const int e = t + 256 * i;
            As[TA ? e / GT : e % GK][TA ? e % GT : e / GK] = va[i];
            Bs[TB ? e % GK : e / GT][TB ? e / GK : e % GT] = vb[i];
        }
        __syncthreads();
        const int kn = min(GK, K - k0);
#pragma unroll 4
        for (int kk = g; kk < kn; kk += GG) {
            float a[4], b[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) a[r] = As[kk][ty + 8 * r];
#pragma unroll
            for (int q = 0; q < 4; ++q) b[q] = Bs[kk][tx + 8 * q];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                rs[r] += a[r];
#pragma unroll
                for (int q = 0; q < 4; ++q) acc[r][q] = fmaf(a[r], b[q], acc[r][q]);
            }
        }
    }
    // the four groups' partial tiles, one after the other through shared memory
    __shared__ float part[GG - 1][64][20];
    __syncthreads();
    if (g > 0) {
        float *p = part[g - 1][t & 63];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            p[16 + r] = rs[r];
#pragma unroll
            for (int q = 0; q < 4; ++q) p[4 * r + q] = acc[r][q];
        }
    }
    __syncthreads();
    if (g > 0) return;
#pragma unroll
    for (int h = 0; h < GG - 1; ++h) {
        const float *p = part[h][t];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            rs[r] += p[16 + r];
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[r][q] += p[4 * r + q];
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int gm = m0 + ty + 8 * r;
        if (gm >= M) continue;
        if (rowsum && blockIdx.x == 0 && tx == 0) rowsum[gm] = rs[r];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int gn = n0 + tx + 8 * q;
            if (gn >= N) continue;
            float v = acc[r][q];
            if (bias) v += bias[gn];
            if (relu) v = fmaxf(v, 0.f);
            if (mask && !(mask[(int64_t)gm * N + gn] > 0.f)) v = 0.f;
            C[(int64_t)gm * N + gn] = v;
        }
    }
}

static cudaError_t gemm(bool ta, bool tb, const float *A, const float *B, float *C, int M, int N,
                        int K, const float *bias, bool relu, const float *mask, float *rowsum, cudaStream_t st)
{
    // A launch's row tiles lie along gridDim.y, so more rows take more launches
    // (only the products over a minibatch's rows have that many, never op(A) = A^T).
    // All tiles along gridDim.x would need no loop, but the tile's division
    // changed the code for the worse: backward pass of 65536 rows 6.02 ms, 4.91 so.
    if (ta && M > MLP_ROWS) return cudaErrorInvalidValue;
    for (int64_t m0 = 0; m0 < M; m0 += MLP_ROWS) {
        const int rows = (int)std::min<int64_t>(M - m0, MLP_ROWS);
        const dim3 grid((N + GT - 1) / GT, (rows + GT - 1) / GT);
        const int64_t o = m0 * N;
        const float *a = A + m0 * K, *mk = mask ? mask + o : nullptr;
        if (ta) {
            k_gemm<true, false><<<grid, 256, 0, st>>>(A, B, C, M, N, K, bias, relu, mask, rowsum);
        } else if (tb) {
            k_gemm<false, true><<<grid, 256, 0, st>>>(a, B, C + o, rows, N, K, bias, relu, mk, rowsum);
        } else {
            k_gemm<false, false><<<grid, 256, 0, st>>>(a, B, C + o, rows, N, K, bias, relu, mk, rowsum);
        }
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Mean pinball loss of Y [B x 2K] against T [B x K] and its gradient.
__global__ void k_pinball(const float *__restrict__ Y, const float *__restrict__ T, int B, int K,
                          float tau_lo, float tau_hi, float *dY, float *loss)
{
    const int64_t n = (int64_t)B * 2 * K;
    const float inv = 1.f / (float)n;
    float part = 0.f;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = e / (2 * K);
        const int o = (int)(e % (2 * K));
        const float tau = (o & 1) ? tau_hi : tau_lo;
        const float r = T[b * K + (o >> 1)] - Y[e];
        part += (r >= 0.f) ? tau * r : (tau - 1.f) * r;
        dY[e] = ((r >= 0.f) ? -tau : 1.f - tau) * inv;
    }
    if (loss) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(FULL, part, o);
        if ((threadIdx.x & 31) == 0) atomicAdd(loss, part * inv);
    }
}

__global__ void k_adam(float *p, const float *__restrict__ g, float *m, float *v, int64_t n,
                       float lr, float b1, float b2, float eps, float c1, float c2)
{
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const float ge = g[e];
        const float me = b1 * m[e] + (1.f - b1) * ge;
        const float ve = b2 * v[e] + (1.f - b2) * ge * ge;
        m[e] = me;
        v[e] = ve;
        p[e] -= lr * (me / c1) / (sqrtf(ve / c2) + eps);
    }
}

// Parameter blocks inside the flat vector.
struct MlpView {
    const float *W1, *b1, *W2, *b2, *W3, *b3;
};
__host__ __device__ inline MlpView mlp_view(const float *p)
{
    MlpView v;
    v.W1 = p;
    v.b1 = v.W1 + HIDDEN * FEATURES;
    v.W2 = v.b1 + HIDDEN;
    v.b2 = v.W2 + HIDDEN * HIDDEN;
    v.W3 = v.b2 + HIDDEN;
    v.b3 = v.W3 + MLP_OUT * HIDDEN;
    return v;
}

cudaError_t mlp_forward(const float *params, const float *X, int B, float *Y, float *acts,
                        cudaStream_t st)
{
    const MlpView v = mlp_view(params);
    float *H1 = acts, *H2 = acts + (int64_t)B * HIDDEN;
    cudaError_t e;
    if ((e = gemm(false, true, X, v.W1, H1, B, HIDDEN, FEATURES, v.b1, true, nullptr, nullptr, st))) return e;
    if ((e = gemm(false, true, H1, v.W2, H2, B, HIDDEN, HIDDEN, v.b2, true, nullptr, nullptr, st))) return e;
    return gemm(false, true, H2, v.W3, Y, B, MLP_OUT, HIDDEN, v.b3, false, nullptr, nullptr, st);
}

cudaError_t mlp_backward(const float *params, const float *X, const float *acts, const float *Y,
                         const float *T, int B, float tau_lo, float tau_hi, float *grads,
                         float *loss, float *scratch, cudaStream_t st)
{
    const MlpView v = mlp_view(params);
    const float *H1 = acts, *H2 = acts + (int64_t)B * HIDDEN;
    float *gW1 = grads, *gb1 = gW1 + HIDDEN * FEATURES, *gW2 = gb1 + HIDDEN,
          *gb2 = gW2 + HIDDEN * HIDDEN, *gW3 = gb2 + HIDDEN, *gb3 = gW3 + MLP_OUT * HIDDEN;
    float *dY = scratch, *dZ2 = dY + (int64_t)B * MLP_OUT, *dZ1 = dZ2 + (int64_t)B * HIDDEN;
    cudaError_t e;
    if (loss && (e = cudaMemsetAsync(loss, 0, sizeof(float), st))) return e;
    const int64_t n = (int64_t)B * MLP_OUT;
    k_pinball<<<(int)std::min<int64_t>((n + 255) / 256, 1024), 256, 0, st>>>(
        Y, T, B, MLP_OUT / 2, tau_lo, tau_hi, dY, loss);
    if ((e = cudaGetLastError())) return e;
    // each layer: weight and bias gradients in one launch, then the gradient
    // of its input
    if ((e = gemm(true, false, dY, H2, gW3, MLP_OUT, HIDDEN, B, nullptr, false, nullptr, gb3, st))) return e;
    if ((e = gemm(false, false, dY, v.W3, dZ2, B, HIDDEN, MLP_OUT, nullptr, false, H2, nullptr, st))) return e;
    if ((e = gemm(true, false, dZ2, H1, gW2, HIDDEN, HIDDEN, B, nullptr, false, nullptr, gb2, st))) return e;
    if ((e = gemm(false, false, dZ2, v.W2, dZ1, B, HIDDEN, HIDDEN, nullptr, false, H1, nullptr, st))) return e;
    if ((e = gemm(true, false, dZ1, X, gW1, HIDDEN, FEATURES, B, nullptr, false, nullptr, gb1, st))) return e;
    return cudaGetLastError();
}

cudaError_t adam_step(float *p, const float *g, float *m, float *v, int64_t n, int t, float lr,
                      float b1, float b2, float eps, cudaStream_t st)
{
    const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
    k_adam<<<(int)std::min<int64_t>((n + 255) / 256, 2048), 256, 0, st>>>(p, g, m, v, n, lr, b1, b2,
                                                                          eps, c1, c2);
    return cudaGetLastError();
}

// ------------------------------------------------------------ training data
// Labels of the network: T[s][k] = ln(max(eps[s][k], 2^-126)) - c[s], the
// thresholds in the centred log scale of the sketch features.
__global__ void k_log_labels(const float *__restrict__ eps, const float *__restrict__ centre, int S,
                             int K, float *__restrict__ T)
{
    const int64_t n = (int64_t)S * K;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x)
        T[e] = logf(fmaxf(eps[e], 0x1p-126f)) - centre[e / K];
}

cudaError_t launch_log_labels(const float *eps, const float *centre, int S, int K, float *T,
                              cudaStream_t st)
{
    const int64_t n = (int64_t)S * K;
    k_log_labels<<<(int)std::min<int64_t>((n + 255) / 256, 1024), 256, 0, st>>>(eps, centre, S, K, T);
    return cudaGetLastError();
}

// Validation of a bracket network over B rows: the summed pinball loss of the
// 2K outputs (lower ends at tau_lo, upper at tau_hi), the targets inside
// [lo - margin, hi + margin] and the summed width hi - lo + 2 margin.
__global__ void k_bracket_eval(const float *__restrict__ Y, const float *__restrict__ T, int B,
                               int K, float tau_lo, float tau_hi, float margin, double *loss_sum,
                               unsigned long long *inside, double *width_sum)
{
    double l = 0.0, w = 0.0;
    unsigned long long in = 0;
    const int64_t n = (int64_t)B * K;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t b = e / K;
        const int k = (int)(e % K);
        const float t = T[e];
        const float lo = Y[b * 2 * K + 2 * k], hi = Y[b * 2 * K + 2 * k + 1];
        const float rl = t - lo, rh = t - hi;
        l += (double)((rl >= 0.f) ? tau_lo * rl : (tau_lo - 1.f) * rl);
        l += (double)((rh >= 0.f) ? tau_hi * rh : (tau_hi - 1.f) * rh);
        in += (t >= lo - margin && t <= hi + margin) ? 1ull : 0ull;
        w += (double)((hi + margin) - (lo - margin));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        l += __shfl_xor_sync(FULL, l, o);
        w += __shfl_xor_sync(FULL, w, o);
        in += __shfl_xor_sync(FULL, in, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(loss_sum, l);
        atomicAdd(width_sum, w);
        atomicAdd(inside, in);
    }
}

cudaError_t launch_bracket_eval(const float *Y, const float *T, int B, int K, float tau_lo,
                                float tau_hi, float margin, double *loss_sum,
                                unsigned long long *inside, double *width_sum, cudaStream_t st)
{
    cudaError_t e;
    if ((e = cudaMemsetAsync(loss_sum, 0, sizeof(double), st))) return e;
    if ((e = cudaMemsetAsync(width_sum, 0, sizeof(double), st))) return e;
    if ((e = cudaMemsetAsync(inside, 0, sizeof(unsigned long long), st))) return e;
    const int64_t n = (int64_t)B * K;
    k_bracket_eval<<<(int)std::min<int64_t>((n + 255) / 256, 512), 256, 0, st>>>(
        Y, T, B, K, tau_lo, tau_hi, margin, loss_sum, inside, width_sum);
    return cudaGetLastError();
}

// dst row r = src row idx[r], rows of `width` floats (a minibatch gather).
__global__ void k_gather_rows(const float *__restrict__ src, const int64_t *__restrict__ idx, int n,
                              int width, float *__restrict__ dst)
{
    const int64_t total = (int64_t)n * width;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e / width;
        dst[e] = src[idx[r] * width + (e - r * width)];
    }
}

cudaError_t launch_gather_rows(const float *src, const int64_t *idx, int n, int width, float *dst,
                               cudaStream_t st)
{
    const int64_t total = (int64_t)n * width;
    k_gather_rows<<<(int)std::min<int64_t>((total + 255) / 256, 2048), 256, 0, st>>>(src, idx, n, width, dst);
    return cudaGetLastError();
}

// ------------------------------------------------------------ bracket
// Coarse buckets to split in the first counting round.  Per target the
// interval runs from the bucket of exp(c + lo - margin) to that of
// exp(c + hi + margin).  If all of them fit in NSUB_MAX buckets, every bucket
// from the lowest to the highest end is split (and up to two below); else the
// buckets nearest each target's middle bucket first, then the narrowest gaps
// between split buckets.  Keys between the first and the last split bucket
// are counted either way (unsplit buckets at coarse resolution).  One thread
// marks them (a few dozen steps); all 256 number the marks, eight buckets each,
// instead of one thread over the table's 2048 entries (with the sketch above:
// bracket phase of four series of 1e4 225 -> 191 us).
constexpr int BRACKET_T = 256;
static_assert(NCOARSE == 8 * BRACKET_T, "eight buckets per thread");
__global__ void __launch_bounds__(BRACKET_T)
k_bracket(const float *__restrict__ Yb, const float *__restrict__ centre,
                          float margin, int K, const uint8_t *__restrict__ dom, int8_t *tab_sub,
                          int32_t *n_sub, uint32_t *range)
{
    __shared__ uint16_t lo_b[KMAX], hi_b[KMAX], mid_b[KMAX];
    __shared__ __align__(8) int8_t tb[NCOARSE];
    __shared__ int wsum[BRACKET_T / 32];
    const int s = blockIdx.x;
    if (!dom[s]) {  // outside the network's domain: the full selection takes it
        int8_t *tab = tab_sub + (int64_t)s * NCOARSE;
        for (int x = threadIdx.x; x < NCOARSE; x += blockDim.x) tab[x] = -1;
        if (threadIdx.x == 0) {
            n_sub[s] = 0;
            range[2 * s] = 0xffffffffu;
            range[2 * s + 1] = 0u;
        }
        return;
    }
    for (int x = threadIdx.x; x < NCOARSE; x += blockDim.x) tb[x] = -1;
    if (threadIdx.x < K) {
        const float c = centre[s];
        float lo = Yb[(int64_t)s * MLP_OUT + 2 * threadIdx.x] - margin;
        float hi = Yb[(int64_t)s * MLP_OUT + 2 * threadIdx.x + 1] + margin;
        if (!(lo <= hi)) {  // crossed or NaN ends: a narrow interval around their mean
            float mm = 0.5f * (lo + hi);
            if (!(mm == mm)) mm = 0.f;
            lo = mm - margin;
            hi = mm + margin;
        }
        auto bucket = [](float ln_v) {
            const float v = expf(fminf(fmaxf(ln_v, -87.f), 88.f));
            return (uint16_t)(__float_as_uint(v) >> COARSE_SHIFT);
        };
        lo_b[threadIdx.x] = bucket(c + lo);
        hi_b[threadIdx.x] = bucket(c + hi);
        mid_b[threadIdx.x] = bucket(c + 0.5f * (lo + hi));
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int lo_all = NCOARSE, hi_all = -1;
        for (int k = 0; k < K; ++k) {
            lo_all = min(lo_all, (int)lo_b[k]);
            hi_all = max(hi_all, (int)hi_b[k]);
        }
        const int span = hi_all - lo_all + 1;
        if (span <= NSUB_MAX) {
            // every bucket from the lowest to the highest interval end: a
            // threshold between two targets' intervals is found too; up to
            // two more buckets below (they hold few keys)
            const int a = max(0, lo_all - min(2, NSUB_MAX - span));
            for (int b = a; b <= hi_all; ++b) tb[b] = 0;
        } else {
            // rings around each target's most likely bucket, inside its
            // interval, all targets alike, until the split budget is spent
            int used = 0, first = NCOARSE - 1, last = 0;  // marked buckets
            for (int r = 0; used < NSUB_MAX; ++r) {
                bool any = false;
                for (int k = 0; k < K; ++k) {
                    for (int side = -1; side <= 1; side += 2) {
                        if (r == 0 && side > 0) continue;
                        const int b = (int)mid_b[k] + side * r;
                        if (b < (int)lo_b[k] || b > (int)hi_b[k]) continue;
                        any = true;
                        if (tb[b] != 0 && used < NSUB_MAX) {
                            tb[b] = 0;
                            ++used;
                            first = min(first, b);
                            last = max(last, b);
                        }
                    }
                }
                if (!any) break;
            }
            // the rest of the budget closes the narrowest gaps between them
            for (;;) {
                int best_a = -1, best_n = NCOARSE;
                for (int b = first; b <= last; ++b) {
                    if (tb[b] == 0) continue;
                    int e = b;
                    while (tb[e] != 0) ++e;  // tb[last] is marked: ends inside
                    if (e - b < best_n) {
                        best_n = e - b;
                        best_a = b;
                    }
                    b = e;
                }
                if (best_a < 0 || used + best_n > NSUB_MAX) break;
                for (int b = best_a; b < best_a + best_n; ++b) tb[b] = 0;
                used += best_n;
            }
        }
    }
    __syncthreads();
    // marked buckets numbered in ascending order; keys the bracket round counts:
    // from its first to its last split bucket
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint2 eight = *reinterpret_cast<const uint2 *>(tb + 8 * t);
    bool mark[8];
    int own = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        mark[i] = (((i < 4 ? eight.x : eight.y) >> (8 * (i & 3))) & 0xffu) == 0u;
        own += mark[i] ? 1 : 0;
    }
    int incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(FULL, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int g = incl - own, total = 0;
    for (int w = 0; w < BRACKET_T / 32; ++w) {
        if (w < warp) g += wsum[w];
        total += wsum[w];
    }
    total = min(total, NSUB_MAX);
    int8_t *tab = tab_sub + (int64_t)s * NCOARSE;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const bool in = mark[i] && g < total;
        const uint32_t b = (uint32_t)(8 * t + i);
        tab[b] = in ? (int8_t)g : (int8_t)-1;
        if (in && g == 0) range[2 * s] = b << COARSE_SHIFT;
        if (in && g == total - 1) range[2 * s + 1] = ((b + 1u) << COARSE_SHIFT) - 1u;
        g += mark[i] ? 1 : 0;
    }
    if (t == 0) {
        n_sub[s] = total;
        if (total == 0) {
            range[2 * s] = 0xffffffffu;
            range[2 * s + 1] = 0u;
        }
    }
}

cudaError_t launch_bracket(const float *Y, const float *centre, float margin, int S, int K,
                           const uint8_t *dom, int8_t *tab_sub, int32_t *n_sub, uint32_t *range,
                           cudaStream_t st)
{
    if (!dom) return cudaErrorInvalidValue;
    k_bracket<<<S, BRACKET_T, 0, st>>>(Y, centre, margin, K, dom, tab_sub, n_sub, range);
    return cudaGetLastError();
}

// Hits and misses of a bracketed selection: a target hit when its key
// prefix was fixed by the split round (level 2 right after it); series
// outside the network's domain (dom[s] == 0) are not counted.
__global__ void k_bracket_stats(const uint8_t *level, const uint8_t *dom, int S, int K,
                                unsigned long long *hm)
{
    unsigned long long h = 0, m = 0;
    const int64_t n = (int64_t)S * K;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        if (!dom[e / K]) continue;
        if (level[e] == 2) ++h;
        else ++m;
    }
    atomicAdd(hm, h);
    atomicAdd(hm + 1, m);
}

cudaError_t launch_bracket_stats(const uint8_t *level, const uint8_t *dom, int S, int K,
                                 unsigned long long *hm, cudaStream_t st)
{
    if (!dom || S < 1 || K < 1) return cudaErrorInvalidValue;
    const int64_t n = (int64_t)S * K;
    k_bracket_stats<<<(int)std::min<int64_t>((n + 255) / 256, 256), 256, 0, st>>>(level, dom, S, K, hm);
    return cudaGetLastError();
}

}  // namespace rqa
