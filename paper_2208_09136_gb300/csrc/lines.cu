// Line pass launches: the kernel variant for the batch's embedding on a
// persistent grid (the kernel is in lines_kernel.cuh, its instantiations in
// lines_*.cu).
#include <algorithm>

#include "lines_kernel.cuh"

namespace rqa {


// The kernel of an embedding variant (full: a sweep of LINE_KMAX thresholds,
// which the special embeddings' diagonal pass has its own variant for).
static LinesKernel lines_kernel(int embed, bool vert, bool full)
{
    switch (embed) {
    case E_M3T3: return lines_kernel_m3t3(vert, full);
    case E_M3T1: return lines_kernel_m3t1(vert, full);
    case E_M1T1: return lines_kernel_m1t1(vert, full);
    case E_M2: case E_M3: case E_M4: return lines_kernel_generic(embed, vert);
    default: return lines_kernel_generic(0, vert);
    }
}

// Join the lines that meet at the chunk boundaries of a band: a thread per
// diagonal and threshold walks down the band's chunks.  Where the last row of
// one chunk and the first row of the next are both recurrent, the two counted
// pieces x and y are one line of length x + y; a piece as long as its chunk
// goes on to the next boundary.  The cells of the lines stay the same, so C_k
// does.  Only edge lengths that k_lines wrote in this launch are read: it writes
// none for a series that it skips.
//
// Bound by the latency of a band's loads and of the atomics at the end, so the
// bands that have boundaries (CellArgs::mprefix) are spread over all CTAs, each
// taking a run of them, whatever series they are of, and flushing once per
// series.  (With the same number of CTAs for every series the long one of a mixed
// batch was joined by a single CTA: line pass of one series of 10^4 and 1000 of
// 300, 2.01 ms, 0.29 so; one of 5 10^4 and 500 of 100, 6.24 and 2.79; 4 of 10^4
// alike.)
constexpr int MERGE_CTAS = 6;  // per SM, two of them resident
template <bool VERT>
__global__ void __launch_bounds__(LD * KT, 2) k_merge(CellArgs a, LineBufs lb, int K, const uint16_t *edges)
{
    __shared__ uint32_t net[LSH][KT];  // changes of P_k(1..LSH) of the current series
    __shared__ uint32_t lmx[KT];
    const int t = threadIdx.x, lane = t % LD, k = t / LD;
    // n MERGE_CTAS SMs < 2^32: cut bands are fewer than 8 per resident warp
    const uint32_t n = (uint32_t)a.n_merge;
    int f = (int)(n * blockIdx.x / gridDim.x);
    const int f_end = (int)(n * (blockIdx.x + 1) / gridDim.x);
    int pos = 0;  // the last with mprefix[pos] <= f, counted by all threads together
    for (int p0 = 1; p0 < a.n_pos; p0 += LD * KT)
        pos += __syncthreads_count(p0 + t < a.n_pos && a.mprefix[p0 + t] <= f);
    for (int i = t; i < LSH * KT; i += LD * KT) (&net[0][0])[i] = 0;
    if (t < KT) lmx[t] = 0;
    while (f < f_end) {
        const int f0 = (int)a.mprefix[pos], f1 = min((int)a.mprefix[pos + 1], f_end);
        const int s = a.order[pos], ne = a.series[s].ne;
        const int64_t o = (int64_t)s * lb.kstride + lb.k0;
        const int hrow = ne - 1 + (VERT && lb.loi ? 1 : 0);
        auto add = [&](int len, bool more) {
            if (len > hrow) {
                set_status(a.status, 10 /*INTERNAL*/);
            } else if (len <= LSH) {
                atomicAdd(&net[len - 1][k], more ? 1u : ~0u);
            } else if (lb.hist) {
                uint64_t *const h = lb.hist + lb.hist_off[s] + (int64_t)(lb.k0 + k) * hrow + (len - 1);
                atomicAdd(reinterpret_cast<unsigned long long *>(h), more ? 1ull : ~0ull);
            }
        };
        bool ok = true;
        if (t < K) {
            const uint32_t v = threshold_key(lb.eps[o + t]);
            ok = threshold_ok(v) && (t == 0 || threshold_key(lb.eps[o + t - 1]) <= v);
        }
        const bool skipped = __syncthreads_or(!ok);  // by k_lines
        for (; f < f1; ++f) {
            if (skipped || k >= K) continue;
            const int b = f - f0, rows = VERT ? ne : ne - 1 - b * LD;
            int64_t base = a.uprefix[pos];  // first unit of the chunk
            int open = 0;                   // length up to the boundary of the line that touches it
            for (int r0 = 0; r0 < rows; r0 += a.rc) {
                const uint16_t *e = edges + ((base + b / a.nb) * a.nb + b % a.nb) * (2 * KT * LD) + k * LD + lane;
                const int y = r0 ? e[0] : 0;
                int z = r0 + a.rc < rows ? e[KT * LD] : 0;
                if (open && y) {
                    add(open, false);
                    add(y, false);
                    add(open + y, true);
                    atomicMax(&lmx[k], (uint32_t)(open + y));
                    if (z == a.rc) z += open;  // the whole chunk
                }
                open = z;
                const int bands = VERT ? (ne + LD - 1) / LD : (ne - 1 - r0 + LD - 1) / LD;
                base += (bands + a.nb - 1) / a.nb;
            }
        }
        __syncthreads();
        for (int i = t; i < LSH * KT; i += LD * KT) {
            const int l = i / KT, q = i - l * KT;
            const int32_t v = (int32_t)net[l][q];
            if (v) {
                atomicAdd(reinterpret_cast<unsigned long long *>(lb.hshort + (o + q) * LSH + l),
                          (unsigned long long)(long long)v);
                net[l][q] = 0;
            }
        }
        if (t < KT && lmx[t]) {
            atomicMax(lb.lmax + o + t, lmx[t]);
            lmx[t] = 0;
        }
        ++pos;
    }
}

template <bool VERT>
static cudaError_t launch_lines_v(const CellArgs &a, const LineBufs &lb, int K, int grid, int embed,
                                  bool chunks, uint16_t *edges, cudaStream_t st)
{
    if (!a.y || !a.series || !a.order || !a.uprefix || !a.queue || !a.status || !lb.eps ||
        !lb.count || !lb.lmax || !lb.hshort || (lb.hist && !lb.hist_off) || K < 1 ||
        K > LINE_KMAX || lb.k0 < 0 || lb.k0 + K > lb.kstride || grid < 1 || a.n_units < 1 ||
        a.n_pos < 1 || a.nb < 1 || a.rc < 32 || a.rc % 32 || (chunks && (!edges || !a.mprefix || a.n_merge < 1)))
        return cudaErrorInvalidValue;
    LinesKernel kern = lines_kernel(embed, VERT, K == LINE_KMAX);
    const int smem = lines_smem_bytes();
    cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    grid *= WARPS / LWARPS;  // the caller counts CTAs of WARPS warps
    grid = persistent_cap(reinterpret_cast<const void *>(kern), smem, grid, LTHREADS);
    if (a.line_ctas > 0) grid = std::min(grid, sm_count_current() * a.line_ctas);
    kern<<<grid, LTHREADS, smem, st>>>(a, lb, K, edges);
    if ((e = cudaGetLastError()) != cudaSuccess || !chunks) return e;
    const int mg = (int)std::min<int64_t>(a.n_merge, sm_count_current() * MERGE_CTAS);
    k_merge<VERT><<<mg, LD * KT, 0, st>>>(a, lb, K, edges);
    return cudaGetLastError();
}

cudaError_t launch_lines(const CellArgs &a, const LineBufs &lb, int K, int grid, int embed, bool vert,
                         bool chunks, uint16_t *edges, cudaStream_t st)
{
    return vert ? launch_lines_v<true>(a, lb, K, grid, embed, chunks, edges, st)
                : launch_lines_v<false>(a, lb, K, grid, embed, chunks, edges, st);
}

}  // namespace rqa
