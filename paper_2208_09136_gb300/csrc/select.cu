// Exact selection of the thresholds that give the chosen recurrence rates
// (Sect. 2: RR is fixed first and eps follows from it; Eq. 3).
//
// eps_k is the T_k-th smallest upper-triangle distance.  Distances are never
// stored: every counting round recomputes them over diagonal bands and
// histograms one digit of their FP32 bit pattern (the "key"; non-negative
// floats order like their bit patterns).  Rounds:
//   R_COARSE      bits 30..20 of every key                    -> 2048 bins
//   R_COARSE_SUB  as R_COARSE, but coarse buckets a learned bracket marks are
//                 split at once by bits 19..10 (skips R_MID for those targets)
//   R_MID         bits 19..10 of keys in a target's coarse bucket
//   R_FINAL       bits 9..0 of keys in a target's 21-bit prefix
// After each round a select kernel turns the histogram into (prefix, rank,
// below) per target.  After R_FINAL the key is complete: eps_k, and
// #{d < eps_k} = below, #{d <= eps_k} = below + (keys equal to eps_k).
#include <cstdint>
#include <type_traits>
#include "dense.cuh"

namespace rqa {

// ------------------------------------------------------------ finiteness
__global__ void k_check_finite(const float *__restrict__ y, int64_t n, int *status)
{
    int bad = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        bad |= !isfinite(y[i]);
    if (__any_sync(FULL, bad) && (threadIdx.x & 31) == 0) set_status(status, 3 /*NONFINITE*/);
}

cudaError_t launch_check_finite(const float *y, int64_t n, int *status, cudaStream_t st)
{
    if (n <= 0) return cudaSuccess;
    int64_t blocks = (n + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    k_check_finite<<<(int)blocks, 256, 0, st>>>(y, n, status);
    return cudaGetLastError();
}

// ------------------------------------------------------------ counting
// Dynamic shared memory of a counting CTA: the warps' windows, the bins
// (32-bit) and the lookup table of its round.
constexpr int CT = 256;        // threads per CTA
constexpr int CW = CT / 32;
constexpr int SUB_WIN = 512;   // coarse buckets of a sparse bracket round counted in shared memory
constexpr int DENSE_FINAL = 48 * NFINE;  // prefixes the final round's byte table can span

static int count_bins(int round, int K)
{
    switch (round) {
    case R_COARSE: return NCOARSE;
    case R_COARSE_SUB: return SUB_WIN + NSUB_MAX * NFINE;
    case R_MID: {
        const int g = K < MID_GROUPS ? K : MID_GROUPS;
        return (g > NSUB_MAX ? g : NSUB_MAX) * NFINE + 4;  // dense: a bin below and one above the range
    }
    default: return 0;
    }
}

static int count_smem_bytes(int round, int K, int win_words)
{
    const int win = CW * win_words * 4;
    switch (round) {
    case R_COARSE: return win + NCOARSE * 4;
    case R_COARSE_SUB: case R_MID: return win + count_bins(round, K) * 4 + NCOARSE;
    default: return win + (DENSE_FINAL + 16 > NHASH * 4 ? DENSE_FINAL + 16 : NHASH * 4);
    }
}

// One persistent launch over the work units.  A CTA keeps the bins of one
// series in shared memory over all the units of it that it takes and adds
// the non-zero ones to the series' 64-bit global histogram when the series
// changes (or before a 32-bit bin could overflow).
//
// Bins of a cell:
//   R_COARSE      key >> 20.
//   split ranges  (bracket round; middle round when the targets' coarse
//                 buckets span at most NSUB_MAX) the 21-bit prefix relative to
//                 the range, clamped to one bin below and one above it: a
//                 shift, one DPX clamp and one unconditional reduction per
//                 cell.  The hardware merges the lanes that meet in a bin, so
//                 the crowded outer bins cost nothing (measured: 2.1 cycles
//                 per SM and warp reduction with 80 % of the lanes in one
//                 bin, 2.5 with all lanes spread; a predicated reduction of
//                 20 % of the lanes 4.2).
//   other ranges  through the group table of the coarse buckets.
//   R_FINAL       keys of a target's 21-bit prefix are rare and go straight
//                 to the global bins: the prefix relative to the range is
//                 looked up in a byte table (spans up to DENSE_FINAL), else
//                 in a hashed table (slot = prefix x multiplier >> 20; the
//                 slot holds the only target prefix that can map there), else
//                 by binary search.
//
// Bound by shared-memory reductions and issue: one reduction and 5 to 9
// instructions per cell (32 cells: per warp).  Units are row chunks of a few
// bands (dense.cuh), so a batch of four 10^4-value series fills the chip.
template <int ROUND, class Src>
__global__ void __launch_bounds__(CT, 2) k_count(CellArgs a, SelBufs sb, int K, int nbins)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ Unit unit;
    __shared__ int next_part, unit_rows;
    __shared__ uint32_t sink[32];  // lane x's reductions of cells that count nowhere (never read)
    __shared__ uint32_t pfx[KMAX + 1];  // final round: the distinct target prefixes, ascending
    __shared__ int n_pfx;
    __shared__ unsigned fbits[4];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *win = reinterpret_cast<uint32_t *>(smem) + warp * Src::WORDS;
    uint32_t *h = reinterpret_cast<uint32_t *>(smem) + CW * Src::WORDS;
    int8_t *t1 = reinterpret_cast<int8_t *>(h + nbins);                   // sparse ranges
    unsigned char *t8 = reinterpret_cast<unsigned char *>(h);             // final round, byte table
    uint32_t *th = h;                                                     // final round, hashed table

    for (int x = threadIdx.x; x < nbins; x += CT) h[x] = 0;

    int cur = -1;
    bool busy = false;              // the current series has work in this round
    uint64_t acc = 0;               // cells counted since the last flush
    uint32_t klo = 0, kspan = 0;    // key range of the filtered rounds: key - klo <= kspan
    int nfine = 0;                  // bins of the series' groups in this launch
    bool dense = false;
    uint32_t hmul = 0;
    uint64_t below = 0;             // sparse bracket round: this lane's keys under the range
    int32_t qoff = 0, qtop = 0;     // dense: clamp of the relative prefix

    auto flush = [&]() {
        if (cur < 0 || !busy || ROUND == R_FINAL) return;
        __syncthreads();
        unsigned long long *gh =
            reinterpret_cast<unsigned long long *>(sb.hist + (int64_t)cur * sb.hstride);
        auto add = [&](unsigned long long *dst, int x) {
            const uint32_t v = h[x];
            if (v) {
                if (dst) atomicAdd(dst, (unsigned long long)v);
                h[x] = 0;
            }
        };
        const int clo = (int)(klo >> COARSE_SHIFT);
        if (ROUND == R_COARSE) {
            for (int x = threadIdx.x; x < NCOARSE; x += CT) add(gh + x, x);
        } else if (dense) {
            // bin 0: keys under the range; they only count in the bracket
            // round, kept in the coarse bucket just below it
            for (int x = threadIdx.x; x < nfine + 2; x += CT) {
                unsigned long long *dst = gh + NCOARSE + x - 1;
                if (x == 0) dst = ROUND == R_COARSE_SUB && clo > 0 ? gh + clo - 1 : nullptr;
                if (x == nfine + 1) dst = nullptr;
                add(dst, x);
            }
        } else if (ROUND == R_COARSE_SUB) {
            for (int x = threadIdx.x; x < SUB_WIN; x += CT) add(clo + x < NCOARSE ? gh + clo + x : nullptr, x);
            for (int x = threadIdx.x; x < nfine; x += CT) add(gh + NCOARSE + x, SUB_WIN + x);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) below += __shfl_xor_sync(FULL, below, o);
            if (lane == 0 && below && clo > 0) atomicAdd(gh + clo - 1, (unsigned long long)below);
            below = 0;
        } else {
            for (int x = threadIdx.x; x < nfine; x += CT) add(gh + NCOARSE + (int64_t)a.g0 * NFINE + x, x);
        }
        acc = 0;
        __syncthreads();
    };

    for (;;) {
        __syncthreads();  // every warp done with the unit before
        if (threadIdx.x == 0) {
            const unsigned t = atomicAdd(a.queue, 1u);
            if ((int64_t)t < a.n_units) {
                unit = unit_of<false>(a, (int64_t)t);
                next_part = 0;
                unit_rows = part_rows(unit, CW);
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
            if (ROUND == R_COARSE) {
                busy = sb.redo[cur] != 0;
            } else {
                klo = sb.range[2 * (int64_t)cur];
                kspan = sb.range[2 * (int64_t)cur + 1] - klo;
                const int ng = ROUND == R_COARSE_SUB ? sb.n_sub[cur]
                             : ROUND == R_MID ? max(0, min(sb.n_mid[cur] - a.g0, a.gn)) : sb.n_fin[cur];
                nfine = ng * NFINE;
                busy = ng > 0;
                // every coarse bucket of the range is a group of its own, in order
                dense = (kspan >> COARSE_SHIFT) + 1u == (uint32_t)ng && ng <= NSUB_MAX && a.g0 == 0;
                if (ROUND == R_FINAL) {
                    nfine = (int)(kspan >> 10) + 1;
                    dense = kspan < (uint32_t)DENSE_FINAL << 10;
                }
                qoff = 1 - (int32_t)(klo >> 10);
                qtop = nfine + 1;
            }
            if (busy && ROUND == R_FINAL) {
                // the targets' prefixes ascend: one entry per run of equal ones
                const int k = threadIdx.x;
                uint32_t p = 0;
                bool first = false;
                if (k < K) {
                    const uint32_t *pk = sb.prefix + (int64_t)cur * K + k;
                    p = pk[0];
                    first = k == 0 || pk[-1] != p;
                }
                const unsigned fb = __ballot_sync(FULL, first);
                if (lane == 0 && warp < 4) fbits[warp] = fb;
                __syncthreads();
                if (k < 128) {
                    int g = __popc(fb & ((1u << lane) - 1u));
                    for (int x = 0; x < warp; ++x) g += __popc(fbits[x]);
                    if (first) pfx[g] = p;
                    if (k == 127) n_pfx = g + (first ? 1 : 0);
                }
                hmul = !dense && sb.hash_mul ? sb.hash_mul[cur] : 0u;
                if (dense) {
                    for (int x = threadIdx.x; x < (nfine + 2 + 3) / 4; x += CT) h[x] = 0;
                } else if (hmul) {
                    const uint4 *src = reinterpret_cast<const uint4 *>(sb.tab_hash + (int64_t)cur * NHASH);
                    for (int x = threadIdx.x; x < NHASH / 4; x += CT) reinterpret_cast<uint4 *>(th)[x] = src[x];
                }
                __syncthreads();
                if (dense && (int)threadIdx.x < n_pfx)
                    t8[(int32_t)pfx[threadIdx.x] + qoff] = (unsigned char)(threadIdx.x + 1);
                __syncthreads();
            } else if (busy && ROUND != R_COARSE && !dense) {
                const int8_t *src = (ROUND == R_COARSE_SUB ? sb.tab_sub : sb.tab_mid) + (int64_t)cur * NCOARSE;
                for (int x = threadIdx.x; x < NCOARSE; x += CT) t1[x] = src[x];
                __syncthreads();
            }
        }
        if (!busy) continue;  // no target of this series needs this round
        const uint64_t cells = (uint64_t)(w.b_hi - w.b_lo) * DB * (uint64_t)(w.r_hi - w.r_lo);
        if (acc + cells > 0xffffffffull) flush();  // 32-bit bins stay exact
        acc += cells;

        unsigned long long *gbins =
            reinterpret_cast<unsigned long long *>(sb.hist + (int64_t)cur * sb.hstride + NCOARSE);
        const uint32_t sink_a = static_cast<uint32_t>(__cvta_generic_to_shared(&sink[lane]));
        const uint32_t h_a = static_cast<uint32_t>(__cvta_generic_to_shared(h));
        Src src;
        src.init(a.y + sd.off, sd, lane, win);
        auto bands = [&](auto &&f) {
            each_part(unit, unit_rows, &next_part, lane,
                      [&](int d0, int r_lo, int r_hi) { walk_keys(src, sd.ne, d0, r_lo, r_hi, lane, f); });
        };
        // f(key, ok) for the sixteen cells of a step, one after the other
        auto each = [&](auto &&f) {
            bands([&](const float (&d)[4][DPL], auto valid) {
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int j = 0; j < DPL; ++j) f(__float_as_uint(d[r][j]), valid(r, j));
            });
        };
        // keys of finite or NaN distances have bit 31 clear, so key >> 20
        // indexes the 2048-entry tables
        if (ROUND == R_COARSE) {
            each([&](uint32_t key, bool valid) {
                red_shared(valid ? h_a + ((key >> COARSE_SHIFT) << 2) : sink_a);
            });
        } else if (dense && ROUND != R_FINAL) {
            each([&](uint32_t key, bool valid) {
                const int q = __viaddmin_s32_relu((int)(key >> 10), qoff, qtop);
                red_shared(valid ? h_a + ((uint32_t)q << 2) : sink_a);
            });
        } else if (ROUND == R_COARSE_SUB) {
            const uint32_t clo = klo >> COARSE_SHIFT;
            each([&](uint32_t key, bool valid) {
                below += (valid && key < klo) ? 1u : 0u;
                const uint32_t c = key >> COARSE_SHIFT;
                const int g = t1[c];
                const uint32_t fine = (key >> 10) & (NFINE - 1);
                const bool in = valid && key - klo <= kspan;
                const uint32_t bin = g < 0 ? c - clo : SUB_WIN + (uint32_t)g * NFINE + fine;
                if (in && g < 0 && bin >= (uint32_t)SUB_WIN)  // a range of over 64 octaves: never seen
                    atomicAdd(gbins - NCOARSE + c, 1ull);
                else
                    red_shared(in ? h_a + (bin << 2) : sink_a);
            });
        } else if (ROUND == R_MID) {
            const uint32_t top = (uint32_t)nfine / NFINE - 1u;
            bands([&](const float (&d)[4][DPL], auto valid) {
                // groups outside this launch's window [g0, g0 + gn) wait for another
                uint32_t gw[4][DPL];
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int j = 0; j < DPL; ++j)
                        gw[r][j] = (uint32_t)((int)t1[__float_as_uint(d[r][j]) >> COARSE_SHIFT] - a.g0);
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int j = 0; j < DPL; ++j) {
                        const uint32_t fine = (__float_as_uint(d[r][j]) >> 10) & (NFINE - 1);
                        red_shared(valid(r, j) && gw[r][j] <= top ? h_a + ((gw[r][j] * NFINE + fine) << 2) : sink_a);
                    }
            });
        } else {
            // final round: hit[r][j] = group + 1 of a target's key, 0 for all
            // others; one branch per sixteen cells around the rare hits
            auto finals = [&](auto &&look) {
                bands([&](const float (&d)[4][DPL], auto valid) {
                    uint32_t hit[4][DPL], any = 0;
#pragma unroll
                    for (int r = 0; r < 4; ++r)
#pragma unroll
                        for (int j = 0; j < DPL; ++j) hit[r][j] = look(__float_as_uint(d[r][j]));
#pragma unroll
                    for (int r = 0; r < 4; ++r)
#pragma unroll
                        for (int j = 0; j < DPL; ++j) any |= hit[r][j];
                    if (any == 0u) return;
#pragma unroll
                    for (int r = 0; r < 4; ++r)
#pragma unroll
                        for (int j = 0; j < DPL; ++j)
                            if (valid(r, j) && hit[r][j])
                                atomicAdd(gbins + (int64_t)(hit[r][j] - 1) * NFINE +
                                              (__float_as_uint(d[r][j]) & (NFINE - 1)), 1ull);
                });
            };
            if (dense) {
                finals([&](uint32_t key) -> uint32_t {
                    return t8[__viaddmin_s32_relu((int)(key >> 10), qoff, qtop)];
                });
            } else if (hmul) {
                finals([&](uint32_t key) -> uint32_t {
                    // empty slots hold group 0 with prefix 0x1fffff, which only a
                    // NaN key (already an error) can match, inside group 0's bins
                    const uint32_t p = key >> 10;
                    const uint32_t e = th[(p * hmul) >> (32 - NHASH_BITS)];
                    return ((e ^ p) & 0x1FFFFFu) == 0u ? (e >> 21) + 1u : 0u;
                });
            } else {
                const int np = n_pfx;
                finals([&](uint32_t key) -> uint32_t {
                    const uint32_t p = key >> 10;
                    int lo = 0;  // last prefix <= p, or the first; all lanes in step
#pragma unroll 1
                    for (int step = (KMAX + 1) / 2; step; step >>= 1) {
                        const int c = lo + step;
                        lo = (c < np) & (pfx[min(c, np - 1)] <= p) ? c : lo;
                    }
                    return pfx[lo] == p ? (uint32_t)lo + 1u : 0u;
                });
            }
        }
    }
    flush();
}

template <int ROUND>
static cudaError_t launch_count_m(const CellArgs &a, const SelBufs &sb, int K, int grid,
                                  int embed, cudaStream_t st)
{
    void (*kern)(CellArgs, SelBufs, int, int);
    int words = WIN_WORDS;
    switch (embed) {
    case E_M1T1: kern = k_count<ROUND, DiagSrc<1, 1>>; break;
    case E_M3T1: kern = k_count<ROUND, DiagSrc<3, 1>>; break;
    case E_M3T3: kern = k_count<ROUND, DiagSrc<3, 3>>; break;
    default:
        // the bracket and middle rounds' bins leave no room for windows per
        // coordinate beside a second CTA on the SM
        if ((ROUND == R_COARSE || ROUND == R_FINAL) && a.m_max <= WinSrc::MAXM) {
            kern = k_count<ROUND, WinSrc>;
            words = WinSrc::WORDS;
        } else {
            kern = k_count<ROUND, GenSrc>;
            words = GenSrc::WORDS;
        }
    }
    const int smem = count_smem_bytes(ROUND, K, words);
    cudaError_t e = allow_smem(kern, count_smem_bytes(ROUND, KMAX, words));
    if (e != cudaSuccess) return e;
    grid = persistent_cap(reinterpret_cast<const void *>(kern), smem, grid, CT);
    kern<<<grid, CT, smem, st>>>(a, sb, K, count_bins(ROUND, K));
    return cudaGetLastError();
}

cudaError_t launch_count(int round, const CellArgs &a, const SelBufs &sb, int K, int grid,
                         int embed, cudaStream_t st)
{
    if (!a.y || !a.series || !a.order || !a.uprefix || !a.queue || !a.status || !sb.hist || K < 1 ||
        K > KMAX || grid < 1 || a.n_units < 1 || a.n_units > 0x7fffffff || a.n_pos < 1 || a.m_max < 1 || a.nb < 1 ||
        a.rc < RB || a.rc % RB)
        return cudaErrorInvalidValue;
    if (round == R_MID && (a.g0 < 0 || a.gn < 1 || a.gn > MID_GROUPS)) return cudaErrorInvalidValue;
    switch (round) {
    case R_COARSE: return launch_count_m<R_COARSE>(a, sb, K, grid, embed, st);
    case R_COARSE_SUB: return launch_count_m<R_COARSE_SUB>(a, sb, K, grid, embed, st);
    case R_MID: return launch_count_m<R_MID>(a, sb, K, grid, embed, st);
    default: return launch_count_m<R_FINAL>(a, sb, K, grid, embed, st);
    }
}

// ------------------------------------------------------------ selection
constexpr int ST = 512;  // threads per series
constexpr int SW = ST / 32;

// In-place inclusive scan of n 64-bit values in shared memory (n a multiple
// of ST).
__device__ void block_scan_u64(uint64_t *v, int n, uint64_t *warp_tot)
{
    const int per = n / ST;
    const int t = threadIdx.x;
    uint64_t s = 0;
    for (int x = 0; x < per; ++x) {
        s += v[t * per + x];
        v[t * per + x] = s;
    }
    uint64_t incl = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t u = __shfl_up_sync(FULL, incl, o);
        if ((t & 31) >= o) incl += u;
    }
    if ((t & 31) == 31) warp_tot[t >> 5] = incl;
    __syncthreads();
    uint64_t wpre = 0;
    for (int w = 0; w < (t >> 5); ++w) wpre += warp_tot[w];
    const uint64_t excl = wpre + incl - s;
    for (int x = 0; x < per; ++x) v[t * per + x] += excl;
    __syncthreads();
}

// Smallest index x with a[x] >= v (n if none).
__device__ __forceinline__ int lower_bound_u64(const uint64_t *a, int n, uint64_t v)
{
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (a[mid] < v) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ uint64_t warp_scan_u64(uint64_t v, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint64_t u = __shfl_up_sync(FULL, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// One warp: the bin x of the NFINE bins at src whose cumulative count first
// reaches R (NFINE if none), the counts below it and in it.  Two levels of 32,
// so a target costs two scans and no barrier (a scan of the whole group by
// the CTA per target took 3 us and four barriers each).
__device__ __forceinline__ int warp_search(const uint64_t *src, uint64_t R, int lane, uint64_t &below,
                                           uint64_t &in)
{
    static_assert(NFINE == 32 * 32, "two levels of 32");
    uint64_t seg = 0;  // lane: bins 32 lane .. 32 lane + 31
    const ulonglong2 *p = reinterpret_cast<const ulonglong2 *>(src) + lane * 16;
#pragma unroll
    for (int x = 0; x < 16; ++x) {
        const ulonglong2 v = p[x];
        seg += v.x + v.y;
    }
    const uint64_t cs = warp_scan_u64(seg, lane);
    const unsigned hit = __ballot_sync(FULL, cs >= R);
    below = 0;
    in = 0;
    if (!hit) return NFINE;
    const int sl = __ffs(hit) - 1;
    const uint64_t base = __shfl_sync(FULL, cs - seg, sl);
    const uint64_t v = src[32 * sl + lane];
    const uint64_t cv = base + warp_scan_u64(v, lane);
    const int bl = __ffs(__ballot_sync(FULL, cv >= R)) - 1;
    below = __shfl_sync(FULL, cv - v, bl);
    in = __shfl_sync(FULL, v, bl);
    return 32 * sl + bl;
}

// Number of distinct values up to each of the K ascending values v (threads
// t < K; K <= 128): grp = index of v[t] among them; returns their count.
__device__ int distinct_groups(const uint32_t *v, int K, int *grp, unsigned *bits)
{
    const int t = threadIdx.x;
    if (t < 128) {
        const bool first = t < K && (t == 0 || v[t] != v[t - 1]);
        const unsigned b = __ballot_sync(FULL, first);
        if ((t & 31) == 0) bits[t >> 5] = b;
    }
    __syncthreads();
    int n = 0;
    for (int w = 0; w < 4; ++w) n += __popc(bits[w]);
    if (t < K) {
        int g = __popc(bits[t >> 5] & (0xffffffffu >> (31 - (t & 31)))) - 1;
        for (int w = 0; w < (t >> 5); ++w) g += __popc(bits[w]);
        grp[t] = g;
    }
    __syncthreads();
    return n;
}

// One CTA per series, a warp per target.  ROUND is the counting round whose
// histogram is read.
template <int ROUND>
__global__ void __launch_bounds__(ST)
k_select(SelBufs sb, int s_begin, int K, float *eps_out, uint64_t *le_out, uint64_t *lt_out, int *status)
{
    __shared__ uint64_t cum[ROUND == R_COARSE || ROUND == R_COARSE_SUB ? NCOARSE : 1];
    __shared__ uint64_t wt[SW];
    __shared__ uint32_t pre[KMAX + 1];
    __shared__ uint8_t lev[KMAX + 1];
    __shared__ uint64_t rnk[KMAX + 1], blw[KMAX + 1];
    __shared__ int grp[KMAX + 1];
    __shared__ unsigned bits[4];
    const int s = s_begin + blockIdx.x;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int64_t sk = (int64_t)s * K;
    const uint64_t *gh = sb.hist + (int64_t)s * sb.hstride;
    const uint64_t *gfine = gh + NCOARSE;

    // targets of group grp[k] (>= 0): the middle digit, one warp each
    auto middle_digit = [&]() {
        for (int k = warp; k < K; k += SW) {
            if (grp[k] < 0) continue;
            uint64_t below, in;
            const int x = warp_search(gfine + (int64_t)grp[k] * NFINE, rnk[k], lane, below, in);
            __syncwarp();
            if (lane == 0) {
                if (x >= NFINE) {
                    set_status(status, 10 /*INTERNAL*/);
                } else {
                    pre[k] = (pre[k] << 10) | (uint32_t)x;
                    lev[k] = 2;
                    rnk[k] -= below;
                    blw[k] += below;
                }
            }
        }
        __syncthreads();
    };

    if (ROUND == R_COARSE && !sb.redo[s]) return;  // the bracket settled this series
    if (ROUND == R_COARSE || ROUND == R_COARSE_SUB) {
        __shared__ int hard;  // bracket round: some target outside the bracket
        if (t == 0) hard = 0;
        // bucket totals; a split bucket's keys sit in its fine group
        for (int x = t; x < NCOARSE; x += ST) cum[x] = gh[x];
        __syncthreads();
        const int8_t *tab = ROUND == R_COARSE_SUB ? sb.tab_sub + (int64_t)s * NCOARSE : nullptr;
        const int nsub = ROUND == R_COARSE_SUB ? sb.n_sub[s] : 0;
        if (ROUND == R_COARSE_SUB) {
            __shared__ int inv[NSUB_MAX];
            if (t < NSUB_MAX) inv[t] = -1;
            __syncthreads();
            for (int c = t; c < NCOARSE; c += ST) {
                const int g = tab[c];
                if (g >= 0 && g < NSUB_MAX) inv[g] = c;
            }
            __syncthreads();
            for (int g = warp; g < nsub; g += SW) {
                uint64_t part = 0;
                for (int x = lane; x < NFINE; x += 32) part += gfine[(int64_t)g * NFINE + x];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(FULL, part, o);
                if (lane == 0 && inv[g] >= 0) cum[inv[g]] += part;
            }
            __syncthreads();
        }
        block_scan_u64(cum, NCOARSE, wt);
        // bracket round: only the bracket's buckets were counted (keys under it
        // lumped into the bucket just below, keys above it not at all)
        const int sub_lo = (int)(sb.range[2 * (int64_t)s] >> COARSE_SHIFT);
        const int sub_hi = (int)(sb.range[2 * (int64_t)s + 1] >> COARSE_SHIFT);
        if (t < K) {
            const uint64_t R = sb.T[sk + t];
            const int c = lower_bound_u64(cum, NCOARSE, R);
            if (ROUND == R_COARSE_SUB && (nsub == 0 || c >= NCOARSE || c < sub_lo || c > sub_hi)) {
                pre[t] = 0; lev[t] = 0; rnk[t] = R; blw[t] = 0;  // outside: full selection
                hard = 1;
            } else if (c >= NCOARSE || R == 0) {
                set_status(status, 10 /*INTERNAL*/);
                pre[t] = 0; lev[t] = 1; rnk[t] = 1; blw[t] = 0;
            } else {
                const uint64_t below = c ? cum[c - 1] : 0;
                pre[t] = (uint32_t)c;
                lev[t] = 1;
                rnk[t] = R - below;
                blw[t] = below;
            }
            grp[t] = ROUND == R_COARSE_SUB && lev[t] == 1 ? tab[pre[t]] : -1;
        }
        __syncthreads();
        if (ROUND == R_COARSE_SUB) {
            middle_digit();
            if (t == 0) sb.redo[s] = (uint8_t)hard;
            if (hard) {  // the plain rounds redo this series; levels kept for the statistics
                if (t < K) sb.level[sk + t] = lev[t];
                return;
            }
        }
        // middle-round table: coarse bucket -> group, for targets at level 1
        // (ascending buckets).  Buckets that span at most NSUB_MAX make every
        // bucket of the span a group, so the counting kernel needs no table.
        __shared__ int n_mid, c_lo, c_hi;
        int8_t *tm = sb.tab_mid + (int64_t)s * NCOARSE;
        for (int x = t; x < NCOARSE / 4; x += ST) reinterpret_cast<uint32_t *>(tm)[x] = 0xffffffffu;
        if (t == 0) {
            int lo = NCOARSE, hi = -1;
            for (int k = 0; k < K; ++k)
                if (lev[k] == 1) {
                    lo = min(lo, (int)pre[k]);
                    hi = max(hi, (int)pre[k]);
                }
            c_lo = lo;
            c_hi = hi;
            n_mid = hi < lo ? 0 : hi - lo + 1;
        }
        __syncthreads();
        if (n_mid > 0 && n_mid <= NSUB_MAX) {
            if (t < n_mid) tm[c_lo + t] = (int8_t)t;
        } else if (n_mid > 0) {
            __syncthreads();  // every thread has read n_mid
            if (t == 0) {
                int g = 0;
                for (int k = 0; k < K; ++k)
                    if (lev[k] == 1 && tm[pre[k]] < 0) tm[pre[k]] = (int8_t)g++;
                n_mid = g;
            }
            __syncthreads();
        }
        if (t == 0) {
            sb.n_mid[s] = n_mid;
            sb.range[2 * (int64_t)s] = n_mid ? (uint32_t)c_lo << COARSE_SHIFT : 0xffffffffu;
            sb.range[2 * (int64_t)s + 1] = n_mid ? (((uint32_t)c_hi + 1u) << COARSE_SHIFT) - 1u : 0u;
        }
        if (t < K) {
            sb.prefix[sk + t] = pre[t];
            sb.level[sk + t] = lev[t];
            sb.rank[sk + t] = rnk[t];
            sb.below[sk + t] = blw[t];
        }
        return;
    }

    // R_MID and R_FINAL: state from global memory
    if (t < K) {
        pre[t] = sb.prefix[sk + t];
        lev[t] = sb.level[sk + t];
        rnk[t] = sb.rank[sk + t];
        blw[t] = sb.below[sk + t];
    }
    __syncthreads();

    if (ROUND == R_MID) {
        const int8_t *tm = sb.tab_mid + (int64_t)s * NCOARSE;
        if (t < K) grp[t] = (lev[t] == 1) ? tm[pre[t]] : -1;
        __syncthreads();
        middle_digit();
        // final round: the distinct prefixes (every target is at level 2 now,
        // ascending) are its groups, in order
        const int nfin = distinct_groups(pre, K, grp, bits);
        const uint32_t lo = pre[0] << 10, hi = ((pre[K - 1] + 1u) << 10) - 1u;
        if (t == 0) {
            sb.n_fin[s] = nfin;
            sb.range[2 * (int64_t)s] = lo;
            sb.range[2 * (int64_t)s + 1] = hi;
        }
        if (t < K) {
            sb.prefix[sk + t] = pre[t];
            sb.level[sk + t] = lev[t];
            sb.rank[sk + t] = rnk[t];
            sb.below[sk + t] = blw[t];
        }
        // hashed table of the prefixes, read when their span exceeds the
        // counting kernel's byte table: the first odd multiplier of a fixed
        // sequence that puts them in distinct slots (none among 64: the
        // kernel searches)
        if (sb.tab_hash && hi - lo >= (uint32_t)DENSE_FINAL << 10) {
            uint32_t *fh = sb.tab_hash + (int64_t)s * NHASH;
            __shared__ uint32_t pg[KMAX + 1];
            if (t < K) pg[grp[t]] = pre[t];
            for (int x = t; x < NHASH; x += ST) fh[x] = 0x1fffffu;  // group 0, no finite key
            __syncthreads();
            uint32_t mul = 0;
            for (int at = 0; at < 64 && !mul; ++at) {
                const uint32_t m = (0x9E3779B1u + 0x6A09E668u * (uint32_t)at) | 1u;
                bool clash = false;
                for (int x = t; x < nfin * nfin; x += ST) {
                    const int i = x / nfin, j = x - i * nfin;
                    clash |= j < i && ((pg[i] * m) >> (32 - NHASH_BITS)) == ((pg[j] * m) >> (32 - NHASH_BITS));
                }
                if (!__syncthreads_or(clash)) mul = m;
            }
            if (mul && t < nfin) fh[(pg[t] * mul) >> (32 - NHASH_BITS)] = pg[t] | ((uint32_t)t << 21);
            if (t == 0) sb.hash_mul[s] = mul;
        }
        return;
    }

    // R_FINAL: the low digit completes the key
    distinct_groups(pre, K, grp, bits);
    for (int k = warp; k < K; k += SW) {
        uint64_t below, in;
        const int x = warp_search(gfine + (int64_t)grp[k] * NFINE, rnk[k], lane, below, in);
        if (lane == 0) {
            if (x >= NFINE) {
                set_status(status, 10);
            } else {
                const uint64_t lt = blw[k] + below;
                eps_out[sk + k] = __uint_as_float((pre[k] << 10) | (uint32_t)x);
                if (le_out) le_out[sk + k] = lt + in;
                if (lt_out) lt_out[sk + k] = lt;
            }
        }
    }
}

cudaError_t launch_select(int round, const SelBufs &sb, int s_begin, int n_series, int K, float *eps_out,
                          uint64_t *le_out, uint64_t *lt_out, int *status, cudaStream_t st)
{
    if (n_series <= 0) return cudaSuccess;
    switch (round) {
    case R_COARSE:
        k_select<R_COARSE><<<n_series, ST, 0, st>>>(sb, s_begin, K, eps_out, le_out, lt_out, status);
        break;
    case R_COARSE_SUB:
        k_select<R_COARSE_SUB><<<n_series, ST, 0, st>>>(sb, s_begin, K, eps_out, le_out, lt_out, status);
        break;
    case R_MID:
        k_select<R_MID><<<n_series, ST, 0, st>>>(sb, s_begin, K, eps_out, le_out, lt_out, status);
        break;
    default:
        k_select<R_FINAL><<<n_series, ST, 0, st>>>(sb, s_begin, K, eps_out, le_out, lt_out, status);
        break;
    }
    return cudaGetLastError();
}

// ------------------------------------------------------------ short series
// The whole selection of one short series by one CTA: the finiteness check and
// the three radix rounds on bins in shared memory, the distances recomputed
// in each round from the series' copy there.  A call on a few short series is
// bound by its launches, not its cells: at N = 100 the general rounds are
// twelve launches and memsets that take 71 us for 4950 cells.
//
// Groups as in the general rounds: the distinct coarse buckets of the
// targets, then their distinct 21-bit prefixes; both ascend with the targets.
constexpr int SM_T = 512;
constexpr int SM_K = 24;  // targets: two sets of SM_K x NFINE bins fit in shared memory

int small_select_smem(int n_max) { return (NCOARSE + 2 * SM_K * NFINE + n_max) * 4 + NCOARSE; }

__global__ void __launch_bounds__(SM_T)
k_select_small(const float *__restrict__ y, const SeriesDev *series, const uint64_t *T, int K, float *eps_out,
               uint64_t *le_out, uint64_t *lt_out, int *status)
{
    extern __shared__ __align__(16) unsigned char smem[];
    uint32_t *h1 = reinterpret_cast<uint32_t *>(smem);    // coarse bins, then their cumulative counts
    uint32_t *h2 = h1 + NCOARSE, *h3 = h2 + SM_K * NFINE;  // middle and low digits, per group
    float *ys = reinterpret_cast<float *>(h3 + SM_K * NFINE);
    __shared__ uint32_t pre[SM_K], rnk[SM_K], blw[SM_K], wsum[SM_T / 32];
    __shared__ int grp[SM_K];
    const int s = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const SeriesDev sd = series[s];
    int8_t *t1 = reinterpret_cast<int8_t *>(ys + sd.n);  // coarse bucket -> group
    const int64_t sk = (int64_t)s * K;
    bool bad = false;
    for (int i = t; i < sd.n; i += SM_T) {
        const float v = y[sd.off + i];
        ys[i] = v;
        bad |= !isfinite(v);
    }
    if (__any_sync(FULL, bad) && lane == 0) set_status(status, 3 /*NONFINITE*/);
    for (int i = t; i < NCOARSE + 2 * SM_K * NFINE; i += SM_T) h1[i] = 0;
    for (int i = t; i < NCOARSE; i += SM_T) t1[i] = -1;
    __syncthreads();

    // f(key) for every pair: a warp per row, lanes along the columns
    auto cells = [&](auto &&f) {
        for (int i = warp; i < sd.ne - 1; i += SM_T / 32)
            for (int j = i + 1 + lane; j < sd.ne; j += 32) {
                float d = fabsf(ys[i] - ys[j]);
                for (int q = 1; q < sd.m; ++q) d = fmaxf(d, fabsf(ys[i + q * sd.tau] - ys[j + q * sd.tau]));
                f(__float_as_uint(d));
            }
        __syncthreads();
    };
    // targets 0 .. K-1: grp[k] = index of v[k] among the distinct ascending values
    auto groups = [&](const uint32_t *v) {
        if (warp == 0) {
            const unsigned b = __ballot_sync(FULL, lane < K && (lane == 0 || v[lane] != v[lane - 1]));
            if (lane < K) grp[lane] = __popc(b & (0xffffffffu >> (31 - lane))) - 1;
        }
        __syncthreads();
    };
    // a warp: the bin of the NFINE at src whose cumulative count first reaches R
    auto search = [&](const uint32_t *src, uint32_t R, uint32_t &below, uint32_t &in) -> int {
        uint32_t seg = 0;
        for (int i = 0; i < 32; ++i) seg += src[32 * lane + ((i + lane) & 31)];
        uint32_t cs = seg;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(FULL, cs, o);
            if (lane >= o) cs += u;
        }
        const unsigned hit = __ballot_sync(FULL, cs >= R);
        below = in = 0;
        if (!hit) return NFINE;
        const int sl = __ffs(hit) - 1;
        const uint32_t base = __shfl_sync(FULL, cs - seg, sl);
        const uint32_t v = src[32 * sl + lane];
        uint32_t cv = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(FULL, cv, o);
            if (lane >= o) cv += u;
        }
        cv += base;
        const int bl = __ffs(__ballot_sync(FULL, cv >= R)) - 1;
        below = __shfl_sync(FULL, cv - v, bl);
        in = __shfl_sync(FULL, v, bl);
        return 32 * sl + bl;
    };

    cells([&](uint32_t key) { atomicAdd(&h1[key >> COARSE_SHIFT], 1u); });
    {   // cumulative coarse counts in place (four bins per thread)
        uint32_t v[NCOARSE / SM_T], sum = 0;
#pragma unroll
        for (int i = 0; i < NCOARSE / SM_T; ++i) v[i] = sum += h1[t * (NCOARSE / SM_T) + i];
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(FULL, incl, o);
            if (lane >= o) incl += u;
        }
        if (lane == 31) wsum[warp] = incl;
        __syncthreads();
        uint32_t excl = incl - sum;
        for (int w = 0; w < warp; ++w) excl += wsum[w];
#pragma unroll
        for (int i = 0; i < NCOARSE / SM_T; ++i) h1[t * (NCOARSE / SM_T) + i] = excl + v[i];
        __syncthreads();
    }
    if (t < K) {
        const uint32_t R = (uint32_t)T[sk + t];
        int lo = 0, hi = NCOARSE;  // first bucket whose cumulative count reaches R
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (h1[mid] < R) lo = mid + 1;
            else hi = mid;
        }
        if (lo >= NCOARSE || R == 0) {
            set_status(status, 10 /*INTERNAL*/);
            lo = NCOARSE - 1;
        }
        blw[t] = lo ? h1[lo - 1] : 0u;
        pre[t] = (uint32_t)lo;
        rnk[t] = R - blw[t];
    }
    __syncthreads();
    groups(pre);
    if (t < K) t1[pre[t]] = (int8_t)grp[t];
    __syncthreads();
    cells([&](uint32_t key) {
        const int g = t1[key >> COARSE_SHIFT];
        if (g >= 0) atomicAdd(&h2[g * NFINE + ((key >> 10) & (NFINE - 1))], 1u);
    });
    for (int k = warp; k < K; k += SM_T / 32) {
        uint32_t below, in;
        const int x = search(h2 + grp[k] * NFINE, rnk[k], below, in);
        __syncwarp();
        if (lane == 0) {
            if (x >= NFINE) set_status(status, 10);
            pre[k] = pre[k] << 10 | (uint32_t)min(x, NFINE - 1);
            rnk[k] -= below;
            blw[k] += below;
        }
    }
    __syncthreads();
    // the middle bins become the table (coarse group, middle digit) -> prefix
    // group + 1, zero for the others
    for (int i = t; i < SM_K * NFINE; i += SM_T) h2[i] = 0;
    __syncthreads();
    uint32_t slot = 0;
    if (t < K) slot = (uint32_t)grp[t] * NFINE + (pre[t] & (NFINE - 1));
    groups(pre);
    if (t < K) h2[slot] = (uint32_t)grp[t] + 1u;
    __syncthreads();
    cells([&](uint32_t key) {
        const int g1 = t1[key >> COARSE_SHIFT];
        if (g1 < 0) return;
        const uint32_t g = h2[g1 * NFINE + ((key >> 10) & (NFINE - 1))];
        if (g) atomicAdd(&h3[(g - 1u) * NFINE + (key & (NFINE - 1))], 1u);
    });
    for (int k = warp; k < K; k += SM_T / 32) {
        uint32_t below, in;
        const int x = search(h3 + grp[k] * NFINE, rnk[k], below, in);
        if (lane == 0) {
            if (x >= NFINE) {
                set_status(status, 10);
            } else {
                eps_out[sk + k] = __uint_as_float(pre[k] << 10 | (uint32_t)x);
                if (le_out) le_out[sk + k] = (uint64_t)blw[k] + below + in;
                if (lt_out) lt_out[sk + k] = (uint64_t)blw[k] + below;
            }
        }
    }
}

bool small_select_ok(int K, int32_t ne_max, int64_t n_max, uint64_t total_cells, int sm_count)
{
    return K <= SM_K && ne_max <= SMALL_NE && n_max <= 2 * SMALL_NE && total_cells <= (uint64_t)sm_count << 17;
}

cudaError_t launch_select_small(const float *y, const SeriesDev *series, int S, int n_max, const uint64_t *T, int K,
                                float *eps_out, uint64_t *le_out, uint64_t *lt_out, int *status, cudaStream_t st)
{
    if (!y || !series || !T || !eps_out || !status || S < 1 || K < 1 || K > SM_K || n_max < 2 ||
        n_max > 2 * SMALL_NE)
        return cudaErrorInvalidValue;
    const int smem = small_select_smem(n_max);
    cudaError_t e = allow_smem(k_select_small, small_select_smem(2 * SMALL_NE));
    if (e != cudaSuccess) return e;
    k_select_small<<<S, SM_T, smem, st>>>(y, series, T, K, eps_out, le_out, lt_out, status);
    return cudaGetLastError();
}

}  // namespace rqa
