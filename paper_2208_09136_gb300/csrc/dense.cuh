// The cell walk shared by the counting rounds, the grid search and the line
// passes: a warp owns a band of 128 consecutive diagonals (or columns) of the
// never-materialised distance matrix and walks down it in blocks of 28 rows;
// lane x holds the four neighbouring diagonals d0 + 4x .. d0 + 4x + 3, so the
// cells of a lane follow each other along their diagonals.
//
// Why this shape: the cell loop is bound by instruction issue.  Along a
// diagonal the coordinate difference e(s) = y[s] - y[s + d] of row s serves
// the cells of rows s, s - tau, .., s - (m-1) tau, so a lane that walks down
// its diagonals needs one subtraction and (m = 3) one three-input maximum per
// cell, where a lane that holds one row needs m subtractions.  Four
// neighbouring diagonals share their column values (row r, diagonal j reads
// value r + j of a window), so four rows of a lane's sixteen cells take one
// 16-byte shared load for the columns and one (broadcast) for the rows.
#pragma once
#include <cstdint>
#include <type_traits>
#include "rqa_common.cuh"

namespace rqa {

constexpr int DPL = 4;             // diagonals per lane
constexpr int RB = ROW_BLOCK;      // 28 rows per block: a multiple of 4 and of the ring of m = tau = 3
constexpr int COLW = DB + RB + 4;  // column window of a block, in values
constexpr int ROWW = 32;           // row window
constexpr int WIN_WORDS = COLW + ROWW;  // 32-bit words of a warp's windows (16-byte multiples)
// The windows reach up to 158 values past the end of a series, whose length
// goes up to 2^31 - 65: an index that may pass the end is unsigned.
static_assert(DB == 32 * DPL && RB % 4 == 0 && COLW % 32 == 0 && WIN_WORDS % 4 == 0, "band shape");

// Work unit u of a launch: bands [b_lo, b_hi) of series s over rows
// [r_lo, r_hi).  The units of a series are its row chunks of a.rc rows, each
// cut into groups of a.nb bands; the chunk at r_lo has the bands whose
// longest diagonal reaches it (diagonal pass) or every band (vertical pass).
struct Unit {
    int s, b_lo, b_hi, r_lo, r_hi;
};
// W: diagonals (columns) per band.
template <bool VERT, int W = DB>
__device__ __forceinline__ Unit unit_of(const CellArgs &a, int64_t u)
{
    int lo = 0, hi = a.n_pos;  // last pos with uprefix[pos] <= u
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (a.uprefix[mid] <= u) lo = mid;
        else hi = mid;
    }
    Unit w;
    w.s = a.order[lo];
    const int ne = a.series[w.s].ne;
    int64_t rem = u - a.uprefix[lo];
    int bands = 0;
    w.r_lo = 0;
    for (;;) {
        bands = VERT ? (ne + W - 1) / W : (ne - 1 - w.r_lo + W - 1) / W;
        const int items = (bands + a.nb - 1) / a.nb;
        if (rem < items || w.r_lo + a.rc >= ne) break;
        rem -= items;
        w.r_lo += a.rc;
    }
    w.b_lo = (int)rem * a.nb;
    w.b_hi = min(w.b_lo + a.nb, bands);
    w.r_hi = min(w.r_lo + a.rc, ne);
    return w;
}

// How the warps of a CTA share a unit: one band at a time, so that no warp
// idles while another still has several left; a unit of fewer bands than warps
// is cut further, into parts of part_rows(w, warps) rows (a multiple of RB).
// Short series have fewer bands: @@
__device__ __forceinline__ int part_rows(const Unit &w, int warps)
{
    const int nb = w.b_hi - w.b_lo, blocks = (w.r_hi - w.r_lo + RB - 1) / RB;
    if (nb >= warps) return blocks * RB;
    const int parts = min((warps + nb - 1) / nb, blocks);
    return (blocks + parts - 1) / parts * RB;
}
// f(first diagonal, first row, end row) for every part that this warp takes.
// All arguments lie in shared memory and are read again for each part, which
// costs less than their registers; next: the unit's counter, 0 at its start.
template <class F>
__device__ __forceinline__ void each_part(const Unit &w, const int &rows, int *next, int lane, F &&f)
{
    for (;;) {
        int i = 0;
        if (lane == 0) i = atomicAdd(next, 1);
        i = __shfl_sync(FULL, i, 0);
        const int nb = w.b_hi - w.b_lo, part = i < nb ? 0 : i / nb, r = w.r_lo + part * rows;
        if (r >= w.r_hi) break;
        f(1 + (w.b_lo + i - part * nb) * DB, r, min(r + rows, w.r_hi));
    }
}

// Distances of the compile-time embedding (M, TAU): the ring e[] holds the
// coordinate differences of the last (M-1) TAU rows of each diagonal.  Eight
// rows long, so that two steps of four rows bring it back to the same
// registers and a block is a loop of such pairs (each_quad).  With all 28 rows
// unrolled the loops did not stay in the instruction cache (the three radix
// rounds over 8e8 cells, m = tau = 3: 1.00 ms, 0.85 ms in this form).
template <int M, int TAU>
struct DiagSrc {
    static constexpr int H = (M - 1) * TAU, RS = 8;
    static_assert(H < RS, "history rows");
    static constexpr int WORDS = WIN_WORDS;  // shared memory per warp
    float e[RS][DPL];
    float pc[COLW / 32], pr;  // the next block's windows on their way from memory
    float4 c0;
    const float *ys;
    int n, d0, lane;
    float *cw, *rw;

    __device__ __forceinline__ void init(const float *y, const SeriesDev &sd, int lane_, uint32_t *win)
    {
        ys = y;
        n = sd.n;
        lane = lane_;
        cw = reinterpret_cast<float *>(win);
        rw = cw + COLW;
    }
    __device__ __forceinline__ void fetch(int i0)
    {
        const int cb = i0 + H + d0 + lane, rr = i0 + H + lane;
#pragma unroll
        for (int x = 0; x < COLW / 32; ++x) pc[x] = cb + 32 * x < n ? __ldg(ys + cb + 32 * x) : 0.f;
        pr = lane < RB && rr < n ? __ldg(ys + rr) : 0.f;
    }
    // first block of a walk: the differences of the rows above its ring
    __device__ __forceinline__ void begin(int d, int i0)
    {
        d0 = d;
#pragma unroll
        for (int s = 0; s < H; ++s)
#pragma unroll
            for (int j = 0; j < DPL; ++j) {
                const int c = i0 + s + d0 + DPL * lane + j;
                e[s][j] = c < n ? __ldg(ys + i0 + s) - __ldg(ys + c) : 0.f;
            }
        fetch(i0);
    }
    // the windows of block i0 into shared memory, those of the next one requested
    __device__ __forceinline__ void enter(int i0)
    {
        __syncwarp();
#pragma unroll
        for (int x = 0; x < COLW / 32; ++x) cw[lane + 32 * x] = pc[x];
        rw[lane] = pr;
        __syncwarp();
        fetch(i0 + RB);
        c0 = *reinterpret_cast<const float4 *>(cw + DPL * lane);
    }
    // distances of rows 4u .. 4u+3 of the block; PH = u mod 2 picks the ring's registers
    template <bool CHECK, int PH>
    __device__ __forceinline__ void quad(int u, int, float (&d)[4][DPL])
    {
        const float4 r4 = *reinterpret_cast<const float4 *>(rw + 4 * u);
        const float4 c1 = *reinterpret_cast<const float4 *>(cw + 4 * u + 4 + DPL * lane);
        const float rv[4] = {r4.x, r4.y, r4.z, r4.w};
        const float cv[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int j = 0; j < DPL; ++j) {
                const int t = 4 * PH + r;
                e[(t + H) % RS][j] = rv[r] - cv[r + j];
                float x[M];
#pragma unroll
                for (int q = 0; q < M; ++q) x[q] = e[(t + q * TAU) % RS][j];
                d[r][j] = maxnorm<M>(x);
            }
        c0 = c1;
    }
    __device__ __forceinline__ void leave()
    {
        if constexpr (H > 0) {  // seven steps of four rows: the ring's other half comes first again
            float t[RS][DPL];
#pragma unroll
            for (int s = 0; s < RS; ++s)
#pragma unroll
                for (int j = 0; j < DPL; ++j) t[s][j] = e[(s + RB) % RS][j];
#pragma unroll
            for (int s = 0; s < RS; ++s)
#pragma unroll
                for (int j = 0; j < DPL; ++j) e[s][j] = t[s][j];
        }
    }
};

// Any embedding (m and tau at run time, also unlike between the series of a
// batch): the values are read through L1, two coordinates per step so that
// one three-input maximum serves both.  CHECK: indexes past the series are
// pulled back to its last value (the caller discards those cells).
struct GenSrc {
    static constexpr int WORDS = 0;
    const float *ys;
    int n, d0, lane, m, tau;

    __device__ __forceinline__ void init(const float *y, const SeriesDev &sd, int lane_, uint32_t *)
    {
        ys = y;
        n = sd.n;
        m = sd.m;
        tau = sd.tau;
        lane = lane_;
    }
    __device__ __forceinline__ void begin(int d, int) { d0 = d; }
    __device__ __forceinline__ void enter(int) {}
    template <bool CHECK>
    __device__ __forceinline__ float at(uint32_t i) const
    {
        return __ldg(ys + (CHECK ? min(i, (uint32_t)n - 1u) : i));
    }
    template <bool CHECK>
    __device__ __forceinline__ void diff(uint32_t ri, float (&x)[4][DPL]) const
    {
        const uint32_t ci = ri + (uint32_t)(d0 + DPL * lane);
        float rv[4], cv[3 + DPL];
#pragma unroll
        for (int r = 0; r < 4; ++r) rv[r] = at<CHECK>(ri + r);
#pragma unroll
        for (int c = 0; c < 3 + DPL; ++c) cv[c] = at<CHECK>(ci + c);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int j = 0; j < DPL; ++j) x[r][j] = rv[r] - cv[r + j];
    }
    template <bool CHECK, int PH>
    __device__ __forceinline__ void quad(int u, int i0, float (&d)[4][DPL])
    {
        const uint32_t i = (uint32_t)(i0 + 4 * u);
        diff<CHECK>(i, d);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int j = 0; j < DPL; ++j) d[r][j] = fabsf(d[r][j]);
        int q = 1;
        for (; q + 1 < m; q += 2) {
            float a[4][DPL], b[4][DPL];
            diff<CHECK>(i + q * tau, a);
            diff<CHECK>(i + (q + 1) * tau, b);
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int j = 0; j < DPL; ++j) d[r][j] = fmax3(d[r][j], fabsf(a[r][j]), fabsf(b[r][j]));
        }
        if (q < m) {
            float a[4][DPL];
            diff<CHECK>(i + q * tau, a);
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int j = 0; j < DPL; ++j) d[r][j] = fmaxf(d[r][j], fabsf(a[r][j]));
        }
    }
    __device__ __forceinline__ void leave() {}
};

// Any embedding with at most MAXM coordinates: a window of rows and one of
// columns per coordinate in shared memory, so that four rows of a lane's
// sixteen cells take three 16-byte loads per coordinate, nine wavefronts.
// Through L1 (GenSrc) the column reads of one coordinate are seven loads that
// stride over four lines each, 28 wavefronts, and bind the rounds: four series
// of 2e4 samples, all rounds, m = 2, 4, 6, 8: 1.62, 2.61, 3.65, 4.72 ms through
// L1 and 1.28, 1.87, 2.47, 3.13 ms here.  Eight windows leave two CTAs on an
// SM in the rounds that use them; larger m keeps GenSrc.
struct WinSrc {
    static constexpr int MAXM = 8, WORDS = MAXM * WIN_WORDS;
    const float *ys;
    int n, d0, lane, m, tau;
    float *win;  // [q]: COLW columns, ROWW rows

    __device__ __forceinline__ void init(const float *y, const SeriesDev &sd, int lane_, uint32_t *w)
    {
        ys = y;
        n = sd.n;
        m = sd.m;
        tau = sd.tau;
        lane = lane_;
        win = reinterpret_cast<float *>(w);
    }
    __device__ __forceinline__ void begin(int d, int) { d0 = d; }
    __device__ __forceinline__ void enter(int i0)
    {
        __syncwarp();
        for (int q = 0; q < m; ++q) {
            float *w = win + q * WIN_WORDS + lane;
            const uint32_t r = (uint32_t)(q * tau) + (uint32_t)(i0 + lane);
            const uint32_t c = r + (uint32_t)d0, end = (uint32_t)n - 1u;
            float v[COLW / 32 + 1];
#pragma unroll
            for (uint32_t x = 0; x < COLW / 32; ++x) v[x] = __ldg(ys + min(c + 32u * x, end));
            v[COLW / 32] = __ldg(ys + min(r, end));
#pragma unroll
            for (int x = 0; x <= COLW / 32; ++x) w[32 * x] = v[x];
        }
        __syncwarp();
    }
    __device__ __forceinline__ void diff(const float *w, int u, float (&x)[4][DPL]) const
    {
        const float4 c0 = *reinterpret_cast<const float4 *>(w + 4 * u + DPL * lane);
        const float4 c1 = *reinterpret_cast<const float4 *>(w + 4 * u + 4 + DPL * lane);
        const float4 r4 = *reinterpret_cast<const float4 *>(w + COLW + 4 * u);
        const float rv[4] = {r4.x, r4.y, r4.z, r4.w};
        const float cv[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int j = 0; j < DPL; ++j) x[r][j] = rv[r] - cv[r + j];
    }
    template <bool CHECK, int PH>
    __device__ __forceinline__ void quad(int u, int, float (&d)[4][DPL])
    {
        diff(win, u, d);
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int j = 0; j < DPL; ++j) d[r][j] = fabsf(d[r][j]);
        int q = 1;
        for (; q + 1 < m; q += 2) {
            float a[4][DPL], b[4][DPL];
            diff(win + q * WIN_WORDS, u, a);
            diff(win + (q + 1) * WIN_WORDS, u, b);
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int j = 0; j < DPL; ++j) d[r][j] = fmax3(d[r][j], fabsf(a[r][j]), fabsf(b[r][j]));
        }
        if (q < m) {
            float a[4][DPL];
            diff(win + q * WIN_WORDS, u, a);
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int j = 0; j < DPL; ++j) d[r][j] = fmaxf(d[r][j], fabsf(a[r][j]));
        }
    }
    __device__ __forceinline__ void leave() {}
};

// A block's steps of four rows: q(phase, u) for u = 0 .. 6.
template <class Q>
__device__ __forceinline__ void each_quad(Q &&q)
{
    static_assert(RB == 28, "three pairs and one");
#pragma unroll 1
    for (int u = 0; u < 6; u += 2) {
        q(std::integral_constant<int, 0>{}, u);
        q(std::integral_constant<int, 1>{}, u + 1);
    }
    q(std::integral_constant<int, 0>{}, 6);
}

struct AllValid {
    __device__ __forceinline__ constexpr bool operator()(int, int) const { return true; }
};
struct MaskValid {
    uint32_t m;
    __device__ __forceinline__ bool operator()(int r, int j) const { return (m >> (4 * r + j)) & 1u; }
};
// Walk rows [r_lo, r_hi) of the band at diagonal d0 and hand the distances of
// every lane's four rows x four diagonals to f(d[4][DPL], valid): valid(r, j) is
// a compile-time true inside the triangle and a bit of a run-time mask in blocks
// that reach over its edge.  f sees sixteen cells at once so that it can issue
// their lookups together before it uses any.
template <class Src, class F>
__device__ __forceinline__ void walk_keys(Src &src, int ne, int d0, int r_lo, int r_hi, int lane, F &&f)
{
    const int r_end = min(r_hi, ne - d0);           // rows of the longest diagonal
    const int r_in = min(r_end, ne - d0 - DB + 1);  // rows where all 128 diagonals have a cell
    if (r_lo >= r_end) return;
    src.begin(d0, r_lo);
    const int lim = ne - d0 - DPL * lane;  // rows of the lane's first diagonal
    for (int i0 = r_lo; i0 < r_end; i0 += RB) {
        src.enter(i0);
        if (i0 + RB <= r_in) {
            each_quad([&](auto ph, int u) {
                float d[4][DPL];
                src.template quad<false, decltype(ph)::value>(u, i0, d);
                f(d, AllValid{});
            });
        } else {
            each_quad([&](auto ph, int u) {
                float d[4][DPL];
                src.template quad<true, decltype(ph)::value>(u, i0, d);
                uint32_t m = 0;
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int j = 0; j < DPL; ++j) m |= i0 + 4 * u + r < lim - j ? 1u << (4 * r + j) : 0u;
                f(d, MaskValid{m});
            });
        }
        src.leave();
    }
}

}  // namespace rqa
