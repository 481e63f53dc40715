// The line pass kernel (template).  Diagonal lines of the never-materialised recurrence matrices for all K
// thresholds at once (Eq. 4; Sect. 4: upper triangle, cells computed on the
// fly, line lengths from the beginnings and ends of runs).
//
// A warp owns a band of LD = 32 consecutive diagonals and walks down it 32
// rows at a time.  Each 32 x 32 row block takes two phases:
//
//  cells  the rank r = #{k : eps_k < d} of every cell (one lookup in a bucket
//         table of the thresholds, or a 5-step search over them).
//         m <= 4: lane j walks down diagonal j (column j) and packs the ranks
//         of its 32 cells into eight registers.  m > 4 and mixed batches:
//         lane t holds row i0+t and stores r as a byte of row j of a
//         32 x 32 rank matrix in shared memory, which lane j then reads.
//         (m = 3, cycles per SM quarter and 32 cells of the whole pass, mixed
//         signals: 56.7 by diagonals, 65.1 by rows; tau = 1: 76 and 85.)
//  runs   lane j holds diagonal j.  It gathers the five bit planes of its ranks:
//         two words of four ranks are interleaved bit by bit, so one mask and
//         one multiply bring bit p of eight ranks into the top byte of a
//         product, and byte permutes put four such bytes together (the rows
//         are stored in the byte order this produces); then, for every
//         threshold k, rebuilds the 32-row recurrence word {t : r_t <= k} (the
//         borrow out of r - (k+1), two LOP3s).  A line ends at row t-1 where
//         row t-1 is recurrent and row t is not; copies of the word shifted
//         down by 1..4 rows (the rows above the block come from the state
//         carried from the previous block) tell whether that line is at least
//         2, 3 or 4 long, so lines of length >= 1, 2 and 3 are counted with
//         three popcounts per word.  Lines of length >= 4 are measured one by one
//         from the nearest non-recurrent row above their end, or from the
//         carried run length when the run started in an earlier block.
//
// All K thresholds share one distance evaluation per cell, and every lane
// works on its own diagonal in the run phase.  The run state carried from one
// row block to the next (per lane and threshold) is the top four bits of the
// previous word and the length of the run open at its last row.
//
// Outputs per (series, threshold): P_k(l) (lengths 1..3 from packed register
// tallies, less the lines measured one by one for length 3; 4..WSH in the
// warp's shared histogram; both flushed when the warp goes on to another series
// or at 2^33 cells; WSH+1..LSH in the series' global short histogram; longer lines
// to the caller's full histogram), L_max, and C_k = sum of l P_k(l), the
// recurrent cells.
//
// A batch with too few bands to fill the chip is cut into row chunks
// (CellArgs::rc).  A chunk counts its rows as if the matrix ended at them and
// keeps, per diagonal and threshold, the lengths of the lines that touch its
// first and its last row (edges); k_merge (lines.cu) then joins the lines that
// meet at a chunk boundary.  The four 10^4-value series of lorenz-n1e4 have
// 1252 bands for 2432 resident warps, each 10^4 rows long.
//
// The vertical pass (VERT) is the same kernel over bands of 32 consecutive
// columns walked over every row of the matrix: lane c's words are 32 rows of its
// column, so their runs are vertical lines.
#pragma once
#include <cstdint>
#include <type_traits>
#include "dense.cuh"

namespace rqa {

constexpr int LD = 32;        // diagonals (or columns) per band: one per lane in the run phase
constexpr int KT = LINE_KMAX; // thresholds per sweep: per-lane carry state and tallies in registers
constexpr int WSH = 44;       // lines of length 4..WSH counted in the warp's shared histogram
constexpr int HROW = WSH + 1; // rows 0..WSH of that histogram (row 0: lines longer than WSH)
constexpr int TMAX = 384;     // entries of the rank table
constexpr uint32_t CMASK = 0x0FFFFFFFu;  // carry state: length of the open run ...
constexpr uint32_t TOP4 = 0xF0000000u;   // ... and the top four rows of the previous word
constexpr int SETTLE = 60;    // row blocks between tally settles (10-bit fields, <= 17 per block)

static_assert(LSH > WSH, "lengths WSH+1..LSH go to the global short histogram");

// Per-warp shared memory, in 32-bit words:
//   lq    [KT][LD] 8 bytes each: when the word of threshold k of diagonal j
//         ends lines of length >= 4, their end mask and the run state carried
//         into the word (the run open above it in the low 28 bits); they are
//         measured after the threshold loop (the word
//         itself is rebuilt there from the row block's planes).  The same
//         space first holds the row block's rank matrix, [LD][32] bytes (row
//         j: the ranks of diagonal j's 32 cells), read before any slot is
//         written.
//   pl    [LD][4] bit planes 0..3 of the ranks of the current row block (16-byte rows)
//   pl4   [LD]    bit plane 4 (both written by lane j for diagonal j, read back
//                 when the lines of length >= 4 are measured)
//   epsb  [32]    threshold keys of the current series (padding above every key)
//   tab   [TMAX]  rank table
//   hs    [HROW][32] line counts by length, one column (bank) per lane:
//         rows 1..3 from the tallies (row 3: every line of length >= 3),
//         rows 4..WSH one by one, row 0 the lines longer than WSH
constexpr int O_LQ = 0, O_PL = O_LQ + KT * LD * 2, O_PL4 = O_PL + LD * 4, O_EPS = O_PL4 + LD,
              O_TAB = O_EPS + 32, O_HS = O_TAB + TMAX, WARP_WORDS = (O_HS + HROW * 32 + 3) & ~3;

// CTAs of 2 warps: eight fit per SM (shared memory and registers), sixteen warps
constexpr int LTHREADS = 64;
constexpr int LWARPS = LTHREADS / 32;
inline int lines_smem_bytes() { return LWARPS * WARP_WORDS * 4; }

// Recurrence word of threshold k over the 32 rows: bit t = [r_t <= k], i.e.
// the borrow out of r_t - (k+1) rippled through the bit planes B[0..4] of the
// ranks.  k is a compile-time constant after unrolling, so every step is a
// two-input function of (plane, borrow) and the compiler fuses pairs of steps
// into single LOP3s.  Rank 31 (a cell outside the matrix) is recurrent for no
// k <= 30.
__device__ __forceinline__ uint32_t rank_le_word(const uint32_t (&B)[5], int k)
{
    const int c = k + 1;
    uint32_t lt = 0;
    bool on = false;
#pragma unroll
    for (int b = 0; b < 5; ++b) {
        const bool cb = (c >> b) & 1;
        if (!on) {
            if (cb) {
                lt = ~B[b];
                on = true;
            }
        } else {
            lt = cb ? (~B[b] | lt) : (~B[b] & lt);
        }
    }
    return lt;
}

// 3-input bitwise function with an 8-bit truth table (one LOP3 instruction):
// bit i of the table is the output for (a, b, c) = bits of (0xF0, 0xCC, 0xAA).
template <uint32_t LUT>
__device__ __forceinline__ uint32_t lop3(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, %4;" : "=r"(d) : "r"(a), "r"(b), "r"(c), "n"(LUT));
    return d;
}

// The same word for a threshold that differs between lanes: kbm[b] is all
// ones where bit b of k + 1 is set.  Each step is the borrow of one bit
// plane: (~r & c) | (~r & borrow) | (c & borrow), one LOP3.
__device__ __forceinline__ uint32_t rank_le_word_lane(uint32_t b0, uint32_t b1, uint32_t b2,
                                                      uint32_t b3, uint32_t b4,
                                                      const uint32_t (&kbm)[5])
{
    uint32_t w = lop3<0x0C>(b0, kbm[0], 0u);  // ~r0 & c0
    w = lop3<0x8E>(b1, kbm[1], w);
    w = lop3<0x8E>(b2, kbm[2], w);
    w = lop3<0x8E>(b3, kbm[3], w);
    return lop3<0x8E>(b4, kbm[4], w);
}

// Transpose a 32 x 32 bit matrix held one row per lane: on return lane k
// holds column k (bit j of the result = bit k of lane j's word).  Five rounds
// of exchanging off-diagonal blocks with the lane s apart.
__device__ __forceinline__ uint32_t transpose32(uint32_t x, int lane)
{
    constexpr uint32_t MASKS[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int r = 0; r < 5; ++r) {
        const int sh = 16 >> r;
        const uint32_t m = MASKS[r];
        const uint32_t y = __shfl_xor_sync(FULL, x, sh);
        x = (lane & sh) ? ((x & ~m) | ((y & ~m) >> sh)) : ((x & m) | ((y & m) << sh));
    }
    return x;
}

// The key of a caller's threshold (-0 as +0), and whether it is one: neither
// negative nor NaN.  The line pass skips a series with a threshold that is not,
// or with thresholds that do not ascend (RQA_ERR_UNSORTED).
__device__ __forceinline__ uint32_t threshold_key(float eps)
{
    const uint32_t v = __float_as_uint(eps);
    return v == 0x80000000u ? 0u : v;
}
__device__ __forceinline__ bool threshold_ok(uint32_t v) { return !(v & 0x80000000u) && v <= 0x7f800000u; }

// Warp-centric: every warp pulls units from one global queue and keeps its
// own histogram in shared memory, flushed when the series changes.  No CTA-wide
// barrier, so no warp waits for another.
// FK: a full sweep, K = KT thresholds known at compile time (the per-threshold
// code then runs without a test of k against K); the argument is ignored.
template <int M, int TAU, bool VERT, bool FK = false>
__global__ void __launch_bounds__(LTHREADS, 8) k_lines(CellArgs a, LineBufs lb, int K_arg, uint16_t *edges)
{
    const int K = FK ? KT : K_arg;
    constexpr bool WALK = M > 0;            // cells by diagonals (columns), else by rows
    constexpr bool RING = TAU > 0 && !VERT;  // differences kept from row to row
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t *ws = reinterpret_cast<uint32_t *>(smem) + warp * WARP_WORDS;
    uint32_t *pl = ws + O_PL, *pl4 = ws + O_PL4, *epsb = ws + O_EPS, *tab = ws + O_TAB;
    uint32_t *hs = ws + O_HS + lane;  // this lane's column: [l * 32], threshold kk (below)
    uint2 *lqa = reinterpret_cast<uint2 *>(ws + O_LQ);  // [k * LD + j]
    unsigned char *rkm = reinterpret_cast<unsigned char *>(ws + O_LQ);  // rank matrix, row j
    uint2 *lq = lqa + lane;                               // slots of this lane's diagonal
    const bool klane = lane < K;
    // byte of row `lane` in a row of the rank matrix: rows 8h + 2u and 8h + 2u + 1
    // sit four bytes apart (bytes 8h + u and 8h + u + 4), the order the plane
    // gather of the run phase reads them in
    const int rcol = (lane & ~7) | ((lane & 7) >> 1) | ((lane & 1) << 2);
    // Lines of length >= 4: lane k < K measures those of threshold k; the
    // 32 - K lanes left over help the top thresholds (the ones with the most
    // lines), lane L >= K taking threshold L - (32 - K) on the odd diagonals
    // while that threshold's own lane keeps the even ones.  kk: the threshold
    // a lane measures (-1: none); its histogram column is its own.
    const int kpart = lane - (32 - K);  // lane >= K: the threshold it helps (< 0: none)
    const int kk = klane ? lane : kpart;
    const uint32_t dsel = klane ? (lane >= 2 * K - 32 ? 0x55555555u : FULL)
                                : (kpart >= 0 ? 0xAAAAAAAAu : 0u);
    // the bits of kk + 1 as masks, for rebuilding the recurrence words of threshold kk
    uint32_t kbm[5];
#pragma unroll
    for (int b = 0; b < 5; ++b) kbm[b] = (((kk + 1) >> b) & 1) ? FULL : 0u;

    for (int l = 0; l < HROW; ++l) hs[l * 32] = 0;

    __syncwarp();
    uint64_t lmass = 0;  // cells on lines of threshold kk longer than WSH (since the last flush, this lane)
    uint32_t lmx = 0;    // the longest of them

    int cur = -1;
    uint64_t acc = 0;  // cells since the last flush
    bool bad = false;
    SeriesDev sd{};
    int tshift = 0, tbm1 = 0, tnb = 0;
    uint32_t tmul = 0;  // 2^(32 - tshift)
    bool use_tab = false;
    uint32_t tal[KT];   // per threshold: ends of lines >= 1, >= 2, >= 3 minus those >= 4
                        // (10-bit fields at bits 0, 10, 20)
#pragma unroll
    for (int k = 0; k < KT; ++k) tal[k] = 0;
    int nrb = 0;        // row blocks since the last settle

    // tallies -> column k, rows 1..3: P(1) = f1 - f2, P(2) = f2 - f3, P(3) = f3
    auto settle = [&]() {
        uint32_t g1 = 0, g2 = 0, g3 = 0;  // lane k: the sums of threshold k
#pragma unroll
        for (int k = 0; k < KT; ++k) {
            if (k < K) {
                const uint32_t f1 = __reduce_add_sync(FULL, tal[k] & 1023u);
                const uint32_t f2 = __reduce_add_sync(FULL, (tal[k] >> 10) & 1023u);
                const uint32_t f3 = __reduce_add_sync(FULL, tal[k] >> 20);
                if (lane == k) {
                    g1 = f1;
                    g2 = f2;
                    g3 = f3;
                }
            }
            tal[k] = 0;
        }
        if (klane) {
            hs[1 * 32] += g1 - g2;
            hs[2 * 32] += g2 - g3;
            hs[3 * 32] += g3;
        }
        nrb = 0;
        __syncwarp();
    };

    // A lane's column to the short histogram of threshold kk (both lanes of a
    // helped threshold add theirs).  Row 3 of column k holds every line of
    // length >= 3; those of length >= 4 are counted again one by one (rows
    // 4..WSH and row 0, in the columns of threshold k's lane and its helper),
    // so P_k(3) is row 3 less them.  C_k is the line mass, sum over l of
    // l * P_k(l) (every recurrent cell lies on exactly one line of its
    // diagonal), and L_max the longest line.
    auto flush = [&]() {
        if (cur < 0) return;
        settle();
        const int64_t o = (int64_t)cur * lb.kstride + lb.k0 + (kk < 0 ? 0 : kk);
        uint64_t *gs = lb.hshort + o * LSH;
        uint64_t cnt = lmass;
        uint32_t lm = lmx;
        uint32_t longer = hs[0];  // this column's lines of length >= 4
        hs[0] = 0;
        auto put = [&](int l, uint32_t v) {
            if (v) {
                atomicAdd(reinterpret_cast<unsigned long long *>(gs + (l - 1)), (unsigned long long)v);
                cnt += (uint64_t)l * v;
                lm = max(lm, (uint32_t)l);
            }
        };
        if (kk >= 0) {
#pragma unroll 1
            for (int l = 4; l <= WSH; ++l) {  // row l: one bank per lane
                const uint32_t v = hs[l * 32];
                if (v) {
                    hs[l * 32] = 0;
                    longer += v;
                    put(l, v);
                }
            }
        }
        // lane k: the lines of length >= 4 its helper counted
        const uint32_t helped = __shfl_sync(FULL, longer, min(lane + 32 - K, 31));
        if (klane) {
            if (lane >= 2 * K - 32) longer += helped;
            put(1, hs[1 * 32]);
            put(2, hs[2 * 32]);
            put(3, hs[3 * 32] - longer);
            hs[1 * 32] = 0;
            hs[2 * 32] = 0;
            hs[3 * 32] = 0;
        }
        if (kk >= 0) {
            if (cnt) atomicAdd(reinterpret_cast<unsigned long long *>(lb.count + o),
                               (unsigned long long)cnt);
            if (lm) atomicMax(lb.lmax + o, lm);
        }
        lmass = 0;
        lmx = 0;
        __syncwarp();
    };

    for (;;) {
        int64_t u = 0;
        if (lane == 0) u = (int64_t)atomicAdd(reinterpret_cast<unsigned long long *>(a.queue), 1ull);
        u = __shfl_sync(FULL, u, 0);
        if (u >= a.n_units) break;
        const Unit un = unit_of<VERT, LD>(a, u);
        const int s = un.s, ub_lo = un.b_lo, ub_hi = un.b_hi;
        // counts are kept while a warp's units are of one series and stay under
        // 2^33 cells together
        const uint64_t cells = (uint64_t)(ub_hi - ub_lo) * LD * (uint64_t)(un.r_hi - un.r_lo);
        const bool full = acc + cells > (1ull << 33);
        if (s == cur && full) flush();
        acc = (s == cur && !full ? acc : 0ull) + cells;
        if (s != cur) {
            flush();
            cur = s;
            sd = a.series[s];
            uint32_t v = 0xffffffffu;   // padding: above every key
            bool ok = true;
            if (klane) {
                v = threshold_key(lb.eps[(int64_t)s * lb.kstride + lb.k0 + lane]);
                ok = threshold_ok(v);
            }
            const uint32_t prev = __shfl_up_sync(FULL, v, 1);
            if (klane && lane > 0 && prev > v) ok = false;              // not ascending
            bad = !__all_sync(FULL, ok);
            epsb[lane] = v;
            if (bad && lane == 0) set_status(a.status, 8 /*UNSORTED*/);
            // rank table: the widest buckets that still separate every pair
            // of distinct thresholds
            tshift = 22;
            for (; tshift > 0; --tshift) {
                const bool clash = klane && lane > 0 && prev != v && (prev >> tshift) == (v >> tshift);
                if (!__any_sync(FULL, clash)) break;
            }
            const uint32_t vmin = __shfl_sync(FULL, v, 0), vmax = __shfl_sync(FULL, v, K - 1);
            const int tbase = (int)(vmin >> tshift);
            tbm1 = tbase - 1;
            tnb = (int)(vmax >> tshift) - tbase + 1;
            tmul = tshift > 0 ? 1u << (32 - tshift) : 0u;
            use_tab = !bad && tshift > 0 && tnb + 2 <= TMAX;
            __syncwarp();
            if (use_tab) {
                // entry: rank of a key up to the bucket's threshold (bits 0-4),
                // rank of a key above it (bits 5-9), the threshold's offset
                // inside the bucket in the top tshift bits
                for (int q = lane; q < tnb + 2; q += 32) {
                    uint32_t e;
                    if (q == 0) {
                        e = 0u;                    // below every threshold's bucket
                    } else if (q == tnb + 1) {
                        e = (uint32_t)K | ((uint32_t)K << 5);  // above: all K thresholds are smaller
                    } else {
                        uint32_t rlo = 0, cnt = 0, off = 0;
                        for (int k = 0; k < K; ++k) {
                            const uint32_t ek = epsb[k];
                            const int eb = (int)(ek >> tshift) - tbase;
                            if (eb < q - 1) ++rlo;
                            else if (eb == q - 1) { ++cnt; off = ek * tmul; }
                        }
                        e = rlo | ((rlo + cnt) << 5) | off;
                    }
                    tab[q] = e;
                }
            }
            __syncwarp();
        }
        if (bad) continue;

        const float *ys = a.y + sd.off;
        // the full histogram row of threshold k (lane-independent base)
        const int64_t hrow = sd.ne - 1 + (VERT && lb.loi ? 1 : 0);
        uint64_t *const hbase =
            lb.hist ? lb.hist + lb.hist_off[s] + (int64_t)lb.k0 * hrow : nullptr;
        uint64_t *const gshort = lb.hshort + ((int64_t)s * lb.kstride + lb.k0) * LSH;

        // a line of threshold kk longer than WSH (rare): its length into the
        // series' short histogram or the caller's full one
        auto emit_rare = [&](uint32_t len) {
            lmx = max(lmx, len);
            lmass += len;
            hs[0] += 1u;  // row 0 of the lane's column: lines longer than WSH
            if (len <= (uint32_t)LSH)
                atomicAdd(reinterpret_cast<unsigned long long *>(gshort + (int64_t)kk * LSH + (len - 1)),
                          1ull);
            else if (hbase)
                atomicAdd(reinterpret_cast<unsigned long long *>(hbase + (int64_t)kk * hrow + (len - 1)),
                          1ull);
        };

        // Lines of length >= 4.  Lane j's mask has bit k when slot [k][j]
        // holds the word of threshold k of diagonal j; a bit transpose hands
        // lane k the diagonals of its threshold, so every lane adds to its own
        // histogram column.  In a slot, a line ends at row t - 1 for each bit t
        // of the end mask; its first row follows the nearest non-recurrent row
        // above, or it continues the run open above the word (bit 0: a line
        // ending at the previous word's last row).
        //
        // The loop is warp-uniform (its condition is a vote) and takes at most
        // one line per lane per turn with predicated steps and a predicated
        // shared reduction, so no lane's data steers the warp's control flow;
        // only a line longer than WSH branches.
        auto long_lines = [&](uint32_t mask) {
            if (!__any_sync(FULL, mask != 0u)) return;
            __syncwarp();  // every lane's slots written before other lanes read them
            // lane k: diagonals j with lines of threshold k; then the share of the
            // lane's own threshold kk (all, the even or the odd diagonals)
            uint32_t diag = transpose32(mask, lane);
            diag = __shfl_sync(FULL, diag, kk < 0 ? 0 : kk) & dsel;
            uint32_t x = 0, wq = 0, cq = 0;           // the slot being read
            const uint32_t hcol = static_cast<uint32_t>(__cvta_generic_to_shared(hs));
            while (__any_sync(FULL, (x | diag) != 0u)) {
                if (x == 0u && diag != 0u) {  // the next diagonal's slot
                    const int j = __ffs(diag) - 1;
                    diag &= diag - 1u;
                    const uint2 q = lqa[kk * LD + j];
                    x = q.x;
                    cq = q.y & CMASK;
                    const uint4 b4 = *reinterpret_cast<const uint4 *>(pl + j * 4);
                    wq = rank_le_word_lane(b4.x, b4.y, b4.z, b4.w, pl4[j], kbm);
                }
                // the lowest end bit t of the slot (lowb = 2^t; 0 when the lane
                // has no line left); the line ends at row t - 1 and starts below
                // the nearest non-recurrent row above it, or continues the run
                // open above the word when rows 0 .. t - 1 are all recurrent
                // (then clz(zb) = 32): len = t - 32 + clz(zb) + [zb == 0] * cq
                const bool has = x != 0u;
                const uint32_t lowb = x & (0u - x);
                x ^= lowb;
                const uint32_t zb = ~wq & (lowb - 1u);
                const uint32_t cz = __clz(zb);
                const uint32_t len = cz - (uint32_t)__clz(lowb) - 1u + (cz >> 5) * cq;
                red_shared_if_le(hcol + min(len, (uint32_t)WSH) * 128u, has ? len : ~0u, (uint32_t)WSH);
                if (has && len > (uint32_t)WSH) emit_rare(len);
            }
            __syncwarp();  // slots are rewritten by the next block
        };

        // the unit's bands; the rank method is fixed per unit (branch hoisted)
        auto bands = [&](auto use_table) {
            constexpr bool TABLE = decltype(use_table)::value;
            auto rank_of = [&](uint32_t key) -> uint32_t {
                if (TABLE) {
                    const uint64_t pk = (uint64_t)key * tmul;
                    // bucket - (tbase - 1) clamped to [0, tnb + 1]: max(min(a + b, c), 0)
                    const int q = __viaddmin_s32_relu((int)(uint32_t)(pk >> 32), -tbm1, tnb + 1);
                    const uint32_t e = tab[q];
                    return ((uint32_t)pk > e) ? (e >> 5) : e;  // bits 0-4: the rank
                }
                uint32_t rk = 0;
                rk += (epsb[rk + 15] < key) ? 16u : 0u;
                rk += (epsb[rk + 7] < key) ? 8u : 0u;
                rk += (epsb[rk + 3] < key) ? 4u : 0u;
                rk += (epsb[rk + 1] < key) ? 2u : 0u;
                rk += (epsb[rk] < key) ? 1u : 0u;
                return rk;
            };
            for (int b = ub_lo; b < ub_hi; ++b) {
                const int d_lo = 1 + b * LD;                 // diagonal pass: first diagonal
                const int c_lo = b * LD;                     // vertical pass: first column
                const int rows = VERT ? sd.ne : sd.ne - d_lo;  // rows of the band's longest line
                const bool last = un.r_hi >= rows;             // the band's last row chunk
                const int r_end = last ? rows : un.r_hi;
                // lengths of the lines at the chunk's first and last row, [k][lane]
                uint16_t *const edge = edges + (u * a.nb + (b - ub_lo)) * (2 * KT * LD) + lane;
                // thresholds whose line from the chunk's first row has not ended: k >= mr
                int mr = un.r_lo > 0 ? 0 : K;
                bool at_top = un.r_lo > 0;  // some lane has one
                uint32_t st[KT];
#pragma unroll
                for (int k = 0; k < KT; ++k) st[k] = 0;
                // cell phase of the 32 rows i0..i0+31, lane = row: the ranks of
                // every diagonal into the rank matrix.  INTERIOR: every cell of
                // the block inside the matrix (no bounds checks).
                auto cell_phase = [&](int i0, auto interior) {
                    constexpr bool INTERIOR = decltype(interior)::value;
                    const int i = i0 + lane;
#pragma unroll 4
                    for (int j = 0; j < LD; ++j) {
                        const int col = c_lo + j;   // vertical pass: column
                        // diagonal pass: cell (i, i + dl); vertical: (i, col)
                        const int dl = VERT ? col - i : d_lo + j;
                        const bool valid = INTERIOR || (VERT ? i < sd.ne && col < sd.ne && (lb.loi || dl != 0)
                                                             : i < sd.ne - dl);
                        uint32_t r = 31;  // outside the matrix: recurrent for no k
                        if (valid) r = rank_of(__float_as_uint(cell_dist(ys, i, dl, sd.tau, sd.m)));
                        rkm[j * 32 + rcol] = (unsigned char)r;
                    }
                };

                // The same by diagonals (WALK), lane = diagonal, the ranks staying
                // in the lane that needs them (by rows: a byte store per cell and
                // two 16-byte loads per lane).
                //  RING  compile-time embedding: the coordinate difference
                //        e(s) = y[s] - y[s + d] of row s serves the cells of rows
                //        s, s - tau, .., s - (m-1) tau, so a cell takes one
                //        subtraction and one maximum (by rows: m subtractions and
                //        1.3 window loads).
                //  delay known at run time: a window per coordinate, m
                //        subtractions of conflict-free shared loads.
                //  VERT  the lane's column vector in registers, the rows of each
                //        coordinate as a broadcast window.
                // The windows of a block come through the slots' shared memory,
                // requested one block ahead.
                constexpr int NW = RING || M == 0 ? 1 : M;   // windows
                constexpr int H = RING ? (M - 1) * TAU : 0;  // rows of differences kept
                const int tau = TAU > 0 ? TAU : sd.tau;
                float eh[RING ? H + 8 : 1], av[VERT && M > 0 ? M : 1];
                float pc[NW][2], pr[NW];
                float *const rw = reinterpret_cast<float *>(ws + O_LQ), *const cw = rw + 32 * NW;
                auto walk_fetch = [&](int i0) {
#pragma unroll
                    for (int q = 0; q < NW; ++q) {
                        // up to 94 values past the end: unsigned (dense.cuh)
                        const uint32_t r = (uint32_t)(q * tau) + (uint32_t)(i0 + H + lane);
                        const uint32_t c = r + (uint32_t)d_lo, n = (uint32_t)sd.n;
                        pr[q] = r < n ? __ldg(ys + r) : 0.f;
                        if (!VERT) {
                            pc[q][0] = c < n ? __ldg(ys + c) : 0.f;
                            pc[q][1] = c + 32u < n ? __ldg(ys + c + 32u) : 0.f;
                        }
                    }
                };
                auto walk_begin = [&](int i0) {
#pragma unroll
                    for (int x = 0; x < H; ++x) {
                        const int c = i0 + x + d_lo + lane;
                        eh[x] = c < sd.n ? __ldg(ys + i0 + x) - __ldg(ys + c) : 0.f;
                    }
                    if (VERT) {
#pragma unroll
                        for (int q = 0; q < M; ++q) av[q] = __ldg(ys + min(c_lo + lane + q * tau, sd.n - 1));
                    }
                    walk_fetch(i0);
                };
                auto walk = [&](int i0, uint32_t (&R)[8]) {
                    __syncwarp();
#pragma unroll
                    for (int q = 0; q < NW; ++q) {
                        rw[32 * q + lane] = pr[q];
                        if (!VERT) {
                            cw[64 * q + lane] = pc[q][0];
                            cw[64 * q + lane + 32] = pc[q][1];
                        }
                    }
                    __syncwarp();
                    walk_fetch(i0 + 32);
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        uint32_t key[8], r[8];
#pragma unroll
                        for (int g = 0; g < 8; g += 4) {
                            float rv[NW][4];
#pragma unroll
                            for (int q = 0; q < NW; ++q) {
                                const float4 v = *reinterpret_cast<const float4 *>(rw + 32 * q + 8 * h + g);
                                rv[q][0] = v.x;
                                rv[q][1] = v.y;
                                rv[q][2] = v.z;
                                rv[q][3] = v.w;
                            }
#pragma unroll
                            for (int t = 0; t < 4; ++t) {
                                float x[M > 0 ? M : 1];
                                if (RING) eh[RING ? H + g + t : 0] = rv[0][t] - cw[8 * h + g + t + lane];
#pragma unroll
                                for (int q = 0; q < M; ++q)
                                    x[q] = RING   ? eh[RING ? g + t + q * TAU : 0]
                                           : VERT ? rv[RING ? 0 : q][t] - av[VERT ? q : 0]
                                                  : rv[RING ? 0 : q][t] - cw[64 * q + 8 * h + g + t + lane];
                                key[g + t] = __float_as_uint(maxnorm<(M > 0 ? M : 1)>(x));
                            }
                        }
                        if (TABLE) {  // eight lookups in flight before the first is used
                            uint32_t lo[8], e[8];
#pragma unroll
                            for (int t = 0; t < 8; ++t) {
                                const uint64_t pk = (uint64_t)key[t] * tmul;
                                lo[t] = (uint32_t)pk;
                                e[t] = tab[__viaddmin_s32_relu((int)(uint32_t)(pk >> 32), -tbm1, tnb + 1)];
                            }
#pragma unroll
                            for (int t = 0; t < 8; ++t) r[t] = lo[t] > e[t] ? (e[t] >> 5) : e[t];
                        } else {
#pragma unroll
                            for (int t = 0; t < 8; ++t) r[t] = rank_of(key[t]);
                        }
                        // the byte order of the rank matrix: even rows, odd rows
                        R[2 * h] = __byte_perm(__byte_perm(r[0], r[2], 0x0040), __byte_perm(r[4], r[6], 0x0040), 0x5410);
                        R[2 * h + 1] = __byte_perm(__byte_perm(r[1], r[3], 0x0040), __byte_perm(r[5], r[7], 0x0040), 0x5410);
#pragma unroll
                        for (int x = 0; x < H; ++x) eh[x] = eh[RING ? x + 8 : 0];
                    }
                };

                // run phase of the same 32 rows: lane j takes diagonal j.  edge_block:
                // the ranks may hold cells outside the matrix, which become 31
                auto run_phase = [&](int i0, const uint32_t (&R)[8], bool edge_block) {
                    // Words 2h and 2h + 1 hold rows 8h .. 8h + 7 (byte u of word
                    // 2h: row 8h + 2u, of word 2h + 1: row 8h + 2u + 1).  X[h]
                    // interleaves their even bits (bit p of byte u of word 2h
                    // at p + 8u, of word 2h + 1 at p + 1 + 8u), Xo[h] their odd
                    // bits one place lower.  For plane p the two bits of each
                    // byte pair are masked and one multiply by
                    // 2^24 + 2^18 + 2^12 + 2^6 (shifted down by the pair's bit
                    // position) moves the eight of them, rows in order, into
                    // bits 24..31 with no two partial products meeting (so no
                    // carry reaches the top byte); three byte permutes join the
                    // four top bytes into the plane.
                    uint32_t X[4], Xo[4];
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        X[h] = (R[2 * h] & 0x55555555u) | ((R[2 * h + 1] << 1) & 0xAAAAAAAAu);
                        Xo[h] = ((R[2 * h] >> 1) & 0x55555555u) | (R[2 * h + 1] & 0xAAAAAAAAu);
                    }
                    uint32_t B[5];
#pragma unroll
                    for (int p = 0; p < 5; ++p) {
                        const int sh = p & ~1;
                        uint32_t v[4];
#pragma unroll
                        for (int h = 0; h < 4; ++h)
                            v[h] = ((p & 1 ? Xo[h] : X[h]) & (0x03030303u << sh)) * (0x01041040u >> sh);
                        const uint32_t lo = __byte_perm(v[0], v[1], 0x0073);
                        const uint32_t hi = __byte_perm(v[2], v[3], 0x7300);
                        B[p] = __byte_perm(lo, hi, 0x7610);
                    }
                    if (edge_block) {
                        // rows that the lane's diagonal (column) does not have, and
                        // the identity cell of a column unless it counts
                        const int col = c_lo + lane;
                        const int lim = VERT ? (col < rows ? rows - i0 : 0) : rows - lane - i0;
                        uint32_t out = lim >= 32 ? 0u : FULL << max(lim, 0);
                        if (VERT && !lb.loi && (uint32_t)(col - i0) < 32u) out |= 1u << (col - i0);
#pragma unroll
                        for (int p = 0; p < 5; ++p) B[p] |= out;
                    }
                    // this diagonal's planes, for rebuilding words of long lines
                    *reinterpret_cast<uint4 *>(pl + lane * 4) = make_uint4(B[0], B[1], B[2], B[3]);
                    pl4[lane] = B[4];
                    __syncwarp();  // rank rows read before slots overwrite them
                    if (at_top) {
                        // the chunk's first blocks: where the lines that touch its
                        // first row end (thresholds nest, so those still open are
                        // the ones from some rank on)
                        int still = K;
#pragma unroll 1
                        for (int k = 0; k < K; ++k) {
                            uint32_t km[5];
#pragma unroll
                            for (int p = 0; p < 5; ++p) km[p] = (((k + 1) >> p) & 1) ? FULL : 0u;
                            const uint32_t w = rank_le_word_lane(B[0], B[1], B[2], B[3], B[4], km);
                            if (k >= mr) {
                                if (w != FULL) edge[k * LD] = (uint16_t)(i0 - un.r_lo + __ffs(~w) - 1);
                                else still = min(still, k);
                            }
                        }
                        mr = still;
                        at_top = __any_sync(FULL, mr < K);
                    }
                    uint32_t lmask = 0;  // thresholds whose word ends lines of length >= 4
#pragma unroll
                    for (int k = 0; k < KT; ++k) {
                        if (k < K) {
                            const uint32_t w = rank_le_word(B, k);
                            const uint32_t s0 = st[k];
                            // row t of p_n = row t - n (rows above the block: the
                            // previous word's top four rows, kept in the state)
                            const uint32_t p1 = __funnelshift_l(s0, w, 1);
                            const uint32_t p2 = __funnelshift_l(s0, w, 2);
                            const uint32_t p3 = __funnelshift_l(s0, w, 3);
                            const uint32_t p4 = __funnelshift_l(s0, w, 4);
                            // bit t: a line ends at row t - 1 (t = 0: the previous
                            // block's last row) and is at least 1, 2, 3, 4 long
                            const uint32_t e1 = p1 & ~w;
                            const uint32_t e2 = e1 & p2;
                            const uint32_t e3 = e2 & p3;
                            const uint32_t e4 = e3 & p4;
                            // every line counts towards lengths >= 1, 2, 3; those of
                            // length >= 4 are measured one by one after the loop
                            // (rare for noisy series) and taken off length 3 at the flush
                            tal[k] += __popc(e1) + (__popc(e2) << 10) + (__popc(e3) << 20);
                            if (e4) {  // the reader takes the run length from the state's low bits
                                lq[k * LD] = make_uint2(e4, s0);
                                lmask |= 1u << k;
                            }
                            // the new state: top rows of this word and the run open at
                            // its last row.  c = 32 only for an all-ones word, whose run
                            // continues the one open above: c + s0 has the old length
                            // + 32 in its low bits (the sum stays under 2^28), and its
                            // top bits are overwritten by the word's, all ones.
                            const uint32_t c = __clz(~w);
                            st[k] = (w & TOP4) | (s0 * (c >> 5) + c);
                        }
                    }
                    long_lines(lmask);
                };

                // One copy of the block's code for interior blocks and edges: the
                // edges' ranks are corrected in the planes.  With a copy for each
                // (and a select per cell) warps of short series alternated between
                // the two, and both did not stay in the instruction cache: line pass
                // over 10^4 series of 200, K = 13, m = 1, 2, 3 (tau = m): 0.83, 1.07,
                // 0.92 ms with two copies, 0.50, 0.57, 0.55 with one (25 series of
                // 2e4, K = 20: 6.6, 8.9, 6.9 and 6.5, 8.1, 6.9).
                // The packed tallies take SETTLE row blocks before a field could overflow.
                int i0 = un.r_lo;
                if constexpr (WALK) walk_begin(i0);
                for (; i0 < r_end; i0 += 32) {
                    // interior row blocks: every cell inside the matrix (and off the
                    // identity line)
                    // (full sweeps decide before the walk, the others after it, by the
                    // registers that ptxas finds: K = 13, m = tau = 3 6 % less so)
                    auto inside = [&]() -> bool {
                        return VERT ? c_lo + LD <= sd.ne && i0 + 32 <= rows &&
                                          (lb.loi || i0 + 32 <= c_lo || i0 >= c_lo + LD)
                                    : i0 + 32 <= rows - (LD - 1);
                    };
                    uint32_t R[8];
                    const bool early = FK && !inside();
                    if constexpr (WALK) {
                        walk(i0, R);
                    } else {
                        if (inside()) cell_phase(i0, std::true_type{});
                        else cell_phase(i0, std::false_type{});
                        __syncwarp();
                        const uint4 ra = *reinterpret_cast<const uint4 *>(rkm + lane * 32);
                        const uint4 rb = *reinterpret_cast<const uint4 *>(rkm + lane * 32 + 16);
                        R[0] = ra.x; R[1] = ra.y; R[2] = ra.z; R[3] = ra.w;
                        R[4] = rb.x; R[5] = rb.y; R[6] = rb.z; R[7] = rb.w;
                    }
                    run_phase(i0, R, WALK && (FK ? early : !inside()));
                    if (++nrb == SETTLE) settle();
                }
                // lines that reach the end of a diagonal, or of the chunk, exactly at
                // a block's last row: a line of length c ending just above a word
                // (end bit 0)
                uint32_t bmask = 0;
#pragma unroll
                for (int k = 0; k < KT; ++k) {
                    if (k < K) {
                        const uint32_t c = st[k] & CMASK;
                        tal[k] += c == 0 ? 0u : c == 1 ? 1u : c == 2 ? 0x401u : 0x100401u;
                        if (c >= 4) {
                            lq[k * LD] = make_uint2(1u, c);
                            bmask |= 1u << k;
                        }
                        if (!last) edge[(KT + k) * LD] = (uint16_t)c;
                        if (k >= mr) edge[k * LD] = (uint16_t)c;  // from the chunk's first row to its last
                    }
                }
                long_lines(bmask);
            }
        };
        if (use_tab) bands(std::true_type{});
        else bands(std::false_type{});
    }
    flush();
}

}  // namespace rqa

namespace rqa {
using LinesKernel = void (*)(CellArgs, LineBufs, int, uint16_t *);
// Instantiations, one group per translation unit (they compile in parallel).
// full: the diagonal pass's variant for a sweep of exactly LINE_KMAX thresholds
LinesKernel lines_kernel_m3t3(bool vert, bool full);
LinesKernel lines_kernel_m3t1(bool vert, bool full);
LinesKernel lines_kernel_m1t1(bool vert, bool full);
LinesKernel lines_kernel_generic(int m, bool vert);
}  // namespace rqa
