// Internal declarations shared by the host API and the kernels of librqa.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace rqa {

// FP32 distances are non-negative, so their bit patterns ("keys") order like
// the values and use only bits 30..0.  Exact selection splits a key into an
// 11-bit coarse digit (bits 30..20), a 10-bit middle digit (19..10) and a
// 10-bit low digit (9..0).
constexpr int KMAX = 127;        // targets per series and call
constexpr int LINE_KMAX = 20;    // targets per line-pass sweep (per-lane run state in registers)
constexpr int LINE_BAND = 32;    // diagonals (columns) per warp band of the line pass: one per lane
constexpr int MID_GROUPS = 48;   // middle-round groups per launch (4 KB of shared bins each)
constexpr int COARSE_SHIFT = 20;
constexpr int NCOARSE = 1 << 11;   // 2048 coarse buckets
constexpr int NFINE = 1 << 10;     // 1024 bins per middle / low digit group
constexpr int NHASH_BITS = 12;     // final round: hashed table of the targets' 21-bit prefixes
constexpr int NHASH = 1 << NHASH_BITS;
constexpr int NSUB_MAX = 24;       // bracket-subdivided coarse buckets per series
constexpr int LSH = 64;            // line lengths 1..LSH counted in shared memory
constexpr int LMIN_MAX = 8;        // entries of an lmin list
constexpr int THREADS = 256;       // threads per CTA of the cell kernels
constexpr int DB = 128;            // diagonals (columns) per warp band of the cell walk
constexpr int LINE_TILE_DEFAULT = 16;  // rqa_tuning.tile when none was set (reported only)
constexpr int LINE_NE_MAX = (1 << 26) - 1;  // vectors per series the line pass counts exactly
constexpr int64_t COUNT_NE_MAX = (int64_t)3 << 25;  // vectors per series the counting rounds take
constexpr int WARPS = THREADS / 32;

// Counting rounds of the selection.
enum Round : int {
    R_COARSE = 0,      // coarse digit of every key
    R_COARSE_SUB = 1,  // coarse digit, bracket buckets already split by middle digit
    R_MID = 2,         // middle digit of keys whose coarse digit holds a target
    R_FINAL = 3        // low digit of keys whose 21-bit prefix holds a target
};

struct SeriesDev {
    int64_t off;      // first value of the series in the batch buffer
    int32_t n;        // N
    int32_t ne;       // Ne = N - (m-1) tau
    int32_t m, tau;
    uint64_t P;       // Ne (Ne - 1) / 2
};

// Device buffers of the selection state; [s*K + k] unless stated.
struct SelBufs {
    const uint64_t *T;     // target counts
    uint32_t *prefix;      // key bits fixed so far
    uint8_t *level;        // 1: coarse digit known, 2: 21-bit prefix known
    uint64_t *rank;        // rank of the target within its current key interval
    uint64_t *below;       // keys below the current key interval
    int8_t *tab_sub;       // [s][NCOARSE] bracket split buckets -> group, -1
    int8_t *tab_mid;       // [s][NCOARSE] coarse bucket -> middle group, -1
    uint32_t *tab_hash;    // [s][NHASH] final round: prefix | group << 21 at slot (prefix * mul) >> 20,
                           // 0x1fffff empty
    uint32_t *hash_mul;    // [s]: the slot multiplier, 0 = no collision-free one
    int32_t *n_sub, *n_mid, *n_fin;   // [s]
    uint32_t *range;       // [s][2]: keys the next filtered round can count, inclusive
    uint8_t *redo;         // [s]: 1 = the plain coarse round runs for this series
    uint64_t *hist;        // [s][hstride]: NCOARSE coarse bins then fine bins
    int64_t hstride;
};

struct CellArgs {
    const float *y;
    const SeriesDev *series;
    int32_t g0, gn;          // middle round: the groups [g0, g0 + gn) this launch counts
    // work units along the series order[0..n_pos)
    const int32_t *order;    // series, largest first
    const int64_t *uprefix;  // n_pos + 1 prefix of unit counts along order
    int32_t n_pos;
    int32_t m_max;           // largest embedding dimension of the batch
    int32_t nb, rc;          // bands per unit and rows per unit (a multiple of the kernel's row block)
    const int64_t *mprefix;  // line pass: n_pos + 1 prefix of the bands cut into several row chunks ...
    int64_t n_merge;         // ... and their number
    int32_t line_ctas;       // persistent CTAs of the line pass per SM (0: as many as fit)
    int64_t n_units;
    unsigned int *queue;   // ticket counter (64-bit aligned), zeroed before launch
    int *status;
};

// How a launch of the cell walk cuts its work: units of `nb` bands of DB
// diagonals over `rc` rows.
struct Split {
    int nb, rc;
};
constexpr int ROW_BLOCK = 28;  // rows per block of the cell walk (units start on block boundaries)
constexpr int COUNT_NB = 8;  // bands per unit of the counting rounds: one per warp of a CTA
// About six units per CTA (two CTAs per SM) over the whole launch, and rows
// per unit between 8 and 585 blocks: shorter chunks pay their first window
// loads over too few cells (lorenz-n1e4: 771 us with at least 8 blocks, 848 with
// 2), longer ones leave a tail.  A launch with fewer units than CTAs even so is
// bound by one unit's latency and goes down to 2 blocks (two series of 2003
// values: 135 us with 8, 87 with 2).
Split split_cells(uint64_t cells, int nb, int sm_count);
// Units of the line pass over series with these cells and bands of LINE_BAND
// diagonals, one warp each: runs of whole bands, about eight units per resident
// warp (16 per SM), so the tail stays short; below that single bands.  These are
// cut into row chunks for about two units per warp (four: 876 us instead of 805
// for lorenz-n1e4, 391 instead of 346 for three series of 7001), of at least 256
// rows (a chunk's edges and its first window cost about three blocks of 32 rows),
// unless the longest band has at most 32 blocks and at most twice a warp's share of
// all of them: short chunks then cost more than the tail (line pass of a call, whole
// and in chunks: 300 series of 500, 135 and 167 us; 100 of 1000, 162 and 199).
// Longer bands gain from chunks (vertical pass of 30 of 2000: 421 whole, 402), and
// so do short ones that are few (30 of 1000: 137 and 103).  A unit covers at most
// 2^33 cells, so the warp's 32-bit counts of lines of length >= 4 (each line and
// the cell after it: >= 5 cells) stay exact.
Split split_lines(uint64_t cells, int64_t bands, int32_t ne_max, int unit_bands, int sm_count);
// Units of a series of ne vectors with bands of w diagonals (vert: the vertical
// pass, every column over every row).
int64_t units_of_series(int64_t ne, const Split &sp, bool vert, int w = DB);
// Bands of LINE_BAND diagonals (columns) of a series that are longer than a row
// chunk: the lower ones, and all or none in the vertical pass.
int64_t cut_bands(int64_t ne, const Split &sp, bool vert);

// Kernels (launch wrappers return cudaGetLastError()).
cudaError_t launch_check_finite(const float *y, int64_t n, int *status, cudaStream_t st);
// embed: the Embed code of the batch (rqa_common.cuh), picks the distance kernel variant.
cudaError_t launch_count(int round, const CellArgs &a, const SelBufs &sb, int K, int grid,
                         int embed, cudaStream_t st);
cudaError_t launch_select(int round, const SelBufs &sb, int s_begin, int n_series, int K, float *eps_out,
                          uint64_t *le_out, uint64_t *lt_out, int *status, cudaStream_t st);

// The whole selection (and the finiteness check) of short series, one CTA
// each.  Taken when every series has at most SMALL_NE vectors and the batch few
// enough cells that its row-per-warp walk (25 instructions per 32 cells where
// the counting rounds take 7 to 10) stays shorter than their dozen launches:
// 2^17 cells per SM, one series of 512 vectors per SM.
constexpr int SMALL_NE = 512;
bool small_select_ok(int K, int32_t ne_max, int64_t n_max, uint64_t total_cells, int sm_count);
cudaError_t launch_select_small(const float *y, const SeriesDev *series, int S, int n_max, const uint64_t *T, int K,
                                float *eps_out, uint64_t *le_out, uint64_t *lt_out, int *status, cudaStream_t st);

struct LineBufs {
    const float *eps;      // [s*kstride + k], ascending per series
    uint64_t *count;       // [s*kstride + k]
    uint32_t *lmax;        // [s*kstride + k]
    uint64_t *hshort;      // [s][kstride][LSH]: P_k(l) for l = 1..LSH
    uint64_t *hist;        // caller's full histogram or nullptr
    const int64_t *hist_off;  // device [S+1] offsets into hist (nullptr if no hist)
    int32_t k0;            // line pass: first target of this launch's group
    int32_t kstride;       // targets per series in all arrays above (the call's K)
    int32_t loi;           // vertical pass: the cells (j, j) are recurrent
};
// vert: vertical lines of the whole matrix, over columns instead of diagonals.
// chunks: the units are row chunks, so a second kernel joins the lines at their
// boundaries; edges then holds LINE_EDGE_BYTES per unit and band of it: per
// threshold and diagonal the length of the line that touches the chunk's first
// and its last row.
constexpr size_t LINE_EDGE_BYTES = 2 * LINE_KMAX * LINE_BAND * 2;
constexpr int LINE_CHUNK_MAX = 65504;  // rows of a chunk: its line lengths fit 16 bits
cudaError_t launch_lines(const CellArgs &a, const LineBufs &lb, int K, int grid, int embed, bool vert,
                         bool chunks, uint16_t *edges, cudaStream_t st);
cudaError_t launch_finalize_det(const LineBufs &lb, const SeriesDev *series, int S, int K,
                                const int32_t *lmin_dev, int n_lmin, double *det,
                                double *det_avg, bool loi, cudaStream_t st);
cudaError_t launch_line_measures(const uint64_t *hist, const int64_t *hoff_dev, int S, int K,
                                 const int32_t *lmin_dev, int n_lmin, double *L_out,
                                 double *E_out, double *L_avg, double *E_avg, bool loi,
                                 cudaStream_t st);
cudaError_t launch_grid_select(const CellArgs &a, int S, int n_thr, float *thr, uint64_t *hist,
                               const int32_t *rr_num_dev, int rr_den, int K, float *eps_out,
                               double *rr_out, uint64_t *count_out, int grid, int embed,
                               cudaStream_t st);
cudaError_t launch_lam_tt(const uint64_t *hist, const int64_t *hoff_dev, int S, int K,
                          const int32_t *vmin_dev, int n_vmin, double *lam_out, double *tt_out,
                          double *lam_avg, double *tt_avg, cudaStream_t st);
cudaError_t launch_finalize_hist(const LineBufs &lb, const SeriesDev *series, int S, int K,
                                 uint64_t *stencil, cudaStream_t st);

}  // namespace rqa
