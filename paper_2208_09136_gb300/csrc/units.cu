// How a launch's work is cut into units (host arithmetic; the rules and their
// reasons stand at the declarations in rqa_internal.h, unit_of in dense.cuh is
// the device's side).
#include <algorithm>
#include <cstdint>

#include "rqa_internal.h"

namespace rqa {

Split split_cells(uint64_t cells, int nb, int sm_count)
{
    const uint64_t block = (uint64_t)nb * DB * ROW_BLOCK, ctas = (uint64_t)sm_count * 2;
    const uint64_t least = std::min<uint64_t>(std::max<uint64_t>(cells / (block * ctas), 2), 8);
    const uint64_t blocks = std::max<uint64_t>(cells / (block * ctas * 6), least);
    // more than 585 blocks only to keep the units, 2^30 of them, in the launch's 31 bits
    const uint64_t most = std::max<uint64_t>(585, cells / (block << 30) + 1);
    return Split{nb, ROW_BLOCK * (int)std::min(blocks, most)};
}

Split split_lines(uint64_t cells, int64_t bands, int32_t ne_max, int unit_bands, int sm_count)
{
    const int64_t warps = (int64_t)sm_count * 16;
    const int64_t cap = std::max<int64_t>(1, ((int64_t)1 << 28) / std::max(ne_max, 1));
    const int32_t whole = (std::max(ne_max, 1) + 31) / 32 * 32;  // rows of the longest band
    Split sp{};
    if (bands >= 8 * warps) {
        sp.nb = (int)std::min<int64_t>(64, bands / (8 * warps));
        sp.rc = whole;
    } else {
        sp.nb = 1;
        const uint64_t blocks = cells / ((uint64_t)LINE_BAND * 32 * (uint64_t)warps * 2);  // half a warp's share
        if (whole <= 32 * 32 && (uint64_t)whole <= 4 * 32 * blocks) sp.rc = whole;
        else sp.rc = (int)std::min<uint64_t>(32 * std::max<uint64_t>(blocks, 8), (uint64_t)std::min(whole, LINE_CHUNK_MAX));
    }
    if (unit_bands > 0) sp.nb = unit_bands;  // a tuned size
    sp.nb = (int)std::min({(int64_t)sp.nb, cap, (int64_t)whole / LINE_BAND});  // edge scratch is sized by nb
    return sp;
}

int64_t units_of_series(int64_t ne, const Split &sp, bool vert, int w)
{
    int64_t n = 0;
    for (int64_t r = 0; r < ne; r += sp.rc) {
        const int64_t bands = vert ? (ne + w - 1) / w : (ne - 1 - r + w - 1) / w;
        n += (bands + sp.nb - 1) / sp.nb;
    }
    return n;
}

int64_t cut_bands(int64_t ne, const Split &sp, bool vert)
{
    const int64_t rows = vert ? ne : ne - 1;
    if (rows <= sp.rc) return 0;
    return ((vert ? ne : rows - sp.rc) + LINE_BAND - 1) / LINE_BAND;
}

}  // namespace rqa
