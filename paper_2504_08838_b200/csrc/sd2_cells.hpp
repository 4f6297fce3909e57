// Cells: the device layout of a GAP4 handle for panels of activation rows, in the order of a tensor-core operand.
//
// The strip layout (sd2_format.hpp) is built to be gathered from, entry by entry; its work grows with every activation
// row.  For several rows a handle also keeps this one: a bitmask (one bit per dense slot) plus the packed kept values,
// arranged so that a warp turns a compressed cell into the B fragments of mma.m16n8k16 (8 weight rows x 16 columns)
// with table look-ups by byte permutation, whatever the pattern:
//
//   - Rows are cut into tiles of 8, columns into cells of 256 = two halves of 128.  A warp takes one cell of one
//     tile.  Lane l = 4 g + t holds weight row g; of half h it owns, for u = 0..3, the eight columns
//     128 h + 32 u + 8 t + i, i = 0..7: a *unit*.  Slots 0..3 of a unit feed one mma step, slots 4..7 the next.
//   - mask[h][l] has bit 8 u + i set iff the slot is kept.
//   - A unit's kept values fill whole 32-bit words from both ends: slots 0..3 from the front (a pair of slots that are
//     both kept takes two halfwords, low slot first; a single one takes one), slots 4..7 from the back (a pair's
//     high slot takes the later halfword).  An odd count leaves one halfword of zero in the middle.  So the four
//     values a step needs sit in the first two or the last two words of the unit, at a place that follows from the
//     mask alone, and two byte permutations per register put them (and zeros) where the tensor core wants them.
//   - The words of a lane's four units of half 0 stand one above the other in column l of a matrix of H rows x 32
//     words, from row 0 up; those of half 1 in column pi(l), from row H - 1 down.  pi matches lanes with many words
//     in half 0 to lanes with few in half 1, which keeps H close to the mean (18.7 rows where 18.0 words are used,
//     at 50 % density).  Whatever rows 32 lanes read, they read 32 different banks.
//
// Two CTAs share a tile: one takes the first ceil(D / 2) cells of its columns, the other the rest.  The cells of each
// share stand together, tile by tile, so that a CTA's run of tiles is one run of bytes.
//
//   cell    u32 mask[2][32], u8 pi[32] (4 x column), u32 words[H][32]
//   sec0    u32 cell_off[T * D + 1] (32-byte units into sec1), in order of share, then tile, then column
//   sec1    cells

#pragma once

#include "sd2_format.hpp"

namespace sd2 {

constexpr int kTileRows = 8;
constexpr int kCellCols = 256;
constexpr int kHalfCols = 128;
constexpr int kCellHeaderBytes = 2 * 128 + 32;

constexpr int kChunkCells = 5;        // consecutive cells of a share that travel in one copy, at most

struct CellGeom {
    int64_t T;        // row tiles
    int D;            // cells per tile
};

// cells of share r (0, 1) of a tile
SD2_HD int share_cells(int D, int r) { return r == 0 ? (D + 1) / 2 : D / 2; }

inline CellGeom cell_geometry(int64_t M, int64_t K)
{
    CellGeom g;
    g.T = (M + kTileRows - 1) / kTileRows;
    g.D = (int)((K + kCellCols - 1) / kCellCols);
    return g;
}

struct CellImage {
    uint8_t* data = nullptr;       // sec0 padded to 256 bytes, then sec1 (malloc)
    size_t sec1_off = 0, bytes = 0;
    int max_chunk = 0;             // bytes of the largest run of kChunkCells cells
    int status = 0;
};

// One cell of the tile that starts at row m0, columns from k0; appended to `out`.
inline void pack_cell(const uint16_t* W, const uint8_t* mask, int64_t M, int64_t K, int64_t m0, int64_t k0, std::vector<uint8_t>& out)
{
    uint32_t bits[2][32];
    uint32_t words[2][32][16];
    uint8_t n_words[2][32];
    std::memset(bits, 0, sizeof bits);
    std::memset(n_words, 0, sizeof n_words);
    for (int g = 0; g < kTileRows && m0 + g < M; ++g) {
        const uint16_t* wr = W + (m0 + g) * K;
        const uint8_t* mr = mask ? mask + (m0 + g) * K : nullptr;
        for (int h = 0; h < 2; ++h)
            for (int u = 0; u < 4; ++u)
                for (int t = 0; t < 4; ++t) {
                    const int l = 4 * g + t;
                    const int64_t c0 = k0 + kHalfCols * h + 32 * u + 8 * t;
                    const int nc = c0 >= K ? 0 : (int)(K - c0 < 8 ? K - c0 : 8);
                    uint32_t b = 0;
                    if (mr) { for (int i = 0; i < nc; ++i) b |= (mr[c0 + i] ? 1u : 0u) << i; }
                    else { for (int i = 0; i < nc; ++i) b |= ((wr[c0 + i] & 0x7FFF) ? 1u : 0u) << i; }
                    if (!b) continue;
                    bits[h][l] |= b << (8 * u);
                    const int nw = (__builtin_popcount(b) + 1) / 2;
                    uint16_t hw[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                    int f = 0, e = 2 * nw - 1;
                    for (int i = 0; i < 4; ++i)
                        if (b >> i & 1) hw[f++] = wr[c0 + i];
                    for (int i = 4; i < 8; i += 2) {
                        if (b >> (i + 1) & 1) hw[e--] = wr[c0 + i + 1];
                        if (b >> i & 1) hw[e--] = wr[c0 + i];
                    }
                    std::memcpy(words[h][l] + n_words[h][l], hw, (size_t)nw * 4);
                    n_words[h][l] = (uint8_t)(n_words[h][l] + nw);
                }
    }
    // lanes of half 0 by words, most first; lanes of half 1 by words, fewest first; equal ranks share a column
    int col_of_rank[32], r = 0, H = 0;
    for (int n = 16; n >= 0; --n)
        for (int l = 0; l < 32; ++l)
            if (n_words[0][l] == n) col_of_rank[r++] = l;
    uint8_t pi[32];
    r = 0;
    for (int n = 0; n <= 16; ++n)
        for (int l = 0; l < 32; ++l)
            if (n_words[1][l] == n) {
                const int c = col_of_rank[r++];
                pi[l] = (uint8_t)(4 * c);
                if (n_words[0][c] + n > H) H = n_words[0][c] + n;
            }
    const size_t at = out.size();
    out.resize(at + kCellHeaderBytes + (size_t)H * 128, 0);
    uint8_t* p = out.data() + at;
    std::memcpy(p, bits, 256);
    std::memcpy(p + 256, pi, 32);
    uint32_t* v = (uint32_t*)(p + kCellHeaderBytes);
    for (int l = 0; l < 32; ++l) {
        for (int w = 0; w < n_words[0][l]; ++w) v[(size_t)w * 32 + l] = words[0][l][w];
        for (int w = 0; w < n_words[1][l]; ++w) v[(size_t)(H - 1 - w) * 32 + pi[l] / 4] = words[1][l][w];
    }
}

inline CellImage pack_cells(const uint16_t* W, const uint8_t* mask, int64_t M, int64_t K)
{
    CellImage im;
    const CellGeom g = cell_geometry(M, K);
    const int64_t n_cells = g.T * g.D;
    if (n_cells > 0x3FFFFFFF) { im.status = -2; return im; }
    const size_t sec1_off = align256((size_t)(n_cells + 1) * 4);
    std::vector<std::vector<uint8_t>> tiles((size_t)g.T * 2);
    std::vector<uint32_t> off((size_t)n_cells + 1);       // first the cells' sizes, then their places
    const int64_t first_cell[2] = {0, g.T * share_cells(g.D, 0)};
#pragma omp parallel for schedule(dynamic, 4)
    for (int64_t i = 0; i < g.T; ++i)
        for (int r = 0, d = 0; r < 2; ++r) {
            const int n = share_cells(g.D, r);
            std::vector<uint8_t>& out = tiles[(size_t)(r * g.T + i)];
            out.reserve((size_t)n * 3072);
            for (int j = 0; j < n; ++j, ++d) {
                const size_t start = out.size();
                pack_cell(W, mask, M, K, i * kTileRows, (int64_t)d * kCellCols, out);
                off[(size_t)(first_cell[r] + i * n + j)] = (uint32_t)((out.size() - start) / 32);
            }
        }
    uint64_t units = 0;
    uint32_t max_run = 0;
    for (int64_t c = 0; c < n_cells; ++c) {
        const uint32_t n = off[(size_t)c];
        off[(size_t)c] = (uint32_t)units;
        units += n;
        const uint32_t from = c >= kChunkCells - 1 ? off[(size_t)(c - (kChunkCells - 1))] : 0u;
        if ((uint32_t)units - from > max_run) max_run = (uint32_t)units - from;
    }
    if (units > 0xFFFFFFF0ull) { im.status = -2; return im; }
    off[(size_t)n_cells] = (uint32_t)units;
    im.data = (uint8_t*)lib_malloc(sec1_off + (size_t)units * 32);
    if (!im.data) { im.status = -3; return im; }
    std::memset(im.data, 0, sec1_off);
    std::memcpy(im.data, off.data(), off.size() * 4);
#pragma omp parallel for schedule(static)
    for (int64_t i = 0; i < g.T; ++i)
        for (int r = 0; r < 2; ++r) {
            const std::vector<uint8_t>& src = tiles[(size_t)(r * g.T + i)];
            if (!src.empty()) std::memcpy(im.data + sec1_off + (size_t)off[(size_t)(first_cell[r] + i * share_cells(g.D, r))] * 32, src.data(), src.size());
        }
    im.sec1_off = sec1_off;
    im.bytes = sec1_off + (size_t)units * 32;
    im.max_chunk = (int)(max_run * 32u);
    return im;
}

}  // namespace sd2
