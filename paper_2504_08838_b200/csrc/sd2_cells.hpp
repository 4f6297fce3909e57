// Cells: the device layout of a GAP4 handle for panels of activation rows, in the order of a tensor-core operand.
//
// The strip layout (sd2_format.hpp) is built to be gathered from, entry by entry; its work grows with every activation
// row.  For several rows a handle also keeps this one, which a warp turns into the A fragments of mma.m16n8k16 (16 weight
// rows x 16 columns) whatever the pattern:
//
//   - Rows are cut into tiles of 16, columns into cells of 128.  A warp takes one cell of one tile.  Lane l = 4 g + t holds
//     weight rows g and g + 8; of each it owns, for u = 0..3, the eight columns 32 u + 8 t + i, i = 0..7: four *pairs*
//     of neighbours.  Pairs 0 and 1 of a unit feed one mma step, pairs 2 and 3 the next.
//   - A pair of which anything is kept is one 32-bit word (the low column in the low half, zero for a dropped one); the
//     others take no room.  mask[l] has bit 16 r + 4 u + i set iff pair i of unit u of row g + 8 r has a word.
//   - The words of a lane's row g stand one above the other in column l of a matrix of H rows x 32 words, from row 0 up;
//     those of row g + 8 in column pi(l), from row H - 1 down.  pi matches lanes with many words in one row to lanes
//     with few in the other, which keeps H close to the mean.  Whatever rows 32 lanes read, they read 32 different banks.
//
// Bytes per dense slot at 50 % density: 1.61 (three of four pairs have a word; the strips take 1.28).  Packing the values
// without the pairs' zeros takes 1.39, but its expansion by byte permutations ran at 18 slots per clock and SM; this
// one, a predicated load per pair, runs at 33 (29 for sixteen activation rows), and HBM brings 15.
//
// Two CTAs share a tile: one takes the first ceil(D / 2) cells of its columns, the other the rest.  The cells of each
// share stand together, tile by tile, so that a CTA's run of tiles is one run of bytes.
//
//   cell    u32 mask[32], u8 pi[32] (4 x column), u32 words[H][32].  Bit 7 of pi[6 k + i] is bit i of the height H of the
//           k-th cell from this one on, k = 0..3: a reader of four consecutive cells finds them from the first one.
//   sec0    u32 cell_off[T * D + 1] (32-byte units into sec1), in order of share, then tile, then column
//   sec1    cells

#pragma once

#include "sd2_format.hpp"

namespace sd2 {

constexpr int kTileRows = 16;
constexpr int kCellCols = 128;
constexpr int kCellHeaderBytes = 128 + 32;

constexpr int kChunkCells = 4;        // consecutive cells of a share that travel in one copy, at most

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
    uint32_t bits[32];
    uint32_t words[2][32][17];
    uint8_t n_words[2][32];
    std::memset(bits, 0, sizeof bits);
    std::memset(n_words, 0, sizeof n_words);
    const int64_t left = K - k0;
    const int cols = left < kCellCols ? (int)left : kCellCols;
    uint16_t wv[kCellCols] = {};
    for (int row = 0; row < kTileRows && m0 + row < M; ++row) {
        // the row's kept values, zero elsewhere, and which of them are kept (no branch on a single one: those are coin tosses)
        const uint16_t* wr = W + (m0 + row) * K + k0;
        uint8_t kept[kCellCols] = {};
        if (mask) {
            const uint8_t* mr = mask + (m0 + row) * K + k0;
            for (int c = 0; c < cols; ++c) kept[c] = mr[c] != 0;
        } else {
            for (int c = 0; c < cols; ++c) kept[c] = (wr[c] & 0x7FFF) != 0;
        }
        for (int c = 0; c < cols; ++c) wv[c] = (uint16_t)(wr[c] & -(int)kept[c]);
        const int r = row >> 3;
        for (int t = 0; t < 4; ++t) {
            const int l = 4 * (row & 7) + t;
            uint32_t n = 0, b = 0;
            for (int u = 0; u < 4; ++u)
                for (int i = 0; i < 4; ++i) {
                    const int c = 32 * u + 8 * t + 2 * i;
                    const uint32_t any = kept[c] | kept[c + 1];
                    words[r][l][n] = (uint32_t)wv[c] | (uint32_t)wv[c + 1] << 16;
                    n += any;
                    b |= any << (4 * u + i);
                }
            bits[l] |= b << (16 * r);
            n_words[r][l] = (uint8_t)n;
        }
    }
    // lanes by the words of their first row, most first, and by those of their second, fewest first; equal ranks share a column
    int place[2][18] = {}, col_of_rank[32], H = 0;
    for (int l = 0; l < 32; ++l) {
        ++place[0][17 - n_words[0][l]];
        ++place[1][n_words[1][l] + 1];
    }
    for (int n = 1; n < 18; ++n) {
        place[0][n] += place[0][n - 1];
        place[1][n] += place[1][n - 1];
    }
    uint8_t pi[32];
    for (int l = 0; l < 32; ++l) col_of_rank[place[0][16 - n_words[0][l]]++] = l;
    for (int l = 0; l < 32; ++l) {
        const int c = col_of_rank[place[1][n_words[1][l]]++];
        pi[l] = (uint8_t)(4 * c);
        if (n_words[0][c] + n_words[1][l] > H) H = n_words[0][c] + n_words[1][l];
    }
    const size_t at = out.size();
    out.resize(at + kCellHeaderBytes + (size_t)H * 128, 0);
    uint8_t* p = out.data() + at;
    std::memcpy(p, bits, 128);
    std::memcpy(p + 128, pi, 32);
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
            if (src.empty()) continue;
            const int64_t c0 = first_cell[r] + i * share_cells(g.D, r);
            uint8_t* dst = im.data + sec1_off + (size_t)off[(size_t)c0] * 32;
            std::memcpy(dst, src.data(), src.size());
            for (int64_t c = c0; c < c0 + share_cells(g.D, r); ++c) {
                uint32_t heights = 0;                     // of this cell and the three that follow it
                for (int64_t k = 0; k < kChunkCells && c + k < n_cells; ++k)
                    heights |= ((off[(size_t)(c + k + 1)] - off[(size_t)(c + k)]) * 32u - kCellHeaderBytes) / 128u << (6 * k);
                uint8_t* pi = im.data + sec1_off + (size_t)off[(size_t)c] * 32 + 128;
                for (int l = 0; l < 6 * kChunkCells; ++l) pi[l] |= (uint8_t)((heights >> l & 1u) << 7);
            }
        }
    im.sec1_off = sec1_off;
    im.bytes = sec1_off + (size_t)units * 32;
    im.max_chunk = (int)(max_run * 32u);
    return im;
}

}  // namespace sd2
