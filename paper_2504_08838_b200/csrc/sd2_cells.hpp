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
// Bytes per dense slot at 50 % density: 1.65 (three of four pairs have a word; the strips take 1.28).  Packing the values
// without the pairs' zeros takes 1.39, but its expansion by byte permutations ran at 18 slots per clock and SM; this
// one, a predicated load per pair, ran at 33 (29 for sixteen activation rows) with chains of mma, and HBM brings 15.
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

// Panel cells: the same words and header for a tensor-memory operand.  A block of 128 rows x 64 columns is a chunk of four cells of
// 32 rows; lane l holds row l of its cell, of which columns 0..31 count as row g above and columns 32..63 as row g + 8: bit
// 16 r + e of mask[l] is pair e (columns 32 r + 2 e and the next).  Blocks stand panel by panel, ascending columns inside a panel.
constexpr int kPanelRowsOfBlock = 128;
constexpr int kPanelBlockCols = 64;

struct CellGeom {
    int64_t T;        // row tiles (panel cells: row panels)
    int D;            // cells per tile (blocks per panel)
    int per;          // cells of a place in this grid: 1 (a block's four)
    int64_t cells() const { return T * D * per; }
};

// cells of share r (0, 1) of a tile
SD2_HD int share_cells(int D, int r) { return r == 0 ? (D + 1) / 2 : D / 2; }

// Whether a kernel on GPU `device` can read weights or a mask (elements of `size` bytes) where they lie.  Memory of another GPU
// is out of its reach unless peer access happens to be on, and host memory takes a copy of its own.
enum MemoryPlace { kPlaceHost, kPlaceDevice, kPlaceManaged };
inline bool readable_in_place(MemoryPlace place, int owner, int device, const void* p, size_t size)
{
    if ((uintptr_t)p % size != 0) return false;
    return place == kPlaceManaged || (place == kPlaceDevice && owner == device);
}

inline CellGeom cell_geometry(int64_t M, int64_t K)
{
    CellGeom g;
    g.T = (M + kTileRows - 1) / kTileRows;
    g.D = (int)((K + kCellCols - 1) / kCellCols);
    g.per = 1;
    return g;
}

inline CellGeom panel_geometry(int64_t M, int64_t K)
{
    CellGeom g;
    g.T = (M + kPanelRowsOfBlock - 1) / kPanelRowsOfBlock;
    g.D = (int)((K + kPanelBlockCols - 1) / kPanelBlockCols);
    g.per = kChunkCells;
    return g;
}

// One cell of a panel's block back into dense weights.  cell: its header; H: its height; row0, col0: its place in W.
inline void unpack_panel_cell(const uint8_t* cell, int H, int64_t row0, int64_t col0, int64_t M, int64_t K, uint16_t* W)
{
    const uint32_t* mask = (const uint32_t*)cell;
    const uint32_t* words = (const uint32_t*)(cell + kCellHeaderBytes);
    for (int l = 0; l < 32 && row0 + l < M; ++l)
        for (int r = 0; r < 2; ++r) {
            const int column = r ? (cell[128 + l] & 0x7F) / 4 : l;
            int at = r ? H - 1 : 0;
            for (int e = 0; e < 16; ++e) {
                if (!(mask[l] >> (16 * r + e) & 1u)) continue;
                const uint32_t w = words[32 * at + column];
                const int64_t col = col0 + 32 * r + 2 * e;
                uint16_t* to = W + (row0 + l) * K + col;
                if (col < K) to[0] = (uint16_t)w;
                if (col + 1 < K) to[1] = (uint16_t)(w >> 16);
                at += r ? -1 : 1;
            }
        }
}

}  // namespace sd2
