// Packing cells (sd2_cells.hpp) on the device: one warp per cell, twice.  The first pass finds every cell's height, the host
// turns those into places, the second pass writes the cells.
//
// It runs when a handle is made, from the dense weights (33 MB for 8192 x 2048: some tenths of a millisecond next to the tens
// that the strips take on the host).  On the host the same work took as long as the strips: 27 MB of cells are new pages.

#pragma once

#include "sd2_cells.hpp"
#include "sd2_kernels.cuh"

namespace sd2 {

constexpr int kPackWarps = 8;

// PANEL: panel cells (sd2_mma_kernel.cuh); T and D are then row panels and blocks of a panel.
// height: [cells] (first pass), or NULL; off: directory (second pass).
// mask: one byte per weight, not zero where it is kept; NULL: a weight that has one of the bits of `nonzero` is kept (0x7FFF: what is
// not +0 or -0; 0xFFFF: what is not +0).
template <bool PANEL>
__global__ void __launch_bounds__(32 * kPackWarps) pack_cells_kernel(const uint16_t* W, const uint8_t* mask, uint32_t nonzero, long long M, long long K,
                                                                    int T, int D, uint32_t* height, const uint32_t* off, unsigned char* cells)
{
    __shared__ uint8_t lane_of_rank[kPackWarps][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long n_cells = (long long)T * D * (PANEL ? kChunkCells : 1), in_first = (long long)T * share_cells(D, 0);
    const long long c = (long long)blockIdx.x * kPackWarps + warp;
    if (c >= n_cells) return;                // (whole warps)
    const int n0 = share_cells(D, 0), n1 = share_cells(D, 1);
    const long long tile = c < in_first ? c / n0 : (c - in_first) / n1;
    const int d = c < in_first ? (int)(c - tile * n0) : n0 + (int)(c - in_first - tile * n1);
    const int g = lane >> 2, t = lane & 3;
    uint32_t bits = 0;
    const long long block = c / kChunkCells, panel = block / D;
    // pair i of unit u of row g + 8 r (PANEL: pair 4 u + i of the row's r-th 32 columns): its word, and whether there is one
    auto pair = [&](int r, int u, int i, uint32_t& word) {
        const long long row = PANEL ? panel * kPanelRowsOfBlock + 32 * (c % kChunkCells) + lane : tile * kTileRows + g + 8 * r;
        uint32_t w = 0;
        bool any = false;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const long long col = PANEL ? (block - panel * D) * kPanelBlockCols + 32 * r + 8 * u + 2 * i + k : (long long)d * kCellCols + 32 * u + 8 * t + 2 * i + k;
            if (row >= M || col >= K) continue;
            const uint32_t v = W[row * K + col];
            const bool kept = mask ? mask[row * K + col] != 0 : (v & nonzero) != 0;
            if (kept) { w |= v << (16 * k); any = true; }
        }
        word = w;
        return any;
    };
    int n[2] = {0, 0};
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            uint32_t w;
            if (pair(r, e >> 2, e & 3, w)) {
                bits |= 1u << (16 * r + e);
                ++n[r];
            }
        }
    // lanes by the words of their first row, most first, and by those of their second, fewest first; equal ranks share a column
    int rank0 = 0, rank1 = 0;
    for (int l = 0; l < 32; ++l) {
        const int a = __shfl_sync(0xFFFFFFFFu, n[0], l), b = __shfl_sync(0xFFFFFFFFu, n[1], l);
        rank0 += a > n[0] || (a == n[0] && l < lane) ? 1 : 0;
        rank1 += b < n[1] || (b == n[1] && l < lane) ? 1 : 0;
    }
    lane_of_rank[warp][rank0] = (uint8_t)lane;
    __syncwarp();
    const int column = lane_of_rank[warp][rank1];
    int H = __shfl_sync(0xFFFFFFFFu, n[0], column) + n[1];
    for (int k = 16; k > 0; k >>= 1) H = max(H, __shfl_xor_sync(0xFFFFFFFFu, H, k));
    if (height) {
        if (lane == 0) height[c] = (uint32_t)H;
        return;
    }
    unsigned char* p = cells + (size_t)off[c] * 32;
    uint32_t heights = 0;                    // of this cell and the three that follow it
    for (int k = 0; k < kChunkCells && c + k < n_cells; ++k)
        heights |= ((off[c + k + 1] - off[c + k]) * 32u - kCellHeaderBytes) / 128u << (6 * k);
    ((uint32_t*)p)[lane] = bits;
    p[128 + lane] = (unsigned char)(4 * column | (lane < 6 * kChunkCells ? (heights >> lane & 1u) << 7 : 0u));
    uint32_t* v = (uint32_t*)(p + kCellHeaderBytes);
    for (int r = 0; r < 2; ++r) {
        int at = 0;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            uint32_t w;
            if (!pair(r, e >> 2, e & 3, w)) continue;
            v[r ? (H - 1 - at) * 32 + column : at * 32 + lane] = w;
            ++at;
        }
    }
}

}  // namespace sd2
