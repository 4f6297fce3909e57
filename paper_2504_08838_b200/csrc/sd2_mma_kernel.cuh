// Tensor-core path of libsd2 for panels of activation rows (GAP4_MMA handles).
//
// Y[n, m] = sum over kept k of W[m, k] X[n, k] for N <= 64 rows per launch.  With that many rows the product is worth a dense
// contraction: the compressed weights still cross HBM once, a warp expands them in registers, and tcgen05.mma takes them from
// tensor memory, so that the expanded weights pass through no shared memory.
//
// On the device the weights of such a handle are *panel cells*: the cells of sd2_cells.hpp (a word per pair of columns of which
// anything is kept, words of 32 lanes in 32 banks) cut for an operand in tensor memory.  A panel is 128 weight rows, a block of
// it 64 columns: four cells of 32 rows, which stand together, block after block, so that a CTA's share is one run of bytes.
// Lane l of cell q holds row 32 q + l: the words of columns 0..31 from the bottom of the cell up, those of columns 32..63 from
// its top down.  That is the tensor memory layout of the A operand (a lane a row, a 32-bit column two elements of K).
//
// A CTA has one panel and one share of its columns; the shares of a panel are a cluster (mma_cluster chooses how many).
//
//   warps 0..15   expand: team t = warp / 4 takes blocks t, t + 4, ...; warp q of a team has cell q, whose rows are the 32 lanes
//                 of tensor memory that the warp can reach.  Then all of them read the sums.
//   warp 16       weights: a bulk asynchronous copy per block (13 KB at 50 % density) into a ring
//   warp 17       activations: a tensor-map copy per block (64 columns of all rows, in the swizzled K-major layout of the B
//                 operand; rows beyond N and columns beyond K arrive as zeros)
//   warps 18..21  issue the four K = 16 tcgen05.mma of a block, one warp for every team (one thread needs 560 cycles a block for its
//                 waits, the products and the commit, whatever they multiply: alone it took twice as long as the expanding).  Every
//                 team has sums of its own, so a chain of truncated sums is a quarter as long; they meet in fp32.
//
// The sums of a cluster meet by stores into the shared memory of the CTA that writes the activation row, in one order: results
// do not depend on timing, and a handle has no state that launches share.
//
// What bounds it: both 3072 x 8192 (24 panels, five shares each, 120 CTAs of 25 or 26 blocks) and 8192 x 3072 (64 panels, two shares,
// 128 CTAs of 24 blocks) have 41.5 MB of panel cells at 50 %, 6.4 us at HBM's rate; in a row of launches the first takes 11.5 us for 16
// rows, the second 13.1 for 64 (11.7 and 13.2 in a graph on cold weights).  The rest stands between launches: the last products, reading
// and exchanging the sums, the next start and its first block.  Before, 16-bit values were scattered into operand tiles in shared
// memory (eight dependent steps of 340 cycles a block) and shares added up by red.add: 20.0 and 35.3.  Half-size CTAs, two to an SM,
// whose successors fetch weights early: 11.2 for 16 rows, but 5.2 to 5.5 for 2048 x 2048 instead of 5.0, and sums twice as far from
// 64 bits; not taken.
//
// Every wait is bounded; a wait that runs out sets the error word and the CTA leaves in order (copies drained, tensor memory
// returned).

#pragma once

#include <cuda.h>

#include "sd2_cell_kernel.cuh"
#include "sd2_format_mma.hpp"

namespace sd2 {

constexpr int kMmaMaxRows = 64;                     // activation rows of one launch
constexpr int kMmaTeams = 4;                        // expanding teams
constexpr int kMmaQuads = kMmaBlockRows / 32;       // cells of a block, warps of a team
constexpr int kMmaExpandWarps = kMmaTeams * kMmaQuads;
constexpr int kMmaWeightWarp = kMmaExpandWarps, kMmaXWarp = kMmaExpandWarps + 1, kMmaIssueWarp = kMmaExpandWarps + 2;
constexpr int kMmaThreads = 32 * (kMmaExpandWarps + 2 + kMmaTeams);
constexpr int kMmaStages = 2 * kMmaTeams;           // blocks expanded or being expanded; stage s belongs to team s % 4
constexpr int kMmaMaxSlots = 16;                    // blocks in the ring, at most; always a multiple of the teams, so that a
                                                    // slot is waited for by one team only, in order
constexpr int kMmaStageCols = kMmaBlockCols / 2;    // tensor memory columns of an expanded block
constexpr int kMmaTmemCols = 512;
constexpr int kMmaSumCols = kMmaStages * kMmaStageCols;   // the sums stand behind the operands
constexpr int kMmaMaxCluster = 8;
static_assert(kMmaSumCols + kMmaTeams * kMmaMaxRows <= kMmaTmemCols, "operands and sums share tensor memory");
static_assert(kMmaQuads == kChunkCells, "a block is a chunk of cells");

struct MmaArgs {
    const uint32_t* off;     // [4 * blocks + 1] cells' places (32-byte units into `cells`)
    const unsigned char* cells;
    const uint16_t* X;       // [N, K] bf16
    void* Y;                 // [N, M] bf16 or fp32
    int M, K, N, npad;       // npad: N rounded up to a multiple of 16
    int KB;                  // blocks of a panel
    int shares;              // CTAs of a cluster
    int y_f32;
    int slot_bytes, n_slots; // ring
    int x_tma;               // 1: X comes through the tensor map; 0: the teams fetch it
    int x_vec;               // x_tma == 0: rows of X can be fetched in 16-byte pieces
    int* err;
    long long budget;        // clock cycles a wait may take
};

struct MmaShared {
    unsigned long long full[kMmaMaxSlots];    // a block landed
    unsigned long long empty[kMmaMaxSlots];   // ... and has been expanded
    unsigned long long xfull[kMmaStages];     // a block's activations have landed
    unsigned long long afull[kMmaStages];     // a block is in tensor memory
    unsigned long long aempty[kMmaStages];    // the products of a block are done
    unsigned long long done;                  // all products are (one arrival per team)
    unsigned long long rfull;                 // the other CTAs' sums have landed
    uint32_t tmem_base;
    int abort_flag;
    int never_flag;                           // stays 0: the exit waits must not be cut short by abort_flag
};

// activation rows are written by the CTAs of a cluster in turn, four at a time; how many such fours a CTA has at most
__host__ __device__ constexpr int mma_own_fours(int npad, int shares) { return (npad / 4 + shares - 1) / shares; }
// room for the others' sums: per CTA of the cluster and four rows 128 x 4 fp32
__host__ __device__ constexpr int mma_recv_bytes(int npad, int shares) { return shares > 1 ? shares * mma_own_fours(npad, shares) * kMmaBlockRows * 16 : 0; }

__device__ __forceinline__ void sts_u16(uint32_t a, uint32_t v)
{
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"((uint16_t)v) : "memory");
}
__device__ __forceinline__ void sts_v4(uint32_t a, uint4 v)
{
    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor of a K-major bf16 tile under the 128-byte swizzle: rows of 128
// bytes, groups of eight rows 1024 bytes apart.  Stepping K by 16 elements inside the 64-column
// atom adds 32 bytes to the start address.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t saddr)
{
    uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);   // start address, 16-byte units
    d |= (uint64_t)1 << 16;                             // leading byte offset (not used by swizzled K-major tiles)
    d |= (uint64_t)(1024 >> 4) << 32;                   // stride byte offset: eight rows
    d |= (uint64_t)1 << 46;                             // descriptor version of this architecture
    d |= (uint64_t)2 << 61;                             // 128-byte swizzle
    return d;
}

// D[128 x npad] (+)= A[128 x 16] B[npad x 16]^T, bf16 in, fp32 out, A in tensor memory, B K-major in shared memory
__device__ __forceinline__ void umma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// the mbarrier gets one arrival when every tcgen05.mma issued so far by this thread has completed
__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// 32 columns of the warp's 32 lanes
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,"
        "%25,%26,%27,%28,%29,%30,%31,%32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
          "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]),
          "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
// four columns (the values are there after tmem_ld_wait)
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float (&r)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];" : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]) : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// one box of the tensor map (64 columns x npad rows of X, swizzled) -> shared memory
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
                 "l"(map), "r"(bar), "r"(c0), "r"(c1)
                 : "memory");
}

// The cell `q` of a block at shared address `block`: the lane's row, as 32 words of two columns each.
__device__ __forceinline__ void expand_row(uint32_t block, int q, int lane, uint32_t (&w)[32])
{
    // where the cells start: the first one's header tells the heights of all four
    const uint32_t heights = __ballot_sync(0xFFFFFFFFu, (lds_u8(block + 128u + lane) & 0x80u) != 0);
    uint32_t H = heights & 63u, before = 0;
#pragma unroll
    for (int k = 1; k < kMmaQuads; ++k)
        if (k <= q) { before += H; H = heights >> (6 * k) & 63u; }
    const uint32_t cell = block + (uint32_t)q * kCellHeaderBytes + before * 128u;
    const uint32_t m = lds_u32(cell + 4 * lane), v0 = cell + kCellHeaderBytes;
    const uint32_t pi = lds_u8(cell + 128u + lane) & 0x7Fu;
    uint32_t lo = v0 + 4u * lane, hi = v0 + (H - 1u) * 128u + pi;
#pragma unroll
    for (int e = 0; e < 16; e += 2) take_words(m, 1u << e, lo, hi, w[e], w[16 + e], w[e + 1], w[17 + e]);
}

#ifdef SD2_CHECKED
__device__ __forceinline__ bool block_fits(uint32_t block, uint32_t bytes, int q, int lane)
{
    const uint32_t heights = __ballot_sync(0xFFFFFFFFu, (lds_u8(block + 128u + lane) & 0x80u) != 0);
    uint32_t total = 0, before = 0;
    for (int k = 0; k < kMmaQuads; ++k) {
        if (k == q) before = total;
        total += heights >> (6 * k) & 63u;
    }
    if (kMmaQuads * (uint32_t)kCellHeaderBytes + total * 128u > bytes) return false;
    const uint32_t cell = block + (uint32_t)q * kCellHeaderBytes + before * 128u, H = heights >> (6 * q) & 63u, m = lds_u32(cell + 4 * lane);
    return __all_sync(0xFFFFFFFFu, (uint32_t)__popc(m & 0xFFFFu) <= H && (uint32_t)__popc(m >> 16) <= H);
}
#endif

// A block's 64 columns of X, rows below N, into the B operand's tile at `xt`, by a team's 128 threads.  (What stands in the
// tile's other rows reaches only sums that nobody reads.)
__device__ __forceinline__ void fetch_x(const MmaArgs& a, int k0, uint32_t xt, int t)
{
    if (a.x_vec) {
        for (int i = t; i < a.N * 8; i += 32 * kMmaQuads) {
            const int n = i >> 3, ch = i & 7;
            const uint32_t dst = xt + (uint32_t)n * 128u + (uint32_t)((ch ^ (n & 7)) << 4);
            sts_v4(dst, k0 + ch * 8 < a.K ? __ldcg((const uint4*)(a.X + (size_t)n * a.K + k0 + ch * 8)) : make_uint4(0u, 0u, 0u, 0u));   // K % 8 == 0
        }
    } else {
        for (int i = t; i < a.N * kMmaBlockCols; i += 32 * kMmaQuads) {
            const int n = i >> 6, c = i & 63;
            const uint32_t v = k0 + c < a.K ? (uint32_t)__ldcg(a.X + (size_t)n * a.K + k0 + c) : 0u;
            sts_u16(xt + (uint32_t)n * 128u + (uint32_t)((((c >> 3) ^ (n & 7)) << 4) | ((c & 7) << 1)), v);
        }
    }
}

// activation rows n .. n + 3 of a weight row
__device__ __forceinline__ void store_four(const MmaArgs& a, int n, int row, const float (&v)[4])
{
    if (row >= a.M) return;
    const size_t at = (size_t)n * a.M + row;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (n + j >= a.N) break;
        if (a.y_f32) ((float*)a.Y)[at + (size_t)j * a.M] = v[j];
        else ((uint16_t*)a.Y)[at + (size_t)j * a.M] = f32_to_bf16_rne(v[j]);
    }
}

__global__ void __launch_bounds__(kMmaThreads, 1) mma_kernel(const __grid_constant__ MmaArgs a, const __grid_constant__ CUtensorMap xmap)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;     // swizzled tiles want 1024-byte alignment
    const uint32_t xbytes = (uint32_t)a.npad * 128u;                 // npad rows x 128 bytes
    const uint32_t recv0 = base + (uint32_t)kMmaStages * xbytes;
    const uint32_t ring0 = recv0 + (uint32_t)mma_recv_bytes(a.npad, a.shares);
    MmaShared* sh = (MmaShared*)(smem_raw + (ring0 - smem_u32(smem_raw)) + (size_t)a.n_slots * a.slot_bytes);

    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
    const int rank = (int)blockIdx.x % a.shares, panel = (int)blockIdx.x / a.shares;
    const int kb0 = (int)((long long)a.KB * rank / a.shares);
    const int nblk = (int)((long long)a.KB * (rank + 1) / a.shares) - kb0;      // at least one
    const WaitCtx wc = {&sh->abort_flag, a.budget};
    const WaitCtx wx = {&sh->never_flag, a.budget};

    pdl_let_next_start();
    if (tid < kMmaMaxSlots) {
        mbar_init(smem_u32(&sh->full[tid]), 1);
        mbar_init(smem_u32(&sh->empty[tid]), kMmaQuads);
        if (tid < kMmaStages) {
            mbar_init(smem_u32(&sh->xfull[tid]), 1);
            mbar_init(smem_u32(&sh->afull[tid]), kMmaQuads);
            mbar_init(smem_u32(&sh->aempty[tid]), 1);
        }
        if (tid == 0) {
            mbar_init(smem_u32(&sh->done), kMmaTeams);
            mbar_init(smem_u32(&sh->rfull), 1);
            sh->abort_flag = 0;
            sh->never_flag = 0;
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kMmaIssueWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sh->tmem_base)), "r"(kMmaTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *(volatile uint32_t*)&sh->tmem_base;
    // waited for before the first store to another CTA of the cluster (which has to run by then)
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");

    if (warp != kMmaWeightWarp) pdl_wait();      // (weights are on their way already)
    if (warp == kMmaWeightWarp) {
        // ---------------------------------------------------------------- weights
        const uint32_t full0 = smem_u32(&sh->full[0]), empty0 = smem_u32(&sh->empty[0]);
        const uint32_t NS = (uint32_t)a.n_slots;
        const uint32_t* off = a.off + ((size_t)panel * a.KB + kb0) * kMmaQuads;
        uint32_t o0 = 0, o1 = 0;                 // the lane's block: its place and its end
        int i = 0;
        bool ok = true;
        // the first blocks, as many as there are slots, are asked for at once, a lane each; then four at a time
        while (i < nblk) {
            if ((i & 31) == 0) {
                const int b = min(i + lane, nblk - 1);
                o0 = __ldg(off + (size_t)b * kMmaQuads);
                o1 = __ldg(off + (size_t)(b + 1) * kMmaQuads);
            }
            const int n = min(i == 0 ? (int)NS : kMmaTeams, nblk - i);
            if (i > 0) {
                if (i == (int)NS) pdl_wait();    // (slots are given back by warps that have waited, which the budget is not meant for)
                for (int k = 0; k < n && ok; ++k) ok = wait_phase_warp(empty0 + 8u * ((uint32_t)(i + k) % NS), ((uint32_t)(i + k) / NS & 1u) ^ 1u, wc);
                if (!ok) break;
            }
            const int k = lane - (i & 31);
            if (k >= 0 && k < n) {
                const uint32_t slot = (uint32_t)(i + k) % NS, bytes = (o1 - o0) * 32u;
                mbar_expect_tx(full0 + 8u * slot, bytes);
                bulk_g2s(ring0 + slot * (uint32_t)a.slot_bytes, a.cells + (size_t)o0 * 32, bytes, full0 + 8u * slot);
            }
            __syncwarp();
            i += n;
        }
        // (teams that gave up have left blocks on their way; where they did not, these have landed)
        for (int k = max(0, i - (int)NS); k < i; ++k) wait_landed(full0 + 8u * ((uint32_t)k % NS), (uint32_t)k / NS & 1u, a.budget);
    } else if (warp == kMmaXWarp) {
        // ---------------------------------------------------------------- activations
        if (lane == 0 && a.x_tma) {
            int i = 0;
            for (; i < nblk; ++i) {
                const int st = i % kMmaStages;
                if (i >= kMmaStages && !wait_phase(smem_u32(&sh->aempty[st]), ((uint32_t)(i / kMmaStages) & 1u) ^ 1u, wc)) break;
                const uint32_t xb = smem_u32(&sh->xfull[st]);
                mbar_expect_tx(xb, xbytes);
                tma_load_2d(base + (uint32_t)st * xbytes, &xmap, (kb0 + i) * kMmaBlockCols, 0, xb);
            }
            for (int k = max(0, i - kMmaStages); k < i; ++k) wait_phase(smem_u32(&sh->xfull[k % kMmaStages]), (uint32_t)(k / kMmaStages) & 1u, wx);
        }
    } else if (warp >= kMmaIssueWarp) {
        // ---------------------------------------------------------------- products
        if (lane == 0) {
            // instruction descriptor: fp32 accumulator, bf16 A and B, both K-major, N = npad, M = 128
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(a.npad >> 3) << 17) | ((128u >> 4) << 24);
            const uint64_t xdesc0 = umma_desc_sw128(base);
            const int team = warp - kMmaIssueWarp;
            const uint32_t d = tmem + (uint32_t)(kMmaSumCols + team * a.npad);
            for (int i = team; i < nblk; i += kMmaTeams) {
                const int st = i % kMmaStages;
                const uint32_t par = (uint32_t)(i / kMmaStages) & 1u;
                if (a.x_tma && !wait_phase(smem_u32(&sh->xfull[st]), par, wc)) break;
                if (!wait_phase(smem_u32(&sh->afull[st]), par, wc)) break;
                tc_fence_after();
                // descriptors differ in their start address only (16-byte units in the low bits)
                const uint64_t xd = xdesc0 + (uint64_t)((uint32_t)st * (xbytes >> 4));
                const uint32_t at = tmem + (uint32_t)(st * kMmaStageCols);
#pragma unroll
                for (int kk = 0; kk < kMmaBlockCols / 16; ++kk)
                    umma_bf16_ts(d, at + 8u * kk, xd + (uint64_t)(2 * kk), idesc, (i < kMmaTeams && kk == 0) ? 0u : 1u);
                umma_commit(smem_u32(&sh->aempty[st]));
            }
            // (nothing of this CTA is left in the tensor pipe when this has been waited for)
            umma_commit(smem_u32(&sh->done));
            wait_phase(smem_u32(&sh->done), 0u, wx);
        }
    } else {
        // ---------------------------------------------------------------- expanding teams
        const int q = warp % kMmaQuads, team = warp / kMmaQuads;
        const uint32_t full0 = smem_u32(&sh->full[0]), empty0 = smem_u32(&sh->empty[0]);
        const uint32_t NS = (uint32_t)a.n_slots;
        bool ok = true;
        uint32_t slot = (uint32_t)team, par = 0u;
        for (int i = team; i < nblk; i += kMmaTeams) {
            const int st = i % kMmaStages;
            if (!(ok = wait_phase_warp(full0 + 8u * slot, par, wc))) break;
            uint32_t w[32];
#ifdef SD2_CHECKED
            // checked build: the cells of a block must lie inside its slot, a lane's words inside its cell; a violation is recorded in the
            // error word (value 2) and the block skipped
            if (!block_fits(ring0 + slot * (uint32_t)a.slot_bytes, (uint32_t)a.slot_bytes, q, lane)) {
                if (lane == 0 && a.err) atomicExch(a.err, 2);
#pragma unroll
                for (int k = 0; k < 32; ++k) w[k] = 0u;
            } else
#endif
            expand_row(ring0 + slot * (uint32_t)a.slot_bytes, q, lane, w);
            __syncwarp();
            mbar_arrive_n(empty0 + 8u * slot, 1u, lane == 0);
            if ((slot += kMmaTeams) >= NS) { slot = (uint32_t)team; par ^= 1u; }
            if (i >= kMmaStages && !(ok = wait_phase_warp(smem_u32(&sh->aempty[st]), ((uint32_t)(i / kMmaStages) & 1u) ^ 1u, wc))) break;
            tc_fence_after();
            tmem_st32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(st * kMmaStageCols), w);
            if (!a.x_tma) {
                fetch_x(a, (kb0 + i) * kMmaBlockCols, base + (uint32_t)st * xbytes, 32 * q + lane);
                fence_async_smem();
            }
            tc_fence_before();
            __syncwarp();
            mbar_arrive_n(smem_u32(&sh->afull[st]), 1u, lane == 0);
        }
        if (ok) ok = wait_phase_warp(smem_u32(&sh->done), 0u, wc);
        tc_fence_after();
        // A team has a quarter of the activation rows, four at a time: rows 4 f .. 4 f + 3 (f = team * fours + k) of weight row
        // 32 q + lane.  They belong to CTA f % C of the cluster.  (Loops, not runs of code: what is gone through once comes from L2,
        // and 500 instructions of it took 2 us.)
        const int teams = min(nblk, kMmaTeams), fours = a.npad / (4 * kMmaTeams), C = a.shares;
        const uint32_t lane_at = (uint32_t)((32 * q + lane) * 16);
        const uint32_t four_bytes = kMmaBlockRows * 16, cta_bytes = (uint32_t)mma_own_fours(a.npad, C) * four_bytes;
        if (C > 1) {
            // (all CTAs of the cluster run, and their mbarriers are there)
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
            if (warp == 0 && lane == 0) mbar_expect_tx(smem_u32(&sh->rfull), (uint32_t)((C - 1) * ((a.npad / 4 - rank + C - 1) / C)) * four_bytes);
        }
#pragma unroll 1
        for (int k = 0; k < fours && ok; ++k) {
            const int f = team * fours + k, owner = f % C;
            const uint32_t t = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(kMmaSumCols + 4 * f);
            float s[kMmaTeams][4];
#pragma unroll
            for (int g = 0; g < kMmaTeams; ++g) {
                if (g < teams) tmem_ld4(t + (uint32_t)(g * a.npad), s[g]);
                else s[g][0] = s[g][1] = s[g][2] = s[g][3] = 0.f;
            }
            tmem_ld_wait();
            float v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = (s[0][j] + s[1][j]) + (s[2][j] + s[3][j]);
            const uint32_t at = recv0 + (uint32_t)rank * cta_bytes + (uint32_t)(f / C) * four_bytes + lane_at;
            if (C == 1) {
                store_four(a, 4 * f, panel * kMmaBlockRows + 32 * q + lane, v);
            } else if (owner == rank) {
                sts_v4(at, make_uint4(__float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]), __float_as_uint(v[3])));
            } else {
                uint32_t to, bar;
                asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(at), "r"(owner));
                asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(bar) : "r"(smem_u32(&sh->rfull)), "r"(owner));
                st_async(to, v, bar);
            }
        }
        tc_fence_before();
        if (C > 1) {
            named_bar_sync(1, 32 * kMmaExpandWarps);                             // the sums that this CTA keeps
            if (ok) ok = wait_phase_warp(smem_u32(&sh->rfull), 0u, wc);          // ... and gets
#pragma unroll 1
            for (int f = rank + C * team; f < a.npad / 4 && ok; f += C * kMmaTeams) {
                const uint32_t at = recv0 + (uint32_t)(f / C) * four_bytes + lane_at;
                float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
                for (int r = 0; r < C; ++r) {                                    // in the order of the columns, whatever came first
                    const uint4 o = lds_v4(at + (uint32_t)r * cta_bytes);
                    v[0] += __uint_as_float(o.x);
                    v[1] += __uint_as_float(o.y);
                    v[2] += __uint_as_float(o.z);
                    v[3] += __uint_as_float(o.w);
                }
                store_four(a, 4 * f, panel * kMmaBlockRows + 32 * q + lane, v);
            }
        }
    }

    // ---------------------------------------------------------------- exit
    // Nobody leaves while another CTA may still write to its memory: a CTA that has got its sums may go (threads that are gone count
    // as arrived), one that gave up waits for the others.
    __syncwarp();
    if (a.shares == 1 || warp >= kMmaExpandWarps) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    if (warp == kMmaIssueWarp) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kMmaTmemCols) : "memory");
    }
    if (*(volatile int*)&sh->abort_flag) {
        if (tid == 0 && a.err) atomicExch(a.err, 1);
        __syncwarp();
        asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}

}  // namespace sd2
