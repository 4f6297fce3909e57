// The streaming kernel over cells (sd2_cells.hpp): programs of dependent stages for panels of up to 16 activation rows.
//
// A launch runs a *program* of stages with one persistent CTA per SM.  A stage is up to four weights that read the same
// activations (q|k|v, or one weight), or a gate and an up projection whose results meet in t = silu(g) * u.
// Consecutive stages depend on each other; a grid-wide barrier separates them.  (Tagged words, the hand-off of
// sd2_kernels.cuh, double the bytes every CTA has to fetch, which is what a panel of rows cannot afford.)
//
// CTAs work in clusters of two.  A cluster owns a run of 16-row tiles; each of its CTAs multiplies one half of the
// columns, so it stages half of the activations only (they are the largest thing in shared memory, and every CTA
// fetches them through L2), and sends its sums of every other tile to the CTA that finishes that tile.
//
// Warps of a CTA (sixteen, four per scheduler):
//   12 consumers, in three groups of four.  A chunk of four cells goes to a group, a cell to each of its warps.  A warp
//              expands its cell in registers and multiplies it with mma.m16n8k16: sixteen weight rows are the A operand,
//              eight (twice eight) activation rows the B operand, so the expanded weights never pass through shared
//              memory.  At the end of a tile a warp leaves its 16 x N partial sums in shared memory and goes on.
//   2 finishers: one takes the tiles this CTA finishes, one those it sends, each in order.  They add a tile's partial sums
//              up in one fixed order (so a row's result depends neither on the launch nor on how many rows are with it, as
//              long as they go over cells; the strips add up in another order).  The sums for the other CTA travel as
//              asynchronous stores that count bytes on its mbarrier.  (When the consumer that brought a tile's last
//              contribution finished it, with flags and fences, it was away for 2400 to 7000 cycles per tile: 80 us for 48
//              rows of an 8192 x 2048 matrix.)
//   1 producer: one bulk asynchronous copy per chunk (13 KB at 50 % density) into the group's own ring slots.  Copies of
//              13 KB reach 7 TB/s with 118 KB in flight per SM, 6.5 TB/s with 52 KB; copies of single cells of 2.7 KB
//              1.6 TB/s from one thread (measured).  Nothing waits for a stage boundary: while the previous stage
//              finishes, the next stages' weights land.
//   1 service warp: waits for the grid barrier, starts the bulk copies of the stage's activation rows, and fetches the
//              next stage's descriptor.
// The last four share their schedulers with three busy warps each and get an instruction in every four to eight cycles: what
// counts for them is the number of instructions.
//
// What bounds it: HBM for large matrices (15 slots per clock and SM at 50 % density against 33 that twelve warps expanded, 29
// for sixteen rows, before the sums were added up in fp32); between stages some 2.8 us: from the last output to the barrier's release 1.2, to the activations 0.6, to
// the first cell 0.9.  One launch with its start and its last sums is 8 us at least, and launches of a stream overlap there.
// Against the strips, which gather row by row (us): 5 rows of 1531 x 3001 18.5 -> 8.7, 48 rows of 8192 x 2048 111 -> 25.5, two
// blocks of 2048/512/8192 for 8 rows 230 -> 67.5, a block of 3072/1024/8192 for 16 rows 342 -> 60.
//
// Every wait (ring barriers, counters, grid barrier) is bounded by a cycle budget: when it runs out the CTA raises the
// error word and winds down instead of hanging.

#pragma once

#include "sd2_cells.hpp"
#include "sd2_kernels.cuh"

namespace sd2 {

constexpr int kCellWarps = 12;
constexpr int kCellGroups = 3;
static_assert(kCellWarps == kCellGroups * kChunkCells, "a group has a warp for every cell of a chunk");
constexpr int kCellConsumers = kCellWarps * 32;
constexpr int kProducerWarp = kCellWarps, kServiceWarp = kCellWarps + 1, kOwnWarp = kCellWarps + 2, kSendWarp = kCellWarps + 3;
constexpr int kCellThreads = 32 * (kCellWarps + 4);
constexpr int kGroupSlots = 4;              // chunks in flight per group, at most
constexpr int kPartSlots = 8;               // groups' partial sums that may wait for a finisher, at most (a power of two)
constexpr int kRecvSlots = 8;               // sums from the other CTA that wait to be used
constexpr int kPairSlots = 8;               // gate tiles whose results wait for the up tile's
constexpr int kPanelRows = 16;              // activation rows of a launch of several stages, at most
constexpr int kWidePanelRows = 32;          // ... of a single stage: a cell is expanded once for all of them (us, in panels of
                                            // 16 / of 32: 24 rows of 8192 x 2048 at 50 % 19.5 / 12.8, 48 rows 29.3 / 25.8)
// A warp's contribution to a tile: for every eight activation rows 16 x 8 fp32, the activation row fastest.  A lane's
// fragment goes there in 8-byte stores and a finisher reads 16 bytes a lane, both without bank conflicts.
constexpr int kPartRowBytes = 32;
__host__ __device__ constexpr int part_slot_bytes(int nr) { return kChunkCells * kTileRows * kPartRowBytes * (nr / 8); }

struct CMat {
    const uint32_t* off;           // [T * D + 1], 32-byte units into `cells`
    const unsigned char* cells;
    void* y;                       // [N * M]
    int M;
    int T;
    int y_f32;                     // 1: fp32 output, 0: bf16
    int reserved;
};

struct CStage {
    CMat mat[kMaxFused];
    const uint16_t* x;     // [N * K] bf16, or NULL: the activation is bf16(silu(g) * u)
    const uint16_t* g;
    const uint16_t* u;
    uint16_t* t_out;       // gate|up stage, or x == NULL: t (may be NULL)
    int K;
    int D;                 // cells per tile
    int tiles_div;         // V / clusters: the cluster with stage-local number c runs tiles_div + (c < tiles_rem) tiles (pairs)
    int tiles_rem;
    int rot;               // the stage's first tile goes to cluster `rot`, so that uneven stages even out over a program
    int pair;              // mat[0] is gate, mat[1] up (equal shapes)
    int count;             // weights
    int V;                 // tiles of all weights; tile pairs in a gate|up stage
};
static_assert(sizeof(CStage) % 8 == 0, "stage descriptors are arrays of 8-byte fields");

struct CArgsBase {
    const CStage* ext;              // device array of stages, or NULL: the inline ones (stage 0 is always inline)
    const uint16_t* x_in;           // replaces stage 0's x when not NULL
    void* y_out;                    // replaces the last stage's mat[0].y when not NULL
    unsigned int* gbar;             // grid barrier: [0] arrivals, [32] exits (two cache lines)
    int* err;                       // device error word
    long long wait_cycles;          // budget of every bounded wait
    int n_stages;
    int N;                          // activation rows of this launch
    int n0;                         // first activation row: every X / Y pointer is advanced by n0 rows
    int part_mask;                  // slots of partial sums per finisher - 1 (a power of two)
    int xbuf_bytes;                 // staged activations
    int chunk_bytes, n_slots;       // a ring slot, slots per group
    int fold_any;                   // host side: launch the FOLD instance
};

// MAXS: inline stages the argument block has room for (a launch of one stage, or of stages in device memory, passes 0.4 KB
// of arguments, not 3 KB)
template <int MAXS>
struct CArgs : CArgsBase {
    CStage inl[MAXS];
    SFold fold[MAXS];               // read by FOLD instances only
};

template <int NR>
struct CellShared {
    unsigned long long full[kCellGroups][kGroupSlots];    // a chunk landed
    unsigned long long empty[kCellGroups][kGroupSlots];   // ... and has been consumed
    unsigned long long dfull;                           // the stage's descriptor is there
    unsigned long long xfull;                           // the stage's activations have landed
    unsigned long long left;                            // consumers and finishers have left the stage: its descriptor and rows are free
    unsigned long long csync;                           // all consumers have come this far
    unsigned long long pfull[2][kPartSlots];            // a group's partial sums are complete: [0] to be sent, [1] to be finished here
    unsigned long long rfull[kRecvSlots];               // sums from the other CTA have landed in recv[]
    unsigned long long credit[2];                       // the other CTA has taken ours out of this half of its recv[]
    unsigned int freed[2][kPartSlots];                  // how often the slot's sums have been read
    uint2 gate[kPairSlots][NR / 8][32];         // bf16 results of gate tiles, as the finisher's lanes hold them
    float4 recv[kRecvSlots][NR / 8][32];
    int abort_flag;                                     // any warp: a bounded wait ran out
    float red[4][kCellWarps];                           // FOLD: per-warp partial sums of squares of some rows
    CStage stage[2];                                    // descriptors of the current and the next stage
};

// wait_phase for a whole warp: its lanes get one answer, and every branch is on a vote.  (mma.sync and other warp-wide
// instructions need the warp whole, and lanes that come back from a wait one by one cost hundreds of cycles to bring together:
// an eight-row drafter step took 76 us with a wait per lane, 127 us with one lane waiting for the others.)
__device__ __forceinline__ bool wait_phase_warp(uint32_t bar, uint32_t parity, const WaitCtx& w)
{
    if (__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity))) return true;
    const long long t0 = clock64();
    uint32_t it = 0;
    while (!__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity))) {
        if ((++it & 15u) == 0u) {
            if (__any_sync(0xFFFFFFFFu, *w.abort_flag != 0)) return false;
            if (__any_sync(0xFFFFFFFFu, clock64() - t0 > w.budget)) {
                *w.abort_flag = 1;
                return false;
            }
        }
    }
    return true;
}

// Until the copies counted by a phase have landed.  For a warp that is about to leave: the abort flag does not cut this short,
// since memory that copies are on their way to must not be given up.
__device__ __forceinline__ void wait_landed(uint32_t bar, uint32_t parity, long long budget)
{
    const long long t0 = clock64();
    while (!__all_sync(0xFFFFFFFFu, mbar_try_wait(bar, parity)))
        if (__any_sync(0xFFFFFFFFu, clock64() - t0 > budget)) return;
}

// Until the shared counter at p has reached `want` (one warp, together).
__device__ __forceinline__ bool wait_count(const unsigned int* p, unsigned int want, const WaitCtx& w)
{
    if (__any_sync(0xFFFFFFFFu, (int)(*(const volatile unsigned int*)p - want) < 0)) {
        const long long t0 = clock64();
        uint32_t it = 0;
        while (__any_sync(0xFFFFFFFFu, (int)(*(const volatile unsigned int*)p - want) < 0)) {
            if ((++it & 15u) == 0u) {
                if (__any_sync(0xFFFFFFFFu, *w.abort_flag != 0)) return false;
                if (__any_sync(0xFFFFFFFFu, clock64() - t0 > w.budget)) {
                    *w.abort_flag = 1;
                    return false;
                }
            }
        }
    }
    __threadfence_block();
    return true;
}

// Until `target` arrivals have been counted.  false: the wait budget is out.
__device__ __forceinline__ bool grid_wait(const unsigned int* gbar, unsigned int target, const WaitCtx& w)
{
    const long long t0 = clock64();
    uint32_t it = 0;
    while ((int)(ld_acquire_gpu(gbar) - target) < 0) {
        if ((++it & 15u) == 0u) {
            if (*w.abort_flag) return false;
            if (clock64() - t0 > w.budget) { *w.abort_flag = 1; return false; }
        }
    }
    return true;
}

// the same shared-memory address in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank)
{
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    return a;
}
// four floats into the other CTA's shared memory, counted in bytes on its mbarrier when they are there
__device__ __forceinline__ void st_async(uint32_t a, const float (&v)[4], uint32_t bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(a), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_remote(uint32_t bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// one lane's arrival, predicated: a branch around it splits the warp
__device__ __forceinline__ void mbar_arrive_n(uint32_t bar, uint32_t n, bool lead)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %2, 0;\n\t@p mbarrier.arrive.shared::cta.b64 _, [%0], %1;\n\t}" ::"r"(bar), "r"(n), "r"((int)lead) : "memory");
}
// ... that also announces a bulk copy, and the copy (with or without an L2 policy)
__device__ __forceinline__ void bulk_chunk(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar, bool lead)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t@p mbarrier.arrive.expect_tx.shared::cta.b64 _, [%3], %2;\n\t"
                 "@p cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n\t}" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar), "r"((int)lead)
                 : "memory");
}
__device__ __forceinline__ void bulk_chunk(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar, bool lead, uint64_t policy)
{
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t@p mbarrier.arrive.expect_tx.shared::cta.b64 _, [%3], %2;\n\t"
                 "@p cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %5;\n\t}" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar), "r"((int)lead), "l"(policy)
                 : "memory");
}

// The runs of consecutive tiles of one weight that a cluster works through in a stage, in order.
struct TileRuns {
    int v, end, half, stop;      // next tile (pair), last + 1; gate|up: which of the two, end of the current group
    __device__ __forceinline__ TileRuns(int cluster, int clusters, int rot, int div, int rem)
    {
        const int c = cluster - rot + (cluster < rot ? clusters : 0);
        v = c * div + (c < rem ? c : rem);
        end = v + div + (c < rem ? 1 : 0);
        half = 0;
        stop = 0;
    }
    // mat: weight, t0: its first tile, nt: tiles.  false: that was all.
    __device__ __forceinline__ bool next(int pair, int count, int T0, int T1, int T2, int& mat, int& t0, int& nt)
    {
        if (v >= end) return false;
        if (pair) {
            if (half == 0) stop = min(v + kPairSlots, end);
            mat = half;
            t0 = v;
            nt = stop - v;
            if (half) v = stop;
            half ^= 1;
            return true;
        }
        int base = 0, T = T0;
        mat = 0;
        if (count > 1 && v >= T0) { base = T0; T = T1; mat = 1; }
        if (count > 2 && v >= T0 + T1) { base = T0 + T1; T = T2; mat = 2; }
        if (count > 3 && v >= T0 + T1 + T2) { base = T0 + T1 + T2; T = end - base; mat = 3; }
        t0 = v - base;
        nt = min(end, base + T) - v;
        v += nt;
        return true;
    }
};

// How a run's cells (nt tiles of Dr each, in order) are dealt to the groups.  Up to kSplitCells cells per tile a group
// takes whole tiles: four contributions per tile for a finisher to add, not twelve.  Longer tiles are few and would leave
// groups idle at the end of a stage: there the chunks go round and each group brings a third of a tile.
constexpr int kSplitCells = 16;
struct RunDeal {
    bool split;
    int tiles;         // per turn of a group
    int cells;         // of a turn (the last one may be shorter)
    int per;           // chunks of a turn
    int turns;         // split: chunks
    int chunks;        // of the run
    __device__ __forceinline__ RunDeal(int Dr, int nt)
    {
        split = Dr > kSplitCells;
        tiles = split ? nt : Dr < kChunkCells ? kChunkCells : (Dr & (kChunkCells - 1)) && Dr < 2 * kChunkCells ? 2 : 1;
        cells = tiles * Dr;
        per = (cells + kChunkCells - 1) / kChunkCells;
        if (split) {
            turns = chunks = per;
            return;
        }
        const int sh = tiles == 4 ? 2 : tiles - 1, whole = nt >> sh, rest = nt - (whole << sh);
        turns = Dr > 0 ? whole + (rest ? 1 : 0) : 0;
        chunks = whole * per + (rest * Dr + kChunkCells - 1) / kChunkCells;
    }
};

// ---- expanding a cell -----------------------------------------------------------------

// d = A B, from zero
__device__ __forceinline__ void mma_rows(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}
// d += s, two sums to an instruction
__device__ __forceinline__ void add_rows(float (&d)[4], const float (&s)[4])
{
    asm("{\n\t.reg .b64 p, q;\n\tmov.b64 p, {%0, %1};\n\tmov.b64 q, {%4, %5};\n\tadd.rn.f32x2 p, p, q;\n\tmov.b64 {%0, %1}, p;\n\t"
        "mov.b64 p, {%2, %3};\n\tmov.b64 q, {%6, %7};\n\tadd.rn.f32x2 p, p, q;\n\tmov.b64 {%2, %3}, p;\n\t}"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "f"(s[0]), "f"(s[1]), "f"(s[2]), "f"(s[3]));
}

// The words of four pairs of a lane, by steps: two from shared address `lo` upward and two from `hi` downward, 128 bytes apart, where the
// mask has the bits `bit` and the next, and those 16 above; zero and no step where it has not.  Four instructions a pair.  (Four
// addresses at once, from prefix sums of the mask's bits, take five and no less time even where a warp has a single cell.  us, prefix sums
// and steps, calls back to back: 512 x 512 for eight rows 4.83 and 4.70, 2048 x 8192 8.89 and 8.58, 8192 x 8192 21.4 and 21.2, steps of
// two blocks of 256/64/1024 for four rows 32.1 and 31.9, of 2048/512/8192 for eight 67.2 and 65.7.)
__device__ __forceinline__ void take_words(uint32_t mask, uint32_t bit, uint32_t& lo, uint32_t& hi, uint32_t& a, uint32_t& b, uint32_t& c, uint32_t& d)
{
    asm volatile("{\n\t.reg .pred p, q, r, s;\n\t.reg .b32 t, u, v, w;\n\t"
                 "and.b32 t, %6, %7;\n\tand.b32 u, %6, %8;\n\tand.b32 v, %6, %9;\n\tand.b32 w, %6, %10;\n\t"
                 "setp.ne.u32 p, t, 0;\n\tsetp.ne.u32 q, u, 0;\n\tsetp.ne.u32 r, v, 0;\n\tsetp.ne.u32 s, w, 0;\n\t"
                 "mov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\tmov.b32 %2, 0;\n\tmov.b32 %3, 0;\n\t"
                 "@p ld.shared.u32 %0, [%4];\n\t@q ld.shared.u32 %1, [%5];\n\t@p add.u32 %4, %4, 128;\n\t@q sub.u32 %5, %5, 128;\n\t"
                 "@r ld.shared.u32 %2, [%4];\n\t@s ld.shared.u32 %3, [%5];\n\t@r add.u32 %4, %4, 128;\n\t@s sub.u32 %5, %5, 128;\n\t}"
                 : "=&r"(a), "=&r"(b), "=&r"(c), "=&r"(d), "+r"(lo), "+r"(hi)
                 : "r"(mask), "r"(bit), "r"(bit << 16), "r"(bit << 1), "r"(bit << 17) : "memory");
}

// One cell: eight mma steps for each eight activation rows.  m: the lane's mask; lo, hi: shared addresses of the first
// words of its rows g and g + 8; xo[h]: of the first eight activations of panel row g + 8 h.
// Every mma starts from zero and its sums are added up in fp32, pair by pair: the tensor core truncates the sum that it
// carries on, so chains of mma drift towards zero.  Relative error of a row of 2048 at 50 % density against 64 bits: chains over
// a warp's cells 9.4e-8 (of one set of sums for 32 activation rows 15.2e-8), chains of a cell 7.5e-8, single steps 6.8e-8, which
// is what the strips' fused multiply-adds have; at 11008 columns 14.9e-8, 8.7e-8, 8.2e-8 (strips 8.9e-8).  The order of the
// sums is that of every instance, so a row has the same sums in every panel.
template <int NR>
__device__ __forceinline__ void multiply_cell(uint32_t m, uint32_t lo, uint32_t hi, const uint32_t (&xo)[NR / 8], uint32_t xd,
                                              float (&c)[NR / 8][4])
{
    float two[NR / 8][4], four[NR / 8][4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        uint32_t a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; i += 2) take_words(m, 1u << (4 * u + i), lo, hi, a[i], b[i], a[i + 1], b[i + 1]);
#pragma unroll
        for (int h = 0; h < NR / 8; ++h) {
            const uint4 x = lds_v4(xo[h] + xd + 64u * u);
            float s[4], t[4];
            mma_rows(s, a[0], b[0], a[1], b[1], x.x, x.y);
            mma_rows(t, a[2], b[2], a[3], b[3], x.z, x.w);
            add_rows(s, t);
            float (&to)[4] = u < 2 ? two[h] : four[h];
            if (u & 1) {
                add_rows(to, s);
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) to[k] = s[k];
            }
            if (u == 3) {
                add_rows(two[h], four[h]);
                add_rows(c[h], two[h]);
            }
        }
    }
}

// ---- staging the activations ------------------------------------------------------------

struct XRows {
    unsigned char* buf;      // staged rows: bf16, row n at n * pitch bytes, zero from column K to the last cell's end
    int pitch;
    int K, N;                // columns staged here
    int ld;                  // columns of a whole row in global memory
};

// Walks the groups (n, k) of a panel of rows, `kq` groups to a row, in steps of the consumer threads.
struct PanelWalk {
    uint32_t n, k, kq, step_n, step_k;
    __device__ __forceinline__ PanelWalk(uint32_t kq_, uint32_t tid) : kq(kq_)
    {
        n = tid / kq;
        k = tid - n * kq;
        step_n = (uint32_t)kCellConsumers / kq;
        step_k = (uint32_t)kCellConsumers - step_n * kq;
    }
    __device__ __forceinline__ void next()
    {
        n += step_n;
        k += step_k;
        if (k >= kq) { k -= kq; ++n; }
    }
};

constexpr int kStageBatch = 8;   // 16-byte (silu: 2-byte) loads a thread keeps in flight while staging

// Rows that a bulk copy cannot bring, because they do not start on 16 bytes: a thread puts eight columns together from the
// two 16-byte words they lie in.  (Column by column five rows of 3001 took 12000 cycles.)  Columns K .. Kp - 1 become zero.
// x: the first staged column of row 0, `before` columns into the row.
__device__ __noinline__ void stage_rows(const XRows& r, const uint16_t* x, int before, int Kp, int ctid)
{
    const uintptr_t lo = (uintptr_t)(x - before), hi = lo + (uintptr_t)r.N * (uintptr_t)r.ld * 2u;     // the rows of the launch
    auto word = [&](uintptr_t p) {           // nothing outside them is read
        if (p >= lo && p + 16 <= hi) return __ldcg((const uint4*)p);
        uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uintptr_t e = p + 2u * i;
            if (e >= lo && e < hi) w[i >> 1] |= (uint32_t)__ldcg((const uint16_t*)e) << (16 * (i & 1));
        }
        return make_uint4(w[0], w[1], w[2], w[3]);
    };
    constexpr int kItems = kStageBatch / 2;
    PanelWalk at((uint32_t)Kp / 8u, (uint32_t)ctid);
    while (at.n < (uint32_t)r.N) {
        uint4 v[kItems][2];
        PanelWalk ahead = at;
#pragma unroll
        for (int b = 0; b < kItems; ++b, ahead.next()) {
            v[b][0] = v[b][1] = make_uint4(0u, 0u, 0u, 0u);
            const int left = r.K - 8 * (int)ahead.k;
            if (ahead.n >= (uint32_t)r.N || left <= 0) continue;
            const uintptr_t p = (uintptr_t)(x + (size_t)ahead.n * r.ld + 8u * ahead.k), w = p & ~(uintptr_t)15;
            v[b][0] = word(w);
            if (w + 16 < p + 2u * (uint32_t)min(left, 8)) v[b][1] = word(w + 16);
        }
#pragma unroll
        for (int b = 0; b < kItems; ++b, at.next()) {
            if (at.n >= (uint32_t)r.N) break;
            const int left = r.K - 8 * (int)at.k;
            const uint32_t off = (uint32_t)(uintptr_t)(x + (size_t)at.n * r.ld) & 15u;                 // (8 columns are 16 bytes)
            uint32_t w[8] = {v[b][0].x, v[b][0].y, v[b][0].z, v[b][0].w, v[b][1].x, v[b][1].y, v[b][1].z, v[b][1].w};
#pragma unroll
            for (int i = 0; i < 6; ++i) w[i] = off & 8u ? w[i + 2] : w[i];
#pragma unroll
            for (int i = 0; i < 5; ++i) w[i] = off & 4u ? w[i + 1] : w[i];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                w[i] = off & 2u ? __funnelshift_r(w[i], w[i + 1], 16) : w[i];
                w[i] = 2 * i + 1 < left ? w[i] : 2 * i < left ? w[i] & 0xFFFFu : 0u;
            }
            *(uint4*)(r.buf + at.n * (uint32_t)r.pitch + 16u * at.k) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// bf16(silu(g) * u) in place of activations; t_out (or NULL) gets it too
__device__ __noinline__ void stage_silu(const XRows& r, const uint16_t* g, const uint16_t* u, uint16_t* t_out, int ctid)
{
    PanelWalk at((uint32_t)r.K, (uint32_t)ctid);
    while (at.n < (uint32_t)r.N) {
        uint16_t v[kStageBatch];
        PanelWalk ahead = at;
#pragma unroll
        for (int b = 0; b < kStageBatch; ++b, ahead.next()) {
            if (ahead.n >= (uint32_t)r.N) break;
            const size_t i = (size_t)ahead.n * r.ld + ahead.k;
            v[b] = silu_mul_bits(__ldcg(g + i), __ldcg(u + i));
            if (t_out) t_out[i] = v[b];
        }
#pragma unroll
        for (int b = 0; b < kStageBatch; ++b, at.next()) {
            if (at.n >= (uint32_t)r.N) break;
            *(uint16_t*)(r.buf + at.n * (uint32_t)r.pitch + 2u * at.k) = v[b];
        }
    }
}

// All consumer warps have come this far (an mbarrier and not bar.sync: the wait is bounded like every other).
struct ConsumerSync {
    uint32_t bar, phase;
    __device__ __forceinline__ bool operator()(const WaitCtx& w, int lane)
    {
        __syncwarp();
        if (lane == 0) mbar_arrive(bar);
        const bool ok = wait_phase_warp(bar, phase, w);
        phase ^= 1u;
        return ok;
    }
};

// rows[n] = rmsnorm(rows[n] [+ res]) * norm_w on the staged columns, two rows at a time.  The sum of squares is over the
// whole row: the columns that the other CTA of the cluster stages are read from global memory.  xg: the rows in global
// memory, from the first column on; c0: first staged column.
// scratch: shared memory that nobody else uses now.
__device__ __noinline__ bool fold_norm(const XRows& r, const SFold& f, const uint16_t* xg, int row0, int c0, bool pub, float (*red)[kCellWarps],
                                       uint16_t* scratch, int scratch_bytes,
                                       ConsumerSync& sync, const WaitCtx& wc, int ctid)
{
    const int lane = ctid & 31;
    // Eight columns of up to four rows to a thread, from the first load to the last store (input, residual and gains asked for together,
    // 16 bytes at a time), where the rows are on 16 bytes and short enough.  Whole rows stand in `scratch` while their squares are added
    // up, in the order of the loop below; the staged copies are written over.
    // From kHeldMin values on.  Below, few threads have a column, and code that is gone through once comes from L2: us of a decode block
    // by the loop and through registers: hidden 256, four and twelve rows 36.2 and 39.1, 57.0 and 57.1; 512, two and six 34.9 and 37.5,
    // 47.4 and 46.7; 768, two, four and eight 39.5 and 42.1, 46.0 and 46.1, 58.5 and 53.7; 1024, two and three 42.0 and 42.3, 47.1 and 44.2;
    // 2048, eight 105 and 66.
    constexpr int kHeldMin = 3072;
    constexpr int kHeld = 4;
    if (r.N * r.ld >= kHeldMin && (r.ld & 7) == 0 && r.ld <= 8 * kCellConsumers && 2 * r.ld <= scratch_bytes &&
        ((((uintptr_t)xg | (uintptr_t)f.res | (uintptr_t)f.norm_w | (uintptr_t)f.sum_out | (uintptr_t)f.norm_out) & 15) == 0)) {
        const int fit = min(kHeld, scratch_bytes / (2 * r.ld));
        const bool mine = ctid < (r.ld >> 3), own = mine && 8 * ctid >= c0 && 8 * ctid < c0 + r.K;
        const uint4 w = own ? __ldg((const uint4*)f.norm_w + ctid) : make_uint4(0u, 0u, 0u, 0u);
        for (int n0 = 0; n0 < r.N; n0 += fit) {
            const int rows = min(fit, r.N - n0);
            const size_t at = (size_t)(row0 + n0) * r.ld;
            uint4 v[kHeld];
#pragma unroll
            for (int q = 0; q < kHeld; ++q)
                v[q] = mine && q < rows ? __ldcg((const uint4*)(xg + (size_t)(n0 + q) * r.ld) + ctid) : make_uint4(0u, 0u, 0u, 0u);
            if (f.res) {
                uint4 a[kHeld];
#pragma unroll
                for (int q = 0; q < kHeld; ++q)
                    a[q] = mine && q < rows ? __ldcg((const uint4*)(f.res + at + (size_t)q * r.ld) + ctid) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int q = 0; q < kHeld; ++q) {
                    v[q] = add_bf16_rows(v[q], a[q]);
                    if (own && pub && f.sum_out && q < rows) ((uint4*)(f.sum_out + at + (size_t)q * r.ld))[ctid] = v[q];
                }
            }
#pragma unroll
            for (int q = 0; q < kHeld; ++q)
                if (mine && q < rows) ((uint4*)(scratch + (size_t)q * r.ld))[ctid] = v[q];
            if (!sync(wc, lane)) return false;
#pragma unroll
            for (int q = 0; q < kHeld; ++q) {
                if (q >= rows) continue;
                float ss = 0.f;
                for (int i = ctid; i < r.ld; i += kCellConsumers) {
                    const float e = bf16_to_f32(scratch[(size_t)q * r.ld + i]);
                    ss += e * e;
                }
                __syncwarp();
                ss = warp_sum(ss);
                if (lane == 0) red[q][ctid >> 5] = ss;
            }
            if (!sync(wc, lane)) return false;
#pragma unroll
            for (int q = 0; q < kHeld; ++q) {
                if (!own || q >= rows) continue;
                float tot = 0.f;
#pragma unroll
                for (int k = 0; k < kCellWarps; ++k) tot += red[q][k];
                const uint4 o = scale_bf16_row(v[q], rsqrtf(tot / (float)r.ld + f.eps), w);
                *(uint4*)(r.buf + (size_t)(n0 + q) * r.pitch + 2 * (8 * ctid - c0)) = o;
                if (pub && f.norm_out) ((uint4*)(f.norm_out + at + (size_t)q * r.ld))[ctid] = o;
            }
        }
        return true;
    }
    for (int n0 = 0; n0 < r.N; n0 += 2) {
        if (!sync(wc, lane)) return false;     // the rows are staged; red is free
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int n = n0 + q;
            if (n >= r.N) continue;
            uint16_t* xl = (uint16_t*)(r.buf + (size_t)n * r.pitch);
            const size_t go = (size_t)(row0 + n) * r.ld, gx = (size_t)n * r.ld;
            float ss = 0.f;
            for (int i = ctid; i < r.ld; i += kCellConsumers) {
                const int j = i - c0;
                const bool own = j >= 0 && j < r.K;
                float v = bf16_to_f32(own ? xl[j] : __ldcg(xg + gx + i));
                if (f.res) {
                    const uint16_t sb = f32_to_bf16_rne(v + bf16_to_f32(__ldcg(f.res + go + i)));
                    if (own) {
                        xl[j] = sb;
                        if (pub && f.sum_out) f.sum_out[go + i] = sb;
                    }
                    v = bf16_to_f32(sb);
                }
                ss += v * v;
            }
            __syncwarp();
            ss = warp_sum(ss);
            if (lane == 0) red[q][ctid >> 5] = ss;
        }
        if (!sync(wc, lane)) return false;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int n = n0 + q;
            if (n >= r.N) continue;
            uint16_t* xl = (uint16_t*)(r.buf + (size_t)n * r.pitch);
            const size_t go = (size_t)(row0 + n) * r.ld;
            float tot = 0.f;
#pragma unroll
            for (int w = 0; w < kCellWarps; ++w) tot += red[q][w];
            const float rs = rsqrtf(tot / (float)r.ld + f.eps);
            // (a column is normalised by the thread that added its residual)
            for (int i = ctid; i < r.ld; i += kCellConsumers) {
                const int j = i - c0;
                if (j < 0 || j >= r.K) continue;
                const uint16_t o = f32_to_bf16_rne(bf16_to_f32(xl[j]) * rs * bf16_to_f32(__ldg(f.norm_w + i)));
                xl[j] = o;
                if (pub && f.norm_out) f.norm_out[go + i] = o;
            }
        }
    }
    return true;
}

// ---- finishing a tile ---------------------------------------------------------------------

// A finisher shares its scheduler with busy warps and gets an instruction in every few cycles, so what counts here is the
// number of instructions per tile.  Lane 2 r + t holds activation rows 4 t .. 4 t + 3 (and those + 8) of weight row r.

// The sum of the C <= 4 contributions of a group, in one order.  p: the lane's place in the first.
template <int NR>
__device__ __forceinline__ void sum_parts(const unsigned char* p, int C, float (&r)[NR / 8][4])
{
    constexpr uint32_t kStep = kTileRows * kPartRowBytes * (NR / 8);
#pragma unroll
    for (int h = 0; h < NR / 8; ++h) {
        float4 v[kChunkCells];
#pragma unroll
        for (int k = 0; k < kChunkCells; ++k) v[k] = k < C ? *(const float4*)(p + (uint32_t)k * kStep + 512u * h) : make_float4(0.f, 0.f, 0.f, 0.f);
        r[h][0] = (v[0].x + v[1].x) + (v[2].x + v[3].x);
        r[h][1] = (v[0].y + v[1].y) + (v[2].y + v[3].y);
        r[h][2] = (v[0].z + v[1].z) + (v[2].z + v[3].z);
        r[h][3] = (v[0].w + v[1].w) + (v[2].w + v[3].w);
    }
}

__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi)
{
    uint32_t d;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
    return d;
}

// bf16 values of up to four activation rows, `ld` elements apart
__device__ __forceinline__ void store_bf16(uint16_t* p, uint2 v, int rows, size_t ld)
{
    if (rows > 0) p[0] = (uint16_t)v.x;
    if (rows > 1) p[ld] = (uint16_t)(v.x >> 16);
    if (rows > 2) p[2 * ld] = (uint16_t)v.y;
    if (rows > 3) p[3 * ld] = (uint16_t)(v.y >> 16);
}

// ---- activations that are not finite --------------------------------------------------------

// The products of an expanded cell take in the weights that were dropped, as zeros, and zero times an infinite or undefined
// activation is NaN: it would reach every output of its row.  So the finishers keep an eye on their sums, and where a stage had
// any that were not finite they form these again, from the kept weights alone.  (To look for such activations instead is a pass
// over every stage's rows.)  What it costs where all is finite (us): five rows of 1531 x 3001 8.4 -> 8.6, 48 rows of 8192 x 2048
// 25.4 -> 25.8, an eight-row step of two blocks of 2048/512/8192 67.8 -> 68.2, a block of 3072/1024/8192 for 16 rows 61.4 -> 61.5.
// With a vote and the slow path in the loop over tiles these took 8.5, 26.4, 69.1, 61.9; a call in the loop over stages, the
// arguments of which tie up the finishers' registers, 8.8, 26.7, 69.5, 63.5.

// the largest magnitude of m, a, b; NaN if one of them is
__device__ __forceinline__ float watch(float m, float a, float b)
{
    asm("max.NaN.abs.f32 %0, %0, %1, %2;" : "+f"(m) : "f"(a), "f"(b));
    return m;
}

// The sum over the Dr cells of a share of a tile for one weight row and one activation row, kept weight by kept weight.  off: the
// share's directory entries; x: the staged activations, in either CTA.  A kept zero counts as dropped.
__device__ __forceinline__ float sum_kept(float sum, const uint32_t* off, const unsigned char* cells, int Dr, int row, const unsigned char* x)
{
    const int second = row >> 3;
#pragma unroll 1
    for (int d = 0; d < Dr; ++d) {
        const unsigned char* cell = cells + (size_t)__ldg(off + d) * 32;
        const int H = (int)((__ldg(off + d + 1) - __ldg(off + d)) * 32u - kCellHeaderBytes) / 128;
        const uint32_t* words = (const uint32_t*)(cell + kCellHeaderBytes);
#pragma unroll 1
        for (int t = 0; t < 4; ++t) {
            const int owner = 4 * (row & 7) + t;
            const int column = second ? (__ldg(cell + 128 + owner) & 0x7F) >> 2 : owner;
            int at = second ? H - 1 : 0;
#pragma unroll 1
            for (uint32_t left = __ldg((const uint32_t*)cell + owner) >> (16 * second) & 0xFFFFu; left; left &= left - 1u, at += second ? -1 : 1) {
                const int e = __ffs((int)left) - 1;
                const uint32_t w = __ldg(words + 32 * at + column);
                const uint32_t xv = *(const uint32_t*)(x + 2 * (d * kCellCols + 32 * (e >> 2) + 8 * t + 2 * (e & 3)));
                if (w & 0x7FFFu) sum = fmaf(bf16_lo(w), bf16_lo(xv), sum);
                if (w & 0x7FFF0000u) sum = fmaf(bf16_hi(w), bf16_hi(xv), sum);
            }
        }
    }
    return sum;
}

// Every tile that this CTA has finished in the stage, once more: outputs that are not finite are replaced.  One warp, with the
// lanes that stored them.  rows: this CTA's staged activations; the other CTA's stay where they are until the grid barrier, or
// its end, for which this warp is still missing.
__device__ __forceinline__ void repair_stage(const CStage& st, int rank, int cluster, int clusters, void* y_last, const unsigned char* rows, int N, int n0)
{
    const int lane = threadIdx.x & 31, D = st.D;
    const bool alone = D == 1;
    TileRuns runs(cluster, clusters, st.rot, st.tiles_div, st.tiles_rem);
    int mat, t0, nt;
    while (runs.next(st.pair, st.count, st.mat[0].T, st.mat[1].T, st.mat[2].T, mat, t0, nt)) {
        const CMat& md = st.mat[mat];
        unsigned char* y = (unsigned char*)(y_last && mat == 0 ? y_last : md.y);
        for (int j = alone ? 0 : rank; j < nt; j += alone ? 1 : 2) {
            const int row = (t0 + j) * kTileRows + (lane >> 1);
#pragma unroll 1
            for (int n = (lane & 1) * 4; n < N && row < md.M; n += (n & 3) == 3 ? 5 : 1) {
                const size_t at = (size_t)(n0 + n) * md.M + row;
                float* f = (float*)y + at;
                uint16_t* b = (uint16_t*)y + at;
                if (md.y_f32 ? !isfinite(*f) : (*b & 0x7F80u) == 0x7F80u) {
                    float sum = 0.f;
#pragma unroll 1
                    for (int r = 0; r < 2; ++r) {
                        uint64_t x;
                        asm("mapa.u64 %0, %1, %2;" : "=l"(x) : "l"((uint64_t)rows), "r"(r));
                        const int Dr = share_cells(D, r);
                        const size_t first = (r ? (size_t)md.T * share_cells(D, 0) : 0) + (size_t)(t0 + j) * Dr;
                        sum = sum_kept(sum, md.off + first, md.cells, Dr, lane >> 1, (const unsigned char*)x + (size_t)n * (2 * Dr * kCellCols + 64));
                    }
                    if (md.y_f32) *f = sum;
                    else *b = (uint16_t)bf16_pair(sum, 0.f);
                }
                if (st.pair && mat == 1 && st.t_out) st.t_out[at] = (uint16_t)silu_mul_pair(((const uint16_t*)st.mat[0].y)[at], *b);
            }
        }
        __syncwarp();
    }
}

// ... out of line, for launches of one stage, which repair it on their way out
__device__ __noinline__ void repair_call(const CStage& st, int rank, int cluster, int clusters, void* y_last, const unsigned char* rows, int N, int n0)
{
    repair_stage(st, rank, cluster, clusters, y_last, rows, N, n0);
}

// ---- the kernel ---------------------------------------------------------------------------

template <int MAXS, int NR, bool FOLD>
__global__ void __launch_bounds__(kCellThreads, 1) cell_kernel(const __grid_constant__ CArgs<MAXS> a)
{
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr uint32_t kPartOff = (uint32_t)((sizeof(CellShared<NR>) + 127) & ~127);
    CellShared<NR>* sh = (CellShared<NR>*)smem;
    constexpr uint32_t kSlotBytes = (uint32_t)part_slot_bytes(NR);
    const uint32_t xoff = kPartOff + 2u * (uint32_t)(a.part_mask + 1) * kSlotBytes;
    const uint32_t ring_off = xoff + (uint32_t)a.xbuf_bytes;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);      // (known to be the same in all lanes)
    const int rank = blockIdx.x & 1, cluster = blockIdx.x >> 1, clusters = gridDim.x >> 1;
    const int G = gridDim.x;
    const int N = a.N;
    const uint32_t NS = (uint32_t)a.n_slots;

    pdl_let_next_start();
    if (tid < kCellGroups * kGroupSlots) {
        mbar_init(smem_u32(&sh->full[0][0]) + 8 * tid, 1);
        mbar_init(smem_u32(&sh->empty[0][0]) + 8 * tid, kChunkCells);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    } else if (tid == 32) {
        mbar_init(smem_u32(&sh->dfull), 1);
        mbar_init(smem_u32(&sh->xfull), 1);
        mbar_init(smem_u32(&sh->left), kCellWarps + 2);
        mbar_init(smem_u32(&sh->csync), kCellWarps);
        sh->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    } else if (tid >= 64 && tid < 64 + 2 * kPartSlots) {
        mbar_init(smem_u32(&sh->pfull[0][0]) + 8 * (tid - 64), kChunkCells);
        (&sh->freed[0][0])[tid - 64] = 0u;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    } else if (tid >= 96 && tid < 96 + kRecvSlots) {
        mbar_init(smem_u32(&sh->rfull[tid - 96]), 1);
        if (tid < 98) mbar_init(smem_u32(&sh->credit[tid - 96]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    // waited for before the first access to the other CTA (only its mbarriers have to be there: fence.mbarrier_init above)
    asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");

    WaitCtx wc;
    wc.abort_flag = &sh->abort_flag;
    wc.budget = a.wait_cycles;

    // word i of a stage's descriptor
    auto stage_word = [&](int s, int i) {
        return a.ext && s > 0 ? ((const uint32_t*)(a.ext + s))[i] : ((const uint32_t*)&a.inl[MAXS == 1 ? 0 : s])[i];
    };
    // Starts the copies of every second activation row of stage s (the service warp's and the sending finisher's halves;
    // a copy takes a warp some 90 cycles to start).  bytes: of all the rows; 0: the consumers fetch them.
    auto start_rows = [&](int s, int part, uint32_t& bytes) {
        const uint32_t xfull = smem_u32(&sh->xfull);
        const CStage& st = sh->stage[s & 1];
        // (the first stage's rows are on their way before its descriptor has been copied to shared memory)
        const int D = s == 0 ? a.inl[0].D : st.D, K = s == 0 ? a.inl[0].K : st.K;
        const int Dr = share_cells(D, rank), xb = rank ? share_cells(D, 0) * kCellCols : 0;
        const int Kr = min(K - xb, Dr * kCellCols);
        const uint16_t* x = s == 0 ? (a.x_in ? a.x_in : a.inl[0].x) : st.x;
        bytes = x && (K & 7) == 0 && (((uintptr_t)x) & 15) == 0 && Kr > 0 ? (uint32_t)(N * Kr * 2) : 0u;
        if (s > 0) {
            // this CTA's warps have left the previous stage, those without a tile in it among them ...
            if (!wait_phase_warp(smem_u32(&sh->left), (uint32_t)(s - 1) & 1u, wc)) return false;
            // ... and every CTA has written its outputs (and has read its activations)
            bool ok = true;
            if (lane == 0) ok = grid_wait(a.gbar, (unsigned int)s * (unsigned int)G, wc);
            if (!__all_sync(0xFFFFFFFFu, ok)) return false;
            asm volatile("fence.proxy.async.global;" ::: "memory");      // ... written through the generic proxy, read by bulk copies
        }
        int n = 2 * lane + part;
        if (bytes && n < N) {
            n += cluster;                                        // (not all CTAs ask for the same row first)
            n -= n / N * N;
            bulk_g2s(smem_u32(smem) + xoff + (uint32_t)(n * (2 * Dr * kCellCols + 64)), x + (size_t)(a.n0 + n) * K + xb, (uint32_t)(Kr * 2), xfull);
        }
        __syncwarp();
        return true;
    };
    constexpr bool kWide = NR > kPanelRows;      // (launches of one stage)
    bool odd = false;                            // (finishers) sums of the stage were not finite
    if (warp != kProducerWarp) pdl_wait();       // (the producer streams weights already)
    if (warp == kProducerWarp) {
        // ---------------------------------------------------------------------- producer
        // Directory entries come in batches of up to 32 chunks of a stage, a chunk to a lane.  (Like the finishers this warp
        // gets an instruction in every few cycles only, and with single cells' entries to look up and to pass on it spent 600
        // cycles per chunk where a chunk's share of HBM's bandwidth is 540.)
        // A stage's descriptor is spread over the lanes, and the next stage's is loaded when the stage begins: its latency
        // (and a chain of dependent loads, 3000 cycles at every run of tiles when they were made one by one) is hidden.
        constexpr int kWords = (int)(sizeof(CStage) / 4);
        static_assert(kWords <= 64, "two words a lane");
        uint32_t w0 = stage_word(0, lane), w1 = 32 + lane < kWords ? stage_word(0, 32 + lane) : 0u, next_w0 = 0, next_w1 = 0;
        auto word = [&](int i) { return __shfl_sync(0xFFFFFFFFu, i < 32 ? w0 : w1, i & 31); };
        auto pointer = [&](int i) {
            const uint32_t lo = word(i), hi = word(i + 1);
            return (const unsigned char*)((unsigned long long)hi << 32 | lo);
        };
#define SD2_WORD(f) ((int)(offsetof(CStage, f) / 4))
        int sa = 0, q0 = 0, n = 0, gb = 0;                       // stage; of the run of tiles: next chunk, cells, first group
        RunDeal deal(0, 0);
        const uint32_t* off = nullptr;
        const unsigned char* cells = nullptr;
        TileRuns runs(0, 0, 0, 0, 0);
        int D = 0, pair = 0, count = 0, T0 = 0, T1 = 0, T2 = 0;
        auto begin_stage = [&]() {
            if (sa + 1 < a.n_stages) {
                next_w0 = stage_word(sa + 1, lane);
                next_w1 = 32 + lane < kWords ? stage_word(sa + 1, 32 + lane) : 0u;
            }
            runs = TileRuns(cluster, clusters, (int)word(SD2_WORD(rot)), (int)word(SD2_WORD(tiles_div)), (int)word(SD2_WORD(tiles_rem)));
            D = (int)word(SD2_WORD(D));
            pair = (int)word(SD2_WORD(pair));
            count = (int)word(SD2_WORD(count));
            T0 = (int)word(SD2_WORD(mat[0].T));
            T1 = (int)word(SD2_WORD(mat[1].T));
            T2 = (int)word(SD2_WORD(mat[2].T));
        };
        begin_stage();
        uint32_t o0 = 0, o1 = 0;             // the lane's chunk: directory entries of its first cell and past its last
        const unsigned char* from = nullptr;
        int from_grp = 0;                    // whose chunk it is
        auto load_batch = [&]() {            // returns the number of chunks; 0: the end
            int got = 0;
            while (got < 32 && sa < a.n_stages) {
                if (q0 < deal.chunks) {
                    const int q = q0 + lane - got;
                    if (lane >= got && q < deal.chunks) {
                        const int turn = deal.split ? q : q / deal.per, i0 = deal.split ? 0 : turn * deal.cells;
                        const int i = i0 + (deal.split ? q : q - turn * deal.per) * kChunkCells;
                        o0 = __ldg(off + i);
                        o1 = __ldg(off + min(i + kChunkCells, deal.split ? n : min(i0 + deal.cells, n)));
                        from = cells;
                        from_grp = (gb + turn) % kCellGroups;
                    }
                    const int take = min(32 - got, deal.chunks - q0);
                    q0 += take;
                    got += take;
                    continue;
                }
                gb = (gb + deal.turns) % kCellGroups;            // on to the next run of tiles, the next stage
                deal = RunDeal(0, 0);
                q0 = 0;
                int mat, t0, nt;
                if (runs.next(pair, count, T0, T1, T2, mat, t0, nt)) {
                    const int Dr = share_cells(D, rank), w = mat * (int)(sizeof(CMat) / 4);
                    n = nt * Dr;
                    deal = RunDeal(Dr, nt);
                    cells = pointer(w + SD2_WORD(mat[0].cells));
                    off = (const uint32_t*)pointer(w + SD2_WORD(mat[0].off)) +
                          (rank ? (size_t)word(w + SD2_WORD(mat[0].T)) * share_cells(D, 0) : 0) + (size_t)t0 * Dr;
                } else {
                    if (++sa < a.n_stages) {
                        w0 = next_w0;
                        w1 = next_w1;
                        begin_stage();
                    }
                    if (got > 0) break;      // (the next descriptor may still be on its way)
                }
            }
            return got;
        };
        // weights are read once: with several stages their lines leave L2 first, so that the stream does not push out
        // the small, shared, re-read activations
        const uint64_t policy = l2_evict_first();
        const bool hinted = a.n_stages > 1;
        const uint32_t full0 = smem_u32(&sh->full[0][0]), empty0 = smem_u32(&sh->empty[0][0]), ring = smem_u32(smem) + ring_off;
        uint32_t next_slot = 0x101010u;      // of each group (a byte each): its next slot, 16 times the parity of the wait for it
        bool ok = true;
        for (int got; ok && (got = load_batch()) > 0;) {
            const uint32_t bytes = (o1 - o0) * 32u;
            for (int k = 0; k < got; ++k) {
                const int grp = __shfl_sync(0xFFFFFFFFu, from_grp, k);
                const uint32_t at = next_slot >> (8 * grp) & 0xFFu, slot = at & 15u;
                const uint32_t s = (uint32_t)(grp * kGroupSlots) + slot, dst = ring + ((uint32_t)grp * NS + slot) * (uint32_t)a.chunk_bytes;
                // (slots are not given back before the consumers are let go, which the budget of a wait is not meant for)
                if (at == 0u) pdl_wait();        // (a group's first slot that has to be given back)
                if (!wait_phase_warp(empty0 + 8 * s, at >> 4, wc)) { ok = false; break; }
                if (hinted) bulk_chunk(dst, from + (size_t)o0 * 32, bytes, full0 + 8 * s, lane == k, policy);
                else bulk_chunk(dst, from + (size_t)o0 * 32, bytes, full0 + 8 * s, lane == k);
                next_slot ^= (at ^ (slot + 1 == NS ? (at ^ 16u) & 16u : at + 1u)) << (8 * grp);
            }
        }
        // (consumers that gave up have left chunks on their way; where they did not, these have landed)
        for (int g = 0; g < kCellGroups; ++g)
            for (uint32_t u = 0; u < NS; ++u) {
                const uint32_t at = next_slot >> (8 * g) & 0xFFu;
                wait_landed(full0 + 8 * (g * kGroupSlots + u), (at >> 4) ^ (u < (at & 15u) ? 1u : 0u), wc.budget);
            }
        __syncwarp();
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    } else if (warp == kServiceWarp) {
        // ---------------------------------------------------------------------- service warp
        const uint32_t xfull = smem_u32(&sh->xfull);
        auto fetch_stage = [&](int s) {
            uint32_t* dst = (uint32_t*)&sh->stage[s & 1];
            for (int i = lane; i < (int)(sizeof(CStage) / 4); i += 32) dst[i] = stage_word(s, i);
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&sh->dfull));
        };
        int started = -1;                                        // the last stage whose rows are on their way
        for (int s = 0; s < a.n_stages; ++s) {
            uint32_t bytes;
            if (!start_rows(s, 0, bytes)) break;
            if (lane == 0) {
                if (bytes) mbar_expect_tx(xfull, bytes);
                else mbar_arrive(xfull);
            }
            started = s;
            if (s == 0) fetch_stage(0);
            if (s + 1 < a.n_stages) fetch_stage(s + 1);
        }
        wait_landed(xfull, (uint32_t)started & 1u, wc.budget);   // (stage 0's at least; no phase is begun before the one before it is through)
        __syncwarp();
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    } else if (warp > kServiceWarp) {
        // ---------------------------------------------------------------------- finishers
        const int own = warp == kOwnWarp ? 1 : 0;
        const uint32_t PM = (uint32_t)a.part_mask;
        const uint32_t pfull0 = smem_u32(&sh->pfull[own][0]);
        const uint32_t recv_off = (uint32_t)lane * 16u;
        const unsigned char* parts = smem + kPartOff + (uint32_t)own * (PM + 1u) * kSlotBytes + recv_off;
        const int n0 = (lane & 1) * 4, r0 = lane >> 1;
        const uint32_t peer_recv = peer_addr(&sh->recv[0][0][0], (uint32_t)(rank ^ 1)) + recv_off;
        const uint32_t peer_rfull = peer_addr(&sh->rfull[0], (uint32_t)(rank ^ 1)), peer_credit = peer_addr(&sh->credit[0], (uint32_t)(rank ^ 1));
        const uint32_t rfull0 = smem_u32(&sh->rfull[0]), credit0 = smem_u32(&sh->credit[0]);
        constexpr uint32_t kRecvBytes = (uint32_t)sizeof(sh->recv[0]);
        uint32_t ps = 0, use = 0, rs = 0, ru = 0;                // slot of partial sums and its use, the same for exchanged sums
        bool ok = true;
        uint32_t bytes;
        int started = 0;                                         // (the sending finisher) the last stage whose rows it has started
        if (!own) start_rows(0, 1, bytes);
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        const uint32_t dfull = smem_u32(&sh->dfull);
        bool ready = wait_phase_warp(dfull, 0u, wc);
        for (int s = 0; s < a.n_stages && ok && ready; ++s) {
            if (!own && s > 0) {
                if (!start_rows(s, 1, bytes)) break;
                started = s;
            }
            const CStage& st = sh->stage[s & 1];
            const int D = st.D, Dr = share_cells(D, rank), C = Dr < kChunkCells ? Dr : kChunkCells;
            const int n_parts = Dr > kSplitCells ? kCellGroups : 1;
            const bool alone = D == 1, pair = st.pair != 0;
            float seen = 0.f;                                    // largest magnitude of the lane's sums
            TileRuns runs(cluster, clusters, st.rot, st.tiles_div, st.tiles_rem);
            int mat, t0, nt;
            while (ok && runs.next(pair, st.count, st.mat[0].T, st.mat[1].T, st.mat[2].T, mat, t0, nt)) {
                if (alone && (rank || !own)) continue;           // CTA 0 has all the cells and finishes all the tiles
                const CMat& md = st.mat[mat];
                const int M = md.M;
                const bool f32 = md.y_f32 != 0;
                unsigned char* y = (unsigned char*)(s == a.n_stages - 1 && a.y_out && mat == 0 ? a.y_out : md.y);
                for (int j = alone ? 0 : own ? rank : rank ^ 1; j < nt; j += alone ? 1 : 2) {
                    float r[NR / 8][4];
                    for (int part = 0; part < n_parts; ++part) {
                        if (!(ok = wait_phase_warp(pfull0 + 8 * ps, use & 1u, wc))) break;
                        if (part == 0) {
                            sum_parts<NR>(parts + ps * kSlotBytes, C, r);
                        } else {
                            float q[NR / 8][4];
                            sum_parts<NR>(parts + ps * kSlotBytes, C, q);
#pragma unroll
                            for (int h = 0; h < NR / 8; ++h)
#pragma unroll
                                for (int k = 0; k < 4; ++k) r[h][k] += q[h][k];
                        }
                        __syncwarp();
                        if (lane == 0) *(volatile unsigned int*)&sh->freed[own][ps] = use + 1u;
                        if (++ps > PM) { ps = 0; ++use; }
                    }
                    if (!ok) break;
                    // (the other CTA is told of every half of recv[] that has been used up: an arrival there that releases
                    // takes some 700 cycles)
                    const uint32_t half = rs / (kRecvSlots / 2);
                    if (!own) {
                        if (ru > 0 && rs % (kRecvSlots / 2) == 0 && !(ok = wait_phase_warp(credit0 + 8 * half, (ru - 1u) & 1u, wc))) break;
#pragma unroll
                        for (int h = 0; h < NR / 8; ++h) st_async(peer_recv + rs * kRecvBytes + 512u * h, r[h], peer_rfull + 8 * rs);
                        if (++rs == kRecvSlots) { rs = 0; ++ru; }
                        continue;
                    }
                    if (!alone) {
                        if (lane == 0) mbar_expect_tx(rfull0 + 8 * rs, 512u * (NR / 8));
                        if (!(ok = wait_phase_warp(rfull0 + 8 * rs, ru & 1u, wc))) break;
#pragma unroll
                        for (int h = 0; h < NR / 8; ++h) {
                            const float4 v = *(const float4*)((const unsigned char*)&sh->recv[rs][0][0] + recv_off + 512u * h);
                            r[h][0] += v.x;
                            r[h][1] += v.y;
                            r[h][2] += v.z;
                            r[h][3] += v.w;
                        }
                        __syncwarp();
                        if ((rs + 1) % (kRecvSlots / 2) == 0 && lane == 0) mbar_arrive_remote(peer_credit + 8 * half);
                        if (++rs == kRecvSlots) { rs = 0; ++ru; }
                    }
#pragma unroll
                    for (int h = 0; h < NR / 8; ++h) seen = watch(watch(seen, r[h][0], r[h][1]), r[h][2], r[h][3]);
                    const int row = (t0 + j) * kTileRows + r0;
                    if (row >= M) continue;
#pragma unroll
                    for (int h = 0; h < NR / 8; ++h) {
                        const int n = n0 + 8 * h, rows = N - n;      // activation rows of the lane that exist
                        const size_t at = (size_t)(a.n0 + n) * M + row;
                        if (f32) {
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                if (k < rows) ((float*)y)[at + (size_t)k * M] = r[h][k];
                            continue;
                        }
                        const uint2 b = make_uint2(bf16_pair(r[h][0], r[h][1]), bf16_pair(r[h][2], r[h][3]));
                        store_bf16((uint16_t*)y + at, b, rows, (size_t)M);
                        if (pair) {
                            // gate tiles of a run wait for the up tiles of the run that follows, written and read by the same lane
                            uint2* gt = &sh->gate[j % kPairSlots][h][lane];
                            if (mat == 0) *gt = b;
                            else if (st.t_out) store_bf16(st.t_out + at, make_uint2(silu_mul_pair(gt->x, b.x), silu_mul_pair(gt->y, b.y)), rows, (size_t)M);
                        }
                    }
                }
            }
            __syncwarp();
            // (a CTA without a tile must not be counted before the stage has begun: the barrier counts arrivals, not stages)
            odd = own && ok && __any_sync(0xFFFFFFFFu, !(seen < INFINITY));
            if (own && ok && ((odd && !kWide) || s + 1 < a.n_stages)) ok = wait_phase_warp(smem_u32(&sh->xfull), (uint32_t)s & 1u, wc);
            if (!kWide && __builtin_expect(odd && ok, 0))
                repair_stage(st, rank, cluster, clusters, s == a.n_stages - 1 ? a.y_out : nullptr, smem + xoff, N, a.n0);
            __syncwarp();
            // this CTA's outputs are visible before the grid barrier counts it (the warp's stores are ordered before this
            // lane's release by the __syncwarp above)
            if (own && ok && s + 1 < a.n_stages && lane == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.gbar) : "memory");
            __syncwarp();
            // (nobody counts as gone from a stage before it has seen the next one's descriptor: dfull never runs two ahead)
            if (s + 1 < a.n_stages) ready = wait_phase_warp(dfull, (uint32_t)(s + 1) & 1u, wc);
            if (lane == 0) mbar_arrive(smem_u32(&sh->left));
        }
        if (!own) wait_landed(smem_u32(&sh->xfull), (uint32_t)started & 1u, wc.budget);
    } else {
        // ---------------------------------------------------------------------- consumers
        const int ctid = tid;
        const int grp = warp / kChunkCells, cj = warp - grp * kChunkCells;
        const uint32_t full0 = smem_u32(&sh->full[grp][0]), empty0 = smem_u32(&sh->empty[grp][0]);
        const uint32_t xfull = smem_u32(&sh->xfull);
        const uint32_t sbase = smem_u32(smem);
        const uint32_t ring = sbase + ring_off + (uint32_t)grp * NS * (uint32_t)a.chunk_bytes;
        const int g = lane >> 2;
        ConsumerSync sync;
        sync.bar = smem_u32(&sh->csync);
        sync.phase = 0;
        uint32_t slot = 0, phase = 0;
        uint32_t cnt[2] = {0, 0};                                // tiles of each finisher before this run
        int gb = 0;                                              // the group that gets the run's first chunk
        const uint32_t dfull = smem_u32(&sh->dfull);
        bool failed = !wait_phase_warp(dfull, 0u, wc);
        for (int s = 0; s < a.n_stages && !failed; ++s) {
            const CStage& st = sh->stage[s & 1];
            const int D = st.D, K = st.K, Dr = share_cells(D, rank), xb = rank ? share_cells(D, 0) * kCellCols : 0;
            const int Kp = Dr * kCellCols, Kr = min(K - xb, Kp);
            const int pitch = 2 * Kp + 64;                       // a multiple of 64 that is not one of 128: rows of one
                                                                 // 128-bit read fall into different banks
            const uint16_t* x = (s == 0 && a.x_in) ? a.x_in : st.x;
            const bool bulk = x && (K & 7) == 0 && (((uintptr_t)x) & 15) == 0;
            TileRuns runs(cluster, clusters, st.rot, st.tiles_div, st.tiles_rem);
            const int pair = st.pair, count = st.count, T0 = st.mat[0].T, T1 = st.mat[1].T, T2 = st.mat[2].T;
            int mat, t0, nt;
            bool more = runs.next(pair, count, T0, T1, T2, mat, t0, nt);
            RunDeal deal(Dr, more ? nt : 0);
            if (!wait_phase_warp(xfull, (uint32_t)s & 1u, wc)) break;    // (all that the descriptor decides is known by now)
            const bool norm = FOLD && a.fold[MAXS == 1 ? 0 : s].norm_w;
            if ((!bulk || Kr < Kp || norm) && Kr > 0) {
                XRows xr;
                xr.buf = smem + xoff;
                xr.pitch = pitch;
                xr.K = Kr;
                xr.N = N;
                xr.ld = K;
                const size_t go = (size_t)a.n0 * K + xb;
                const bool pub = cluster == 0;
                if (!bulk && x) stage_rows(xr, x + go, xb, Kp, ctid);
                else if (!bulk) stage_silu(xr, st.g + go, st.u + go, pub && st.t_out ? st.t_out + go : nullptr, ctid);
                for (int n = 0; n < N && (bulk || !x); ++n)
                    for (int i = Kr + ctid; i < Kp; i += kCellConsumers) *(uint16_t*)(xr.buf + (size_t)n * pitch + 2 * i) = 0;
                if constexpr (FOLD) {
                    // (scratch: the places for partial sums; all those of the stage before have been read before the grid barrier let this one begin)
                    if (norm && !fold_norm(xr, a.fold[MAXS == 1 ? 0 : s], x + (size_t)a.n0 * K, a.n0, xb, pub, sh->red, (uint16_t*)(smem + kPartOff),
                                           2 * (a.part_mask + 1) * (int)kSlotBytes, sync, wc, ctid)) break;
                }
                // (the next stage's rows come here by bulk copies, which do not see these stores in the order of `left` alone)
                fence_async_smem();
                if (!sync(wc, lane)) break;
            }
            const uint32_t C = (uint32_t)(Dr < kChunkCells ? Dr : kChunkCells);
            const bool alone = D == 1;
            uint32_t xl[NR / 8];                                 // rows beyond N repeat row 0; their sums are never read
#pragma unroll
            for (int h = 0; h < NR / 8; ++h) xl[h] = sbase + xoff + (uint32_t)((g + 8 * h < N ? g + 8 * h : 0) * pitch) + 16u * (lane & 3);
            while (!failed && more) {
                const uint32_t n_parts = deal.split ? kCellGroups : 1;
                const int step = deal.split ? kCellWarps : kChunkCells;
                int q = grp - gb;                                // the group's first turn
                if (q < 0) q += kCellGroups;
                float acc[NR / 8][4];
#pragma unroll
                for (int m = 0; m < NR / 8; ++m)
#pragma unroll
                    for (int k = 0; k < 4; ++k) acc[m][k] = 0.f;
                for (int turn = deal.split ? 0 : q; turn < (deal.split ? 1 : deal.turns) && !failed; turn += kCellGroups) {
                int tl = turn * deal.tiles;                      // the warp's tile, its cell in the turn, in the tile
                const int n = min(deal.tiles, nt - tl) * Dr;
                int i = cj + (deal.split ? q * kChunkCells : 0);
                int d = i;
                while (d >= Dr && i < n) { d -= Dr; ++tl; }
                int c0 = d;
                for (int i0 = i - cj; i0 < n; i0 += step, i += step) {
                    if (!wait_phase_warp(full0 + 8 * slot, phase, wc)) { failed = true; break; }
                    if (i < n) {
                        // where the chunk's cells start: the first one's header tells the heights of all four
                        const uint32_t first = ring + slot * (uint32_t)a.chunk_bytes;
                        const uint32_t heights = __ballot_sync(0xFFFFFFFFu, (lds_u8(first + 128u + lane) & 0x80u) != 0);
                        uint32_t H = heights & 63u, before = 0;
#pragma unroll
                        for (int k = 1; k < kChunkCells; ++k)
                            if (k <= cj) { before += H; H = heights >> (6 * k) & 63u; }
                        const uint32_t cell = first + (uint32_t)cj * kCellHeaderBytes + before * 128u;
                        const uint32_t m = lds_u32(cell + 4 * lane), v0 = cell + kCellHeaderBytes;
                        const uint32_t pi = lds_u8(cell + 128u + lane) & 0x7Fu;
                        const uint32_t xd = (uint32_t)d * (2 * kCellCols);
                        multiply_cell<NR>(m, v0 + 4u * lane, v0 + (H - 1u) * 128u + pi, xl, xd, acc);
                    }
                    __syncwarp();
                    mbar_arrive_n(empty0 + 8 * slot, 1u, lane == 0);
                    if (++slot == NS) { slot = 0; phase ^= 1u; }
                    if (i >= n) continue;
                    d += step;
                    if (d < Dr) continue;                        // the next cell belongs to the same tile
                    // the tile's sums go to the finisher in charge
                    {
                        const int own = alone || (tl & 1) == rank ? 1 : 0;
                        const uint32_t k = (own ? cnt[1] : cnt[0]) + (uint32_t)(alone ? tl : tl >> 1) * n_parts + (uint32_t)(c0 / kChunkCells);
                        const uint32_t ps = k & (uint32_t)a.part_mask, use = k / ((uint32_t)a.part_mask + 1u);
                        if (use > 0 && !wait_count(&sh->freed[own][ps], use, wc)) { failed = true; break; }
                        const uint32_t entry = (uint32_t)(c0 % kChunkCells);
                        unsigned char* p = smem + kPartOff + ((uint32_t)own * ((uint32_t)a.part_mask + 1u) + ps) * kSlotBytes +
                                           entry * (kSlotBytes / kChunkCells) + 8u * lane;       // (row g, activation rows 2 t and 2 t + 1)
#pragma unroll
                        for (int h = 0; h < NR / 8; ++h) {
                            *(float2*)(p + 512 * h) = make_float2(acc[h][0], acc[h][1]);
                            *(float2*)(p + 512 * h + 256) = make_float2(acc[h][2], acc[h][3]);
                        }
#pragma unroll
                        for (int m = 0; m < NR / 8; ++m)
#pragma unroll
                            for (int k = 0; k < 4; ++k) acc[m][k] = 0.f;
                        __syncwarp();
                        // the C contributions make four arrivals between them
                        mbar_arrive_n(smem_u32(&sh->pfull[own][ps]), entry == 0 ? kChunkCells + 1u - C : 1u, lane == 0);
                    }
                    do { d -= Dr; ++tl; } while (d >= Dr);
                    c0 = d;
                }
                }
                gb = (gb + deal.turns) % kCellGroups;
                if (alone) {
                    cnt[1] += rank ? 0u : (uint32_t)nt;
                } else {                                         // tile j is finished by CTA j & 1
                    cnt[1] += ((uint32_t)(nt + 1 - rank) >> 1) * n_parts;
                    cnt[0] += ((uint32_t)(nt + rank) >> 1) * n_parts;
                }
                more = runs.next(pair, count, T0, T1, T2, mat, t0, nt);
                if (more) deal = RunDeal(Dr, nt);
            }
            __syncwarp();
            if (s + 1 < a.n_stages && !failed) failed = !wait_phase_warp(dfull, (uint32_t)(s + 1) & 1u, wc);
            if (lane == 0) mbar_arrive(smem_u32(&sh->left));
        }
        __syncwarp();
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    }

    // ---- exit: every role comes here; nobody leaves while the other CTA may still write to this one's memory
    __syncwarp();
    if (kWide && odd && wait_phase_warp(smem_u32(&sh->xfull), 0u, wc))
        repair_call(sh->stage[0], rank, cluster, clusters, a.y_out, smem + xoff, N, a.n0);
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    if (tid != 0) return;
    if (sh->abort_flag) {   // a bounded wait ran out somewhere in this CTA
        if (a.err) atomicExch(a.err, 1);
        return;
    }
    // leave the barrier words as they were found: the last CTA out clears them
    if (a.n_stages > 1) {
        const unsigned int prev = atomicAdd(a.gbar + 32, 1u);
        if (prev == (unsigned int)G - 1u) {
            atomicExch(a.gbar, 0u);
            atomicExch(a.gbar + 32, 0u);
        }
    }
}

}  // namespace sd2
