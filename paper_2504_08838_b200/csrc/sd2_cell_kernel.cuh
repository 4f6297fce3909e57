// The streaming kernel over cells (sd2_cells.hpp): programs of dependent stages for panels of up to 16 activation rows.
//
// One persistent CTA per SM runs a *program* of stages.  A stage is one launch's worth of work: up to four weights
// that read the same activations (q|k|v, or one weight), or a gate and an up projection whose results meet in
// t = silu(g) * u.  Consecutive stages depend on each other.  The hand-off is the one of sd2_kernels.cuh: a grid-wide
// barrier (programs over a caller's workspace) or tagged words (drafters).
//
// Warps of a CTA: 15 consumers, 1 producer (four per scheduler, 128 registers each).
//
//   producer   one bulk asynchronous copy per cell (about 2.7 KB at 50 % density), one lane per consumer warp: lane w fills
//              the few ring slots that warp w alone empties, and the copies of a round are issued by one instruction.
//              Nothing waits for a stage boundary: while the consumers wait for the previous stage's outputs, the next
//              stages' weights land.
//   consumers  the cells of the CTA's tiles, numbered through, go to the 15 warps in turn.  A warp expands a cell in
//              registers and multiplies it with mma.m16n8k16: the activation rows are the A operand (16 rows), eight
//              weight rows the B operand, so the expanded weights never pass through shared memory.  At the end of a
//              tile a warp leaves its 8 x N partial sums in shared memory; the warp that brings the last of a tile's
//              contributions adds them up in one fixed order (so a row's result depends neither on the launch nor on
//              N), rounds and stores.
//
// What bounds it: the expansion, about 75 permute / logic instructions per warp and 1024 slots, which an SM retires at
// two per clock (measured): 27 slots per clock and SM at most, against 17 that arrive from HBM at 50 % density.  The
// activations are staged as plain rows and nothing is gathered, so the work per slot does not grow with N.
//
// Every wait (ring barriers, tag polls, counters, grid barrier) is bounded by a cycle budget: when it runs out the CTA
// raises the error word and winds down instead of hanging.

#pragma once

#include "sd2_cells.hpp"
#include "sd2_kernels.cuh"

namespace sd2 {

constexpr int kCellWarps = 15;
constexpr int kCellConsumers = kCellWarps * 32;
constexpr int kCellThreads = kCellConsumers + 32;
constexpr int kCellSlots = 8;               // cells in flight per consumer warp, at most
constexpr int kPartSlots = 4;               // tiles whose partial sums may be incomplete
constexpr int kPairSlots = 8;               // gate tiles whose results wait for the up tile's
constexpr int kPanelRows = 16;              // activation rows of a launch, at most
constexpr int kRingGuardBytes = 256;        // the two words read past a cell's last row may lie behind the ring

struct CMat {
    const uint32_t* off;           // [T * D + 1], 32-byte units into `cells`
    const unsigned char* cells;
    void* y;                       // [N * M] (may be NULL when yt is set, or in a gate|up stage)
    uint32_t* yt;                  // [N * M] tagged words for the next stage, or NULL
    int M;
    int T;
    int y_f32;                     // 1: fp32 output, 0: bf16
    int reserved;
};

struct CStage {
    CMat mat[kMaxFused];
    const uint16_t* x;     // [N * K] bf16 (or tagged words), or NULL: the activation is bf16(silu(g) * u)
    const uint16_t* g;
    const uint16_t* u;
    uint16_t* t_out;       // gate|up stage, or x == NULL: plain copy of t (may be NULL)
    uint32_t* tt;          // gate|up stage of a tagged program: tagged t
    int K;
    int D;                 // cells per tile
    int tiles_div;         // V / grid size: the CTA with stage-local number c runs tiles_div + (c < tiles_rem) tiles (pairs)
    int tiles_rem;
    int rot;               // the stage's first tile goes to CTA `rot`, so that uneven stages even out over a program
    int tagged_in;         // x points at tagged 32-bit words
    int pair;              // mat[0] is gate, mat[1] up (equal shapes): tile i of both go to one CTA, one after the other
    int V;                 // tiles of all weights; tile pairs in a gate|up stage
    int count;             // weights
    int reserved;
};
static_assert(sizeof(CStage) % 8 == 0, "stage descriptors are arrays of 8-byte fields");

struct CArgsBase {
    const CStage* ext;              // device array of stages, or NULL: the inline ones
    const uint16_t* x_in;           // replaces stage 0's x when not NULL
    void* y_out;                    // replaces the last stage's mat[0].y when not NULL
    unsigned int* gbar;             // grid barrier: [0] arrivals, [32] exits (two cache lines)
    unsigned int* rowseq;           // tagged programs: per activation row, how often it has been produced
    int* err;                       // device error word
    long long wait_cycles;          // budget of every bounded wait
    int n_stages;
    int N;                          // activation rows of this launch
    int n0;                         // first activation row: every X / Y pointer is advanced by n0 rows
    int tagged;                     // 1: stages hand activations over as tagged words, no grid barrier
    int part_bytes;                 // shared memory: one tile's partial sums (kPartSlots of them), staged activations
    int xbuf_bytes[2];              // (two buffers, or one where xbuf_bytes[1] == 0), ring
    int slot_bytes, n_slots;        // a cell's slot, slots per consumer warp
    int fold_any;                   // host side: launch the FOLD instance
};

// MAXS: inline stages the argument block has room for (a single-stage launch passes 0.4 KB of arguments, not 3 KB)
template <int MAXS>
struct CArgs : CArgsBase {
    CStage inl[MAXS];
    SFold fold[MAXS];               // read by FOLD instances only
};

struct CellShared {
    unsigned long long full[kCellWarps][kCellSlots];    // a cell landed
    unsigned long long empty[kCellWarps][kCellSlots];   // ... and has been consumed
    int rows[kCellWarps][kCellSlots];                   // H of the cell in the slot
    unsigned int arrived[kPartSlots];                   // contributions to the tile in the slot so far
    unsigned int finished[kPartSlots];                  // 1 + number of the last tile that was finished in the slot
    unsigned int gate_done[kPairSlots];                 // 1 + number of the last gate tile whose results are in gate[]
    uint16_t gate[kPairSlots][kPanelRows][kTileRows];   // bf16 results of gate tiles
    unsigned int stage_tiles;                           // grid-barrier programs: tiles of the stage finished so far
    int abort_flag;                                     // any warp: a bounded wait ran out
    int stage_dead[2];                                  // thread 0 only: copy of abort_flag taken before a stage's barrier
    unsigned int tag_base[kPanelRows];                  // tagged programs: (production count of row n0 + n & 0xFF) << 8
    float red[2][kCellWarps];                           // FOLD: per-warp partial sums of squares of two rows
    CStage stage[2];                                    // descriptors of the current and the next stage
};

// The lanes of a warp come back from wait_phase one by one, with answers of their own.  This one brings the warp back
// together and with one answer: mma.sync, bar.sync and the like need it whole.
__device__ __forceinline__ bool wait_phase_warp(uint32_t bar, uint32_t parity, const WaitCtx& w)
{
    const bool ok = wait_phase(bar, parity, w);
    return __all_sync(0xFFFFFFFFu, ok);
}

// Until the shared counter at p has reached `want` (one warp, together).
__device__ __forceinline__ bool wait_count(const unsigned int* p, unsigned int want, const WaitCtx& w)
{
    bool ok = true;
    if ((int)(*(const volatile unsigned int*)p - want) < 0) {
        const long long t0 = clock64();
        uint32_t it = 0;
        while ((int)(*(const volatile unsigned int*)p - want) < 0) {
            if ((++it & 15u) == 0u) {
                if (*w.abort_flag) { ok = false; break; }
                if (clock64() - t0 > w.budget) { *w.abort_flag = 1; ok = false; break; }
            }
        }
    }
    ok = __all_sync(0xFFFFFFFFu, ok);
    __threadfence_block();
    return ok;
}

// Until `target` arrivals have been counted (or the wait budget is out).
__device__ __forceinline__ void grid_wait(const unsigned int* gbar, unsigned int target, const WaitCtx& w)
{
    const long long t0 = clock64();
    uint32_t it = 0;
    while ((int)(ld_acquire_gpu(gbar) - target) < 0) {
        if ((++it & 15u) == 0u) {
            if (*w.abort_flag) break;
            if (clock64() - t0 > w.budget) { *w.abort_flag = 1; break; }
        }
    }
    __threadfence();
}

__device__ __forceinline__ void consumer_sync()
{
    __syncwarp();
    named_bar_sync(1, kCellConsumers);
}

// ---- expanding a cell -----------------------------------------------------------------

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t s)
{
    uint32_t d;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(s));
    return d;
}

// c + 128 * byte K8 of p (SGN = 1) or c - 128 * byte K8 of p (SGN = -1): one integer dot-product instruction
template <int SGN, int K8>
__device__ __forceinline__ uint32_t byte_times_128(uint32_t p, uint32_t c)
{
    uint32_t d;
    constexpr uint32_t kWeight = 0x80u << (8 * K8);              // one byte: 128, or -128 where it counts as signed
    if (SGN > 0) asm("dp4a.u32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(p), "r"(kWeight), "r"(c));
    else asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(p), "r"(kWeight), "r"(c));
    return d;
}

__device__ __forceinline__ void mma_rows(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Selector tables for prmt, indexed by the two mask bits of a pair of slots (bit 0: low slot kept).  Bytes 0-3 serve
// front pairs (the next halfword of the stream is the low half of the window), bytes 4-7 back pairs (it is the high
// half).  S: places the window's halfwords in the pair's register, zeros (bytes 4..7 of prmt's second operand) for
// dropped slots.  H: moves the window on by the pair's kept halfwords.
constexpr uint32_t kSFrontLo = 0x10441044u, kSFrontHi = 0x32104444u, kSBackLo = 0x10443244u, kSBackHi = 0x32324444u;
constexpr uint32_t kHFrontLo = 0x54323210u, kHFrontHi = 0x76545432u, kHBackLo = 0x10323254u, kHBackHi = 0x32545476u;

// Half a cell: eight mma steps.  m: the lane's mask; base: byte offset in shared memory of the lane's first word (words
// 128 bytes apart, upward for SGN = 1); xo, xo8: byte offsets of the lane's first eight activations in rows g and g + 8.
template <int NR, int SGN>
__device__ __forceinline__ void half_cell(const unsigned char* smem, uint32_t m, uint32_t base, uint32_t xo, uint32_t xo8,
                                          float (&af)[4], float (&ab)[4])
{
    // words of each unit: (kept + 1) / 2, then their running sum, one byte per unit
    const uint32_t p2 = m - ((m >> 1) & 0x55555555u);
    const uint32_t p4 = (p2 & 0x33333333u) + ((p2 >> 2) & 0x33333333u);
    const uint32_t p8 = (p4 + (p4 >> 4)) & 0x0F0F0F0Fu;
    const uint32_t ends = (((p8 + 0x01010101u) >> 1) & 0x07070707u) * 0x01010101u;
    // selectors of the first (E) and second (O) pair of every group of four slots, byte-wise by table
    const uint32_t E = (m & 0x33333333u) | 0x40404040u, O = ((m >> 2) & 0x33333333u) | 0x40404040u;
    constexpr uint32_t kStep = (uint32_t)(128 * SGN);
    uint32_t start = base;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const uint32_t e = E >> (16 * t), o = O >> (16 * t);
        const uint32_t sl = prmt(kSFrontLo, kSBackLo, e), sh = prmt(kSFrontHi, kSBackHi, e);
        const uint32_t hl = prmt(kHFrontLo, kHBackLo, e), hh = prmt(kHFrontHi, kHBackHi, e);
        const uint32_t ol = prmt(kSFrontLo, kSBackLo, o), oh = prmt(kSFrontHi, kSBackHi, o);
#pragma unroll
        for (int v = 0; v < 2; ++v) {
            const int u = 2 * t + v;
            const uint32_t end = u == 0 ? byte_times_128<SGN, 0>(ends, base) : u == 1 ? byte_times_128<SGN, 1>(ends, base)
                               : u == 2 ? byte_times_128<SGN, 2>(ends, base) : byte_times_128<SGN, 3>(ends, base);
            const uint32_t wa = *(const uint32_t*)(smem + start), wb = *(const uint32_t*)(smem + (start + kStep));
            const uint32_t wz = *(const uint32_t*)(smem + (end - kStep)), wy = *(const uint32_t*)(smem + (end - 2 * kStep));
            const uint4 xv = *(const uint4*)(smem + (xo + 64u * u));
            uint4 xw = make_uint4(0u, 0u, 0u, 0u);
            if (NR > 8) xw = *(const uint4*)(smem + (xo8 + 64u * u));
            const uint32_t pf = v == 0 ? 0x0040u : 0x0062u, pb = v == 0 ? 0x0051u : 0x0073u;   // byte k of the low and of the high result
            const uint32_t f0 = prmt(wa, 0u, prmt(sl, sh, pf));
            const uint32_t f1 = prmt(prmt(wa, wb, prmt(hl, hh, pf)), 0u, prmt(ol, oh, pf));
            mma_rows(af, xv.x, xw.x, xv.y, xw.y, f0, f1);
            const uint32_t b0 = prmt(wz, 0u, prmt(sl, sh, pb));
            const uint32_t b1 = prmt(prmt(wy, wz, prmt(hl, hh, pb)), 0u, prmt(ol, oh, pb));
            mma_rows(ab, xv.z, xw.z, xv.w, xw.w, b0, b1);
            start = end;
        }
    }
}

// ---- staging the activations ------------------------------------------------------------

struct XRows {
    unsigned char* buf;      // staged rows: bf16, row n at n * pitch bytes, zero from column K to the last cell's end
    int pitch;
    int K, N;
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

constexpr int kStageBatch = 4;   // loads a thread keeps in flight while staging

__device__ __forceinline__ bool tags_ok(const uint4& v, uint32_t tag)
{
    return ((((v.x ^ tag) | (v.y ^ tag) | (v.z ^ tag) | (v.w ^ tag)) & 0xFFFFu) == 0u);
}
__device__ __forceinline__ uint4 ld_relaxed_v4(const uint32_t* p)
{
    uint4 v;
    asm volatile("ld.relaxed.gpu.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}

// Rows of tagged words -> bf16 rows, waiting for each word's tag.
__device__ __noinline__ void stage_tagged(const XRows& r, const uint32_t* x, uint32_t tag, const unsigned int* tagb, const WaitCtx& w, int ctid)
{
    if ((r.K & 3) == 0 && (((uintptr_t)x) & 15) == 0) {
        PanelWalk at((uint32_t)r.K >> 2, (uint32_t)ctid);
        while (at.n < (uint32_t)r.N) {
            uint4 v[kStageBatch];
            PanelWalk ahead = at;
#pragma unroll
            for (int b = 0; b < kStageBatch; ++b, ahead.next())
                if (ahead.n < (uint32_t)r.N) v[b] = ld_relaxed_v4(x + 4 * ((size_t)ahead.n * at.kq + ahead.k));
#pragma unroll
            for (int b = 0; b < kStageBatch; ++b, at.next()) {
                if (at.n >= (uint32_t)r.N) break;
                const uint32_t want = tag | tagb[at.n];
                if (!tags_ok(v[b], want)) {
                    const long long t0 = clock64();
                    uint32_t it = 0;
                    do {
                        v[b] = ld_relaxed_v4(x + 4 * ((size_t)at.n * at.kq + at.k));
                        if ((++it & 7u) == 0u) {
                            if (*w.abort_flag) break;
                            if (clock64() - t0 > w.budget) { *w.abort_flag = 1; break; }
                        }
                    } while (!tags_ok(v[b], want));
                }
                *(uint2*)(r.buf + at.n * (uint32_t)r.pitch + 8u * at.k) =
                    make_uint2(__byte_perm(v[b].x, v[b].y, 0x7632), __byte_perm(v[b].z, v[b].w, 0x7632));
            }
        }
        return;
    }
    for (PanelWalk at((uint32_t)r.K, (uint32_t)ctid); at.n < (uint32_t)r.N; at.next()) {
        const uint32_t v = poll_tagged1(x + (size_t)at.n * r.K + at.k, tag | tagb[at.n], w);
        *(uint16_t*)(r.buf + at.n * (uint32_t)r.pitch + 2u * at.k) = (uint16_t)(v >> 16);
    }
}

// Plain bf16 rows, or bf16(silu(g) * u) where x is NULL (CTA 0 then stores t as well).
__device__ __noinline__ void stage_plain(const XRows& r, const uint16_t* x, const uint16_t* g, const uint16_t* u, uint16_t* t_out, int ctid)
{
    const bool pub = !x && t_out && blockIdx.x == 0;
    if ((r.K & 7) == 0 && ((((uintptr_t)x) | ((uintptr_t)g) | ((uintptr_t)u) | ((uintptr_t)t_out)) & 15) == 0) {
        PanelWalk at((uint32_t)r.K >> 3, (uint32_t)ctid);
        while (at.n < (uint32_t)r.N) {
            uint4 v[kStageBatch];
            PanelWalk ahead = at;
#pragma unroll
            for (int b = 0; b < kStageBatch; ++b, ahead.next()) {
                if (ahead.n >= (uint32_t)r.N) break;
                const size_t i = (size_t)ahead.n * at.kq + ahead.k;
                if (x) {
                    v[b] = __ldcg((const uint4*)x + i);
                } else {
                    const uint4 gv = __ldcg((const uint4*)g + i), uv = __ldcg((const uint4*)u + i);
                    v[b] = make_uint4(silu_mul_pair(gv.x, uv.x), silu_mul_pair(gv.y, uv.y), silu_mul_pair(gv.z, uv.z), silu_mul_pair(gv.w, uv.w));
                    if (pub) ((uint4*)t_out)[i] = v[b];
                }
            }
#pragma unroll
            for (int b = 0; b < kStageBatch; ++b, at.next()) {
                if (at.n >= (uint32_t)r.N) break;
                *(uint4*)(r.buf + at.n * (uint32_t)r.pitch + 16u * at.k) = v[b];
            }
        }
        return;
    }
    PanelWalk at((uint32_t)r.K, (uint32_t)ctid);
    while (at.n < (uint32_t)r.N) {
        uint16_t v[2 * kStageBatch];
        PanelWalk ahead = at;
#pragma unroll
        for (int b = 0; b < 2 * kStageBatch; ++b, ahead.next()) {
            if (ahead.n >= (uint32_t)r.N) break;
            const size_t i = (size_t)ahead.n * r.K + ahead.k;
            v[b] = x ? __ldcg(x + i) : silu_mul_bits(__ldcg(g + i), __ldcg(u + i));
            if (pub) t_out[i] = v[b];
        }
#pragma unroll
        for (int b = 0; b < 2 * kStageBatch; ++b, at.next()) {
            if (at.n >= (uint32_t)r.N) break;
            *(uint16_t*)(r.buf + at.n * (uint32_t)r.pitch + 2u * at.k) = v[b];
        }
    }
}

// rows[n] = rmsnorm(rows[n] [+ res]) * norm_w on the staged rows, two at a time
__device__ __noinline__ void fold_norm(const XRows& r, const SFold& f, int row0, float (*red)[kCellWarps], int ctid)
{
    const bool pub = blockIdx.x == 0;
    for (int n0 = 0; n0 < r.N; n0 += 2) {
        consumer_sync();     // the rows are staged; red is free
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int n = n0 + q;
            if (n >= r.N) continue;
            uint16_t* xl = (uint16_t*)(r.buf + (size_t)n * r.pitch);
            const size_t go = (size_t)(row0 + n) * r.K;
            float ss = 0.f;
            for (int i = ctid; i < r.K; i += kCellConsumers) {
                float v = bf16_to_f32(xl[i]);
                if (f.res) {
                    const uint16_t sb = f32_to_bf16_rne(v + bf16_to_f32(__ldcg(f.res + go + i)));
                    xl[i] = sb;
                    if (pub && f.sum_out) f.sum_out[go + i] = sb;
                    v = bf16_to_f32(sb);
                }
                ss += v * v;
            }
            __syncwarp();
            ss = warp_sum(ss);
            if ((ctid & 31) == 0) red[q][ctid >> 5] = ss;
        }
        consumer_sync();
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int n = n0 + q;
            if (n >= r.N) continue;
            uint16_t* xl = (uint16_t*)(r.buf + (size_t)n * r.pitch);
            const size_t go = (size_t)(row0 + n) * r.K;
            float tot = 0.f;
#pragma unroll
            for (int w = 0; w < kCellWarps; ++w) tot += red[q][w];
            const float rs = rsqrtf(tot / (float)r.K + f.eps);
            for (int i = ctid; i < r.K; i += kCellConsumers) {
                const uint16_t o = f32_to_bf16_rne(bf16_to_f32(xl[i]) * rs * bf16_to_f32(__ldg(f.norm_w + i)));
                xl[i] = o;
                if (pub && f.norm_out) f.norm_out[go + i] = o;
            }
        }
    }
}

// ---- finishing a tile ---------------------------------------------------------------------

struct TileOut {
    int n0, N, tagged;
    uint32_t tag;            // stage part
    void* y_out;             // replaces mat[0].y (last stage), or NULL
};

// Stores rows 2 t and 2 t + 1 (values r) of tile v of a stage for panel row n.
__device__ __forceinline__ void store_tile(const CStage& st, int v, int n, int t2, const float (&r)[2], const TileOut& o, const unsigned int* tagb)
{
    int mi = 0;
    for (int m = 0; m + 1 < st.count; ++m)
        if (mi == m && v >= st.mat[m].T) { v -= st.mat[m].T; mi = m + 1; }
    const CMat& md = st.mat[mi];
    void* yp = (o.y_out && mi == 0) ? o.y_out : md.y;
    uint32_t* yt = o.tagged ? md.yt : nullptr;
    const size_t M = (size_t)md.M;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const size_t row = (size_t)v * kTileRows + t2 + j;
        if (row >= M) break;
        const size_t at = (size_t)(o.n0 + n) * M + row;
        if (yt) {
            const uint32_t bits = f32_to_bf16_rne(r[j]);
            st_relaxed_u32(yt + at, (bits << 16) | o.tag | tagb[n]);
            if (yp) ((uint16_t*)yp)[at] = (uint16_t)bits;
        } else if (md.y_f32) {
            ((float*)yp)[at] = r[j];
        } else {
            ((uint16_t*)yp)[at] = f32_to_bf16_rne(r[j]);
        }
    }
}

// The same for a gate|up stage: g, u as plain bf16 (where asked for), t = silu(g) * u plain and tagged.
__device__ __forceinline__ void store_pair(const CStage& st, int v, int n, int t2, const uint16_t* g, const float (&r)[2], const TileOut& o,
                                           const unsigned int* tagb)
{
    const size_t M = (size_t)st.mat[0].M;
    uint16_t *gp = (uint16_t*)st.mat[0].y, *up = (uint16_t*)st.mat[1].y, *tp = st.t_out;
    uint32_t* tt = o.tagged ? st.tt : nullptr;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const size_t row = (size_t)v * kTileRows + t2 + j;
        if (row >= M) break;
        const size_t at = (size_t)(o.n0 + n) * M + row;
        const uint16_t gb = g[j], ub = f32_to_bf16_rne(r[j]), tv = silu_mul_bits(gb, ub);
        if (tt) st_relaxed_u32(tt + at, ((uint32_t)tv << 16) | o.tag | tagb[n]);
        if (tp) tp[at] = tv;
        if (gp) gp[at] = gb;
        if (up) up[at] = ub;
    }
}

// The warp that brought a tile's last contribution: adds the C contributions up (four running sums, then one tree: an
// order that depends neither on N nor on the CTA), and stores.  tl: number of the tile (gate and up apart) in the CTA's
// share of the stage, ord: in the CTA's share of the program.
template <int NR>
__device__ __noinline__ bool finish_tile(CellShared* sh, const CStage& st, const unsigned char* part, int C, int tl, unsigned int ord,
                                         int first, int G, const TileOut& o, const WaitCtx& wc, int lane)
{
    const int t2 = (lane & 3) * 2;
    const uint32_t part_row = (uint32_t)o.N * 32u;               // bytes of one contribution: N x 8 fp32
    float r[NR / 8][2];
#pragma unroll
    for (int q = 0; q < NR / 8; ++q) {
        const int n = (lane >> 2) + 8 * q;
        const unsigned char* p = part + (n < o.N ? n : 0) * 32 + t2 * 4;
        float2 acc[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] = make_float2(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < kCellWarps; ++c)
            if (c < C) {
                const float2 v = *(const float2*)(p + (uint32_t)c * part_row);
                acc[c & 3].x += v.x;
                acc[c & 3].y += v.y;
            }
        r[q][0] = (acc[0].x + acc[1].x) + (acc[2].x + acc[3].x);
        r[q][1] = (acc[0].y + acc[1].y) + (acc[2].y + acc[3].y);
    }
    if (!st.pair) {
#pragma unroll
        for (int q = 0; q < NR / 8; ++q) {
            const int n = (lane >> 2) + 8 * q;
            if (n < o.N) store_tile(st, first + tl * G, n, t2, r[q], o, sh->tag_base);
        }
        return true;
    }
    const unsigned int pair = (ord - (unsigned int)(tl & 1)) >> 1;   // gate tiles are the even ones of the stage, each followed by its up tile
    const unsigned int gs = pair % kPairSlots;
    if (!(tl & 1)) {
        // the gate slot's previous pair must have been finished (one of an earlier stage has been)
        if (tl >= 2 * kPairSlots && !wait_count(&sh->finished[(ord + 1u) % kPartSlots], ord + 2u - 2u * kPairSlots, wc)) return false;
#pragma unroll
        for (int q = 0; q < NR / 8; ++q) {
            const int n = (lane >> 2) + 8 * q;
            if (n < o.N) *(uint32_t*)&sh->gate[gs][n][t2] = (uint32_t)f32_to_bf16_rne(r[q][0]) | ((uint32_t)f32_to_bf16_rne(r[q][1]) << 16);
        }
        __threadfence_block();
        __syncwarp();
        if (lane == 0) *(volatile unsigned int*)&sh->gate_done[gs] = pair + 1u;
        return true;
    }
    if (!wait_count(&sh->gate_done[gs], pair + 1u, wc)) return false;
#pragma unroll
    for (int q = 0; q < NR / 8; ++q) {
        const int n = (lane >> 2) + 8 * q;
        if (n < o.N) store_pair(st, first + (tl >> 1) * G, n, t2, &sh->gate[gs][n][t2], r[q], o, sh->tag_base);
    }
    return true;
}

// ---- the kernel ---------------------------------------------------------------------------

template <int MAXS, int NR, bool FOLD>
__global__ void __launch_bounds__(kCellThreads, 1) cell_kernel(const __grid_constant__ CArgs<MAXS> a)
{
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr uint32_t kPartOff = (uint32_t)((sizeof(CellShared) + 127) & ~127);
    CellShared* sh = (CellShared*)smem;
    const uint32_t xoff0 = kPartOff + (uint32_t)(kPartSlots * a.part_bytes);
    const uint32_t ring_off = xoff0 + (uint32_t)a.xbuf_bytes[0] + (uint32_t)a.xbuf_bytes[1];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cta = blockIdx.x, G = gridDim.x;
    const int N = a.N;
    const uint32_t NS = (uint32_t)a.n_slots;

    if (tid < kCellWarps * kCellSlots) {
        mbar_init(smem_u32(&sh->full[0][0]) + 8 * tid, 1);
        mbar_init(smem_u32(&sh->empty[0][0]) + 8 * tid, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    } else if (tid < kCellWarps * kCellSlots + kPairSlots) {
        const int i = tid - kCellWarps * kCellSlots;
        sh->gate_done[i] = 0u;
        if (i < kPartSlots) sh->arrived[i] = sh->finished[i] = 0u;
        if (i == 0) {
            sh->abort_flag = 0;
            sh->stage_dead[0] = sh->stage_dead[1] = 0;
            sh->stage_tiles = 0u;
        }
    } else if (tid >= 160 && tid < 160 + kPanelRows) {
        const int n = tid - 160;
        sh->tag_base[n] = (a.tagged && n < N) ? ((*(volatile unsigned int*)(a.rowseq + a.n0 + n)) & 0xFFu) << 8 : 0u;
    }
    __syncthreads();

    WaitCtx wc;
    wc.abort_flag = &sh->abort_flag;
    wc.budget = a.wait_cycles;

    if (warp == kCellWarps) {
        // ---------------------------------------------------------------------- producer
        // Rounds of up to 15 cells, one per lane, through all stages.  A round's directory entries are loaded four rounds
        // ahead and a stage's fields one stage ahead, so the latencies stay off the ring's critical path.
        struct PStage {
            int count, D, nsub, first, n_cells;
            int T[kMaxFused - 1];
            const uint32_t* off[kMaxFused];
            const unsigned char* cells[kMaxFused];
        };
        struct PCell {
            uint32_t bytes;
            const unsigned char* src;
        };
        auto stage_of = [&](const CStage& st) {
            PStage p;
            p.count = st.count;
            p.D = st.D;
            p.nsub = st.pair ? 2 : 1;
            p.first = cta - st.rot + (cta < st.rot ? G : 0);
            p.n_cells = (st.tiles_div + (p.first < st.tiles_rem ? 1 : 0)) * p.nsub * p.D;
#pragma unroll
            for (int m = 0; m < kMaxFused; ++m) {
                if (m + 1 < kMaxFused) p.T[m] = st.mat[m].T;
                p.off[m] = st.mat[m].off;
                p.cells[m] = st.mat[m].cells;
            }
            return p;
        };
        auto load_stage = [&](int s) { return a.ext ? stage_of(a.ext[s]) : stage_of(a.inl[MAXS == 1 ? 0 : s]); };
        // position of the look-ahead: stage sa (fields in `cur`), first cell of the next round ia, warp that gets cell 0 fb
        int sa = 0, ia = 0, fb = 0;
        PStage cur = load_stage(0);
        PStage nxt = a.n_stages > 1 ? load_stage(1) : cur;
        auto load_round = [&]() {
            PCell c;
            c.bytes = 0u;
            c.src = nullptr;
            while (sa < a.n_stages && ia >= cur.n_cells) {       // on to the next stage that has cells for this CTA
                fb = (fb + cur.n_cells) % kCellWarps;
                ++sa;
                ia = 0;
                cur = nxt;
                if (sa + 1 < a.n_stages) nxt = load_stage(sa + 1);
            }
            if (sa >= a.n_stages) return c;
            const int r = lane - fb;
            const int i = ia + (r < 0 ? r + kCellWarps : r);
            if (lane < kCellWarps && i < cur.n_cells) {
                const int tl = i / cur.D, d = i - tl * cur.D;
                int mi = 0, v;
                if (cur.nsub == 2) {
                    mi = tl & 1;
                    v = cur.first + (tl >> 1) * G;
                } else {
                    v = cur.first + tl * G;
#pragma unroll
                    for (int m = 0; m + 1 < kMaxFused; ++m)
                        if (mi == m && m + 1 < cur.count && v >= cur.T[m]) { v -= cur.T[m]; mi = m + 1; }
                }
                const uint32_t* off = cur.off[0];
                const unsigned char* ce = cur.cells[0];
#pragma unroll
                for (int m = 1; m < kMaxFused; ++m)
                    if (mi == m) { off = cur.off[m]; ce = cur.cells[m]; }
                const uint32_t o0 = __ldg(off + (size_t)v * cur.D + d), o1 = __ldg(off + (size_t)v * cur.D + d + 1);
                c.bytes = (o1 - o0) * 32u;
                c.src = ce + (size_t)o0 * 32;
            }
            ia += kCellWarps;
            return c;
        };
        // weights are read once: with several stages their lines leave L2 first, so that the stream does not push out
        // the small, shared, re-read hand-off words
        const uint64_t policy = l2_evict_first();
        const bool hinted = a.n_stages > 1;
        const uint32_t bar = 8u * (uint32_t)kCellSlots * (uint32_t)lane;
        const uint32_t full0 = smem_u32(&sh->full[0][0]) + bar, empty0 = smem_u32(&sh->empty[0][0]) + bar;
        const uint32_t ring = smem_u32(smem) + ring_off + (uint32_t)lane * NS * (uint32_t)a.slot_bytes;
        uint32_t slot = 0, phase = 1, issued = 0;                // of this lane's warp
        bool ok = true;
        PCell c0 = load_round(), c1 = load_round(), c2 = load_round(), c3 = load_round();
        while (__any_sync(0xFFFFFFFFu, (c0.bytes | c1.bytes | c2.bytes | c3.bytes) != 0u)) {
            bool good = true;
            if (c0.bytes) good = wait_phase(empty0 + 8 * slot, phase, wc);
            if (!__all_sync(0xFFFFFFFFu, good)) { ok = false; break; }
            if (c0.bytes) {
                sh->rows[lane][slot] = (int)(c0.bytes - kCellHeaderBytes) >> 7;
                mbar_expect_tx(full0 + 8 * slot, c0.bytes);
                const uint32_t dst = ring + slot * (uint32_t)a.slot_bytes;
                if (hinted) bulk_g2s(dst, c0.src, c0.bytes, full0 + 8 * slot, policy);
                else bulk_g2s(dst, c0.src, c0.bytes, full0 + 8 * slot);
                ++issued;
                if (++slot == NS) { slot = 0; phase ^= 1u; }
            }
            __syncwarp();
            c0 = c1;
            c1 = c2;
            c2 = c3;
            c3 = load_round();
        }
        if (!ok && lane < kCellWarps) {
            // give the copies already issued time to land before this CTA's memory is released
            for (uint32_t t = issued > NS ? issued - NS : 0u; t != issued; ++t) {
                const long long t0 = clock64();
                while (!mbar_try_wait(full0 + 8 * (t % NS), (t / NS) & 1u))
                    if (clock64() - t0 > wc.budget) break;
            }
        }
    } else {
        // ---------------------------------------------------------------------- consumers
        const int ctid = tid;
        struct CUse {
            const uint16_t* x;
            int K, D, nsub, first, n_tiles, tagged_in;
        };
        auto use_of = [&](const CStage& st) {
            CUse c;
            c.x = st.x;
            c.K = st.K;
            c.D = st.D;
            c.nsub = st.pair ? 2 : 1;
            c.first = cta - st.rot + (cta < st.rot ? G : 0);
            c.n_tiles = (st.tiles_div + (c.first < st.tiles_rem ? 1 : 0)) * c.nsub;
            c.tagged_in = st.tagged_in;
            return c;
        };
        auto load_use = [&](int s) { return a.ext ? use_of(a.ext[s]) : use_of(a.inl[MAXS == 1 ? 0 : s]); };
        auto fetch_stage = [&](int s) {                          // one warp: the descriptor for those who finish tiles
            uint32_t* dst = (uint32_t*)&sh->stage[s & 1];
            for (int i = lane; i < (int)(sizeof(CStage) / 4); i += 32)
                dst[i] = a.ext ? ((const uint32_t*)(a.ext + s))[i] : ((const uint32_t*)&a.inl[s])[i];
        };
        const uint32_t full0 = smem_u32(&sh->full[warp][0]), empty0 = smem_u32(&sh->empty[warp][0]);
        const uint32_t ring = ring_off + (uint32_t)warp * NS * (uint32_t)a.slot_bytes;
        const int g = lane >> 2;
        const int xrow = g < N ? g : 0, xrow8 = g + 8 < N ? g + 8 : 0;   // rows beyond N repeat row 0; their sums are never read
        uint32_t slot = 0, phase = 0;
        unsigned int ord0 = 0;                                   // tiles of the CTA before this stage
        int fb = 0;                                              // the warp that gets the stage's first cell
        bool failed = false;
        CUse use = load_use(0);
        if (MAXS > 1 && warp == kCellWarps - 1) fetch_stage(0);  // visible behind the first staging barrier
        for (int s = 0; s < a.n_stages; ++s) {
            const int K = use.K, D = use.D;
            const uint32_t xoff = xoff0 + ((s & 1) && a.xbuf_bytes[1] ? (uint32_t)a.xbuf_bytes[0] : 0u);
            const int Kp = D * kCellCols;
            XRows xr;
            xr.buf = smem + xoff;
            xr.K = K;
            xr.pitch = 2 * Kp + 64;                              // a multiple of 64 that is not one of 128: rows of one
            xr.N = N;                                            // 128-bit read fall into different banks
            const bool first_x = s == 0 && a.x_in;
            const uint16_t* x = first_x ? a.x_in : use.x;
            if (s > 0 && (!a.xbuf_bytes[1] || !a.tagged)) {
                // one buffer: everybody has left the previous stage's rows.  Grid barrier: every CTA has written the
                // previous stage's outputs; one that has no tiles now arrives for this stage at once.
                if (!a.tagged && ctid == 0) {
                    grid_wait(a.gbar, (unsigned int)s * (unsigned int)G, wc);
                    if (use.n_tiles == 0 && s + 1 < a.n_stages) atomicAdd(a.gbar, 1u);
                }
                consumer_sync();
            } else if (s == 0 && !a.tagged && a.n_stages > 1 && use.n_tiles == 0 && ctid == 0) {
                atomicAdd(a.gbar, 1u);
            }
            const size_t go = (size_t)a.n0 * K;
            if (a.tagged && use.tagged_in && !first_x) {
                stage_tagged(xr, (const uint32_t*)x + go, (uint32_t)s, sh->tag_base, wc, ctid);
            } else if (x) {
                stage_plain(xr, x + go, nullptr, nullptr, nullptr, ctid);
            } else {
                const CStage& st = a.inl[MAXS == 1 ? 0 : s];     // (glue mode: inline programs only)
                stage_plain(xr, nullptr, st.g + go, st.u + go, st.t_out ? st.t_out + go : nullptr, ctid);
            }
            for (int n = 0; n < N; ++n)
                for (int i = K + ctid; i < Kp; i += kCellConsumers) *(uint16_t*)(xr.buf + (size_t)n * xr.pitch + 2 * i) = 0;
            if constexpr (FOLD) {
                if (a.fold[MAXS == 1 ? 0 : s].norm_w) fold_norm(xr, a.fold[MAXS == 1 ? 0 : s], a.n0, sh->red, ctid);
            }
            if (ctid == 0) sh->stage_dead[s & 1] = sh->abort_flag;
            consumer_sync();
            if (sh->stage_dead[s & 1]) break;
            const int n_tiles = use.n_tiles, first = use.first, n_cells = n_tiles * D;
            if (s + 1 < a.n_stages) {
                use = load_use(s + 1);
                if (warp == kCellWarps - 1) fetch_stage(s + 1);
            }
            const CStage& st = MAXS == 1 ? a.inl[0] : sh->stage[s & 1];
            TileOut to;
            to.n0 = a.n0;
            to.N = N;
            to.tagged = a.tagged;
            to.tag = (uint32_t)(s + 1);
            to.y_out = s == a.n_stages - 1 ? a.y_out : nullptr;

            const int C = D < kCellWarps ? D : kCellWarps;
            const uint32_t xl = xoff + (uint32_t)(xrow * xr.pitch) + 16u * (lane & 3), xl8 = xoff + (uint32_t)(xrow8 * xr.pitch) + 16u * (lane & 3);
            int i = warp - fb;
            if (i < 0) i += kCellWarps;
            int tl = i / D, d = i - tl * D, c0 = d;
            float af[4] = {0.f, 0.f, 0.f, 0.f}, ab[4] = {0.f, 0.f, 0.f, 0.f};
            while (i < n_cells && !failed) {   // (after a failure the barriers ahead are attended; thread 0 reads abort_flag there)
                if (!wait_phase_warp(full0 + 8 * slot, phase, wc)) { failed = true; break; }
                const uint32_t cell = ring + slot * (uint32_t)a.slot_bytes;
                {
                    const uint32_t H = (uint32_t)sh->rows[warp][slot];
                    const uint32_t ma = *(const uint32_t*)(smem + cell + 4 * lane), mb = *(const uint32_t*)(smem + cell + 128 + 4 * lane);
                    const uint32_t pi = *(smem + cell + 256 + lane);
                    const uint32_t xd = (uint32_t)d * (2 * kCellCols), v0 = cell + kCellHeaderBytes;
                    half_cell<NR, 1>(smem, ma, v0 + 4u * lane, xl + xd, xl8 + xd, af, ab);
                    if (d * kCellCols + kHalfCols < K)
                        half_cell<NR, -1>(smem, mb, v0 + (H - 1u) * 128u + pi, xl + xd + 2 * kHalfCols, xl8 + xd + 2 * kHalfCols, af, ab);
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(empty0 + 8 * slot);
                if (++slot == NS) { slot = 0; phase ^= 1u; }
                i += kCellWarps;
                d += kCellWarps;
                if (d < D) continue;                             // the next cell belongs to the same tile
                // the tile's sums go to shared memory; who completes them finishes the tile
                const unsigned int ord = ord0 + (unsigned int)tl;
                const uint32_t ps = ord % kPartSlots;
                if (ord >= kPartSlots && !wait_count(&sh->finished[ps], ord + 1u - kPartSlots, wc)) { failed = true; break; }
                unsigned char* part = smem + kPartOff + ps * (uint32_t)a.part_bytes;
                {
                    unsigned char* p = part + (uint32_t)(c0 * N + g) * 32u + (lane & 3) * 8;
                    if (g < N) *(float2*)p = make_float2(af[0] + ab[0], af[1] + ab[1]);
                    if (NR > 8 && g + 8 < N) *(float2*)(p + 256) = make_float2(af[2] + ab[2], af[3] + ab[3]);
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) af[k] = ab[k] = 0.f;
                __threadfence_block();
                __syncwarp();
                unsigned int before = 0;
                if (lane == 0) before = atomicAdd(&sh->arrived[ps], 1u);
                before = __shfl_sync(0xFFFFFFFFu, before, 0);
                if (before == (unsigned int)C - 1u) {
                    __threadfence_block();
                    if (!finish_tile<NR>(sh, st, part, C, tl, ord, first, G, to, wc, lane)) { failed = true; break; }
                    const bool barrier = !a.tagged && s + 1 < a.n_stages;
                    if (barrier) __threadfence();                // the tile's outputs are visible before the grid barrier counts them
                    __syncwarp();
                    if (lane == 0) {
                        sh->arrived[ps] = 0u;
                        __threadfence_block();
                        *(volatile unsigned int*)&sh->finished[ps] = ord + 1u;
                        if (barrier && atomicAdd(&sh->stage_tiles, 1u) + 1u == (unsigned int)n_tiles) {
                            sh->stage_tiles = 0u;                // nobody of this CTA is past the barrier yet
                            __threadfence();
                            atomicAdd(a.gbar, 1u);
                        }
                    }
                    __syncwarp();
                }
                do { d -= D; ++tl; } while (d >= D);
                c0 = d;
            }
            ord0 += (unsigned int)n_tiles;
            fb = (fb + n_cells) % kCellWarps;
        }
    }

    // ---- exit: every role comes here
    __syncwarp();
    __syncthreads();
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
            if (a.tagged)   // the launch's activation rows have been produced once more: their next tags differ
                for (int n = 0; n < N; ++n) atomicAdd(a.rowseq + a.n0 + n, 1u);
        }
    }
}

}  // namespace sd2
