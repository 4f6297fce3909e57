// C ABI of libsd2 (see include/sd2.h): handle management, host format builder entry
// points, kernel dispatch.  No torch types, no exceptions across the boundary.

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <mutex>
#include <new>
#include <unordered_set>
#include <vector>

#include "../../include/sd2.h"
#include "sd2_format.hpp"
#include "sd2_format_mma.hpp"
#include "sd2_kernels.cuh"
#include "sd2_cell_kernel.cuh"
#include "sd2_cells_pack.cuh"
#include "sd2_mma_kernel.cuh"
#include "sd2_glue.cuh"

using namespace sd2;

struct sd2_handle_s {
    int64_t M, K, nnz, compressed_bytes, blob_bytes;
    int format, y_dtype, device;
    uint8_t* d_blob;
    const uint32_t* d_sec0;
    const uint32_t* d_sec1;
    const void* d_sec2;
    // GAP4 geometry
    int S, B, T, max_tile_bytes, V;
    int paired;   // GAP4: rows 2i, 2i+1 share a tile (header field `pairing`)
    // GAP4: the same weights as cells (sd2_cells.hpp), for panels of rows (d_image NULL: none); GAP4_MMA: the weights as panel
    // cells (and nothing else: d_blob has room for their heights)
    uint8_t* d_image;
    const unsigned char* d_cells;
    int64_t cell_bytes;        // what a launch reads of them
    int64_t device_bytes;      // all that the handle owns
    int cell_T, cell_D, max_chunk;
};

// What a program over cells needs from shared memory.
int cell_pitch(int D) { return 2 * share_cells(D, 0) * kCellCols + 64; }

struct CellNeeds {
    int pitch = 0;             // bytes of a staged activation row: the largest
    int max_chunk = 0;
    int tiles_max = 0;         // most tiles of any stage
    bool split = false;        // a stage's tiles are split over the groups
    void add(sd2_handle h)
    {
        const int p = cell_pitch(h->cell_D);
        if (p > pitch) pitch = p;
        if (h->max_chunk > max_chunk) max_chunk = h->max_chunk;
        if (share_cells(h->cell_D, 0) > kSplitCells) split = true;
    }
};

struct sd2_drafter_s {
    int L, device;
    int64_t n_max;
    int n_stages;
    int y_f32;                 // dtype of the last block's output
    int64_t hidden, out_dim;
    std::vector<sd2_handle> handles;
    std::vector<sd2_handle> owned;      // paired gate|up stacks the drafter built for itself
    std::vector<int> pair_block;        // the block each of them belongs to
    std::vector<int64_t> ws_off;        // per block: offsets of q,k,v,hdn,g,u,t and the block output inside d_ws
    int64_t x_off;             // a copy of the step's input inside d_ws, or -1 (see sd2_drafter_create)
    uint8_t* d_ws;
    SStage* d_stages;
    unsigned int* d_gbar;
    uint32_t* d_tags;          // tagged copies of q, hdn, g, u and the block output of every block (or NULL)
    int64_t tags_bytes;
    int K_max, max_tile;       // what decides the shared-memory split
    int free_tiles;            // every stage has enough tiles per CTA for free tile assignment
    int xs_need[3];            // bytes of staged activations at panel widths 1, 2, 4
    // the same blocks as a program over cells, with barrier words of its own; NULL: a handle has no cells
    CStage* d_cstages;
    CStage first_cstage;       // the first stages of both programs go along with a launch
    SStage first_stage;
    unsigned int* d_cbar;
    int n_cstages;
    CellNeeds cell_needs;
};

namespace {

// cudaMalloc behind the same failure plan as the host allocations (see lib_alloc_fails)
cudaError_t dev_malloc(void** p, size_t n)
{
    if (lib_alloc_fails()) { *p = nullptr; return cudaErrorMemoryAllocation; }
    return cudaMalloc(p, n);
}
template <class T>
cudaError_t dev_malloc(T** p, size_t n) { return dev_malloc((void**)p, n); }

// NVTX range over a call (a profiler's timeline then shows the library's calls by name; without a profiler
// attached the push and pop are a pointer test each)
struct Range {
    explicit Range(const char* name) { nvtxRangePushA(name); }
    ~Range() { nvtxRangePop(); }
};

std::mutex g_mu;
std::unordered_set<sd2_handle> g_live;
std::unordered_set<sd2_drafter> g_live_drafters;

// A launch that may start while the kernel before it in the stream ends (see pdl_wait).
cudaLaunchAttribute pdl_attribute()
{
    cudaLaunchAttribute a;
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    return a;
}
template <class... P, class... A>
cudaError_t launch_pdl(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr = pdl_attribute();
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

constexpr int kMaxDevices = 64;
constexpr int kBarrierPool = 64;             // grid-barrier word pairs handed out round-robin
constexpr int kBarrierStrideWords = 64;      // 256 bytes apart
constexpr int kSmemMax = 227 * 1024;         // dynamic shared memory a CTA may opt in to
constexpr int kMaxBlockRows = 1 << 16;       // activation rows a block step accepts (taken in panels)
constexpr int kDrafterWordsBytes = 512;      // a drafter's device words: barrier (two lines), then 64 production counts

struct DeviceState {
    bool ready;
    int sms;
    int clock_khz;
    int* err_word;
    unsigned int* barriers;
    int mma_clusters[kMmaMaxCluster + 1];    // how many clusters of so many CTAs of mma_kernel run at once
};
DeviceState g_dev[kMaxDevices];
std::atomic<unsigned> g_next_barrier{0};

bool live(sd2_handle h)
{
    if (!h) return false;
    std::lock_guard<std::mutex> lk(g_mu);
    return g_live.count(h) != 0;
}

bool live(sd2_drafter d)
{
    if (!d) return false;
    std::lock_guard<std::mutex> lk(g_mu);
    return g_live_drafters.count(d) != 0;
}

sd2_status from_pack(int s)
{
    switch (s) {
        case 0: return SD2_OK;
        case -2: return SD2_ERR_SHAPE;
        case -3: return SD2_ERR_ALLOC;
        case -5: return SD2_ERR_UNSUPPORTED;
        case -6: return SD2_ERR_CORRUPT;
        default: return SD2_ERR_INVALID_ARG;
    }
}

constexpr int kFoldStaticBytes = 256;   // static shared memory of the kernel instances that fold a norm into staging

template <int MAXS, int NT>
cudaError_t set_smem_attr()
{
    cudaError_t e = cudaFuncSetAttribute(stream_kernel<MAXS, NT, kNoFold>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(stream_kernel<MAXS, NT, kFoldShared>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax - kFoldStaticBytes);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(stream_kernel<MAXS, NT, kFoldHeld>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax - kFoldStaticBytes);
}

template <int MAXS, int NR>
cudaError_t set_cell_attr()
{
    cudaError_t e = cudaFuncSetAttribute(cell_kernel<MAXS, NR, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(cell_kernel<MAXS, NR, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
}

sd2_status count_mma_clusters(int* room);

// Once per device: SM count, shared-memory opt-in, the error word and the barrier pool.
sd2_status ensure_device(int* dev_out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return SD2_ERR_CUDA; }
    if (dev < 0 || dev >= kMaxDevices) return SD2_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lk(g_mu);
    DeviceState& ds = g_dev[dev];
    if (!ds.ready) {
        int sms = 0, khz = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, dev) != cudaSuccess) { cudaGetLastError(); return SD2_ERR_CUDA; }
        constexpr int kMany = kMaxStagesInline;
        if (set_smem_attr<1, 1>() != cudaSuccess || set_smem_attr<1, 2>() != cudaSuccess || set_smem_attr<1, 4>() != cudaSuccess ||
            set_smem_attr<kMany, 1>() != cudaSuccess || set_smem_attr<kMany, 2>() != cudaSuccess || set_smem_attr<kMany, 4>() != cudaSuccess ||
            set_cell_attr<1, 8>() != cudaSuccess || set_cell_attr<1, 16>() != cudaSuccess ||
            set_cell_attr<kMany, 8>() != cudaSuccess || set_cell_attr<kMany, 16>() != cudaSuccess ||
            cudaFuncSetAttribute(cell_kernel<1, kWidePanelRows, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) != cudaSuccess ||
            cudaFuncSetAttribute(mma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) != cudaSuccess ||
            cudaFuncSetAttribute(lm_head_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) != cudaSuccess ||
            cudaFuncSetAttribute(lm_head_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) != cudaSuccess ||
            cudaFuncSetAttribute(lm_head_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) != cudaSuccess ||
            cudaFuncSetAttribute(lm_head_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax) != cudaSuccess) {
            cudaGetLastError();
            return SD2_ERR_CUDA;
        }
        const sd2_status counted = count_mma_clusters(ds.mma_clusters);
        if (counted != SD2_OK) return counted;
        int* err = nullptr;
        unsigned int* bars = nullptr;
        const size_t bar_bytes = (size_t)kBarrierPool * kBarrierStrideWords * 4;
        if (dev_malloc((void**)&err, 256) != cudaSuccess) { cudaGetLastError(); return SD2_ERR_ALLOC; }
        if (dev_malloc((void**)&bars, bar_bytes) != cudaSuccess) { cudaGetLastError(); cudaFree(err); return SD2_ERR_ALLOC; }
        if (cudaMemset(err, 0, 256) != cudaSuccess || cudaMemset(bars, 0, bar_bytes) != cudaSuccess) {
            cudaGetLastError();
            cudaFree(err);
            cudaFree(bars);
            return SD2_ERR_CUDA;
        }
        ds.err_word = err;
        ds.barriers = bars;
        ds.sms = sms;
        ds.clock_khz = khz > 0 ? khz : 2000000;
        ds.ready = true;
    }
    *dev_out = dev;
    return SD2_OK;
}

// The SM count alone, for calls that need nothing else of a device: they allocate nothing, so that the first call of a program may
// be one that is captured.
sd2_status device_sms(int* sms)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return SD2_ERR_CUDA;
    }
    return SD2_OK;
}

int resolve_format(const sd2_options* opt, int64_t M, int64_t K)
{
    int f = opt ? opt->format : SD2_FORMAT_AUTO;
    if (f == SD2_FORMAT_AUTO) f = gap4_geometry(M, K).S > 0 ? SD2_FORMAT_GAP4 : SD2_FORMAT_BITMASK;
    // SD2_FORMAT_GAP4_PAIRED stays as asked: only the packer tells it from GAP4.  SD2_FORMAT_GAP4_STRIPS is GAP4 to the packer.
    return f == SD2_FORMAT_GAP4_STRIPS ? (int)SD2_FORMAT_GAP4 : f;
}

sd2_status check_pack(int64_t M, int64_t K, const sd2_options* opt)
{
    if (M < 1 || K < 1 || M > 0x7FFFFFF0ll || K > 0x7FFFFFF0ll || M * K > (1ll << 40)) return SD2_ERR_SHAPE;
    return opt && opt->y_dtype != SD2_DTYPE_BF16 && opt->y_dtype != SD2_DTYPE_F32 ? SD2_ERR_INVALID_ARG : SD2_OK;
}

sd2_status pack_any(const uint16_t* W, const uint8_t* mask, int64_t M, int64_t K, const sd2_options* opt,
                    uint8_t** blob, int64_t* bytes)
{
    if (!W || !blob || !bytes) return SD2_ERR_INVALID_ARG;
    const sd2_status checked = check_pack(M, K, opt);
    if (checked != SD2_OK) return checked;
    const int y_dtype = opt ? opt->y_dtype : SD2_DTYPE_BF16;
    const int f = resolve_format(opt, M, K);
    PackResult r;
    try {
        if (f == SD2_FORMAT_BITMASK) r = pack_bitmask(W, mask, M, K, y_dtype);
        else if (f == SD2_FORMAT_GAP4) r = pack_gap4(W, mask, M, K, y_dtype);
        else if (f == SD2_FORMAT_GAP4_PAIRED) r = pack_gap4(W, mask, M, K, y_dtype, true);
        else if (f == SD2_FORMAT_GAP4_MMA) r = pack_gap4_mma(W, mask, M, K, y_dtype);
        else return SD2_ERR_INVALID_ARG;
    } catch (const std::bad_alloc&) {
        return SD2_ERR_ALLOC;
    }
    if (r.status != 0) return from_pack(r.status);
    *blob = r.blob;
    *bytes = r.bytes;
    return SD2_OK;
}

int unpack_any(const BlobHeader& hd, const uint8_t* blob, uint16_t* dense)
{
    if (hd.format == (uint32_t)kFormatBitmask) return unpack_bitmask(hd, blob, dense);
    if (hd.format == (uint32_t)kFormatGap4Mma) return unpack_gap4_mma(hd, blob, dense);
    return unpack_gap4(hd, blob, dense);
}

// A handle with a blob's facts, and its sections on the GPU (GAP4_MMA: without, the GPU has no use for the records and they need not
// be there).
sd2_status upload(const uint8_t* blob, int64_t bytes, const BlobHeader& hd, sd2_handle* out)
{
    int dev = 0;
    sd2_status st = ensure_device(&dev);
    if (st != SD2_OK) return st;
    sd2_handle h = lib_alloc_fails() ? nullptr : new (std::nothrow) sd2_handle_s();
    if (!h) return SD2_ERR_ALLOC;
    void* d = nullptr;
    // (with room behind a GAP4 blob for the heights of its cells while they are packed: an allocation of their own took
    // longer than the packing)
    const bool mma = hd.format == (uint32_t)kFormatGap4Mma;
    const size_t heights = hd.format == (uint32_t)kFormatGap4 ? (size_t)cell_geometry(hd.M, hd.K).cells() * 4
                         : mma ? (size_t)panel_geometry(hd.M, hd.K).cells() * 4 : 0;
    if (mma) bytes = 0;
    if (dev_malloc(&d, align256((size_t)bytes) + heights) != cudaSuccess) { cudaGetLastError(); delete h; return SD2_ERR_ALLOC; }
    if (bytes && cudaMemcpy(d, blob, (size_t)bytes, cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(d);
        delete h;
        return SD2_ERR_CUDA;
    }
    h->M = hd.M; h->K = hd.K; h->nnz = hd.nnz;
    h->compressed_bytes = hd.compressed_bytes;
    h->blob_bytes = bytes;
    h->format = (int)hd.format;
    h->y_dtype = (int)hd.y_dtype;
    h->device = dev;
    h->d_blob = (uint8_t*)d;
    h->d_sec0 = mma ? nullptr : (const uint32_t*)(h->d_blob + hd.sec_off[0]);
    h->d_sec1 = mma ? nullptr : (const uint32_t*)(h->d_blob + hd.sec_off[1]);
    h->d_sec2 = mma ? nullptr : (const void*)(h->d_blob + hd.sec_off[2]);
    h->S = (int)hd.strips;
    h->B = (int)hd.strip_cols;
    h->T = (int)hd.n_tiles;
    h->max_tile_bytes = (int)hd.max_tile_bytes;
    h->V = (int)hd.overlap;
    h->paired = (int)hd.pairing;
    h->d_image = nullptr;
    h->device_bytes = (int64_t)(align256((size_t)bytes) + heights);
    {
        std::lock_guard<std::mutex> lk(g_mu);
        g_live.insert(h);
    }
    *out = h;
    return SD2_OK;
}

MemoryPlace place_of(const void* p, int* owner)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) { cudaGetLastError(); return kPlaceHost; }
    *owner = a.device;
    return a.type == cudaMemoryTypeManaged ? kPlaceManaged : a.type == cudaMemoryTypeDevice ? kPlaceDevice : kPlaceHost;
}

bool is_device_ptr(const void* p)
{
    int owner = 0;
    return place_of(p, &owner) != kPlaceHost;
}

bool kernel_reads(const void* p, size_t size, int device)
{
    int owner = -1;
    const MemoryPlace place = place_of(p, &owner);
    return readable_in_place(place, owner, device, p, size);
}

// Where a fresh handle's dense weights come from while its cells are packed: `fetch` puts the rows row0 .. row0 + rows - 1 of the weights and
// of the mask (NULL: see pack_cells_kernel) in reach of a kernel.  It is asked for `step` rows at a time, in order, and twice for each of
// them where step is less than all rows.
struct CellSource {
    int64_t step;
    uint32_t nonzero;
    std::function<sd2_status(int64_t row0, int64_t rows, const uint16_t** W, const uint8_t** mask)> fetch;
};

// Gives a fresh handle its cells (GAP4_MMA: panel cells).
sd2_status pack_cells(sd2_handle h, const CellSource& src)
{
    const bool panel = h->format == SD2_FORMAT_GAP4_MMA;
    const CellGeom g = panel ? panel_geometry(h->M, h->K) : cell_geometry(h->M, h->K);
    const int64_t n_cells = g.cells();
    if (n_cells > 0x3FFFFFFF) return SD2_ERR_UNSUPPORTED;
    const size_t dir_bytes = align256((size_t)(n_cells + 1) * 4);
    std::vector<uint32_t> off((size_t)n_cells + 1);          // first the cells' heights, then their places
    uint32_t* d_height = (uint32_t*)(h->d_blob + align256((size_t)h->blob_bytes));
    uint8_t* image = nullptr;
    const uint16_t* W = nullptr;
    const uint8_t* mask = nullptr;
    // one pass over the weights: heights, or, once there is an image, the cells
    auto pass = [&]() {
        for (int64_t row0 = 0; row0 < h->M; row0 += src.step) {
            const int64_t rows = std::min(src.step, h->M - row0);
            if (!image || src.step < h->M) {
                const sd2_status st = src.fetch(row0, rows, &W, &mask);
                if (st != SD2_OK) return st;
            }
            const CellGeom part = panel ? panel_geometry(rows, h->K) : g;
            const int64_t first = panel ? row0 / kPanelRowsOfBlock * g.D * g.per : 0;
            const unsigned grid = (unsigned)((part.cells() + kPackWarps - 1) / kPackWarps);
            auto* const kernel = panel ? pack_cells_kernel<true> : pack_cells_kernel<false>;
            kernel<<<grid, 32 * kPackWarps>>>(W, mask, src.nonzero, rows, h->K, (int)part.T, g.D, image ? nullptr : d_height + first,
                                              image ? (const uint32_t*)image + first : nullptr, image ? image + dir_bytes : nullptr);
            if (cudaGetLastError() != cudaSuccess) return SD2_ERR_CUDA;
        }
        return SD2_OK;
    };
    sd2_status st = pass();
    if (st != SD2_OK) return st;
    if (cudaMemcpy(off.data(), d_height, (size_t)n_cells * 4, cudaMemcpyDeviceToHost) != cudaSuccess) return SD2_ERR_CUDA;
    uint64_t units = 0;
    uint32_t max_run = 0;
    for (int64_t c = 0; c < n_cells; ++c) {
        const uint32_t n = (kCellHeaderBytes + off[(size_t)c] * 128u) / 32u;
        off[(size_t)c] = (uint32_t)units;
        units += n;
        const uint32_t from = c >= kChunkCells - 1 ? off[(size_t)(c - (kChunkCells - 1))] : 0u;
        if ((uint32_t)units - from > max_run) max_run = (uint32_t)units - from;
    }
    if (units > 0xFFFFFFF0ull) return SD2_ERR_UNSUPPORTED;
    off[(size_t)n_cells] = (uint32_t)units;
    const size_t bytes = dir_bytes + (size_t)units * 32;
    if (dev_malloc(&image, bytes) != cudaSuccess) return SD2_ERR_ALLOC;
    h->d_image = image;                                       // (sd2_free has it from here on)
    h->d_cells = image + dir_bytes;
    cudaError_t e = cudaMemset(image, 0, bytes);
    if (e == cudaSuccess) e = cudaMemcpy(image, off.data(), off.size() * 4, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return SD2_ERR_CUDA;
    if ((st = pass()) != SD2_OK) return st;
    if (cudaStreamSynchronize(0) != cudaSuccess) return SD2_ERR_CUDA;       // the weights may go away now
    h->device_bytes += (int64_t)bytes;
    h->cell_bytes = (n_cells + 1) * 4 + (int64_t)units * 32;
    h->cell_T = (int)g.T;
    h->cell_D = g.D;
    h->max_chunk = (int)(max_run * 32u);
    return SD2_OK;
}

// The same from weights and a mask that lie in host memory or where the handle's GPU can read them, or from the records of a GAP4_MMA blob
// (which have been checked).  The cells of a GAP4 handle are a second image of the weights: where there is no memory for them, or for the
// dense weights that they are made from, the handle goes without, and calls of several rows read its strips.  Panel cells are all that
// a GAP4_MMA handle has: they are made kPanelScratch weights at a time, so that little memory is needed beside them.  On any other
// failure the handle is freed.
constexpr int64_t kPanelScratch = 1 << 24;
sd2_status add_cells(sd2_handle h, const uint16_t* W, const uint8_t* mask, uint32_t nonzero = 0x7FFFu, const BlobHeader* hd = nullptr,
                     const uint8_t* blob = nullptr)
{
    const bool w_here = W && kernel_reads(W, sizeof *W, h->device), m_here = !mask || kernel_reads(mask, sizeof *mask, h->device);
    CellSource src;
    src.nonzero = nonzero;
    src.step = h->M;
    if (h->format == SD2_FORMAT_GAP4_MMA && !(w_here && m_here))
        src.step = std::min(h->M, std::max<int64_t>(kPanelScratch / h->K / kPanelRowsOfBlock, 1) * kPanelRowsOfBlock);
    const size_t n = (size_t)(src.step * h->K);
    uint16_t *w_dev = nullptr, *rows_host = nullptr;
    uint8_t* m_dev = nullptr;
    sd2_status st = SD2_OK;
    if (!w_here && dev_malloc(&w_dev, n * 2) != cudaSuccess) st = SD2_ERR_ALLOC;
    if (st == SD2_OK && !m_here && dev_malloc(&m_dev, n) != cudaSuccess) st = SD2_ERR_ALLOC;
    if (st == SD2_OK && blob && !(rows_host = (uint16_t*)lib_malloc(n * 2))) st = SD2_ERR_ALLOC;
    auto fetch = [&](int64_t row0, int64_t rows, const uint16_t** w, const uint8_t** m) {
        const size_t at = (size_t)(row0 * h->K), count = (size_t)(rows * h->K);
        if (blob) unpack_mma_panels(*hd, blob, row0 / kMmaBlockRows, (row0 + rows + kMmaBlockRows - 1) / kMmaBlockRows, rows_host);
        *w = w_here ? W + at : w_dev;
        *m = m_here ? (mask ? mask + at : nullptr) : m_dev;
        if (!w_here && cudaMemcpy(w_dev, blob ? rows_host : W + at, count * 2, cudaMemcpyHostToDevice) != cudaSuccess) return SD2_ERR_CUDA;
        if (!m_here && cudaMemcpy(m_dev, mask + at, count, cudaMemcpyHostToDevice) != cudaSuccess) return SD2_ERR_CUDA;
        return SD2_OK;
    };
    try {
        src.fetch = std::ref(fetch);
        if (st == SD2_OK) st = pack_cells(h, src);
    } catch (const std::bad_alloc&) {
        st = SD2_ERR_ALLOC;
    }
    cudaFree(w_dev);
    cudaFree(m_dev);
    std::free(rows_host);
    if (st == SD2_OK) return st;
    cudaGetLastError();
    if (h->format == SD2_FORMAT_GAP4 && (st == SD2_ERR_ALLOC || st == SD2_ERR_UNSUPPORTED)) return SD2_OK;
    sd2_free(h);
    return st;
}


// ------------------------------------------------------------------ BITMASK launches

int bitmask_grid(int64_t rows_total, int sms)
{
    int64_t want = (rows_total + kWarpsPerCta - 1) / kWarpsPerCta;
    int64_t cap = (int64_t)sms * 8;
    return (int)(want < cap ? want : cap);
}

template <int NT>
sd2_status launch_bitmask_nt(const LaunchGroup& grp, int grid, cudaStream_t s)
{
    launch_pdl(bitmask_kernel<NT>, grid, kThreads, 0, s, grp);
    if (cudaGetLastError() != cudaSuccess) return SD2_ERR_CUDA;
    return SD2_OK;
}

int round_nt(int n, int cap) { int r = n <= 1 ? 1 : n <= 2 ? 2 : n <= 4 ? 4 : 8; return r > cap ? cap : r; }

// One launch per panel of at most 8 activation rows.  Exactly one of x / (g, u) is set.
sd2_status run_bitmask(const sd2_handle* hs, int count, const uint16_t* x, const uint16_t* g, const uint16_t* u,
                       uint16_t* t_out, void* const* Y, int64_t N, bool y_force_bf16, int dev, cudaStream_t s)
{
    const int64_t K = hs[0]->K;
    LaunchGroup grp;
    std::memset(&grp, 0, sizeof grp);
    grp.count = count;
    grp.K = (int)K;
    int64_t rows_total = 0, bytes_total = 0;
    for (int i = 0; i < count; ++i) { rows_total += hs[i]->M; bytes_total += hs[i]->compressed_bytes; }
    const int grid_total = bitmask_grid(rows_total, g_dev[dev].sms);
    int grid = 0;
    for (int i = 0; i < count; ++i) {
        MatDesc& md = grp.mat[i];
        md.sec0 = hs[i]->d_sec0;
        md.sec1 = hs[i]->d_sec1;
        md.sec2 = hs[i]->d_sec2;
        md.M = (int)hs[i]->M;
        md.y_f32 = (!y_force_bf16 && hs[i]->y_dtype == SD2_DTYPE_F32) ? 1 : 0;
        md.cta_begin = grid;
        int64_t share = (int64_t)((double)grid_total * (double)hs[i]->compressed_bytes / (double)bytes_total + 0.5);
        const int64_t need = (hs[i]->M + kWarpsPerCta - 1) / kWarpsPerCta;
        if (share > need) share = need;
        if (share < 1) share = 1;
        md.cta_count = (int)share;
        grid += md.cta_count;
    }
    for (int64_t n0 = 0; n0 < N; n0 += 8) {
        const int n = (int)((N - n0) < 8 ? (N - n0) : 8);
        grp.N = n;
        grp.x = x ? x + n0 * K : nullptr;
        grp.g = g ? g + n0 * K : nullptr;
        grp.u = u ? u + n0 * K : nullptr;
        grp.t_out = t_out ? t_out + n0 * K : nullptr;
        for (int i = 0; i < count; ++i) {
            const size_t esz = grp.mat[i].y_f32 ? 4 : 2;
            grp.mat[i].y = (char*)Y[i] + (size_t)n0 * (size_t)hs[i]->M * esz;
        }
        sd2_status st;
        switch (round_nt(n, 8)) {
            case 1: st = launch_bitmask_nt<1>(grp, grid, s); break;
            case 2: st = launch_bitmask_nt<2>(grp, grid, s); break;
            case 4: st = launch_bitmask_nt<4>(grp, grid, s); break;
            default: st = launch_bitmask_nt<8>(grp, grid, s); break;
        }
        if (st != SD2_OK) return st;
    }
    return SD2_OK;
}

// ------------------------------------------------------------------ GAP4 programs

// Largest panel width (4, 2, 1) whose staged activations leave room for a ring that holds
// `max_tile` bytes at least twice; 0 if even one row does not fit.
struct SmemPlan {
    int nt, xs_bytes, xlin_bytes, ring_bytes;
};

int xs_bytes_for(int S, int B, int V, int nt)
{
    const int groups = 32 / xs_words(nt);
    const int planes = S > groups ? S / groups : 1;
    return planes * ((B + 2 * V + kGap4Slack + 3) & ~3) * 128;
}

bool plan_smem(int nt, int xs_max, int K_max, int max_tile, SmemPlan* p)
{
    const int fixed = (int)((sizeof(StreamShared) + 127) & ~127);
    const int xlin = ((2 * K_max + 127) & ~127) * (nt > 2 ? 2 : 1);   // panels of 4 go two rows at a time
    const int ring = (kSmemMax - fixed - xs_max - xlin) & ~127;
    if (ring < 2 * max_tile + 256) return false;
    p->nt = nt;
    p->xs_bytes = xs_max;
    p->xlin_bytes = xlin;
    p->ring_bytes = ring;
    return true;
}

template <int MAXS, int NT>
sd2_status launch_stream_nt(const SArgsT<MAXS>& a, int grid, int smem, bool cooperative, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kStreamThreads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    if (!cooperative) attr[0] = pdl_attribute();
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    auto* const kernel = a.fold_any == kNoFold ? stream_kernel<MAXS, NT, kNoFold> : a.fold_any == kFoldHeld ? stream_kernel<MAXS, NT, kFoldHeld>
                       : stream_kernel<MAXS, NT, kFoldShared>;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, a);
    if (e != cudaSuccess) { cudaGetLastError(); return SD2_ERR_CUDA; }
    if (cudaGetLastError() != cudaSuccess) return SD2_ERR_CUDA;
    return SD2_OK;
}

template <int MAXS>
sd2_status launch_stream(int nt, const SArgsT<MAXS>& a, int grid, bool cooperative, cudaStream_t s)
{
    const int smem = a.xs_bytes + a.xlin_bytes + (int)((sizeof(StreamShared) + 127) & ~127) + a.ring_bytes;
    switch (nt) {
        case 1: return launch_stream_nt<MAXS, 1>(a, grid, smem, cooperative, s);
        case 2: return launch_stream_nt<MAXS, 2>(a, grid, smem, cooperative, s);
        default: return launch_stream_nt<MAXS, 4>(a, grid, smem, cooperative, s);
    }
}

void set_stage_grid(SStage& st, int grid)
{
    st.tiles_div = st.T_total / grid;
    st.tiles_rem = st.T_total % grid;
}

// Fills one stage from `count` GAP4 handles of equal K and S, to be run by `grid` CTAs.
void fill_stage(SStage& st, const sd2_handle* hs, int count, const uint16_t* x, const uint16_t* g, const uint16_t* u,
                uint16_t* t_out, void* const* Y, bool y_force_bf16, int grid, uint32_t* const* YT = nullptr,
                int tagged_in = 0)
{
    std::memset(&st, 0, sizeof st);
    st.count = count;
    st.K = (int)hs[0]->K;
    st.S = hs[0]->S;
    st.B = hs[0]->B;
    st.V = hs[0]->V;
    st.hdr_bytes = gap4_tile_header_bytes(32 / hs[0]->S);
    st.log2S = 0;
    while ((1 << st.log2S) < hs[0]->S) ++st.log2S;
    st.x = x;
    st.g = g;
    st.u = u;
    st.t_out = t_out;
    int T = 0;
    for (int i = 0; i < count; ++i) {
        SMat& m = st.mat[i];
        m.tile_off = hs[i]->d_sec0;
        m.stream = (const unsigned char*)hs[i]->d_sec1;
        m.y = Y[i];
        m.yt = YT ? YT[i] : nullptr;
        m.M = (int)hs[i]->M;
        m.T = hs[i]->T;
        m.y_f32 = (!y_force_bf16 && hs[i]->y_dtype == SD2_DTYPE_F32) ? 1 : 0;
        T += hs[i]->T;
    }
    st.T_total = T;
    st.tagged_in = tagged_in;
    set_stage_grid(st, grid);
}

long long wait_budget(int dev)
{
    // about two seconds of SM clock; SD2_WAIT_MS overrides (tests use a short one)
    long long ms = 2000;
    if (const char* e = std::getenv("SD2_WAIT_MS")) { long long v = std::atoll(e); if (v >= 1 && v <= 60000) ms = v; }
    return ms * (long long)g_dev[dev].clock_khz;
}

// Tracks what a program needs from shared memory.
struct ProgramNeeds {
    int K_max = 0, max_tile = 0, tiles_max = 0;
    int tiles_min = 0x7FFFFFFF;   // fewest tiles of any stage
    int xs_need[3] = {0, 0, 0};   // staged activations at panel widths 1, 2, 4: the largest over all stages
    // Free tile assignment pays where every stage gives a CTA about as many tiles as it has consumer
    // warps, or more; with fewer, the fixed deal is faster (see the consumer loop of stream_kernel).
    int free_tiles(int grid) const { return tiles_min >= 12 * grid ? 1 : 0; }
    void add(const sd2_handle* hs, int count)
    {
        int T = 0;
        for (int i = 0; i < count; ++i) {
            // elements of the linear staging row: the strips, the zero pads on both sides, read-ahead
            const int lin = hs[i]->S * hs[i]->B + 2 * hs[i]->V + 64;
            if (lin > K_max) K_max = lin;
            if (hs[i]->max_tile_bytes > max_tile) max_tile = hs[i]->max_tile_bytes;
            for (int w = 0; w < 3; ++w) {
                const int need = xs_bytes_for(hs[i]->S, hs[i]->B, hs[i]->V, 1 << w);
                if (need > xs_need[w]) xs_need[w] = need;
            }
            T += hs[i]->T;
        }
        if (T > tiles_max) tiles_max = T;
        if (T < tiles_min) tiles_min = T;
    }
};

int nt_index(int nt) { return nt == 1 ? 0 : nt == 2 ? 1 : 2; }

// Widest panel (4, 2, 1 rows; four and more take the cells) whose staged activations still leave room for the ring; 0 if none.
int widest_panel(const int xs_need[3], int K_max, int max_tile)
{
    // a wide panel whose activations crowd out the ring cannot stream: ask for a ring of at
    // least 96 KB first, and settle for whatever fits only if no width leaves that much
    SmemPlan p;
    for (int nt = 4; nt >= 1; nt >>= 1)
        if (plan_smem(nt, xs_need[nt_index(nt)], K_max, max_tile, &p) && p.ring_bytes >= 96 * 1024) return nt;
    for (int nt = 4; nt >= 1; nt >>= 1)
        if (plan_smem(nt, xs_need[nt_index(nt)], K_max, max_tile, &p)) return nt;
    return 0;
}

// Launches a program over all N rows, in panels of at most `nt_cap` rows (rows are independent).
sd2_status run_panels(SArgs& a, int64_t N, const int xs_need[3], int K_max, int max_tile, int grid, cudaStream_t s)
{
    const int nt_cap = widest_panel(xs_need, K_max, max_tile);
    if (nt_cap == 0) return SD2_ERR_UNSUPPORTED;
    const bool small = a.n_stages == 1 || a.ext;             // one inline stage at most is all that the launch reads
    SArgsT<1> one;
    if (small) {
        one.inl[0] = a.inl[0];
        one.fold[0] = a.fold[0];
    }
    for (int64_t n0 = 0; n0 < N; n0 += nt_cap) {
        const int n = (int)((N - n0) < nt_cap ? (N - n0) : nt_cap);
        const int nt = round_nt(n, nt_cap);
        SmemPlan p;   // the narrower the panel, the more room for the ring
        if (!plan_smem(nt, xs_need[nt_index(nt)], K_max, max_tile, &p)) return SD2_ERR_UNSUPPORTED;
        a.N = n;
        a.n0 = (int)n0;
        a.xs_bytes = p.xs_bytes;
        a.xlin_bytes = p.xlin_bytes;
        a.ring_bytes = p.ring_bytes;
        if (a.fold_any) a.ring_bytes -= kFoldStaticBytes;   // those instances keep a little static shared memory (the ring still holds two tiles)
        sd2_status st;
        if (small) {
            static_cast<SArgsBase&>(one) = a;
            st = launch_stream(nt, one, grid, a.n_stages > 1, s);
        } else {
            st = launch_stream(nt, a, grid, a.n_stages > 1, s);
        }
        if (st != SD2_OK) return st;
    }
    return SD2_OK;
}

// How a program of inline stages takes its norms.  Threads hold rows that are on 16 bytes and no longer than eight columns of each, from 768
// columns on: us of a decode block of one row by shared memory and held, hidden 512 28.4 and 29.1, 768 30.7 and 30.5, 1024 31.9 and 31.8,
// 1536 37.0 and 36.3, 2048 46.0 and 44.5, 4096 71.4 and 62.3; of 256 for three rows 41.6 and 43.8.
int fold_of(const SArgs& a)
{
    for (int i = 0; i < a.n_stages; ++i) {
        const SFold& f = a.fold[i];
        if (!f.norm_w) continue;
        const SStage& st = a.inl[i];
        if (!st.x || st.K % 8 || st.K < 768 || st.K > 8 * kConsumerThreads ||
            (((uintptr_t)st.x | (uintptr_t)f.res | (uintptr_t)f.norm_w | (uintptr_t)f.sum_out | (uintptr_t)f.norm_out) & 15))
            return kFoldShared;
    }
    return kFoldHeld;
}

// Runs a program of inline stages.
sd2_status run_program(SArgs& a, int dev, int64_t N, const ProgramNeeds& needs, cudaStream_t s)
{
    const bool coop = a.n_stages > 1;
    int grid = g_dev[dev].sms;
    if (!coop && needs.tiles_max < grid) grid = needs.tiles_max < 1 ? 1 : needs.tiles_max;
    if (!coop) set_stage_grid(a.inl[0], grid);
    a.err = g_dev[dev].err_word;
    a.wait_cycles = wait_budget(dev);
    a.free_tiles = needs.free_tiles(grid);
    if (a.fold_any) a.fold_any = fold_of(a);
    a.gbar = coop ? g_dev[dev].barriers + (size_t)(g_next_barrier.fetch_add(1) % kBarrierPool) * kBarrierStrideWords : nullptr;
    return run_panels(a, N, needs.xs_need, needs.K_max, needs.max_tile, grid, s);
}

// ------------------------------------------------------------------ programs over cells

struct CellPlan {
    int fixed_bytes, n_parts, part_bytes, xbuf_bytes, chunk_bytes, n_slots;
};

template <int NR>
constexpr int cell_fixed_bytes() { return (int)((sizeof(CellShared<NR>) + 127) & ~127); }

int cell_instance(int n) { return n <= 8 ? 8 : n <= 16 ? 16 : 32; }

// Shared memory of a launch of n rows.  false: not even two chunks per group fit beside the staged rows.
bool plan_cells(int n, const CellNeeds& needs, CellPlan* p)
{
    p->chunk_bytes = (needs.max_chunk + 127) & ~127;
    p->xbuf_bytes = (n * needs.pitch + 127) & ~127;
    // (n_parts: per finisher) the ring comes first: nine chunks in flight cover HBM's latency, then sums may wait, then more.
    // A tile of split stages takes three of the slots for sums.
    const int nr = cell_instance(n);
    p->fixed_bytes = nr == 8 ? cell_fixed_bytes<8>() : nr == 16 ? cell_fixed_bytes<16>() : cell_fixed_bytes<32>();
    static const int tries[][2] = {{4, 8}, {3, 8}, {3, 4}, {2, 4}, {2, 2}};
    for (const int* t : tries) {
        if (t[1] < 4 && needs.split) break;
        p->part_bytes = 2 * t[1] * part_slot_bytes(nr);
        const int ring = kSmemMax - p->fixed_bytes - p->part_bytes - p->xbuf_bytes;
        p->n_parts = t[1];
        p->n_slots = ring > 0 ? ring / (kCellGroups * p->chunk_bytes) : 0;
        if (p->n_slots > kGroupSlots) p->n_slots = kGroupSlots;
        if (p->n_slots >= t[0]) return true;
    }
    return false;
}

// Most rows a launch of the program can take; 0 if none.
int widest_cell_panel(const CellNeeds& needs, int most = kPanelRows)
{
    CellPlan p;
    for (int n = most; n >= 1; --n)
        if (plan_cells(n, needs, &p)) return n;
    return 0;
}


template <int MAXS>
sd2_status launch_cell_kernel(void (*kernel)(CArgs<MAXS>), const CArgs<MAXS>& a, int grid, int smem, cudaStream_t s)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kCellThreads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeCooperative;
    attr[1].val.cooperative = 1;
    if (a.n_stages == 1) attr[1] = pdl_attribute();
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, a);
    if (e != cudaSuccess) { cudaGetLastError(); return SD2_ERR_CUDA; }
    return SD2_OK;
}

template <int MAXS, int NR>
sd2_status launch_cells(const CArgs<MAXS>& a, int grid, int smem, cudaStream_t s)
{
    return launch_cell_kernel<MAXS>(a.fold_any ? cell_kernel<MAXS, NR, true> : cell_kernel<MAXS, NR, false>, a, grid, smem, s);
}
sd2_status launch_wide_cells(const CArgs<1>& a, int grid, int smem, cudaStream_t s)
{
    return launch_cell_kernel<1>(cell_kernel<1, kWidePanelRows, false>, a, grid, smem, s);
}

void set_stage_clusters(CStage& st, int clusters)
{
    st.tiles_div = st.V / clusters;
    st.tiles_rem = st.V % clusters;
}

// Stages of a program over cells while it is put together.
struct CellBuilder {
    CStage* stages;
    CellNeeds needs;
    int n = 0, clusters, rot = 0;
    CellBuilder(CStage* s, int sms) : stages(s), clusters(sms / 2) {}

    // One stage of `count` handles of equal K.  pair: hs[0] and hs[1] are gate and up.
    CStage& add(const sd2_handle* hs, int count, const uint16_t* x, void* const* Y, bool y_force_bf16, bool pair = false)
    {
        CStage& st = stages[n];
        std::memset(&st, 0, sizeof st);
        st.count = count;
        st.K = (int)hs[0]->K;
        st.D = hs[0]->cell_D;
        st.x = x;
        st.pair = pair ? 1 : 0;
        for (int i = 0; i < count; ++i) {
            CMat& m = st.mat[i];
            m.off = (const uint32_t*)hs[i]->d_image;
            m.cells = hs[i]->d_cells;
            m.y = Y[i];
            m.M = (int)hs[i]->M;
            m.T = hs[i]->cell_T;
            m.y_f32 = (!y_force_bf16 && hs[i]->y_dtype == SD2_DTYPE_F32) ? 1 : 0;
            if (!pair || i == 0) st.V += m.T;
            needs.add(hs[i]);
        }
        if (st.V > needs.tiles_max) needs.tiles_max = st.V;
        st.rot = rot;
        rot = (int)(((int64_t)rot + st.V) % clusters);
        set_stage_clusters(st, clusters);
        ++n;
        return st;
    }
};

// Launches a program over all N rows, in panels of equal size (rows are independent).
sd2_status run_cell_panels(CArgs<kMaxStagesInline>& a, int64_t N, const CellNeeds& needs, int grid, cudaStream_t s)
{
    if (a.ext && a.fold_any) return SD2_ERR_UNSUPPORTED;     // stages in device memory carry no norms
    const int cap = widest_cell_panel(needs, a.n_stages == 1 && !a.fold_any ? kWidePanelRows : kPanelRows);
    if (cap == 0) return SD2_ERR_UNSUPPORTED;
    const int64_t panels = (N + cap - 1) / cap;
    const int64_t rows = (N + panels - 1) / panels;
    CArgs<1> one;
    const bool small = a.n_stages == 1 || a.ext;             // one inline stage is all that the launch reads
    if (small) {
        one.inl[0] = a.inl[0];
        one.fold[0] = a.fold[0];
    }
    for (int64_t n0 = 0; n0 < N; n0 += rows) {
        a.N = (int)((N - n0) < rows ? (N - n0) : rows);
        a.n0 = (int)n0;
        CellPlan p;
        if (!plan_cells(a.N, needs, &p)) return SD2_ERR_UNSUPPORTED;
        a.part_mask = p.n_parts - 1;
        a.xbuf_bytes = p.xbuf_bytes;
        a.chunk_bytes = p.chunk_bytes;
        a.n_slots = p.n_slots;
        const int smem = p.fixed_bytes + p.part_bytes + p.xbuf_bytes + kCellGroups * p.n_slots * p.chunk_bytes;
        sd2_status st;
        if (small) {
            static_cast<CArgsBase&>(one) = a;
            st = a.N > 16 ? launch_wide_cells(one, grid, smem, s) : a.N > 8 ? launch_cells<1, 16>(one, grid, smem, s) : launch_cells<1, 8>(one, grid, smem, s);
        } else {
            st = a.N > 8 ? launch_cells<kMaxStagesInline, 16>(a, grid, smem, s) : launch_cells<kMaxStagesInline, 8>(a, grid, smem, s);
        }
        if (st != SD2_OK) return st;
    }
    return SD2_OK;
}

// Runs a program of inline stages.
sd2_status run_cell_program(CArgs<kMaxStagesInline>& a, const CellBuilder& b, int dev, int64_t N, cudaStream_t s)
{
    a.n_stages = b.n;
    const bool coop = a.n_stages > 1;
    int clusters = b.clusters;
    if (!coop && b.needs.tiles_max < clusters) {
        clusters = b.needs.tiles_max;
        set_stage_clusters(a.inl[0], clusters);
    }
    const int grid = 2 * clusters;
    a.err = g_dev[dev].err_word;
    a.wait_cycles = wait_budget(dev);
    if (!a.gbar && coop) a.gbar = g_dev[dev].barriers + (size_t)(g_next_barrier.fetch_add(1) % kBarrierPool) * kBarrierStrideWords;
    return run_cell_panels(a, N, b.needs, grid, s);
}

// Attention by attention_kernel.  A head's positions are split over CTAs while each keeps more than 128 and the SMs are not
// yet taken twice.
template <bool ROPE>
sd2_status launch_attention(uint16_t* q, const uint16_t* k, const uint16_t* v, uint16_t* kc, uint16_t* vc, uint16_t* out, int64_t N,
                            int64_t Hq, int64_t Hkv, int64_t d, int64_t T, int64_t T_max, const RopeTable& tab, int sms, cudaStream_t s)
{
    int64_t S = 1;
    while (S < kAttnMaxCluster && T > 128 * S && N * Hq * 2 * S <= 2 * sms) S *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(N * Hq * S));
    cfg.blockDim = dim3(kAttnThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0] = pdl_attribute();
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)S;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, attention_kernel<ROPE>, q, k, v, kc, vc, out, (int)Hq, (int)Hkv, (int)d, (int)T, (int)T_max,
                                             (int)S, tab);
    if (e != cudaSuccess) { cudaGetLastError(); return SD2_ERR_CUDA; }
    return SD2_OK;
}

// An LM head of NT activation rows at most.
template <int NT>
sd2_status launch_lm_head(const uint16_t* x, const uint16_t* w, float* logits, int n, int V, int H, int sms, cudaStream_t s)
{
    const size_t smem = (size_t)NT * (size_t)H * 2;
    int per_sm = (int)((size_t)(200 * 1024) / smem);
    per_sm = per_sm < 1 ? 1 : per_sm > head_ctas(NT) ? head_ctas(NT) : per_sm;
    int64_t grid = ((int64_t)V + kGlueThreads / 32 - 1) / (kGlueThreads / 32);
    if (grid > (int64_t)sms * per_sm) grid = (int64_t)sms * per_sm;
    launch_pdl(lm_head_kernel<NT>, (unsigned)grid, kGlueThreads, smem, s, x, w, logits, n, V, H);
    return cudaGetLastError() == cudaSuccess ? SD2_OK : SD2_ERR_CUDA;
}

// Whether N rows over these GAP4 handles are faster by their cells.  Cells bring 1.3 times the strips' bytes but expand them
// once for all rows, the strips gather row by row.  Measured (us, cold caches, strips / cells): 2048 x 8192 at 50 %: N = 1
// 14.4 / 16.4, N = 2 18.4 / 16.4, N = 3 24.6 / 16.4; the same at 30 %: 12.3 / 14.5, 15.4 / 16.4, 20.5 / 16.3; two blocks of
// 2048/512/8192 at 50 %: 60 / 70, 75 / 70, 116 / 72.  From four rows on cells are faster at every density, though the strips'
// work shrinks with it: at 10 % 2048 x 2048 for N = 4 about 10 / 6, 640 x 640 9.4 / 5.7, 2048 x 11008 20.6 / 11.3, 1024 x 15360
// (where a launch takes twelve rows) 22 / 10 and for N = 64 345 / 63.  Below a million slots three rows would gain too (640 x
// 640: 8.8 / 5.7, two rows 6.5 / 5.7) and stay with the strips all the same, whose sums do not depend on how many rows a
// call has: small steps give the bits of one-row steps.
bool cells_pay(const sd2_handle* hs, int count, int64_t N)
{
    if (N >= 4) return true;
    if (N < 2) return false;
    int64_t slots = 0, kept = 0, largest = 0;
    for (int i = 0; i < count; ++i) {
        const int64_t n = hs[i]->M * hs[i]->K;
        slots += n;
        kept += hs[i]->nnz;
        if (n > largest) largest = n;
    }
    return largest >= (1 << 20) && (N > 2 || 5 * kept >= 2 * slots);
}

// ... and whether the call can take them.
bool use_cells(const sd2_handle* hs, int count, int64_t N)
{
    CellNeeds needs;
    for (int i = 0; i < count; ++i) {
        if (!hs[i]->d_image) return false;
        needs.add(hs[i]);
    }
    return cells_pay(hs, count, N) && widest_cell_panel(needs) > 0;
}

// Shared by sd2_spmm and sd2_spmm_fused (and by block steps that mix formats).
// cuTensorMapEncodeTiled through the runtime (no link against the driver library).  NULL: not available.
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled_fn()
{
    static std::atomic<void*> cached{nullptr};
    static std::atomic<int> tried{0};
    if (!tried.load()) {
        void* fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) != cudaSuccess || q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            fn = nullptr;
        }
        cached.store(fn);
        tried.store(1);
    }
    return (EncodeTiledFn)cached.load();
}

// Tensor map over X [N, K] bf16 whose boxes are 64 columns x npad rows, stored with the 128-byte swizzle;
// what a box reaches beyond N rows or K columns is filled with zeros.  false: X cannot be described
// (unaligned base or row pitch), the kernel's groups fetch it themselves.
bool make_x_map(CUtensorMap* map, const uint16_t* X, int64_t N, int64_t K, int npad)
{
    EncodeTiledFn enc = encode_tiled_fn();
    if (!enc || (((uintptr_t)X) & 15) || (K & 7) || K < kMmaBlockCols) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)N};
    const cuuint64_t strides[1] = {(cuuint64_t)K * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kMmaBlockCols, (cuuint32_t)npad};
    const cuuint32_t estr[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)X, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Shared memory of a launch of mma_kernel.  false: not even one block for each team fits.
bool plan_mma(const MmaArgs& a, int block_bytes, int* slot_bytes, int* n_slots, int* smem)
{
    const int fixed = 1024 + kMmaStages * a.npad * 128 + mma_recv_bytes(a.npad, a.shares) + (int)((sizeof(MmaShared) + 127) & ~127);
    *slot_bytes = (block_bytes + 127) & ~127;
    int slots = (kSmemMax - fixed) / *slot_bytes / kMmaTeams * kMmaTeams;
    const int most = (((a.KB + a.shares - 1) / a.shares) + kMmaTeams - 1) / kMmaTeams * kMmaTeams;
    if (slots > kMmaMaxSlots) slots = kMmaMaxSlots;
    if (slots > most) slots = most;
    if (slots < kMmaTeams) return false;
    *n_slots = slots;
    *smem = fixed + slots * *slot_bytes;
    // all of an SM's tensor memory goes to one CTA: another one of the launch must not come to the SM, where it would wait for it
    if (*smem < kSmemMax / 2 + 1024) *smem = kSmemMax / 2 + 1024;
    return true;
}

// How many CTAs share a panel's columns: the fewest steps of a CTA, in blocks.  What a CTA does beside its blocks (start, last sums)
// is worth about four of them, the exchange of sums three more.
int mma_cluster(int64_t P, int KB, const int* room)
{
    int best = 1;
    int64_t least = 0;
    for (int c = 1; c <= kMmaMaxCluster && c <= KB; ++c) {
        if (room[c] < 1) continue;
        const int64_t waves = (P + room[c] - 1) / room[c];
        const int64_t steps = waves * ((KB + c - 1) / c + 4) + (c > 1 ? 3 : 0);
        if (c == 1 || steps < least) { best = c; least = steps; }
    }
    return best;
}

cudaError_t launch_mma(const MmaArgs& a, const CUtensorMap& xmap, int64_t P, int smem, cudaStream_t s, int* room = nullptr)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(P * a.shares));
    cfg.blockDim = dim3(kMmaThreads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)a.shares;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1] = pdl_attribute();
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    if (room) {                              // how many clusters of this size run at once
        cfg.numAttrs = 1;
        return cudaOccupancyMaxActiveClusters(room, mma_kernel, &cfg);
    }
    return cudaLaunchKernelEx(&cfg, mma_kernel, a, xmap);
}

sd2_status count_mma_clusters(int* room)
{
    room[0] = 0;
    for (int c = 1; c <= kMmaMaxCluster; ++c) {
        MmaArgs a;
        std::memset(&a, 0, sizeof a);
        a.shares = c;
        room[c] = 0;
        if (launch_mma(a, CUtensorMap{}, 1, kSmemMax, nullptr, &room[c]) != cudaSuccess) {
            cudaGetLastError();
            room[c] = 0;
        }
    }
    return room[1] > 0 ? SD2_OK : SD2_ERR_CUDA;
}

// GAP4_MMA: one launch per 64 activation rows.
sd2_status run_mma(sd2_handle h, const uint16_t* x, void* Y, int64_t N, bool y_force_bf16, int dev, cudaStream_t s)
{
    MmaArgs a;
    std::memset(&a, 0, sizeof a);
    a.off = (const uint32_t*)h->d_image;
    a.cells = h->d_cells;
    a.M = (int)h->M;
    a.K = (int)h->K;
    const int64_t P = h->cell_T;
    a.KB = h->cell_D;
    a.shares = mma_cluster(P, a.KB, g_dev[dev].mma_clusters);
    a.y_f32 = (!y_force_bf16 && h->y_dtype == SD2_DTYPE_F32) ? 1 : 0;
    a.err = g_dev[dev].err_word;
    a.budget = wait_budget(dev);
    const size_t esz = a.y_f32 ? 4 : 2;
    for (int64_t n0 = 0; n0 < N; n0 += kMmaMaxRows) {
        a.N = (int)((N - n0) < kMmaMaxRows ? (N - n0) : kMmaMaxRows);
        a.npad = (a.N + 15) & ~15;
        a.X = x + n0 * h->K;
        a.Y = (char*)Y + (size_t)n0 * (size_t)h->M * esz;
        CUtensorMap xmap;
        std::memset(&xmap, 0, sizeof xmap);
        a.x_tma = make_x_map(&xmap, a.X, a.N, h->K, a.npad) ? 1 : 0;
        a.x_vec = ((h->K & 7) == 0 && (((uintptr_t)a.X) & 15) == 0) ? 1 : 0;
        int smem = 0;
        if (!plan_mma(a, h->max_chunk, &a.slot_bytes, &a.n_slots, &smem)) return SD2_ERR_UNSUPPORTED;
        if (launch_mma(a, xmap, P, smem, s) != cudaSuccess) { cudaGetLastError(); return SD2_ERR_CUDA; }
    }
    return SD2_OK;
}

sd2_status run_group(const sd2_handle* hs, int count, const uint16_t* x, const uint16_t* g, const uint16_t* u,
                     uint16_t* t_out, void* const* Y, int64_t N, bool y_force_bf16, cudaStream_t s)
{
    if (count < 1 || count > kMaxFused) return SD2_ERR_INVALID_ARG;
    for (int i = 0; i < count; ++i)
        if (!live(hs[i]) || !Y[i]) return SD2_ERR_INVALID_ARG;
    if (N < 0) return SD2_ERR_SHAPE;
    if (N == 0) return SD2_OK;
    const int64_t K = hs[0]->K;
    for (int i = 1; i < count; ++i)
        if (hs[i]->K != K) return SD2_ERR_SHAPE;
    bool same = true;
    for (int i = 1; i < count; ++i)
        if (hs[i]->format != hs[0]->format || hs[i]->S != hs[0]->S) same = false;
    if (!same) {  // weights that cannot share a stage: one launch each
        for (int j = 0; j < count; ++j) {
            sd2_status sj = run_group(hs + j, 1, x, g, u, j == 0 ? t_out : nullptr, Y + j, N, y_force_bf16, s);
            if (sj != SD2_OK) return sj;
        }
        return SD2_OK;
    }
    int dev = 0;
    sd2_status st = ensure_device(&dev);
    if (st != SD2_OK) return st;
    for (int i = 0; i < count; ++i)
        if (hs[i]->device != dev) return SD2_ERR_INVALID_ARG;
    if (hs[0]->format == SD2_FORMAT_BITMASK) return run_bitmask(hs, count, x, g, u, t_out, Y, N, y_force_bf16, dev, s);
    if (hs[0]->format == SD2_FORMAT_GAP4_MMA) {
        if (!x || g || u || t_out) return SD2_ERR_UNSUPPORTED;     // plain products only
        for (int i = 0; i < count; ++i) {
            sd2_status si = run_mma(hs[i], x, Y[i], N, y_force_bf16, dev, s);
            if (si != SD2_OK) return si;
        }
        return SD2_OK;
    }
    if (use_cells(hs, count, N)) {
        CArgs<kMaxStagesInline> a = {};
        CellBuilder b(a.inl, g_dev[dev].sms);
        CStage& sg = b.add(hs, count, x, Y, y_force_bf16);
        sg.g = g;
        sg.u = u;
        sg.t_out = t_out;
        return run_cell_program(a, b, dev, N, s);
    }
    SArgs a;
    std::memset(&a, 0, sizeof a);
    a.n_stages = 1;
    fill_stage(a.inl[0], hs, count, x, g, u, t_out, Y, y_force_bf16, g_dev[dev].sms);
    ProgramNeeds needs;
    needs.add(hs, count);
    return run_program(a, dev, N, needs, s);
}

struct BlockDims {
    int64_t hidden, kv, q_out, inter, out;
};

sd2_status block_dims(const sd2_handle* h, BlockDims* d)
{
    if (!h) return SD2_ERR_INVALID_ARG;
    for (int i = 0; i < 7; ++i)
        if (!live(h[i])) return SD2_ERR_INVALID_ARG;
    const sd2_handle q = h[0], k = h[1], v = h[2], o = h[3], ga = h[4], up = h[5], dn = h[6];
    d->hidden = q->K;
    if (k->K != d->hidden || v->K != d->hidden) return SD2_ERR_SHAPE;
    if (k->M != v->M) return SD2_ERR_SHAPE;
    d->kv = k->M;
    d->q_out = q->M;
    if (o->K != q->M) return SD2_ERR_SHAPE;           // attention stub: a = q
    if (ga->K != o->M || up->K != o->M) return SD2_ERR_SHAPE;
    if (ga->M != up->M) return SD2_ERR_SHAPE;
    d->inter = ga->M;
    if (dn->K != d->inter) return SD2_ERR_SHAPE;
    d->out = dn->M;
    return SD2_OK;
}

int64_t a256(int64_t x) { return (x + 255) & ~int64_t(255); }

void block_layout(const sd2_handle* h, const BlockDims& d, int64_t N, int64_t off[8])
{
    const int64_t dims[7] = {d.q_out, d.kv, d.kv, h[3]->M, d.inter, d.inter, d.inter};
    int64_t o = 0;
    for (int i = 0; i < 7; ++i) {
        off[i] = o;
        o = a256(o + 2 * N * dims[i]);
    }
    off[7] = o;
}

// Tagged 32-bit copies of a block's activations (value << 16 | stage tag) through which the
// stages of a tagged program hand their outputs to the next stage without a grid barrier.
struct BlockTags {
    const uint32_t* x_t;   // the block's input as tagged words, or NULL (plain bf16 input)
    uint32_t *q_t, *hdn_t, *g_t, *u_t, *out_t;   // out_t NULL: the block's output is not handed on
    uint32_t* t_t;                               // tagged t = silu(g) * u, one slice per CTA
};

// Appends one group of linears that share an input to `stages` (plain hand-off): one stage if they share a strip
// geometry, else a stage each.  Returns the new stage count.
int append_group(SStage* stages, int n, ProgramNeeds* needs, const sd2_handle* hs, int count, const uint16_t* xin,
                 const uint16_t* gg, const uint16_t* uu, uint16_t* tt, void* const* Y, bool force_bf16, int grid)
{
    bool same = true;
    for (int i = 1; i < count; ++i)
        if (hs[i]->S != hs[0]->S) same = false;
    if (same) {
        fill_stage(stages[n++], hs, count, xin, gg, uu, tt, Y, force_bf16, grid);
        needs->add(hs, count);
    } else {
        for (int i = 0; i < count; ++i) {
            fill_stage(stages[n++], hs + i, 1, xin, gg, uu, i == 0 ? tt : nullptr, Y + i, force_bf16, grid);
            needs->add(hs + i, 1);
        }
    }
    return n;
}

// Appends the stages of one block (h[0..6] = q,k,v,o,gate,up,down) to `stages`.  Weights of a
// group that do not share a strip geometry get a stage each.  Returns the number appended.
int append_block_stages(SStage* stages, const sd2_handle* h, const uint16_t* x, uint16_t* q, uint16_t* k, uint16_t* v,
                        uint16_t* hdn, uint16_t* g, uint16_t* u, uint16_t* t, void* y, bool y_force_bf16,
                        ProgramNeeds* needs, int grid, const BlockTags* tg = nullptr, sd2_handle gu_pair = nullptr)
{
    int n = 0;
    auto group = [&](const sd2_handle* hs, int count, const uint16_t* xin, const uint16_t* gg, const uint16_t* uu,
                     uint16_t* tt, void* const* Y, bool force, uint32_t* const* YT, int tin) {
        bool same = true;
        for (int i = 1; i < count; ++i)
            if (hs[i]->S != hs[0]->S) same = false;
        if (same) {
            fill_stage(stages[n++], hs, count, xin, gg, uu, tt, Y, force, grid, YT, tin);
            needs->add(hs, count);
        } else {
            for (int i = 0; i < count; ++i) {
                fill_stage(stages[n++], hs + i, 1, xin, gg, uu, i == 0 ? tt : nullptr, Y + i, force, grid, YT ? YT + i : nullptr, tin);
                needs->add(hs + i, 1);
            }
        }
    };
    void* y_qkv[3] = {q, k, v};
    void* y_o[1] = {hdn};
    void* y_gu[2] = {g, u};
    void* y_d[1] = {y};
    if (!tg) {
        group(h + 0, 3, x, nullptr, nullptr, nullptr, y_qkv, true, nullptr, 0);
        group(h + 3, 1, q, nullptr, nullptr, nullptr, y_o, true, nullptr, 0);
        group(h + 4, 2, hdn, nullptr, nullptr, nullptr, y_gu, true, nullptr, 0);
        group(h + 6, 1, nullptr, g, u, t, y_d, y_force_bf16, nullptr, 0);
    } else {
        uint32_t* t_qkv[3] = {tg->q_t, nullptr, nullptr};
        uint32_t* t_o[1] = {tg->hdn_t};
        uint32_t* t_gu[2] = {tg->g_t, tg->u_t};
        uint32_t* t_d[1] = {tg->out_t};
        group(h + 0, 3, tg->x_t ? (const uint16_t*)tg->x_t : x, nullptr, nullptr, nullptr, y_qkv, true, t_qkv, tg->x_t ? 1 : 0);
        group(h + 3, 1, (const uint16_t*)tg->q_t, nullptr, nullptr, nullptr, y_o, true, t_o, 1);
        if (gu_pair) {
            // one stacked matrix, gate row i and up row i in one tile: the stage writes g, u and t
            // as plain bf16 and t as tagged words, and the down stage reads t like any activation
            void* y_none[1] = {nullptr};
            SStage& st = stages[n++];
            fill_stage(st, &gu_pair, 1, (const uint16_t*)tg->hdn_t, nullptr, nullptr, nullptr, y_none, true, grid, nullptr, 1);
            needs->add(&gu_pair, 1);
            st.paired = 1;
            st.g = g;
            st.u = u;
            st.t_out = t;
            st.tt = tg->t_t;
            group(h + 6, 1, (const uint16_t*)tg->t_t, nullptr, nullptr, nullptr, y_d, y_force_bf16, t_d, 1);
        } else {
            group(h + 4, 2, (const uint16_t*)tg->hdn_t, nullptr, nullptr, nullptr, y_gu, true, t_gu, 1);
            const int before = n;
            group(h + 6, 1, nullptr, (const uint16_t*)tg->g_t, (const uint16_t*)tg->u_t, t, y_d, y_force_bf16, t_d, 1);
            for (int i = before; i < n; ++i) stages[i].tt = tg->t_t;
        }
    }
    return n;   // at most 7
}

// Appends the four stages of one block (h[0..6] = q,k,v,o,gate,up,down) to a program over cells.  t = silu(g) * u is
// formed where g and u are produced.
void append_block_cells(CellBuilder& b, const sd2_handle* h, const uint16_t* x, uint16_t* q, uint16_t* k, uint16_t* v, uint16_t* hdn,
                        uint16_t* g, uint16_t* u, uint16_t* t, void* y, bool y_force_bf16)
{
    void* y_qkv[3] = {q, k, v};
    void* y_o[1] = {hdn};
    void* y_gu[2] = {g, u};
    void* y_d[1] = {y};
    b.add(h + 0, 3, x, y_qkv, true);
    b.add(h + 3, 1, q, y_o, true);
    b.add(h + 4, 2, hdn, y_gu, true, true).t_out = t;
    b.add(h + 6, 1, t, y_d, y_force_bf16);
}

// A block step over cells.  gbar: barrier words of the caller's, or NULL.
// One program of four stages where its panels are no narrower than the rest of the block needs them.  Where the down
// projection's long rows of activations fill shared memory, it goes apart, in panels of its own: sixteen rows of
// 3072/1024/8192 at 50 % took 94 us as two panels of eight through all stages.
sd2_status run_block_cells(const sd2_handle* h, const uint16_t* x, uint16_t* q, uint16_t* k, uint16_t* v, uint16_t* hdn, uint16_t* g, uint16_t* u,
                           uint16_t* t, void* y, unsigned int* gbar, int dev, int64_t N, cudaStream_t s)
{
    CArgs<kMaxStagesInline> a = {};
    CellBuilder b(a.inl, g_dev[dev].sms);
    append_block_cells(b, h, x, q, k, v, hdn, g, u, t, y, false);
    a.gbar = gbar;
    CArgs<kMaxStagesInline> d = {};
    CellBuilder down(d.inl, g_dev[dev].sms), rest(a.inl, g_dev[dev].sms);
    void* y_d[1] = {y};
    down.add(h + 6, 1, t, y_d, false);
    for (int i = 0; i < 6; ++i) rest.needs.add(h[i]);
    rest.needs.tiles_max = b.needs.tiles_max;
    rest.n = b.n - 1;
    const int64_t all = widest_cell_panel(b.needs), most = widest_cell_panel(rest.needs);
    if ((N + most - 1) / most >= (N + all - 1) / all) return run_cell_program(a, b, dev, N, s);
    const sd2_status st = run_cell_program(a, rest, dev, N, s);
    return st != SD2_OK ? st : run_cell_program(d, down, dev, N, s);
}

// Builds the paired stack of a block's gate and up (row 2i = gate row i, row 2i+1 = up row i)
// from the decoded contents of the two handles.  *out stays NULL where the shape has no paired
// form (fewer than two rows per tile); the caller then keeps the two weights apart.
sd2_status build_gate_up_pair(sd2_handle gate, sd2_handle up, sd2_handle* out)
{
    *out = nullptr;
    const int64_t I = gate->M, K = gate->K;
    if (up->M != I || up->K != K) return SD2_OK;
    const Gap4Geom g = gap4_geometry(2 * I, K, true);
    if (g.S == 0 || g.R < 2) return SD2_OK;
    uint16_t* dense = (uint16_t*)lib_malloc((size_t)(2 * I * K) * 2);
    uint16_t* one = (uint16_t*)lib_malloc((size_t)(I * K) * 2);
    sd2_status st = (dense && one) ? SD2_OK : SD2_ERR_ALLOC;
    for (int w = 0; w < 2 && st == SD2_OK; ++w) {
        st = sd2_decompress(w == 0 ? gate : up, one);
        if (st != SD2_OK) break;
#pragma omp parallel for schedule(static)
        for (int64_t i = 0; i < I; ++i) std::memcpy(dense + (size_t)(2 * i + w) * K, one + (size_t)i * K, (size_t)K * 2);
    }
    std::free(one);
    uint8_t* blob = nullptr;
    int64_t bytes = 0;
    if (st == SD2_OK) {
        // no mask: what decoded to +0 was masked out (or was a kept zero, which adds nothing)
        sd2_options opt = {SD2_FORMAT_GAP4_PAIRED, SD2_DTYPE_BF16};
        st = pack_any(dense, nullptr, 2 * I, K, &opt, &blob, &bytes);
    }
    std::free(dense);
    if (st != SD2_OK) return st;
    BlobHeader hd;
    std::memcpy(&hd, blob, sizeof hd);
    st = upload(blob, bytes, hd, out);
    std::free(blob);
    return st;
}

}  // namespace

extern "C" {

const char* sd2_status_string(sd2_status s)
{
    switch (s) {
        case SD2_OK: return "ok";
        case SD2_ERR_INVALID_ARG: return "invalid argument";
        case SD2_ERR_SHAPE: return "bad or inconsistent shape";
        case SD2_ERR_ALLOC: return "allocation failed";
        case SD2_ERR_CUDA: return "CUDA runtime error";
        case SD2_ERR_UNSUPPORTED: return "unsupported request";
        case SD2_ERR_CORRUPT: return "corrupt blob";
        case SD2_ERR_TIMEOUT: return "device-side wait timed out";
        default: return "unknown status";
    }
}

sd2_status sd2_pack_host(const void* weight_bf16, const uint8_t* mask, int64_t M, int64_t K,
                         const sd2_options* opt, void** blob, int64_t* blob_bytes)
{
    uint8_t* b = nullptr;
    int64_t n = 0;
    sd2_status st = pack_any((const uint16_t*)weight_bf16, mask, M, K, opt, &b, &n);
    if (st != SD2_OK) return st;
    *blob = b;
    *blob_bytes = n;
    return SD2_OK;
}

sd2_status sd2_unpack_host(const void* blob, int64_t blob_bytes, void* dense_bf16_out, int64_t* M, int64_t* K,
                           int64_t* nnz, int64_t* compressed_bytes, int32_t* format)
{
    if (!blob) return SD2_ERR_INVALID_ARG;
    BlobHeader hd;
    if (check_header((const uint8_t*)blob, blob_bytes, hd, true) != 0) return SD2_ERR_CORRUPT;
    int rc;
    try {
        rc = unpack_any(hd, (const uint8_t*)blob, (uint16_t*)dense_bf16_out);
    } catch (const std::bad_alloc&) {
        return SD2_ERR_ALLOC;
    }
    if (rc != 0) return SD2_ERR_CORRUPT;
    if (M) *M = hd.M;
    if (K) *K = hd.K;
    if (nnz) *nnz = hd.nnz;
    if (compressed_bytes) *compressed_bytes = hd.compressed_bytes;
    if (format) *format = (int32_t)hd.format;
    return SD2_OK;
}

sd2_status sd2_blob_free(void* blob)
{
    if (!blob) return SD2_ERR_INVALID_ARG;
    std::free(blob);
    return SD2_OK;
}

sd2_status sd2_compress(const void* weight_bf16, const uint8_t* mask, int64_t M, int64_t K, const sd2_options* opt,
                        sd2_handle* out)
{
    Range range_("sd2_compress");
    if (!weight_bf16 || !out) return SD2_ERR_INVALID_ARG;
    if (M < 1 || K < 1 || M * K > (1ll << 40)) return SD2_ERR_SHAPE;
    const uint16_t* W = (const uint16_t*)weight_bf16;
    const uint8_t* const mask_in = mask;
    uint16_t* w_tmp = nullptr;
    uint8_t* m_tmp = nullptr;
    sd2_status st = SD2_OK;
    if (is_device_ptr(weight_bf16)) {
        w_tmp = (uint16_t*)lib_malloc((size_t)(M * K) * 2);
        if (!w_tmp) return SD2_ERR_ALLOC;
        if (cudaMemcpy(w_tmp, weight_bf16, (size_t)(M * K) * 2, cudaMemcpyDeviceToHost) != cudaSuccess) { cudaGetLastError(); st = SD2_ERR_CUDA; }
        W = w_tmp;
    }
    if (st == SD2_OK && mask && is_device_ptr(mask)) {
        m_tmp = (uint8_t*)lib_malloc((size_t)(M * K));
        if (!m_tmp) st = SD2_ERR_ALLOC;
        else if (cudaMemcpy(m_tmp, mask, (size_t)(M * K), cudaMemcpyDeviceToHost) != cudaSuccess) { cudaGetLastError(); st = SD2_ERR_CUDA; }
        mask = m_tmp;
    }
    uint8_t* blob = nullptr;
    int64_t bytes = 0;
    BlobHeader hd;
    if (st == SD2_OK && resolve_format(opt, M, K) == SD2_FORMAT_GAP4_MMA) {       // (its handles keep no records)
        st = check_pack(M, K, opt);
        if (st == SD2_OK) st = from_pack(size_gap4_mma(W, mask, M, K, opt->y_dtype, &hd));
    } else if (st == SD2_OK) {
        st = pack_any(W, mask, M, K, opt, &blob, &bytes);
        if (st == SD2_OK) std::memcpy(&hd, blob, sizeof hd);
    }
    if (st == SD2_OK) {
        sd2_handle h = nullptr;
        st = upload(blob, bytes, hd, &h);
        std::free(blob);
        const bool cells = h && (h->format == SD2_FORMAT_GAP4_MMA || (h->format == SD2_FORMAT_GAP4 && !(opt && opt->format == SD2_FORMAT_GAP4_STRIPS)));
        if (st == SD2_OK && cells)    // (from the host's copies of what lies on another GPU)
            st = add_cells(h, kernel_reads(weight_bf16, sizeof *W, h->device) ? (const uint16_t*)weight_bf16 : W,
                           mask_in && kernel_reads(mask_in, sizeof *mask_in, h->device) ? mask_in : mask);
        if (st == SD2_OK) *out = h;
    }
    std::free(w_tmp);
    std::free(m_tmp);
    return st;
}

sd2_status sd2_load_blob(const void* blob, int64_t blob_bytes, sd2_handle* out)
{
    if (!blob || !out) return SD2_ERR_INVALID_ARG;
    BlobHeader hd;
    if (check_header((const uint8_t*)blob, blob_bytes, hd, true) != 0) return SD2_ERR_CORRUPT;
    // M and K are believed once the directory bears them out (the checksum does not cover the header); full structural
    // validation before anything reaches a kernel
    uint16_t* dense = nullptr;
    if (hd.format == (uint32_t)kFormatGap4) {
        if (check_gap4(hd, (const uint8_t*)blob) != 0) return SD2_ERR_CORRUPT;
        dense = (uint16_t*)lib_malloc((size_t)(hd.M * hd.K) * 2);     // for the cells; NULL: the handle goes without
    }
    int rc;
    try {
        rc = unpack_any(hd, (const uint8_t*)blob, dense);
        if (rc != 0 && dense) {              // a column that two lanes share has a sum in strips, but no dense form
            std::free(dense);
            dense = nullptr;
            rc = unpack_any(hd, (const uint8_t*)blob, nullptr);
        }
    } catch (const std::bad_alloc&) {
        std::free(dense);
        return SD2_ERR_ALLOC;
    }
    sd2_handle h = nullptr;
    sd2_status st = rc != 0 ? SD2_ERR_CORRUPT : upload((const uint8_t*)blob, blob_bytes, hd, &h);
    // for the cells what decoded to +0 or -0 was masked out, or was a kept zero, which adds nothing (panel cells are what a handle
    // is decompressed from: they keep a -0)
    if (st == SD2_OK && dense) st = add_cells(h, dense, nullptr);
    else if (st == SD2_OK && h->format == SD2_FORMAT_GAP4_MMA) st = add_cells(h, nullptr, nullptr, 0xFFFFu, &hd, (const uint8_t*)blob);
    std::free(dense);
    if (st == SD2_OK) *out = h;
    return st;
}

sd2_status sd2_decompress(sd2_handle h, void* dense_bf16_out)
{
    if (!live(h) || !dense_bf16_out) return SD2_ERR_INVALID_ARG;
    const bool panel = h->format == SD2_FORMAT_GAP4_MMA;
    const CellGeom geom = panel_geometry(h->M, h->K);
    const size_t dir_bytes = align256((size_t)(geom.cells() + 1) * 4);
    const size_t image_bytes = panel ? dir_bytes + (size_t)h->cell_bytes - (size_t)(geom.cells() + 1) * 4 : (size_t)h->blob_bytes;
    uint8_t* blob = (uint8_t*)lib_malloc(image_bytes);
    if (!blob) return SD2_ERR_ALLOC;
    sd2_status st = SD2_OK;
    if (cudaMemcpy(blob, panel ? h->d_image : h->d_blob, image_bytes, cudaMemcpyDeviceToHost) != cudaSuccess) { cudaGetLastError(); st = SD2_ERR_CUDA; }
    const size_t dense_bytes = (size_t)(h->M * h->K) * 2;
    const bool to_dev = is_device_ptr(dense_bf16_out);
    uint16_t* host_out = to_dev ? (uint16_t*)lib_malloc(dense_bytes) : (uint16_t*)dense_bf16_out;
    if (!host_out) st = SD2_ERR_ALLOC;
    if (st == SD2_OK && !panel) st = sd2_unpack_host(blob, h->blob_bytes, host_out, nullptr, nullptr, nullptr, nullptr, nullptr);
    if (st == SD2_OK && panel) {
        const uint32_t* off = (const uint32_t*)blob;
#pragma omp parallel for schedule(static)
        for (int64_t p = 0; p < geom.T; ++p) {
            const int64_t first = p * kPanelRowsOfBlock, rows = std::min<int64_t>(kPanelRowsOfBlock, h->M - first);
            std::memset(host_out + first * h->K, 0, (size_t)(rows * h->K) * 2);
            for (int64_t c = p * geom.D * geom.per; c < (p + 1) * geom.D * geom.per; ++c)
                unpack_panel_cell(blob + dir_bytes + (size_t)off[c] * 32, (int)(((off[c + 1] - off[c]) * 32u - kCellHeaderBytes) / 128u),
                                  first + 32 * (c % geom.per), (c / geom.per - p * geom.D) * kPanelBlockCols, h->M, h->K, host_out);
        }
    }
    if (st == SD2_OK && to_dev &&
        cudaMemcpy(dense_bf16_out, host_out, dense_bytes, cudaMemcpyHostToDevice) != cudaSuccess) { cudaGetLastError(); st = SD2_ERR_CUDA; }
    if (to_dev) std::free(host_out);
    std::free(blob);
    return st;
}

sd2_status sd2_info(sd2_handle h, int64_t* M, int64_t* K, int64_t* nnz, int64_t* compressed_bytes, int32_t* format)
{
    if (!live(h)) return SD2_ERR_INVALID_ARG;
    if (M) *M = h->M;
    if (K) *K = h->K;
    if (nnz) *nnz = h->nnz;
    if (compressed_bytes) *compressed_bytes = h->compressed_bytes;
    if (format) *format = h->format;
    return SD2_OK;
}

sd2_status sd2_free(sd2_handle h)
{
    if (!h) return SD2_ERR_INVALID_ARG;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (!g_live.erase(h)) return SD2_ERR_INVALID_ARG;
    }
    sd2_status st = SD2_OK;
    if (cudaFree(h->d_blob) != cudaSuccess) { cudaGetLastError(); st = SD2_ERR_CUDA; }
    if (h->d_image && cudaFree(h->d_image) != cudaSuccess) { cudaGetLastError(); st = SD2_ERR_CUDA; }
    delete h;
    return st;
}

sd2_status sd2_stream_check(void* cuda_stream)
{
    int dev = 0;
    sd2_status st = ensure_device(&dev);
    if (st != SD2_OK) return st;
    if (cudaStreamSynchronize((cudaStream_t)cuda_stream) != cudaSuccess) { cudaGetLastError(); return SD2_ERR_CUDA; }
    int flag = 0;
    if (cudaMemcpy(&flag, g_dev[dev].err_word, sizeof flag, cudaMemcpyDeviceToHost) != cudaSuccess) { cudaGetLastError(); return SD2_ERR_CUDA; }
    if (flag) {
        // a kernel that gave up leaves its barrier words behind: wait for the device, clear everything
        cudaDeviceSynchronize();
        cudaMemset(g_dev[dev].err_word, 0, sizeof flag);
        cudaMemset(g_dev[dev].barriers, 0, (size_t)kBarrierPool * kBarrierStrideWords * 4);
        {
            std::lock_guard<std::mutex> lk(g_mu);
            for (sd2_drafter d : g_live_drafters)
                if (d->device == dev) {   // barrier words, production counts and every tagged word start over
                    cudaMemset(d->d_gbar, 0, kDrafterWordsBytes);
                    if (d->d_tags) cudaMemset(d->d_tags, 0, (size_t)d->tags_bytes);
                    if (d->d_cbar) cudaMemset(d->d_cbar, 0, kDrafterWordsBytes);
                }
        }
        cudaGetLastError();
        return flag == 2 ? SD2_ERR_CORRUPT : SD2_ERR_TIMEOUT;      // 2: an index check of a checked build failed
    }
    return SD2_OK;
}

// ------------------------------------------------------------------ decode-step glue

sd2_status sd2_rmsnorm(const void* x, const void* w, void* y, int64_t N, int64_t H, float eps, void* cuda_stream)
{
    Range range_("sd2_rmsnorm");
    if (!x || !w || !y) return SD2_ERR_INVALID_ARG;
    if (N < 0 || H < 1 || N > 0x7FFFFFFF || H > 0x7FFFFFFF) return SD2_ERR_SHAPE;
    if (N == 0) return SD2_OK;
    const bool vec = (H & 7) == 0 && ((((uintptr_t)x) | ((uintptr_t)w) | ((uintptr_t)y)) & 15) == 0;
    const int64_t loads = (H / 8 + kGlueThreads - 1) / kGlueThreads;       // 16-byte loads of a thread
    auto* const kernel = !vec ? rmsnorm_kernel<kNormPlain> : loads <= 1 ? rmsnorm_kernel<1> : loads <= 2 ? rmsnorm_kernel<2>
                       : loads <= 4 ? rmsnorm_kernel<4> : rmsnorm_kernel<kNormLoop>;
    launch_pdl(kernel, (unsigned)N, kGlueThreads, 0, (cudaStream_t)cuda_stream, (const uint16_t*)x, (const uint16_t*)w, (uint16_t*)y, (int)H, eps);
    return cudaGetLastError() == cudaSuccess ? SD2_OK : SD2_ERR_CUDA;
}

namespace {
RopeTable rope_table(int64_t head_dim, int64_t pos, double theta)
{
    RopeTable t;
    std::memset(&t, 0, sizeof t);
    for (int64_t i = 0; i < head_dim / 2 && i < kRopeMaxHalf; ++i) {
        const double ang = (double)pos * std::pow(theta, -2.0 * (double)i / (double)head_dim);
        t.c[i] = (float)std::cos(ang);
        t.s[i] = (float)std::sin(ang);
    }
    return t;
}
}  // namespace

sd2_status sd2_add_rmsnorm(const void* a, const void* b, void* sum, const void* w, void* y, int64_t N, int64_t H, float eps,
                           void* cuda_stream)
{
    Range range_("sd2_add_rmsnorm");
    if (!a || !b || !sum || !w || !y) return SD2_ERR_INVALID_ARG;
    if (N < 0 || H < 1 || N > 0x7FFFFFFF || H > 0x7FFFFFFF) return SD2_ERR_SHAPE;
    if (N == 0) return SD2_OK;
    launch_pdl(add_rmsnorm_kernel, (unsigned)N, kGlueThreads, 0, (cudaStream_t)cuda_stream, (const uint16_t*)a, (const uint16_t*)b, (uint16_t*)sum,
                                                                                     (const uint16_t*)w, (uint16_t*)y, (int)H, eps);
    return cudaGetLastError() == cudaSuccess ? SD2_OK : SD2_ERR_CUDA;
}

sd2_status sd2_rope_cache(void* q, const void* k, const void* v, void* k_cache, void* v_cache, int64_t N, int64_t heads_q,
                          int64_t heads_kv, int64_t head_dim, int64_t pos, int64_t T_max, double theta, void* cuda_stream)
{
    if (!q || !k || !v || !k_cache || !v_cache) return SD2_ERR_INVALID_ARG;
    if (N < 0 || heads_q < 1 || heads_kv < 1 || head_dim < 2 || (head_dim & 1) || pos < 0 || pos >= T_max || T_max > 0x7FFFFFFF ||
        heads_q > 65536 || heads_kv > 65536 || head_dim > 8192 || N > 0x7FFFFFFF || !(theta > 0.0))
        return SD2_ERR_SHAPE;
    if (N == 0) return SD2_OK;
    if (head_dim > 2 * kRopeMaxHalf) return SD2_ERR_UNSUPPORTED;
    launch_pdl(rope_cache_kernel, (unsigned)N, kGlueThreads, 0, (cudaStream_t)cuda_stream, (uint16_t*)q, (const uint16_t*)k, (const uint16_t*)v,
                                                                                    (uint16_t*)k_cache, (uint16_t*)v_cache, (int)heads_q,
                                                                                    (int)heads_kv, (int)head_dim, (int)pos, (int)T_max,
                                                                                    rope_table(head_dim, pos, theta));
    return cudaGetLastError() == cudaSuccess ? SD2_OK : SD2_ERR_CUDA;
}

sd2_status sd2_attention_decode(const void* q, const void* k_cache, const void* v_cache, void* out, int64_t N, int64_t heads_q,
                                int64_t heads_kv, int64_t head_dim, int64_t T, int64_t T_max, void* cuda_stream)
{
    Range range_("sd2_attention_decode");
    if (!q || !k_cache || !v_cache || !out) return SD2_ERR_INVALID_ARG;
    if (N < 0 || heads_q < 1 || heads_kv < 1 || heads_q % heads_kv || head_dim < 1 || T < 1 || T > T_max || T_max > 0x7FFFFFFF ||
        N * heads_q > 0x7FFFFFFF)
        return SD2_ERR_SHAPE;
    if (head_dim > 128 || T > kAttnMaxT) return SD2_ERR_UNSUPPORTED;
    if (N == 0) return SD2_OK;
    int sms = 0;
    const sd2_status st = device_sms(&sms);
    if (st != SD2_OK) return st;
    const bool pow2 = (head_dim & (head_dim - 1)) == 0;
    const int vec = (pow2 && head_dim >= 8 && ((((uintptr_t)k_cache) | ((uintptr_t)v_cache)) & 15) == 0) ? 1 : 0;
    if (vec)
        return launch_attention<false>((uint16_t*)q, nullptr, nullptr, (uint16_t*)k_cache, (uint16_t*)v_cache, (uint16_t*)out, N, heads_q,
                                       heads_kv, head_dim, T, T_max, RopeTable{}, sms, (cudaStream_t)cuda_stream);
    launch_pdl(attention_any_kernel, (unsigned)(N * heads_q), kAttnThreads, (size_t)T * 4, (cudaStream_t)cuda_stream,
               (const uint16_t*)q, (const uint16_t*)k_cache, (const uint16_t*)v_cache, (uint16_t*)out, (int)heads_q, (int)heads_kv,
               (int)head_dim, (int)T, (int)T_max);
    return cudaGetLastError() == cudaSuccess ? SD2_OK : SD2_ERR_CUDA;
}

sd2_status sd2_rope_attention(void* q, const void* k, const void* v, void* k_cache, void* v_cache, void* out, int64_t N,
                              int64_t heads_q, int64_t heads_kv, int64_t head_dim, int64_t pos, int64_t T_max, double theta,
                              void* cuda_stream)
{
    Range range_("sd2_rope_attention");
    if (!q || !k || !v || !k_cache || !v_cache || !out) return SD2_ERR_INVALID_ARG;
    if (N < 0 || heads_q < 1 || heads_kv < 1 || heads_q % heads_kv || head_dim < 2 || (head_dim & 1) || pos < 0 || pos >= T_max ||
        T_max > 0x7FFFFFFF || N * heads_q > 0x7FFFFFFF || !(theta > 0.0))
        return SD2_ERR_SHAPE;
    if (head_dim > 128 || pos + 1 > kAttnMaxT) return SD2_ERR_UNSUPPORTED;
    if (N == 0) return SD2_OK;
    int sms = 0;
    const sd2_status st = device_sms(&sms);
    if (st != SD2_OK) return st;
    const bool pow2 = (head_dim & (head_dim - 1)) == 0;
    const int vec = (pow2 && head_dim >= 8 && ((((uintptr_t)k_cache) | ((uintptr_t)v_cache)) & 15) == 0) ? 1 : 0;
    if (vec)
        return launch_attention<true>((uint16_t*)q, (const uint16_t*)k, (const uint16_t*)v, (uint16_t*)k_cache, (uint16_t*)v_cache,
                                      (uint16_t*)out, N, heads_q, heads_kv, head_dim, pos, T_max, rope_table(head_dim, pos, theta),
                                      sms, (cudaStream_t)cuda_stream);
    launch_pdl(rope_attention_any_kernel, (unsigned)(N * heads_q), kAttnThreads, (size_t)(pos + 1) * 4, (cudaStream_t)cuda_stream,
               (uint16_t*)q, (const uint16_t*)k, (const uint16_t*)v, (uint16_t*)k_cache, (uint16_t*)v_cache, (uint16_t*)out, (int)heads_q,
               (int)heads_kv, (int)head_dim, (int)pos, (int)T_max, rope_table(head_dim, pos, theta));
    return cudaGetLastError() == cudaSuccess ? SD2_OK : SD2_ERR_CUDA;
}

sd2_status sd2_add(const void* a, const void* b, void* y, int64_t count, void* cuda_stream)
{
    if (!a || !b || !y) return SD2_ERR_INVALID_ARG;
    if (count < 0) return SD2_ERR_SHAPE;
    if (count == 0) return SD2_OK;
    int64_t grid = (count + kGlueThreads - 1) / kGlueThreads;
    if (grid > 148 * 8) grid = 148 * 8;
    launch_pdl(add_kernel, (unsigned)grid, kGlueThreads, 0, (cudaStream_t)cuda_stream, (const uint16_t*)a, (const uint16_t*)b, (uint16_t*)y, (long long)count);
    return cudaGetLastError() == cudaSuccess ? SD2_OK : SD2_ERR_CUDA;
}

sd2_status sd2_embedding(const int32_t* tokens, const void* table, void* x, int64_t N, int64_t V, int64_t H, void* cuda_stream)
{
    if (!tokens || !table || !x) return SD2_ERR_INVALID_ARG;
    if (N < 0 || V < 1 || H < 1 || N > 0x7FFFFFFF || V > 0x7FFFFFFF || H > 0x7FFFFFFF) return SD2_ERR_SHAPE;
    if (N == 0) return SD2_OK;
    const int vec = ((H & 7) == 0 && ((((uintptr_t)table) | ((uintptr_t)x)) & 15) == 0) ? 1 : 0;
    launch_pdl(embedding_kernel, (unsigned)N, kGlueThreads, 0, (cudaStream_t)cuda_stream, tokens, (const uint16_t*)table, (uint16_t*)x, (int)H, (int)V, vec);
    return cudaGetLastError() == cudaSuccess ? SD2_OK : SD2_ERR_CUDA;
}

sd2_status sd2_lm_head(const void* x, const void* w_out, float* logits, int32_t* tokens, int64_t N, int64_t V, int64_t H,
                       void* cuda_stream)
{
    Range range_("sd2_lm_head");
    if (!x || !w_out || !logits) return SD2_ERR_INVALID_ARG;
    if (N < 0 || V < 1 || H < 1 || V > 0x7FFFFFFF || H > 0x7FFFFFFF) return SD2_ERR_SHAPE;
    if ((H & 7) || (((uintptr_t)w_out) & 15)) return SD2_ERR_UNSUPPORTED;
    if ((size_t)kHeadMaxRows * (size_t)H * 4 > (size_t)kSmemMax) return SD2_ERR_UNSUPPORTED;
    int dev = 0;
    sd2_status st = ensure_device(&dev);
    if (st != SD2_OK) return st;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    for (int64_t n0 = 0; n0 < N; n0 += kHeadMaxRows) {
        const int n = (int)((N - n0) < kHeadMaxRows ? (N - n0) : kHeadMaxRows);
        const uint16_t* xp = (const uint16_t*)x + n0 * H;
        float* lp = logits + n0 * V;
        st = n == 1 ? launch_lm_head<1>(xp, (const uint16_t*)w_out, lp, n, (int)V, (int)H, g_dev[dev].sms, s)
           : n == 2 ? launch_lm_head<2>(xp, (const uint16_t*)w_out, lp, n, (int)V, (int)H, g_dev[dev].sms, s)
           : n <= 4 ? launch_lm_head<4>(xp, (const uint16_t*)w_out, lp, n, (int)V, (int)H, g_dev[dev].sms, s)
                    : launch_lm_head<8>(xp, (const uint16_t*)w_out, lp, n, (int)V, (int)H, g_dev[dev].sms, s);
        if (st != SD2_OK) return st;
    }
    if (tokens && N > 0) {
        const int vec = ((V & 3) == 0 && (((uintptr_t)logits) & 15) == 0) ? 1 : 0;
        launch_pdl(argmax_kernel, (unsigned)(N * kArgmaxCtas), 512, 0, s, logits, tokens, (int)V, vec);
        if (cudaGetLastError() != cudaSuccess) return SD2_ERR_CUDA;
    }
    return SD2_OK;
}

sd2_status sd2_decoder_workspace_bytes(const sd2_handle* h, int64_t N, int64_t* bytes)
{
    if (!bytes) return SD2_ERR_INVALID_ARG;
    if (N < 0 || N > kMaxBlockRows) return SD2_ERR_SHAPE;
    BlockDims d;
    sd2_status st = block_dims(h, &d);
    if (st != SD2_OK) return st;
    int64_t off[8];
    block_layout(h, d, N, off);
    // the linears' intermediates, then xn (normalised input), att (attention output), x1 (after the first residual), down
    *bytes = off[7] + 2 * a256(2 * N * d.hidden) + a256(2 * N * d.q_out) + a256(2 * N * d.out);
    return SD2_OK;
}

sd2_status sd2_decoder_block_step(const sd2_handle* h, const void* norm_attn, const void* norm_ffn, const void* x, void* y,
                                  void* k_cache, void* v_cache, int64_t N, int64_t heads_q, int64_t heads_kv, int64_t pos,
                                  int64_t T_max, float eps, double theta, void* workspace, void* cuda_stream)
{
    Range range_("sd2_decoder_block_step");
    if (!norm_attn || !norm_ffn || !x || !y || !k_cache || !v_cache || !workspace) return SD2_ERR_INVALID_ARG;
    if (N < 0 || N > kMaxBlockRows) return SD2_ERR_SHAPE;
    BlockDims d;
    sd2_status st = block_dims(h, &d);
    if (st != SD2_OK) return st;
    if (heads_q < 1 || heads_kv < 1 || d.q_out % heads_q || d.kv % heads_kv || d.q_out / heads_q != d.kv / heads_kv ||
        d.out != d.hidden || h[3]->M != d.hidden)
        return SD2_ERR_SHAPE;
    if (((uintptr_t)workspace) & 255) return SD2_ERR_INVALID_ARG;
    if (N == 0) return SD2_OK;
    const int64_t hd = d.q_out / heads_q;
    int64_t off[8];
    block_layout(h, d, N, off);
    char* ws = (char*)workspace;
    uint16_t *q = (uint16_t*)(ws + off[0]), *k = (uint16_t*)(ws + off[1]), *v = (uint16_t*)(ws + off[2]);
    uint16_t *hdn = (uint16_t*)(ws + off[3]), *g = (uint16_t*)(ws + off[4]), *u = (uint16_t*)(ws + off[5]), *t = (uint16_t*)(ws + off[6]);
    int64_t o = off[7];
    uint16_t* xn = (uint16_t*)(ws + o); o += a256(2 * N * d.hidden);
    uint16_t* x1 = (uint16_t*)(ws + o); o += a256(2 * N * d.hidden);
    uint16_t* att = (uint16_t*)(ws + o); o += a256(2 * N * d.q_out);
    uint16_t* dn = (uint16_t*)(ws + o);
    cudaStream_t s = (cudaStream_t)cuda_stream;
    bool all_gap4 = true;
    for (int i = 0; i < 7; ++i)
        if (h[i]->format != SD2_FORMAT_GAP4) all_gap4 = false;
    if (all_gap4) {
        // Four launches: (1) q|k|v with the first norm folded into their staging pass, (2) rotation + cache append +
        // attention, (3) one persistent launch for o, gate|up and down, the residual and the second norm folded into
        // the staging pass of gate|up (CTA 0 stores x1 and the normalised row for whoever wants to look), (4) the
        // last residual.
        int dev = 0;
        if ((st = ensure_device(&dev)) != SD2_OK) return st;
        for (int i = 0; i < 7; ++i)
            if (h[i]->device != dev) return SD2_ERR_INVALID_ARG;
        const int grid = g_dev[dev].sms;
        if (use_cells(h, 7, N)) {
            {
                CArgs<kMaxStagesInline> a = {};
                CellBuilder b(a.inl, grid);
                void* yqkv[3] = {q, k, v};
                b.add(h, 3, (const uint16_t*)x, yqkv, true);
                a.fold[0].norm_w = (const uint16_t*)norm_attn;
                a.fold[0].eps = eps;
                a.fold_any = 1;
                Range r_("q|k|v");
                if ((st = run_cell_program(a, b, dev, N, s)) != SD2_OK) return st;
            }
            if ((st = sd2_rope_attention(q, k, v, k_cache, v_cache, att, N, heads_q, heads_kv, hd, pos, T_max, theta, s)) != SD2_OK) return st;
            {
                CArgs<kMaxStagesInline> a = {};
                CellBuilder b(a.inl, grid);
                void* yo[1] = {hdn};
                void* ygu[2] = {g, u};
                void* yd[1] = {dn};
                b.add(h + 3, 1, att, yo, true);
                SFold& f = a.fold[b.n];
                f.res = (const uint16_t*)x;
                f.norm_w = (const uint16_t*)norm_ffn;
                f.eps = eps;
                f.sum_out = x1;
                f.norm_out = xn;
                a.fold_any = 1;
                b.add(h + 4, 2, hdn, ygu, true, true).t_out = t;
                b.add(h + 6, 1, t, yd, true);
                Range r_("o, gate|up, down");
                if ((st = run_cell_program(a, b, dev, N, s)) != SD2_OK) return st;
            }
            return sd2_add(x1, dn, y, N * d.hidden, s);
        }
        {
            SArgs a;
            std::memset(&a, 0, sizeof a);
            ProgramNeeds needs;
            void* yqkv[3] = {q, k, v};
            a.n_stages = append_group(a.inl, 0, &needs, h, 3, (const uint16_t*)x, nullptr, nullptr, nullptr, yqkv, true, grid);
            for (int i = 0; i < a.n_stages; ++i) {
                a.fold[i].norm_w = (const uint16_t*)norm_attn;
                a.fold[i].eps = eps;
            }
            a.fold_any = 1;
            Range r_("q|k|v");
            if ((st = run_program(a, dev, N, needs, s)) != SD2_OK) return st;
        }
        if ((st = sd2_rope_attention(q, k, v, k_cache, v_cache, att, N, heads_q, heads_kv, hd, pos, T_max, theta, s)) != SD2_OK) return st;
        {
            SArgs a;
            std::memset(&a, 0, sizeof a);
            ProgramNeeds needs;
            void* yo[1] = {hdn};
            void* ygu[2] = {g, u};
            void* yd[1] = {dn};
            int n = append_group(a.inl, 0, &needs, h + 3, 1, att, nullptr, nullptr, nullptr, yo, true, grid);
            const int first_gu = n;
            n = append_group(a.inl, n, &needs, h + 4, 2, hdn, nullptr, nullptr, nullptr, ygu, true, grid);
            for (int i = first_gu; i < n; ++i) {
                a.fold[i].res = (const uint16_t*)x;
                a.fold[i].norm_w = (const uint16_t*)norm_ffn;
                a.fold[i].eps = eps;
                a.fold[i].sum_out = x1;
                a.fold[i].norm_out = xn;
            }
            a.fold_any = 1;
            n = append_group(a.inl, n, &needs, h + 6, 1, nullptr, g, u, t, yd, true, grid);
            a.n_stages = n;
            Range r_("o, gate|up, down");
            if ((st = run_program(a, dev, N, needs, s)) != SD2_OK) return st;
        }
        return sd2_add(x1, dn, y, N * d.hidden, s);
    }
    // attention module: x1 = x + Wo attention(rope(Wq n), cache + rope(Wk n), cache + Wv n), n = rmsnorm(x)
    if ((st = sd2_rmsnorm(x, norm_attn, xn, N, d.hidden, eps, s)) != SD2_OK) return st;
    void* yqkv[3] = {q, k, v};
    nvtxRangePushA("q|k|v");
    st = run_group(h, 3, xn, nullptr, nullptr, nullptr, yqkv, N, true, s);
    nvtxRangePop();
    if (st != SD2_OK) return st;
    if ((st = sd2_rope_attention(q, k, v, k_cache, v_cache, att, N, heads_q, heads_kv, hd, pos, T_max, theta, s)) != SD2_OK) return st;
    void* yo[1] = {hdn};
    nvtxRangePushA("o");
    st = run_group(h + 3, 1, att, nullptr, nullptr, nullptr, yo, N, true, s);
    nvtxRangePop();
    if (st != SD2_OK) return st;
    // feed-forward module: y = x1 + Wd (silu(Wg m) * Wu m), m = rmsnorm(x1); the residual and the norm in one launch
    if ((st = sd2_add_rmsnorm(x, hdn, x1, norm_ffn, xn, N, d.hidden, eps, s)) != SD2_OK) return st;
    void* ygu[2] = {g, u};
    nvtxRangePushA("gate|up");
    st = run_group(h + 4, 2, xn, nullptr, nullptr, nullptr, ygu, N, true, s);
    nvtxRangePop();
    if (st != SD2_OK) return st;
    void* yd[1] = {dn};
    nvtxRangePushA("down");
    st = run_group(h + 6, 1, nullptr, g, u, t, yd, N, true, s);
    nvtxRangePop();
    if (st != SD2_OK) return st;
    return sd2_add(x1, dn, y, N * d.hidden, s);
}

sd2_status sd2_debug_fail_allocations(int64_t skip, int64_t fail)
{
    if (skip < 0 || fail < 0) return SD2_ERR_INVALID_ARG;
    std::lock_guard<std::mutex> lk(g_mu);
    alloc_plan().skip_left = skip;
    alloc_plan().fail_left = fail;
    return SD2_OK;
}

sd2_status sd2_selftest_timeout(void* cuda_stream)
{
    int dev = 0;
    sd2_status st = ensure_device(&dev);
    if (st != SD2_OK) return st;
    wait_selftest_kernel<<<1, 32, 0, (cudaStream_t)cuda_stream>>>(g_dev[dev].err_word, wait_budget(dev));
    if (cudaGetLastError() != cudaSuccess) return SD2_ERR_CUDA;
    return SD2_OK;
}

sd2_status sd2_spmm(sd2_handle h, const void* X, void* Y, int64_t N, void* cuda_stream)
{
    Range range_("sd2_spmm");
    if (!X || !Y) return SD2_ERR_INVALID_ARG;
    void* ys[1] = {Y};
    return run_group(&h, 1, (const uint16_t*)X, nullptr, nullptr, nullptr, ys, N, false, (cudaStream_t)cuda_stream);
}

sd2_status sd2_spmm_query(sd2_handle h, int64_t N, int64_t* out)
{
    if (!live(h) || !out) return SD2_ERR_INVALID_ARG;
    if (N < 1) return SD2_ERR_SHAPE;
    int path = SD2_PATH_STRIPS, cap = 0;
    if (h->format == SD2_FORMAT_BITMASK) {
        path = SD2_PATH_BITMASK;
        cap = 8;
    } else if (h->format == SD2_FORMAT_GAP4_MMA) {
        path = SD2_PATH_MMA;
        cap = kMmaMaxRows;
    } else if (use_cells(&h, 1, N)) {
        path = SD2_PATH_CELLS;
        CellNeeds needs;
        needs.add(h);
        cap = widest_cell_panel(needs, kWidePanelRows);
    } else {
        ProgramNeeds needs;
        needs.add(&h, 1);
        cap = widest_panel(needs.xs_need, needs.K_max, needs.max_tile);
    }
    if (cap == 0) return SD2_ERR_UNSUPPORTED;
    out[0] = (N + cap - 1) / cap;
    out[1] = cap;
    out[2] = h->device_bytes;
    out[3] = path == SD2_PATH_CELLS || path == SD2_PATH_MMA ? h->cell_bytes : h->compressed_bytes;
    out[4] = path;
    return SD2_OK;
}

sd2_status sd2_spmm_fused(const sd2_handle* h, int32_t count, const void* X, void* const* Y, int64_t N,
                          void* cuda_stream)
{
    Range range_("sd2_spmm_fused");
    if (!h || !X || !Y) return SD2_ERR_INVALID_ARG;
    return run_group(h, count, (const uint16_t*)X, nullptr, nullptr, nullptr, Y, N, false, (cudaStream_t)cuda_stream);
}

sd2_status sd2_block_workspace_bytes(const sd2_handle* h, int64_t N, int64_t* bytes)
{
    if (!bytes) return SD2_ERR_INVALID_ARG;
    if (N < 0 || N > kMaxBlockRows) return SD2_ERR_SHAPE;
    BlockDims d;
    sd2_status st = block_dims(h, &d);
    if (st != SD2_OK) return st;
    int64_t off[8];
    block_layout(h, d, N, off);
    *bytes = off[7];
    return SD2_OK;
}

sd2_status sd2_block_workspace_layout(const sd2_handle* h, int64_t N, int64_t* offsets)
{
    if (!offsets) return SD2_ERR_INVALID_ARG;
    if (N < 0 || N > kMaxBlockRows) return SD2_ERR_SHAPE;
    BlockDims d;
    sd2_status st = block_dims(h, &d);
    if (st != SD2_OK) return st;
    int64_t off[8];
    block_layout(h, d, N, off);
    for (int i = 0; i < 7; ++i) offsets[i] = off[i];
    return SD2_OK;
}

sd2_status sd2_block_step(const sd2_handle* h, const void* x, void* y, int64_t N, void* workspace, void* cuda_stream)
{
    Range range_("sd2_block_step");
    if (!x || !y || !workspace) return SD2_ERR_INVALID_ARG;
    if (N < 0 || N > kMaxBlockRows) return SD2_ERR_SHAPE;
    BlockDims d;
    sd2_status st = block_dims(h, &d);
    if (st != SD2_OK) return st;
    if (N == 0) return SD2_OK;
    if (((uintptr_t)workspace) & 255) return SD2_ERR_INVALID_ARG;
    int64_t off[8];
    block_layout(h, d, N, off);
    char* ws = (char*)workspace;
    uint16_t* q = (uint16_t*)(ws + off[0]);
    uint16_t* k = (uint16_t*)(ws + off[1]);
    uint16_t* v = (uint16_t*)(ws + off[2]);
    uint16_t* hdn = (uint16_t*)(ws + off[3]);
    uint16_t* g = (uint16_t*)(ws + off[4]);
    uint16_t* u = (uint16_t*)(ws + off[5]);
    uint16_t* t = (uint16_t*)(ws + off[6]);
    cudaStream_t s = (cudaStream_t)cuda_stream;
    bool all_gap4 = true;
    for (int i = 0; i < 7; ++i)
        if (h[i]->format != SD2_FORMAT_GAP4) all_gap4 = false;
    if (all_gap4) {
        // one persistent launch: the stages of the block separated by grid barriers
        int dev = 0;
        st = ensure_device(&dev);
        if (st != SD2_OK) return st;
        for (int i = 0; i < 7; ++i)
            if (h[i]->device != dev) return SD2_ERR_INVALID_ARG;
        if (use_cells(h, 7, N)) {
            return run_block_cells(h, (const uint16_t*)x, q, k, v, hdn, g, u, t, y, nullptr, dev, N, s);
        }
        SArgs a;
        std::memset(&a, 0, sizeof a);
        ProgramNeeds needs;
        a.n_stages = append_block_stages(a.inl, h, (const uint16_t*)x, q, k, v, hdn, g, u, t, y, false, &needs, g_dev[dev].sms);
        return run_program(a, dev, N, needs, s);
    }
    void* y_qkv[3] = {q, k, v};
    st = run_group(h + 0, 3, (const uint16_t*)x, nullptr, nullptr, nullptr, y_qkv, N, true, s);
    if (st != SD2_OK) return st;
    void* y_o[1] = {hdn};
    st = run_group(h + 3, 1, q, nullptr, nullptr, nullptr, y_o, N, true, s);
    if (st != SD2_OK) return st;
    void* y_gu[2] = {g, u};
    st = run_group(h + 4, 2, hdn, nullptr, nullptr, nullptr, y_gu, N, true, s);
    if (st != SD2_OK) return st;
    void* y_d[1] = {y};
    return run_group(h + 6, 1, nullptr, g, u, t, y_d, N, false, s);
}

// ---- block step without allocation -----------------------------------------------------

// Scratch of sd2_block_step_static: grid-barrier words (first 256 bytes), then the block's
// intermediates.  It lives in the library image, so every GPU that loads the library holds
// it until the process exits.
constexpr int64_t kStaticWorkspaceMax = 1 << 20;
static __device__ __align__(256) unsigned char g_static_scratch[256 + kStaticWorkspaceMax];

namespace {
unsigned char* g_static_ptr[kMaxDevices];   // device address of g_static_scratch, per device
}

sd2_status sd2_block_step_static(const sd2_handle* h, const void* x, void* y, int64_t N, void* cuda_stream)
{
    Range range_("sd2_block_step_static");
    if (!x || !y) return SD2_ERR_INVALID_ARG;
    if (N < 0 || N > kMaxBlockRows) return SD2_ERR_SHAPE;
    BlockDims d;
    sd2_status st = block_dims(h, &d);
    if (st != SD2_OK) return st;
    if (N == 0) return SD2_OK;
    for (int i = 0; i < 7; ++i)
        if (h[i]->format != SD2_FORMAT_GAP4) return SD2_ERR_UNSUPPORTED;
    int64_t off[8];
    block_layout(h, d, N, off);
    if (off[7] > kStaticWorkspaceMax) return SD2_ERR_UNSUPPORTED;   // intermediates do not fit the built-in scratch
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return SD2_ERR_CUDA; }
    if (dev < 0 || dev >= kMaxDevices || !g_dev[dev].ready) return SD2_ERR_INVALID_ARG;   // live handles imply a ready device
    for (int i = 0; i < 7; ++i)
        if (h[i]->device != dev) return SD2_ERR_INVALID_ARG;
    {
        // once per device, with that device current: the array's name is only a host-side stand-in
        std::lock_guard<std::mutex> lk(g_mu);
        if (!g_static_ptr[dev]) {
            unsigned char* p = nullptr;
            if (cudaGetSymbolAddress((void**)&p, g_static_scratch) != cudaSuccess || !p) { cudaGetLastError(); return SD2_ERR_CUDA; }
            g_static_ptr[dev] = p;
        }
    }
    unsigned char* base = g_static_ptr[dev];
    cudaStream_t s = (cudaStream_t)cuda_stream;
    // the barrier words must start at zero whatever the last call left behind
    if (cudaMemsetAsync(base, 0, 256, s) != cudaSuccess) { cudaGetLastError(); return SD2_ERR_CUDA; }
    char* ws = (char*)base + 256;
    if (use_cells(h, 7, N)) {
        return run_block_cells(h, (const uint16_t*)x, (uint16_t*)(ws + off[0]), (uint16_t*)(ws + off[1]), (uint16_t*)(ws + off[2]),
                               (uint16_t*)(ws + off[3]), (uint16_t*)(ws + off[4]), (uint16_t*)(ws + off[5]), (uint16_t*)(ws + off[6]), y,
                               (unsigned int*)base, dev, N, s);
    }
    SArgs a;
    std::memset(&a, 0, sizeof a);
    ProgramNeeds needs;
    a.n_stages = append_block_stages(a.inl, h, (const uint16_t*)x, (uint16_t*)(ws + off[0]), (uint16_t*)(ws + off[1]),
                                     (uint16_t*)(ws + off[2]), (uint16_t*)(ws + off[3]), (uint16_t*)(ws + off[4]),
                                     (uint16_t*)(ws + off[5]), (uint16_t*)(ws + off[6]), y, false, &needs, g_dev[dev].sms);
    a.err = g_dev[dev].err_word;
    a.wait_cycles = wait_budget(dev);
    a.free_tiles = needs.free_tiles(g_dev[dev].sms);
    a.gbar = (unsigned int*)base;
    return run_panels(a, N, needs.xs_need, needs.K_max, needs.max_tile, g_dev[dev].sms, s);
}

// ---- whole drafter ---------------------------------------------------------------------

sd2_status sd2_drafter_create(const sd2_handle* h, int32_t L, int64_t n_max, sd2_drafter* out)
{
    if (!h || !out) return SD2_ERR_INVALID_ARG;
    if (L < 1 || L > 4096 || n_max < 1 || n_max > 64) return SD2_ERR_SHAPE;
    int dev = 0;
    sd2_status st = ensure_device(&dev);
    if (st != SD2_OK) return st;
    std::vector<BlockDims> dims((size_t)L);
    for (int b = 0; b < L; ++b) {
        st = block_dims(h + 7 * b, &dims[(size_t)b]);
        if (st != SD2_OK) return st;
        for (int i = 0; i < 7; ++i) {
            if (h[7 * b + i]->format != SD2_FORMAT_GAP4) return SD2_ERR_UNSUPPORTED;
            if (h[7 * b + i]->device != dev) return SD2_ERR_INVALID_ARG;
        }
        if (b > 0 && dims[(size_t)b].hidden != dims[(size_t)b - 1].out) return SD2_ERR_SHAPE;
    }
    sd2_drafter d = lib_alloc_fails() ? nullptr : new (std::nothrow) sd2_drafter_s();
    if (!d) return SD2_ERR_ALLOC;
    d->L = L;
    d->device = dev;
    d->n_max = n_max;
    d->hidden = dims[0].hidden;
    d->out_dim = dims[(size_t)L - 1].out;
    d->y_f32 = h[7 * (L - 1) + 6]->y_dtype == SD2_DTYPE_F32;
    d->handles.assign(h, h + 7 * (size_t)L);
    d->d_ws = nullptr;
    d->d_stages = nullptr;
    d->d_gbar = nullptr;
    d->d_cstages = nullptr;
    d->d_cbar = nullptr;
    d->n_cstages = 0;
    // workspace: per block q,k,v,hdn,g,u,t and the block's bf16 output (the next block's input)
    d->ws_off.assign((size_t)L * 8 + 1, 0);
    int64_t o = 0;
    for (int b = 0; b < L; ++b) {
        int64_t off[8];
        block_layout(h + 7 * b, dims[(size_t)b], n_max, off);
        for (int i = 0; i < 7; ++i) d->ws_off[(size_t)b * 8 + i] = o + off[i];
        d->ws_off[(size_t)b * 8 + 7] = o + off[7];
        o = a256(o + off[7] + 2 * n_max * dims[(size_t)b].out);
    }
    // A launch replaces the input of its first stage.  Where q, k and v of the first block are cut into strips differently they take a
    // stage each, and read a copy.  (A condition in the kernel, for which stages to replace it, cost every single launch 0.04 us of 4.84.)
    d->x_off = -1;
    if (h[1]->S != h[0]->S || h[2]->S != h[0]->S) {
        d->x_off = o;
        o = a256(o + 2 * n_max * d->hidden);
    }
    d->ws_off[(size_t)L * 8] = o;
    std::vector<SStage> stages((size_t)L * 7);
    ProgramNeeds needs;
    bool ok = dev_malloc((void**)&d->d_ws, (size_t)o) == cudaSuccess && cudaMemset(d->d_ws, 0, (size_t)o) == cudaSuccess;
    // Tagged hand-off (stage tags are 8 bits wide): per block q, hdn, g, u, out as 32-bit words.  A stage waits for the tag of the one before
    // it, so weights that share an input must share a stage, which they do not where they are cut into strips differently (q of 4096 x
    // 4096 and k of 1024 x 4096: 16 and 32): such a drafter's stages meet at grid barriers.
    bool tagged = 7 * L <= 254;
    for (int i = 0; i < L; ++i) {
        const sd2_handle* b = h + 7 * i;
        if (b[1]->S != b[0]->S || b[2]->S != b[0]->S || b[5]->S != b[4]->S) tagged = false;
    }
    std::vector<int64_t> tag_off((size_t)L * 6 + 1, 0);
    d->d_tags = nullptr;
    d->tags_bytes = 0;
    if (tagged) {
        int64_t to = 0;
        for (int b = 0; b < L; ++b) {
            const BlockDims& bd = dims[(size_t)b];
            const int64_t w[6] = {bd.q_out, h[7 * b + 3]->M, bd.inter, bd.inter, bd.out, bd.inter};
            for (int i = 0; i < 6; ++i) {
                tag_off[(size_t)b * 6 + i] = to;
                to = a256(to + 4 * n_max * w[i]);
            }
        }
        d->tags_bytes = to;
        ok = ok && dev_malloc((void**)&d->d_tags, (size_t)to) == cudaSuccess && cudaMemset(d->d_tags, 0, (size_t)to) == cudaSuccess;
    }
    int n = 0;
    std::vector<sd2_handle> pairs((size_t)L, nullptr);
    if (ok && tagged) {
        for (int b = 0; b < L && st == SD2_OK; ++b) {
            st = build_gate_up_pair(h[7 * b + 4], h[7 * b + 5], &pairs[(size_t)b]);
            if (pairs[(size_t)b]) { d->owned.push_back(pairs[(size_t)b]); d->pair_block.push_back(b); }
        }
        if (st != SD2_OK) {
            for (sd2_handle p : d->owned) sd2_free(p);
            cudaFree(d->d_ws); cudaFree(d->d_tags);
            cudaGetLastError();
            delete d;
            return st;
        }
    }
    if (ok) {
        for (int b = 0; b < L; ++b) {
            uint8_t* base = d->d_ws;
            const int64_t* wo = &d->ws_off[(size_t)b * 8];
            const int64_t x_off = b == 0 ? d->x_off : d->ws_off[(size_t)(b - 1) * 8 + 7];
            const uint16_t* xin = x_off < 0 ? nullptr : (const uint16_t*)(base + x_off);
            void* yout = base + wo[7];
            BlockTags tg;
            if (tagged) {
                uint8_t* tb = (uint8_t*)d->d_tags;
                const int64_t* to = &tag_off[(size_t)b * 6];
                tg.x_t = b == 0 ? nullptr : (const uint32_t*)(tb + tag_off[(size_t)(b - 1) * 6 + 4]);
                tg.q_t = (uint32_t*)(tb + to[0]);
                tg.hdn_t = (uint32_t*)(tb + to[1]);
                tg.g_t = (uint32_t*)(tb + to[2]);
                tg.u_t = (uint32_t*)(tb + to[3]);
                tg.out_t = b + 1 < L ? (uint32_t*)(tb + to[4]) : nullptr;
                tg.t_t = (uint32_t*)(tb + to[5]);
            }
            n += append_block_stages(stages.data() + n, h + 7 * b, xin, (uint16_t*)(base + wo[0]), (uint16_t*)(base + wo[1]),
                                     (uint16_t*)(base + wo[2]), (uint16_t*)(base + wo[3]), (uint16_t*)(base + wo[4]),
                                     (uint16_t*)(base + wo[5]), (uint16_t*)(base + wo[6]), yout, b + 1 < L, &needs, g_dev[dev].sms,
                                     tagged ? &tg : nullptr, pairs[(size_t)b]);
        }
        d->n_stages = n;
        d->first_stage = stages[0];
        ok = dev_malloc((void**)&d->d_stages, sizeof(SStage) * (size_t)n) == cudaSuccess &&
             cudaMemcpy(d->d_stages, stages.data(), sizeof(SStage) * (size_t)n, cudaMemcpyHostToDevice) == cudaSuccess &&
             dev_malloc((void**)&d->d_gbar, kDrafterWordsBytes) == cudaSuccess && cudaMemset(d->d_gbar, 0, kDrafterWordsBytes) == cudaSuccess;
    }
    bool cells = true;
    for (const sd2_handle hh : d->handles)
        if (!hh->d_image) cells = false;
    if (ok && cells && n_max >= 2) {
        // the same blocks over cells, for steps of several rows
        std::vector<CStage> cstages((size_t)L * 4);
        CellBuilder bld(cstages.data(), g_dev[dev].sms);
        for (int b = 0; b < L; ++b) {
            uint8_t* base = d->d_ws;
            const int64_t* wo = &d->ws_off[(size_t)b * 8];
            const uint16_t* xin = b == 0 ? nullptr : (const uint16_t*)(base + d->ws_off[(size_t)(b - 1) * 8 + 7]);
            append_block_cells(bld, h + 7 * b, xin, (uint16_t*)(base + wo[0]), (uint16_t*)(base + wo[1]), (uint16_t*)(base + wo[2]),
                               (uint16_t*)(base + wo[3]), (uint16_t*)(base + wo[4]), (uint16_t*)(base + wo[5]), (uint16_t*)(base + wo[6]),
                               base + wo[7], b + 1 < L);
        }
        d->n_cstages = bld.n;
        d->first_cstage = cstages[0];
        d->cell_needs = bld.needs;
        if (dev_malloc((void**)&d->d_cstages, sizeof(CStage) * (size_t)bld.n) == cudaSuccess && dev_malloc((void**)&d->d_cbar, kDrafterWordsBytes) == cudaSuccess) {
            ok = cudaMemcpy(d->d_cstages, cstages.data(), sizeof(CStage) * (size_t)bld.n, cudaMemcpyHostToDevice) == cudaSuccess &&
                 cudaMemset(d->d_cbar, 0, kDrafterWordsBytes) == cudaSuccess;
        } else {                                             // no memory: steps of several rows go through the strips
            cudaGetLastError();
            cudaFree(d->d_cstages);
            d->d_cstages = nullptr;
            d->n_cstages = 0;
        }
    }
    auto drop = [&]() {
        cudaGetLastError();
        for (sd2_handle p : d->owned) sd2_free(p);
        cudaFree(d->d_ws); cudaFree(d->d_stages); cudaFree(d->d_gbar); cudaFree(d->d_tags);
        cudaFree(d->d_cstages); cudaFree(d->d_cbar);
        cudaGetLastError();
    };
    if (ok && widest_panel(needs.xs_need, needs.K_max, needs.max_tile) == 0) {
        drop();
        delete d;
        return SD2_ERR_UNSUPPORTED;
    }
    if (!ok) {
        drop();
        delete d;
        return SD2_ERR_ALLOC;
    }
    d->K_max = needs.K_max;
    d->free_tiles = needs.free_tiles(g_dev[dev].sms);
    d->max_tile = needs.max_tile;
    for (int w = 0; w < 3; ++w) d->xs_need[w] = needs.xs_need[w];
    {
        std::lock_guard<std::mutex> lk(g_mu);
        g_live_drafters.insert(d);
    }
    *out = d;
    return SD2_OK;
}

namespace {
bool drafter_uses_cells(sd2_drafter d, int64_t N)
{
    return d->d_cstages && cells_pay(d->handles.data(), 7 * d->L, N) && widest_cell_panel(d->cell_needs) > 0;
}
}  // namespace

sd2_status sd2_drafter_step(sd2_drafter d, const void* x, void* y, int64_t N, void* cuda_stream)
{
    Range range_("sd2_drafter_step");
    if (!live(d) || !x || !y) return SD2_ERR_INVALID_ARG;
    if (N < 0 || N > d->n_max) return SD2_ERR_SHAPE;
    if (N == 0) return SD2_OK;
    int dev = 0;
    sd2_status st = ensure_device(&dev);
    if (st != SD2_OK) return st;
    if (dev != d->device) return SD2_ERR_INVALID_ARG;
    if (drafter_uses_cells(d, N)) {
        CArgs<kMaxStagesInline> c = {};
        c.ext = d->d_cstages;
        c.inl[0] = d->first_cstage;
        c.n_stages = d->n_cstages;
        c.x_in = (const uint16_t*)x;
        c.y_out = y;
        c.gbar = d->d_cbar;
        c.err = g_dev[dev].err_word;
        c.wait_cycles = wait_budget(dev);
        return run_cell_panels(c, N, d->cell_needs, 2 * (g_dev[dev].sms / 2), (cudaStream_t)cuda_stream);
    }
    SArgs a;
    std::memset(&a, 0, sizeof a);
    a.ext = d->d_stages;
    a.inl[0] = d->first_stage;
    a.n_stages = d->n_stages;
    a.x_in = (const uint16_t*)x;
    if (d->x_off >= 0) {
        a.x_in = nullptr;
        if (cudaMemcpyAsync(d->d_ws + d->x_off, x, (size_t)(2 * N * d->hidden), cudaMemcpyDefault, (cudaStream_t)cuda_stream) != cudaSuccess) {
            cudaGetLastError();
            return SD2_ERR_CUDA;
        }
    }
    a.y_out = y;
    a.gbar = d->d_gbar;
    a.free_tiles = d->free_tiles;
    a.err = g_dev[dev].err_word;
    a.wait_cycles = wait_budget(dev);
    if (d->d_tags) {
        a.tagged = 1;
        // How often each activation row has been produced is the first half of every tag.  A word left by
        // an earlier launch (or by launches that covered other rows) can never show the tag this launch
        // waits for: a row's count moves only when the row is produced, so its previous tag is always one
        // behind.  Steps of any N, eager or replayed from a CUDA graph, can therefore follow each other.
        a.rowseq = d->d_gbar + 64;
    }
    // Rows of X are independent through the whole drafter: panels run one after another.  Row n
    // of every buffer starts at n * width, whatever N is.
    return run_panels(a, N, d->xs_need, d->K_max, d->max_tile, g_dev[dev].sms, (cudaStream_t)cuda_stream);
}

sd2_status sd2_drafter_query(sd2_drafter d, int64_t N, int64_t* out)
{
    if (!live(d) || !out) return SD2_ERR_INVALID_ARG;
    if (N < 1 || N > d->n_max) return SD2_ERR_SHAPE;
    const bool cells = drafter_uses_cells(d, N);
    const int cap = cells ? widest_cell_panel(d->cell_needs) : widest_panel(d->xs_need, d->K_max, d->max_tile);
    if (cap == 0) return SD2_ERR_UNSUPPORTED;
    int64_t streamed = 0, owned = 0, kept = 0;
    // what a step streams: every handle once, except that a block's gate and up are read from the
    // drafter's own paired stack where it has one
    std::vector<char> paired((size_t)d->L, 0);
    for (sd2_handle p : d->owned) { streamed += p->compressed_bytes; owned += p->device_bytes; }
    owned += (int64_t)sizeof(CStage) * d->n_cstages + (d->d_cbar ? kDrafterWordsBytes : 0);
    size_t oi = 0;
    for (int b = 0; b < d->L; ++b) {
        // (owned stacks were built in block order, one per block that could be paired)
        const bool has_pair = oi < d->owned.size() && d->owned[oi]->M == 2 * d->handles[(size_t)7 * b + 4]->M &&
                              d->pair_block.size() > oi && d->pair_block[oi] == b;
        if (has_pair) ++oi;
        for (int i = 0; i < 7; ++i) {
            const sd2_handle h = d->handles[(size_t)7 * b + i];
            kept += h->nnz;
            if (!(has_pair && (i == 4 || i == 5))) streamed += h->compressed_bytes;
        }
    }
    if (cells) {
        streamed = 0;
        for (const sd2_handle h : d->handles) streamed += h->cell_bytes;
    }
    out[0] = (N + cap - 1) / cap;                                  // launches per step of N rows
    out[1] = cap;                                                  // rows of the widest panel
    out[2] = owned + d->ws_off.back() + d->tags_bytes + (int64_t)sizeof(SStage) * d->n_stages + kDrafterWordsBytes;
    out[3] = streamed;                                             // bytes of compressed weights read per launch
    out[4] = cells ? d->n_cstages : d->n_stages;
    out[5] = kept;
    return SD2_OK;
}

sd2_status sd2_drafter_buffers(sd2_drafter d, int32_t block, void** ptrs)
{
    if (!live(d) || !ptrs) return SD2_ERR_INVALID_ARG;
    if (block < 0 || block >= d->L) return SD2_ERR_SHAPE;
    for (int i = 0; i < 8; ++i) ptrs[i] = d->d_ws + d->ws_off[(size_t)block * 8 + i];
    return SD2_OK;
}

sd2_status sd2_drafter_free(sd2_drafter d)
{
    if (!d) return SD2_ERR_INVALID_ARG;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (!g_live_drafters.erase(d)) return SD2_ERR_INVALID_ARG;
    }
    sd2_status st = SD2_OK;
    if (cudaFree(d->d_ws) != cudaSuccess) st = SD2_ERR_CUDA;
    if (cudaFree(d->d_stages) != cudaSuccess) st = SD2_ERR_CUDA;
    if (cudaFree(d->d_gbar) != cudaSuccess) st = SD2_ERR_CUDA;
    if (d->d_tags && cudaFree(d->d_tags) != cudaSuccess) st = SD2_ERR_CUDA;
    if (d->d_cstages && cudaFree(d->d_cstages) != cudaSuccess) st = SD2_ERR_CUDA;
    if (d->d_cbar && cudaFree(d->d_cbar) != cudaSuccess) st = SD2_ERR_CUDA;
    for (sd2_handle p : d->owned)
        if (sd2_free(p) != SD2_OK) st = SD2_ERR_CUDA;
    cudaGetLastError();
    delete d;
    return st;
}

}  // extern "C"
