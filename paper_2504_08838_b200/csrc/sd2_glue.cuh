// Glue of one drafter decode step around the sparse linears: RMSNorm, rotary embedding with the
// key/value cache append, grouped-query attention of one new token over the cache, residual add,
// embedding look-up, dense LM head with greedy token.  The paper leaves the embedding and the LM
// head dense (Section "Results") and says a block is an attention module and a feed-forward module
// (Section "Layer pruning"); what those compute is the published definition of the Llama / Qwen
// family.  All of it is small beside the linears (activations of a few KB per row), except the LM
// head, which streams vocab x hidden bf16 weights from HBM once per step.
//
// bf16 in and out, fp32 arithmetic (rotary angles in fp64), one rounding per output.

#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "sd2_kernels.cuh"

namespace sd2 {

constexpr int kGlueThreads = 256;
constexpr int kAttnThreads = 256;
constexpr int kAttnMaxT = 8192;            // cached positions whose scores fit the kernel's shared memory
constexpr int kHeadMaxRows = 8;            // activation rows one LM-head launch keeps in shared memory
constexpr int kRopeMaxHalf = 64;           // head widths up to 128

// cos and sin of the head_dim / 2 rotary angles of one position, computed on the host in fp64 (pos * theta^(-2i/d))
// and handed to the kernels by value: no double-precision transcendental on the device
struct RopeTable {
    float c[kRopeMaxHalf];
    float s[kRopeMaxHalf];
};

__device__ __forceinline__ float block_sum(float v, float* red)
{
    for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    float t = l < nw ? red[l] : 0.f;
    for (int d = 16; d > 0; d >>= 1) t += __shfl_xor_sync(0xFFFFFFFFu, t, d);
    return t;
}

__device__ __forceinline__ float block_max(float v, float* red)
{
    for (int d = 16; d > 0; d >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, d));
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
    __syncthreads();
    if (l == 0) red[w] = v;
    __syncthreads();
    float t = l < nw ? red[l] : -INFINITY;
    for (int d = 16; d > 0; d >>= 1) t = fmaxf(t, __shfl_xor_sync(0xFFFFFFFFu, t, d));
    return t;
}

// the squares of eight values, added to `ss` in the order that every instance below has
__device__ __forceinline__ float add_squares(float ss, uint4 v)
{
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) ss += bf16_lo(u[j]) * bf16_lo(u[j]) + bf16_hi(u[j]) * bf16_hi(u[j]);
    return ss;
}

// y[n, :] = x[n, :] / sqrt(mean(x[n, :]^2) + eps) * w;  one CTA per row.
// HELD > 0: H is a multiple of 8 and x, w, y are 16-byte aligned, so a thread moves eight values per load, and holds its share of row
// and gains, up to HELD such loads of each, from one round of loads to the stores.  kNormLoop: the same for any H; the second pass finds
// the row in L1.  kNormPlain: two bytes at a time.  What bounds it is the latency of the loads for a few rows and HBM for many, where
// registers that a narrow row has no use for keep CTAs off the SM: hence an instance for every number of loads.
constexpr int kNormLoop = 0, kNormPlain = -1;
template <int HELD>
__global__ void __launch_bounds__(kGlueThreads) rmsnorm_kernel(const uint16_t* x, const uint16_t* w, uint16_t* y, int H, float eps)
{
    pdl_let_next_start();
    pdl_wait();
    __shared__ float red[32];
    const uint16_t* xr = x + (size_t)blockIdx.x * H;
    uint16_t* yr = y + (size_t)blockIdx.x * H;
    float ss = 0.f;
    if constexpr (HELD > 0) {
        uint4 v[HELD], g[HELD];
#pragma unroll
        for (int k = 0; k < HELD; ++k) {
            const int i = threadIdx.x + k * kGlueThreads;
            v[k] = i < H / 8 ? ((const uint4*)xr)[i] : make_uint4(0u, 0u, 0u, 0u);
            g[k] = i < H / 8 ? ((const uint4*)w)[i] : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int k = 0; k < HELD; ++k) ss = add_squares(ss, v[k]);
        const float r = rsqrtf(block_sum(ss, red) / (float)H + eps);
#pragma unroll
        for (int k = 0; k < HELD; ++k) {
            const int i = threadIdx.x + k * kGlueThreads;
            if (i < H / 8) ((uint4*)yr)[i] = scale_bf16_row(v[k], r, g[k]);
        }
    } else if constexpr (HELD == kNormLoop) {
        for (int i = threadIdx.x; i < H / 8; i += kGlueThreads) ss = add_squares(ss, ((const uint4*)xr)[i]);
        const float r = rsqrtf(block_sum(ss, red) / (float)H + eps);
        for (int i = threadIdx.x; i < H / 8; i += kGlueThreads) ((uint4*)yr)[i] = scale_bf16_row(((const uint4*)xr)[i], r, ((const uint4*)w)[i]);
    } else {
        for (int i = threadIdx.x; i < H; i += kGlueThreads) {
            const float v = bf16_to_f32(xr[i]);
            ss += v * v;
        }
        const float r = rsqrtf(block_sum(ss, red) / (float)H + eps);
        for (int i = threadIdx.x; i < H; i += kGlueThreads) yr[i] = f32_to_bf16_rne(bf16_to_f32(xr[i]) * r * bf16_to_f32(w[i]));
    }
}

// s = a + b (rounded to bf16 and stored), y = rmsnorm(s) * w: the residual connection and the norm that follows it in
// one pass over the row.  One CTA per row; the second pass re-reads what the same thread stored.
__global__ void __launch_bounds__(kGlueThreads) add_rmsnorm_kernel(const uint16_t* a, const uint16_t* b, uint16_t* sum, const uint16_t* w,
                                                                  uint16_t* y, int H, float eps)
{
    pdl_let_next_start();
    pdl_wait();
    __shared__ float red[32];
    const size_t r0 = (size_t)blockIdx.x * H;
    float ss = 0.f;
    for (int i = threadIdx.x; i < H; i += blockDim.x) {
        const uint16_t sb = f32_to_bf16_rne(bf16_to_f32(a[r0 + i]) + bf16_to_f32(b[r0 + i]));
        sum[r0 + i] = sb;
        const float v = bf16_to_f32(sb);
        ss += v * v;
    }
    const float r = rsqrtf(block_sum(ss, red) / (float)H + eps);
    for (int i = threadIdx.x; i < H; i += blockDim.x) y[r0 + i] = f32_to_bf16_rne(bf16_to_f32(sum[r0 + i]) * r * bf16_to_f32(w[i]));
}

// Rotates q in place and writes the rotated k and the plain v of row n into position `pos` of row n's cache.
// Caches are [N, T_max, Hkv * d].  One CTA per row.
__global__ void __launch_bounds__(kGlueThreads) rope_cache_kernel(uint16_t* q, const uint16_t* k, const uint16_t* v, uint16_t* kc,
                                                                 uint16_t* vc, int Hq, int Hkv, int d, int pos, int T_max,
                                                                 const RopeTable tab)
{
    pdl_let_next_start();
    pdl_wait();
    const int n = blockIdx.x, half = d / 2;
    uint16_t* qr = q + (size_t)n * Hq * d;
    const uint16_t* kr = k + (size_t)n * Hkv * d;
    uint16_t* kdst = kc + ((size_t)n * T_max + pos) * Hkv * d;
    uint16_t* vdst = vc + ((size_t)n * T_max + pos) * Hkv * d;
    for (int p = threadIdx.x; p < (Hq + Hkv) * half; p += blockDim.x) {
        const int h = p / half, i = p % half;
        const float c = tab.c[i], s = tab.s[i];
        if (h < Hq) {
            const float a = bf16_to_f32(qr[h * d + i]), b = bf16_to_f32(qr[h * d + i + half]);
            qr[h * d + i] = f32_to_bf16_rne(a * c - b * s);
            qr[h * d + i + half] = f32_to_bf16_rne(b * c + a * s);
        } else {
            const int hk = h - Hq;
            const float a = bf16_to_f32(kr[hk * d + i]), b = bf16_to_f32(kr[hk * d + i + half]);
            kdst[hk * d + i] = f32_to_bf16_rne(a * c - b * s);
            kdst[hk * d + i + half] = f32_to_bf16_rne(b * c + a * s);
        }
    }
    for (int i = threadIdx.x; i < Hkv * d; i += blockDim.x) vdst[i] = v[(size_t)n * Hkv * d + i];
}

// Attention of one new token per row over T cached positions, by clusters of one to eight CTAs per (row, query head), each
// with its share of the positions.  d is 8, 16, 32, 64 or 128 and the caches are 16-byte aligned: d / 8 lanes share a position,
// a lane holds eight dimensions (one 128-bit load), a warp takes 256 / d positions per step and four steps at a time.
// Latency bounds it (300 positions of 64 dimensions are 38 KB a head), so keys and values are asked for together, and before
// the query is there, and a running maximum takes the place of a pass over the scores with its barriers: with three passes
// (scores, weights, values) by one CTA per head such a step took 19.5 us.
// ROPE: also rotates the query (and writes it back) and the new key, attends over the new token from registers and shared
// memory, and appends it to the caches (the first query head of every group does).
constexpr int kAttnSteps = 4;
constexpr int kAttnMaxCluster = 8;
template <bool ROPE>
__global__ void __launch_bounds__(kAttnThreads) attention_kernel(uint16_t* q, const uint16_t* k, const uint16_t* v, uint16_t* kc, uint16_t* vc,
                                                                 uint16_t* out, int Hq, int Hkv, int d, int T, int T_max, int S,
                                                                 const __grid_constant__ RopeTable tab)
{
    constexpr int kWarps = kAttnThreads / 32;
    __shared__ float qs[128], ks[128];
    __shared__ float part[kWarps + 1][128], pm[kWarps + 1], pl[kWarps + 1];
    __shared__ float cacc[kAttnMaxCluster][128], cm[kAttnMaxCluster], cl[kAttnMaxCluster];   // of rank 0: every CTA's share
    pdl_let_next_start();
    pdl_wait();
    const int rank = blockIdx.x % S, row = blockIdx.x / S;
    const int n = row / Hq, h = row - n * Hq, group = Hq / Hkv, g = h / group;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const size_t pitch = (size_t)Hkv * d, first = (size_t)n * T_max * pitch + (size_t)g * d;
    const int lpp = d >> 3, ppw = 32 / lpp, dl = (lane % lpp) * 8;
    const int begin = (int)((long long)T * rank / S), end = (int)((long long)T * (rank + 1) / S);
    const int w0 = begin + warp * ppw, t0 = w0 + lane / lpp, step = kWarps * ppw;
    const uint16_t* kb = kc + first + (size_t)t0 * pitch + dl;
    const uint16_t* vb = vc + first + (size_t)t0 * pitch + dl;
    uint4 kv[kAttnSteps], vv[kAttnSteps];
    auto load = [&](int at) {                // the four steps from position t0 + at on
#pragma unroll
        for (int i = 0; i < kAttnSteps; ++i) {
            const bool there = t0 + at + i * step < end;
            kv[i] = there ? *(const uint4*)(kb + (size_t)(at + i * step) * pitch) : make_uint4(0u, 0u, 0u, 0u);
            vv[i] = there ? *(const uint4*)(vb + (size_t)(at + i * step) * pitch) : make_uint4(0u, 0u, 0u, 0u);
        }
    };
    load(0);
    uint16_t* qr = q + (size_t)row * d;
    const int half = d / 2;
    uint16_t q0 = 0, q1 = 0, k0 = 0, k1 = 0;
    if (ROPE) {
        if (tid < half) {
            const float c = tab.c[tid], sn = tab.s[tid];
            const uint16_t* kr = k + ((size_t)n * Hkv + g) * d;
            const float a = bf16_to_f32(qr[tid]), b = bf16_to_f32(qr[tid + half]);
            q0 = f32_to_bf16_rne(a * c - b * sn);
            q1 = f32_to_bf16_rne(b * c + a * sn);
            const float ka = bf16_to_f32(kr[tid]), kb2 = bf16_to_f32(kr[tid + half]);
            k0 = f32_to_bf16_rne(ka * c - kb2 * sn);
            k1 = f32_to_bf16_rne(kb2 * c + ka * sn);
            qs[tid] = bf16_to_f32(q0);
            qs[tid + half] = bf16_to_f32(q1);
            ks[tid] = bf16_to_f32(k0);
            ks[tid + half] = bf16_to_f32(k1);
        }
    } else if (tid < d) {
        qs[tid] = bf16_to_f32(qr[tid]);
    }
    __syncthreads();
    if (S > 1) asm volatile("barrier.cluster.arrive.release;" ::: "memory");     // this CTA runs, and has read q
    float qv[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) qv[j] = qs[dl + j];
    const float scale = rsqrtf((float)d);
    float m = -INFINITY, l = 0.f, acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int at = 0; w0 + at < end; at += kAttnSteps * step) {                   // (the same for the whole warp)
        if (at > 0) load(at);
        float s[kAttnSteps], top = m;
#pragma unroll
        for (int i = 0; i < kAttnSteps; ++i) {
            const uint32_t u[4] = {kv[i].x, kv[i].y, kv[i].z, kv[i].w};
            s[i] = 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) s[i] += qv[2 * j] * bf16_lo(u[j]) + qv[2 * j + 1] * bf16_hi(u[j]);
            for (int dd = 1; dd < lpp; dd <<= 1) s[i] += __shfl_xor_sync(0xFFFFFFFFu, s[i], dd);
            s[i] = t0 + at + i * step < end ? s[i] * scale : -INFINITY;
            top = fmaxf(top, s[i]);
        }
        const float base = top == -INFINITY ? 0.f : top;                         // (a lane may have no position yet)
        const float keep = expf(m - base);
        m = top;
        l *= keep;
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] *= keep;
#pragma unroll
        for (int i = 0; i < kAttnSteps; ++i) {
            const float p = expf(s[i] - base);
            const uint32_t u[4] = {vv[i].x, vv[i].y, vv[i].z, vv[i].w};
            l += p;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                acc[2 * j] += p * bf16_lo(u[j]);
                acc[2 * j + 1] += p * bf16_hi(u[j]);
            }
        }
    }
    // the warp's lanes, the CTA's warps, the cluster's CTAs
    float top = m;
    for (int dd = lpp; dd < 32; dd <<= 1) top = fmaxf(top, __shfl_xor_sync(0xFFFFFFFFu, top, dd));
    const float f = m == -INFINITY ? 0.f : expf(m - top);
    l *= f;
    for (int dd = lpp; dd < 32; dd <<= 1) l += __shfl_xor_sync(0xFFFFFFFFu, l, dd);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        float a = acc[j] * f;
        for (int dd = lpp; dd < 32; dd <<= 1) a += __shfl_xor_sync(0xFFFFFFFFu, a, dd);
        if (lane < lpp) part[warp][dl + j] = a;
    }
    if (lane == 0) { pm[warp] = top; pl[warp] = l; }
    const uint16_t* vnew = ROPE ? v + ((size_t)n * Hkv + g) * d : nullptr;
    const int parts = kWarps + (ROPE && rank == 0 ? 1 : 0);                      // rank 0 has the new token
    if (ROPE && rank == 0 && warp == kWarps - 1) {
        float s = 0.f;
        for (int i = lane; i < d; i += 32) {
            s += qs[i] * ks[i];
            part[kWarps][i] = bf16_to_f32(vnew[i]);
        }
        s = warp_sum(s);
        if (lane == 0) { pm[kWarps] = s * scale; pl[kWarps] = 1.f; }
    }
    __syncthreads();
    if (S > 1) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");       // the others run; all have read q
    float A = 0.f, L = 0.f, M = -INFINITY;
    if (tid < d) {
        for (int w = 0; w < parts; ++w) M = fmaxf(M, pm[w]);
        for (int w = 0; w < parts; ++w) {
            const float e = pm[w] == -INFINITY ? 0.f : expf(pm[w] - M);
            L += pl[w] * e;
            A += part[w][tid] * e;
        }
        if (S > 1) {
            uint32_t to_a, to_m, to_l;
            asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(to_a) : "r"(smem_u32(&cacc[rank][tid])));
            asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(to_a), "f"(A) : "memory");
            if (tid == 0) {
                asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(to_m) : "r"(smem_u32(&cm[rank])));
                asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(to_l) : "r"(smem_u32(&cl[rank])));
                asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(to_m), "f"(M) : "memory");
                asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(to_l), "f"(L) : "memory");
            }
        }
    }
    if (S > 1) {
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
        if (rank != 0) return;
        if (tid < d) {
            M = -INFINITY;
            for (int c = 0; c < S; ++c) M = fmaxf(M, cm[c]);
            A = L = 0.f;
            for (int c = 0; c < S; ++c) {
                const float e = cm[c] == -INFINITY ? 0.f : expf(cm[c] - M);
                L += cl[c] * e;
                A += cacc[c][tid] * e;
            }
        }
    }
    if (tid < d) out[(size_t)row * d + tid] = f32_to_bf16_rne(A / L);
    if (ROPE) {
        uint16_t* kdst = kc + first + (size_t)T * pitch;
        uint16_t* vdst = vc + first + (size_t)T * pitch;
        const bool writer = h - g * group == 0;
        if (tid < half) {
            qr[tid] = q0;
            qr[tid + half] = q1;
            if (writer) { kdst[tid] = k0; kdst[tid + half] = k1; }
        }
        if (writer && tid < d) vdst[tid] = vnew[tid];
    }
}

// One new token per row over T cached positions; one CTA per (row, query head); d <= 128.
// For head widths and caches that attention_kernel cannot read in 128-bit words.
__global__ void __launch_bounds__(kAttnThreads) attention_any_kernel(const uint16_t* q, const uint16_t* kc, const uint16_t* vc,
                                                                       uint16_t* out, int Hq, int Hkv, int d, int T, int T_max)
{
    pdl_let_next_start();
    pdl_wait();
    extern __shared__ float sc[];            // T scores, then the weights
    __shared__ float red[32];
    __shared__ float qs[128];
    __shared__ float part[(kAttnThreads / 32) * 128];
    const int n = blockIdx.x / Hq, h = blockIdx.x % Hq, g = h / (Hq / Hkv);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    if (threadIdx.x < d) qs[threadIdx.x] = bf16_to_f32(q[((size_t)n * Hq + h) * d + threadIdx.x]);
    __syncthreads();
    const uint16_t* kb = kc + (size_t)n * T_max * Hkv * d + (size_t)g * d;
    const uint16_t* vb = vc + (size_t)n * T_max * Hkv * d + (size_t)g * d;
    const size_t pitch = (size_t)Hkv * d;
    const float scale = rsqrtf((float)d);
#pragma unroll 4
    for (int t = warp; t < T; t += nw) {
        float s = 0.f;
        for (int i = lane; i < d; i += 32) s += qs[i] * bf16_to_f32(kb[(size_t)t * pitch + i]);
        for (int dd = 16; dd > 0; dd >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, dd);
        if (lane == 0) sc[t] = s * scale;
    }
    __syncthreads();
    float m = -INFINITY;
    for (int t = threadIdx.x; t < T; t += blockDim.x) m = fmaxf(m, sc[t]);
    m = block_max(m, red);
    float z = 0.f;
    for (int t = threadIdx.x; t < T; t += blockDim.x) {
        const float e = expf(sc[t] - m);
        sc[t] = e;
        z += e;
    }
    z = block_sum(z, red);
    __syncthreads();
    // weights times values; the warps' partial sums meet in shared memory
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int t = warp; t < T; t += nw) {
        const float p = sc[t];
        const uint16_t* vr = vb + (size_t)t * pitch;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (lane + 32 * j < d) acc[j] += p * bf16_to_f32(vr[lane + 32 * j]);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (lane + 32 * j < d) part[warp * 128 + lane + 32 * j] = acc[j];
    __syncthreads();
    if (threadIdx.x < d) {
        float a = 0.f;
        for (int w = 0; w < nw; ++w) a += part[w * 128 + threadIdx.x];
        out[((size_t)n * Hq + h) * d + threadIdx.x] = f32_to_bf16_rne(a / z);
    }
}

// sd2_rope_cache and sd2_attention_decode in one launch, one CTA per (row, query head): the CTA rotates its query head
// (and writes it back), rotates the key head of its group for itself, and attends over the cached positions 0..pos-1
// plus the new token, whose key and value it takes from its own shared memory and from `v`, not from the cache; the
// first head of every group also appends the rotated key and the value to the caches.  No CTA reads what another writes.
__global__ void __launch_bounds__(kAttnThreads) rope_attention_any_kernel(uint16_t* q, const uint16_t* k, const uint16_t* v, uint16_t* kc,
                                                                     uint16_t* vc, uint16_t* out, int Hq, int Hkv, int d, int pos,
                                                                     int T_max, const __grid_constant__ RopeTable tab)
{
    pdl_let_next_start();
    pdl_wait();
    extern __shared__ float sc[];            // pos + 1 scores, then the weights
    __shared__ float red[32];
    __shared__ float qs[128], ks[128];
    __shared__ float part[(kAttnThreads / 32) * 128];
    const int n = blockIdx.x / Hq, h = blockIdx.x % Hq, group = Hq / Hkv, g = h / group;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int half = d / 2, T = pos;         // cached positions; the new token is handled apart
    uint16_t* qr = q + ((size_t)n * Hq + h) * d;
    const uint16_t* kr = k + ((size_t)n * Hkv + g) * d;
    const size_t pitch = (size_t)Hkv * d;
    uint16_t* kdst = kc + ((size_t)n * T_max + pos) * pitch + (size_t)g * d;
    uint16_t* vdst = vc + ((size_t)n * T_max + pos) * pitch + (size_t)g * d;
    const uint16_t* vnew = v + ((size_t)n * Hkv + g) * d;
    const bool writer = (h % group) == 0;
    if (threadIdx.x < half) {
        const int i = threadIdx.x;
        const float c = tab.c[i], sn = tab.s[i];
        const float a = bf16_to_f32(qr[i]), b = bf16_to_f32(qr[i + half]);
        const uint16_t q0 = f32_to_bf16_rne(a * c - b * sn), q1 = f32_to_bf16_rne(b * c + a * sn);
        qr[i] = q0;
        qr[i + half] = q1;
        qs[i] = bf16_to_f32(q0);
        qs[i + half] = bf16_to_f32(q1);
        const float ka = bf16_to_f32(kr[i]), kb2 = bf16_to_f32(kr[i + half]);
        const uint16_t k0 = f32_to_bf16_rne(ka * c - kb2 * sn), k1 = f32_to_bf16_rne(kb2 * c + ka * sn);
        ks[i] = bf16_to_f32(k0);
        ks[i + half] = bf16_to_f32(k1);
        if (writer) {
            kdst[i] = k0;
            kdst[i + half] = k1;
        }
    }
    if (writer && threadIdx.x < d) vdst[threadIdx.x] = vnew[threadIdx.x];
    __syncthreads();
    const uint16_t* kb = kc + (size_t)n * T_max * pitch + (size_t)g * d;
    const uint16_t* vb = vc + (size_t)n * T_max * pitch + (size_t)g * d;
    const float scale = rsqrtf((float)d);
#pragma unroll 4
    for (int t = warp; t < T; t += nw) {
        float s = 0.f;
        for (int i = lane; i < d; i += 32) s += qs[i] * bf16_to_f32(kb[(size_t)t * pitch + i]);
        for (int dd = 16; dd > 0; dd >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, dd);
        if (lane == 0) sc[t] = s * scale;
    }
    if (warp == 0) {                         // the new token's own score
        float s = 0.f;
        for (int i = lane; i < d; i += 32) s += qs[i] * ks[i];
        for (int dd = 16; dd > 0; dd >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, dd);
        if (lane == 0) sc[T] = s * scale;
    }
    __syncthreads();
    float m = -INFINITY;
    for (int t = threadIdx.x; t <= T; t += blockDim.x) m = fmaxf(m, sc[t]);
    m = block_max(m, red);
    float z = 0.f;
    for (int t = threadIdx.x; t <= T; t += blockDim.x) {
        const float e = expf(sc[t] - m);
        sc[t] = e;
        z += e;
    }
    z = block_sum(z, red);
    __syncthreads();
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int t = warp; t < T; t += nw) {
        const float p = sc[t];
        const uint16_t* vr = vb + (size_t)t * pitch;
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (lane + 32 * j < d) acc[j] += p * bf16_to_f32(vr[lane + 32 * j]);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (lane + 32 * j < d) part[warp * 128 + lane + 32 * j] = acc[j];
    __syncthreads();
    if (threadIdx.x < d) {
        float a = sc[T] * bf16_to_f32(vnew[threadIdx.x]);
        for (int w = 0; w < nw; ++w) a += part[w * 128 + threadIdx.x];
        out[((size_t)n * Hq + h) * d + threadIdx.x] = f32_to_bf16_rne(a / z);
    }
}

// y = a + b, element by element
__global__ void __launch_bounds__(kGlueThreads) add_kernel(const uint16_t* a, const uint16_t* b, uint16_t* y, long long count)
{
    pdl_let_next_start();
    pdl_wait();
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (long long)gridDim.x * blockDim.x)
        y[i] = f32_to_bf16_rne(bf16_to_f32(a[i]) + bf16_to_f32(b[i]));
}

// x[n, :] = table[token[n], :]
__global__ void __launch_bounds__(kGlueThreads) embedding_kernel(const int32_t* tokens, const uint16_t* table, uint16_t* x, int H, int V, int vec)
{
    pdl_let_next_start();
    pdl_wait();
    const int tok = tokens[blockIdx.x];
    const bool there = tok >= 0 && tok < V;
    if (vec) {                               // H is a multiple of 8, x and table are 16-byte aligned
        for (int i = threadIdx.x; i < H / 8; i += blockDim.x)
            ((uint4*)(x + (size_t)blockIdx.x * H))[i] = there ? ((const uint4*)(table + (size_t)tok * H))[i] : make_uint4(0u, 0u, 0u, 0u);
        return;
    }
    for (int i = threadIdx.x; i < H; i += blockDim.x) x[(size_t)blockIdx.x * H + i] = there ? table[(size_t)tok * H + i] : (uint16_t)0;
}

// logits[n, v] = sum_h W[v, h] x[n, h]: a warp takes kHeadRowsPerWarp vocabulary rows at a time (as many independent
// 128-bit loads in flight per lane and column step) of its share of the table, the activation rows sit in shared memory as
// bf16.  HBM bounds it: 128256 x 2048 takes 80 us for one and two rows (6.5 TB/s), from 102.  What that took:
//   - even shares of rows per warp; steps of four rows dealt out in turn, 3.4 of them per warp, left warps idle: 94 us;
//   - 256-byte requests that pass L1 by and four column steps in flight, on three CTAs per SM: 80 us (asking for the first rows to
//     be brought to L2 while the launches before still run slowed these down by more than it gave);
//   - four rows that share what is read of the activations, and fma.rn.f32x2 (the same fp32 sums, even and odd columns
//     apart): with one row per step every activation row took as long as a pass of its own, four of them 520 us.
constexpr int kHeadRowsPerWarp = 4;
// CTAs per SM of an instance for NT rows, as many as its registers allow
constexpr int head_ctas(int NT) { return NT <= 1 ? 3 : 2; }
__device__ __forceinline__ uint4 ldg_stream(const uint4* p)
{
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::256B.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}
// two bf16 values as a pair of fp32, two fp32 multiply-adds
__device__ __forceinline__ unsigned long long f32_pair(uint32_t w) { return (unsigned long long)(w & 0xFFFF0000u) << 32 | (w << 16); }
__device__ __forceinline__ void fma_pair(unsigned long long& acc, unsigned long long a, unsigned long long b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
template <int NT>
__global__ void __launch_bounds__(kGlueThreads, head_ctas(NT)) lm_head_kernel(const uint16_t* x, const uint16_t* W, float* logits, int N, int V, int H)
{
    pdl_let_next_start();
    pdl_wait();
    extern __shared__ uint4 head_x[];        // [NT][H / 8]: zero beyond row N
    const int groups = H / 8;
    if ((((uintptr_t)x) & 15) == 0) {
        for (int i = threadIdx.x; i < NT * groups; i += blockDim.x) head_x[i] = i < N * groups ? ((const uint4*)x)[i] : make_uint4(0u, 0u, 0u, 0u);
    } else {
        for (int i = threadIdx.x; i < NT * H; i += blockDim.x) ((uint16_t*)head_x)[i] = i < N * H ? x[i] : (uint16_t)0;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const long long warps = (gridDim.x * blockDim.x) >> 5, gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int end = (int)(V * (gw + 1) / warps);
    for (int v0 = (int)(V * gw / warps); v0 < end; v0 += kHeadRowsPerWarp) {
        unsigned long long acc[NT][kHeadRowsPerWarp];
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int r = 0; r < kHeadRowsPerWarp; ++r) acc[n][r] = 0ull;
#pragma unroll(NT <= 2 ? 4 : NT <= 4 ? 2 : 1)
        for (int c = lane; c < groups; c += 32) {
            uint4 w4[kHeadRowsPerWarp];
#pragma unroll
            for (int r = 0; r < kHeadRowsPerWarp; ++r)
                w4[r] = v0 + r < end ? ldg_stream((const uint4*)(W + (size_t)(v0 + r) * H) + c) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                const uint4 xv = head_x[n * groups + c];
                const unsigned long long xw[4] = {f32_pair(xv.x), f32_pair(xv.y), f32_pair(xv.z), f32_pair(xv.w)};
#pragma unroll
                for (int r = 0; r < kHeadRowsPerWarp; ++r) {
                    const uint32_t ww[4] = {w4[r].x, w4[r].y, w4[r].z, w4[r].w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) fma_pair(acc[n][r], f32_pair(ww[j]), xw[j]);
                }
            }
        }
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int r = 0; r < kHeadRowsPerWarp; ++r) {
                const float s = warp_sum(__uint_as_float((uint32_t)acc[n][r]) + __uint_as_float((uint32_t)(acc[n][r] >> 32)));
                if (lane == 0 && n < N && v0 + r < end) logits[(size_t)n * V + v0 + r] = s;
            }
    }
}

// token[n] = index of the largest logit of row n, the lowest index among equals; a cluster of kArgmaxCtas per row (one CTA
// reads 513 KB of logits in 9 us).  vec: V is a multiple of 4 and the row is 16-byte aligned (four logits per load).
constexpr int kArgmaxCtas = 8;
__device__ __forceinline__ void argmax_merge(float& best, int& at, float v, int i)
{
    if (v > best || (v == best && i < at)) { best = v; at = i; }
}
__device__ __forceinline__ void argmax_warp(float& best, int& at)
{
    for (int d = 16; d > 0; d >>= 1) {
        const float ov = __shfl_xor_sync(0xFFFFFFFFu, best, d);
        const int oi = __shfl_xor_sync(0xFFFFFFFFu, at, d);
        argmax_merge(best, at, ov, oi);
    }
}
__global__ void __cluster_dims__(kArgmaxCtas, 1, 1) __launch_bounds__(512) argmax_kernel(const float* logits, int32_t* token, int V, int vec)
{
    pdl_let_next_start();
    pdl_wait();
    __shared__ float bv[32];
    __shared__ int bi[32];
    __shared__ uint2 found[kArgmaxCtas];     // of rank 0: every CTA's best, as bits, and its index
    const int row = blockIdx.x / kArgmaxCtas, rank = blockIdx.x % kArgmaxCtas;
    const float* r = logits + (size_t)row * V;
    float best = -INFINITY;
    int at = 0x7FFFFFFF;
    const int first = rank * blockDim.x + threadIdx.x, step = kArgmaxCtas * blockDim.x;
    if (vec) {
        const float4* r4 = (const float4*)r;
#pragma unroll 8
        for (int i = first; i < V / 4; i += step) {
            const float4 v = r4[i];
            const float c[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (c[j] > best) { best = c[j]; at = 4 * i + j; }      // a thread meets its indices in ascending order
        }
    } else {
        for (int i = first; i < V; i += step) {
            const float v = r[i];
            if (v > best) { best = v; at = i; }
        }
    }
    argmax_warp(best, at);
    if ((threadIdx.x & 31) == 0) { bv[threadIdx.x >> 5] = best; bi[threadIdx.x >> 5] = at; }
    // (both CTAs of a remote store have to be running, and rank 0 may leave only when all stores are there)
    asm volatile("barrier.cluster.arrive;\n\tbarrier.cluster.wait;" ::: "memory");
    if (threadIdx.x < 32) {
        best = threadIdx.x < (blockDim.x >> 5) ? bv[threadIdx.x] : -INFINITY;
        at = threadIdx.x < (blockDim.x >> 5) ? bi[threadIdx.x] : 0x7FFFFFFF;
        argmax_warp(best, at);
        if (threadIdx.x == 0) {
            uint32_t to;
            asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(to) : "r"(smem_u32(&found[rank])));
            asm volatile("st.shared::cluster.v2.b32 [%0], {%1, %2};" ::"r"(to), "r"(__float_as_uint(best)), "r"((uint32_t)at) : "memory");
        }
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive;\n\tbarrier.cluster.wait;" ::: "memory");
    if (rank == 0 && threadIdx.x < 32) {
        best = threadIdx.x < kArgmaxCtas ? __uint_as_float(found[threadIdx.x].x) : -INFINITY;
        at = threadIdx.x < kArgmaxCtas ? (int)found[threadIdx.x].y : 0x7FFFFFFF;
        argmax_warp(best, at);
        if (threadIdx.x == 0) token[row] = at == 0x7FFFFFFF ? 0 : at;
    }
}

}  // namespace sd2
