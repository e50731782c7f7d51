// Append (bf16 -> e4m3 into Recent pages), Demote (FP8 page -> TQ3 record, then publish) and the
// Anchor tag flip.  Algorithm 1 steps 1-2; Section 4 "normalize-rotate-pack".
//
// The TQ3 encoder is specified as a sequence of single IEEE fp32 operations in a fixed order, so
// every arithmetic step below uses a round-to-nearest intrinsic (__fadd_rn, __fmul_rn, __fdiv_rn,
// __fsqrt_rn): the compiler may not fuse or reorder them.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <math_constants.h>

#include <cmath>

#include "mkv_internal.cuh"

namespace mkv {

__device__ __forceinline__ uint16_t f32_to_f16_sat_bits(float x)
{
    x = fminf(fmaxf(x, -65504.f), 65504.f);
    return __half_as_ushort(__float2half_rn(x));
}

// ------------------------------------------------------------------------------------------ append
// Elements 2 pair, 2 pair + 1 of K and V of one token and KV head (scale, round to nearest even, saturate to
// +-448): K token-major, V channel-major.
template <int D>
__device__ __forceinline__ void append_pair(uint8_t* __restrict__ rec, int slot, float inv_k_scale, float inv_v_scale,
                                            __nv_bfloat162 k2, __nv_bfloat162 v2, int pair)
{
    float2 kf = __bfloat1622float2(k2);
    float2 vf = __bfloat1622float2(v2);
    kf.x = __fmul_rn(kf.x, inv_k_scale);
    kf.y = __fmul_rn(kf.y, inv_k_scale);
    vf.x = __fmul_rn(vf.x, inv_v_scale);
    vf.y = __fmul_rn(vf.y, inv_v_scale);
    const __nv_fp8x2_storage_t kq = __nv_cvt_float2_to_fp8x2(kf, __NV_SATFINITE, __NV_E4M3);
    const __nv_fp8x2_storage_t vq = __nv_cvt_float2_to_fp8x2(vf, __NV_SATFINITE, __NV_E4M3);
    const int i = 2 * pair;
    *reinterpret_cast<uint16_t*>(rec + slot * D + i) = kq;             // K: token-major
    rec[16 * D + i * kPage + slot] = (uint8_t)(vq & 0xFF);             // V: channel-major
    rec[16 * D + (i + 1) * kPage + slot] = (uint8_t)(vq >> 8);
}

// Decode-sized calls: one block per (token, KV head).
template <int D>
__global__ void __launch_bounds__(D / 2) append_kernel(uint8_t* __restrict__ fp8, int fp8_pages, int hkv, int tiles,
                                                        float inv_k_scale, float inv_v_scale,
                                                        const __nv_bfloat162* k,
                                                        const __nv_bfloat162* v,
                                                        const int32_t* slots,
                                                        uint32_t* __restrict__ status)
{
    pdl_begin();
    const int tok = blockIdx.x, h = blockIdx.y;
    const int sm = slots[tok];
    if (sm < 0) return;
    // slot_mapping = page * page_tokens + position; a page is `tiles` consecutive 16-token records per head
    const int gt = sm >> 4, slot = sm & 15, page = gt / tiles, m = gt - page * tiles;
    if (page >= fp8_pages) {
        if (threadIdx.x == 0) atomicOr(status, kStBounds);
        return;
    }
    uint8_t* rec = fp8 + (((size_t)page * hkv + h) * tiles + m) * fp8_record_bytes(D);
    const size_t src = ((size_t)tok * hkv + h) * (D / 2);
    append_pair<D>(rec, slot, inv_k_scale, inv_v_scale, k[src + threadIdx.x], v[src + threadIdx.x], threadIdx.x);
}

// eight bf16 (one 16-byte load) -> eight e4m3 bytes
__device__ __forceinline__ uint2 bf16x8_to_e4m3x8(uint4 in, float inv_scale)
{
    const uint32_t w[4] = {in.x, in.y, in.z, in.w};
    uint32_t q[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[i]));
        f.x = __fmul_rn(f.x, inv_scale);
        f.y = __fmul_rn(f.y, inv_scale);
        q[i] = __nv_cvt_float2_to_fp8x2(f, __NV_SATFINITE, __NV_E4M3);
    }
    return make_uint2(q[0] | (q[1] << 16), q[2] | (q[3] << 16));
}

// Prefill-sized calls: one block per (window of 16 consecutive input tokens, KV head).  The block takes the runs
// that START in its window, a run being consecutive tokens that go to consecutive positions of one 16-token tile;
// such a run may reach up to 15 tokens into the next window.  A chunk of a request that starts anywhere inside a
// page therefore still meets whole tiles, one per window.  A run that fills its tile leaves as whole rows: K with
// 8-byte stores, V transposed through shared memory so that every channel's 16 tokens are one 16-byte store (HBM
// bound: 0.97 of the copy bandwidth on 196,608 tokens, 0.81 on 32,845 in five chunks).  Other runs (the ends of a
// request's chunk, scattered or skipped tokens) are stored token by token.  (With windows cut at fixed tokens a chunk that starts inside a page had no whole tile at all
// and every token took the second path: 147 us for 32,845 tokens in five chunks, d = 256.)
template <int D>
__global__ void __launch_bounds__(128) append_run_kernel(uint8_t* __restrict__ fp8, int fp8_pages, int hkv, int tiles,
                                                          float inv_k_scale, float inv_v_scale,
                                                          const __nv_bfloat162* k,
                                                          const __nv_bfloat162* v,
                                                          const int32_t* slots, int n,
                                                          uint32_t* __restrict__ status)
{
    constexpr int VROW = D + 4;                      // padded token row of the transposition tile
    __shared__ __align__(16) uint8_t vt[kPage * VROW];
    __shared__ int32_t slot_s[2 * kPage];            // slots of this window and the next
    __shared__ int32_t rest_s[2 * kPage];            // tokens of the other runs that start in the window
    __shared__ int full_s, n_rest_s;                 // token whose run fills a tile (at most one starts in a window), or -1
    pdl_begin();
    const int t0 = blockIdx.x * kPage, h = blockIdx.y, tid = threadIdx.x;
    if (tid < 32) {
        const int sl = t0 + tid < n ? slots[t0 + tid] : -1;
        const int before = tid == 0 && t0 > 0 ? slots[t0 - 1] : -2;
        slot_s[tid] = sl;
        const int up = __shfl_up_sync(0xffffffffu, sl, 1);
        const int prev = tid == 0 ? before : up;
        __syncwarp();
        int len = 0;
        if (tid < kPage && sl >= 0 && ((sl & 15) == 0 || prev != sl - 1)) {
            len = 1;
            while (len < kPage - (sl & 15) && slot_s[tid + len] == sl + len) ++len;
        }
        const bool full = len == kPage && (sl >> 4) / tiles < fp8_pages;
        const uint32_t m = __ballot_sync(0xffffffffu, full);
        if (full) len = 0;
        int end = len;                               // running count of those tokens
#pragma unroll
        for (int o = 1; o < kPage; o <<= 1) {
            const int before_me = __shfl_up_sync(0xffffffffu, end, o);
            if (tid >= o) end += before_me;
        }
        for (int j = 0; j < len; ++j) rest_s[end - len + j] = tid + j;
        if (tid == 0) full_s = m ? __ffs(m) - 1 : -1;
        if (tid == kPage - 1) n_rest_s = end;
    }
    __syncthreads();
    const int full = full_s;
    if (full >= 0) {
        const int gt = slot_s[full] >> 4, page = gt / tiles;
        uint8_t* rec = fp8 + (((size_t)page * hkv + h) * tiles + (gt - page * tiles)) * fp8_record_bytes(D);
        constexpr int CPT = D / 8, N = kPage * CPT / 128;      // 16-byte input chunks per token, and per thread
        uint4 kin[N], vin[N];                        // all loads before the first store
#pragma unroll
        for (int u = 0; u < N; ++u) {
            const int c = tid + 128 * u;
            const size_t at = ((size_t)(t0 + full + c / CPT) * hkv + h) * CPT + c % CPT;
            kin[u] = reinterpret_cast<const uint4*>(k)[at];
            vin[u] = reinterpret_cast<const uint4*>(v)[at];
        }
#pragma unroll
        for (int u = 0; u < N; ++u) {
            const int c = tid + 128 * u, t = c / CPT, c8 = c % CPT;
            const uint2 kq = bf16x8_to_e4m3x8(kin[u], inv_k_scale);
            const uint2 vq = bf16x8_to_e4m3x8(vin[u], inv_v_scale);
            *reinterpret_cast<uint2*>(rec + t * D + 8 * c8) = kq;
            *reinterpret_cast<uint32_t*>(vt + t * VROW + 8 * c8) = vq.x;
            *reinterpret_cast<uint32_t*>(vt + t * VROW + 8 * c8 + 4) = vq.y;
        }
        __syncthreads();
        // thread c4 owns channels 4 c4 .. 4 c4 + 3: 16 words (one per token) -> 4 x 16 bytes
        for (int c4 = tid; c4 < D / 4; c4 += 128) {
            uint32_t w[kPage];
#pragma unroll
            for (int t = 0; t < kPage; ++t) w[t] = *reinterpret_cast<const uint32_t*>(vt + t * VROW + 4 * c4);
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {
                uint32_t o[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint32_t lo = __byte_perm(w[4 * q], w[4 * q + 1], 0x0040 + 0x0011 * ch);   // bytes ch of t, t+1
                    const uint32_t hi = __byte_perm(w[4 * q + 2], w[4 * q + 3], 0x0040 + 0x0011 * ch);
                    o[q] = __byte_perm(lo, hi, 0x5410);
                }
                *reinterpret_cast<uint4*>(rec + 16 * D + (4 * c4 + ch) * kPage) = make_uint4(o[0], o[1], o[2], o[3]);
            }
        }
    }
    // the rest token by token, the loads of four (token, element pair) items in flight per thread
    const int n_items = n_rest_s * (D / 2);
    for (int i0 = tid; i0 < n_items; i0 += 4 * 128) {
        __nv_bfloat162 kk[4], vv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * 128;
            if (i >= n_items) break;
            const size_t src = ((size_t)(t0 + rest_s[i / (D / 2)]) * hkv + h) * (D / 2) + i % (D / 2);
            kk[u] = k[src];
            vv[u] = v[src];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int i = i0 + u * 128;
            if (i >= n_items) break;
            const int sm = slot_s[rest_s[i / (D / 2)]], gt = sm >> 4, page = gt / tiles;
            if (page >= fp8_pages) {
                if (i % (D / 2) == 0) atomicOr(status, kStBounds);
                continue;
            }
            uint8_t* rec = fp8 + (((size_t)page * hkv + h) * tiles + (gt - page * tiles)) * fp8_record_bytes(D);
            append_pair<D>(rec, sm & 15, inv_k_scale, inv_v_scale, kk[u], vv[u], i % (D / 2));
        }
    }
}

// Decode-sized append into the pools of several layers: one block per (token, KV head, layer).
struct AppendLayers {
    uint8_t* fp8[MKV_MAX_LAYERS_PER_CALL];
    const __nv_bfloat162* k[MKV_MAX_LAYERS_PER_CALL];
    const __nv_bfloat162* v[MKV_MAX_LAYERS_PER_CALL];
    uint32_t* status[MKV_MAX_LAYERS_PER_CALL];
    float inv_k_scale[MKV_MAX_LAYERS_PER_CALL], inv_v_scale[MKV_MAX_LAYERS_PER_CALL];
    int fp8_pages[MKV_MAX_LAYERS_PER_CALL];
};

template <int D>
__global__ void __launch_bounds__(D / 2) append_layers_kernel(const AppendLayers A, int hkv, int tiles,
                                                               const int32_t* slots)
{
    pdl_begin();
    const int tok = blockIdx.x, h = blockIdx.y, layer = blockIdx.z;
    const int sm = slots[tok];
    if (sm < 0) return;
    const int gt = sm >> 4, slot = sm & 15, page = gt / tiles, m = gt - page * tiles;
    if (page >= A.fp8_pages[layer]) {
        if (threadIdx.x == 0) atomicOr(A.status[layer], kStBounds);
        return;
    }
    uint8_t* rec = A.fp8[layer] + (((size_t)page * hkv + h) * tiles + m) * fp8_record_bytes(D);
    const size_t src = ((size_t)tok * hkv + h) * (D / 2);
    append_pair<D>(rec, slot, A.inv_k_scale[layer], A.inv_v_scale[layer], A.k[layer][src + threadIdx.x],
                   A.v[layer][src + threadIdx.x], threadIdx.x);
}

int32_t launch_append_layers(mkv_pool* const* pools, const void* const* k, const void* const* v, const int32_t* slots,
                             int n, int n_layers, cudaStream_t s)
{
    AppendLayers A;
    for (int i = 0; i < n_layers; ++i) {
        A.fp8[i] = pools[i]->fp8;
        A.k[i] = static_cast<const __nv_bfloat162*>(k[i]);
        A.v[i] = static_cast<const __nv_bfloat162*>(v[i]);
        A.status[i] = pools[i]->status_dev;
        A.inv_k_scale[i] = 1.0f / pools[i]->cfg.k_scale;
        A.inv_v_scale[i] = 1.0f / pools[i]->cfg.v_scale;
        A.fp8_pages[i] = pools[i]->cfg.fp8_pages;
    }
    const mkv_pool* p = pools[0];
    dim3 grid(n, p->hkv, n_layers);
    if (p->d == 128) MKV_CUDA(launch_pdl(append_layers_kernel<128>, grid, 64, 0, 1, s, A, p->hkv, p->tiles, slots));
    else MKV_CUDA(launch_pdl(append_layers_kernel<256>, grid, 128, 0, 1, s, A, p->hkv, p->tiles, slots));
    MKV_CUDA(cudaGetLastError());
    return MKV_OK;
}

// Calls of fewer tokens than this take one block per token: a batch's new tokens, each in a page of its own.  At
// 256 tokens both ways take 3.3 us (d = 128, 8 heads); at 64 tokens 2.0 us against 3.2 us.
constexpr int kAppendRun = 256;

int32_t launch_append(mkv_pool* p, const void* k, const void* v, const int32_t* slots, int n, cudaStream_t s)
{
    const float ik = 1.0f / p->cfg.k_scale, iv = 1.0f / p->cfg.v_scale;
    const __nv_bfloat162* kk = (const __nv_bfloat162*)k;
    const __nv_bfloat162* vv = (const __nv_bfloat162*)v;
    if (n >= kAppendRun) {
        dim3 grid((n + kPage - 1) / kPage, p->hkv);
        if (p->d == 128)
            MKV_CUDA(launch_pdl(append_run_kernel<128>, grid, 128, 0, 1, s, p->fp8, p->cfg.fp8_pages, p->hkv, p->tiles, ik, iv, kk, vv, slots, n,
                                                        p->status_dev));
        else
            MKV_CUDA(launch_pdl(append_run_kernel<256>, grid, 128, 0, 1, s, p->fp8, p->cfg.fp8_pages, p->hkv, p->tiles, ik, iv, kk, vv, slots, n,
                                                        p->status_dev));
    } else {
        dim3 grid(n, p->hkv);
        if (p->d == 128)
            MKV_CUDA(launch_pdl(append_kernel<128>, grid, 64, 0, 1, s, p->fp8, p->cfg.fp8_pages, p->hkv, p->tiles, ik, iv, kk, vv, slots, p->status_dev));
        else
            MKV_CUDA(launch_pdl(append_kernel<256>, grid, 128, 0, 1, s, p->fp8, p->cfg.fp8_pages, p->hkv, p->tiles, ik, iv, kk, vv, slots, p->status_dev));
    }
    MKV_CUDA(cudaGetLastError());
    return MKV_OK;
}

// ---- thread-block cluster helpers (Demote and Promote run one cluster per page) ------------------
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// Every thread of every block of the cluster arrives exactly once; no block leaves early.
__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Blocks per page.  A call of few pages (the retier of a decode step) is latency-bound: the heads of a
// page go to the blocks of a cluster, the largest divisor of the head count that a portable cluster
// allows.  A call that fills the GPU with one block per page anyway keeps the heads in one block, which
// amortises the per-block set-up and overlaps one head's copy-out with the next head's encoding.
static int heads_cluster(int hkv, int n_pages, int sms)
{
    if (n_pages > 2 * sms) return 1;
    for (int c = 8; c > 1; --c)
        if (hkv % c == 0) return c;
    return 1;
}

// ------------------------------------------------------------------------------------------ demote
// One thread-block cluster per page, its blocks sharing out the KV heads (block r takes heads r,
// r + cluster size, ...); the cluster's barrier orders every head's record before the page is
// published.  Warps encode key vectors (one token each), threads encode value channels; the 3-bit
// codes meet in shared memory, where every thread assembles one word triple of the record image; the
// image leaves with 16-byte stores.
//
// Shared layout: key codes [token][D + 8] (the 8 pad bytes spread the token rows over the banks for
// the packers, which read rows g and g + 8), value codes [channel][16 tokens], and two record images
// (alternating per head, so that the copy-out of one head overlaps the encoding of the next).

// 16 bytes global -> shared, asynchronously (both addresses 16-byte aligned); completion by cp.async.wait_all
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)), "l"(gmem_src)
                 : "memory");
}

// Two fp32 values in one 64-bit register and the packed operations on them (add, mul, fma, each half rounded to
// nearest even exactly like the scalar instruction): half the instructions for element-wise arithmetic.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b)
{
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// two e4m3 bytes (low byte first) -> two fp32
__device__ __forceinline__ float2 e4m3x2_to_f32(uint32_t two_bytes)
{
    const __half2_raw h = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)two_bytes, __NV_E4M3);
    return __half22float2(__half2(h));
}

// nibble pairs of two bytes -> one byte: (x & 0x000F) | ((x & 0x0F00) >> 4)
__device__ __forceinline__ uint32_t squeeze_nibbles(uint32_t x) { return (x & 0xFu) | ((x >> 4) & 0xF0u); }

// four code bytes -> four nibbles
__device__ __forceinline__ uint32_t squeeze4(uint32_t x)
{
    return (x & 0xFu) | ((x >> 4) & 0xF0u) | ((x >> 8) & 0xF00u) | ((x >> 12) & 0xF000u);
}

// Pages of several tiles are converted by gridDim.y clusters per page (rows of tiles).  When the call publishes
// from inside the kernel, every cluster draws a ticket of its page once all its tiles are written and fenced
// (called by thread 0 of the cluster's first block after the cluster barrier); the cluster that draws the last
// one publishes and leaves the counter at zero.  Nobody waits.  Without tickets (16-token pages: one cluster
// per page) every caller is the last.
__device__ __forceinline__ bool last_cluster_of_page(uint32_t* page_tickets, int page)
{
    if (page_tickets == nullptr) return true;
    const uint32_t prev = atomicAdd(page_tickets + page, 1u);
    if (prev != gridDim.y - 1) return false;
    __threadfence();                    // the other clusters' tiles are ordered before what this thread writes next
    page_tickets[page] = 0u;
    return true;
}

// Constants of the key encoder that depend only on the lane (FMT: the record format's codebook).
template <int D, int FMT>
struct DemoteLane {
    float c0sq, c1sq, c2sq, c3sq;     // squared levels (single fp32 products, as the record's norm correction defines them)
    uint32_t flip[D / 32];            // rotation signs of this lane's key elements, as fp32 sign-bit masks
    float sgn[5];                     // butterfly stage m: lanes with bit m set subtract (-1.0f), the others add (+1.0f)
    __device__ __forceinline__ void init(const SigmaBits& sigma, int lane)
    {
        using CB = KeyCodebook<FMT>;
        c0sq = __fmul_rn(CB::C0, CB::C0);
        c1sq = __fmul_rn(CB::C1, CB::C1);
        c2sq = __fmul_rn(CB::C2, CB::C2);
        c3sq = __fmul_rn(CB::C3, CB::C3);
#pragma unroll
        for (int r = 0; r < D / 32; ++r) {
            const int i = lane * (D / 32) + r;
            flip[r] = ((sigma.w[i >> 5] >> (i & 31)) & 1u) << 31;
        }
#pragma unroll
        for (int b = 0; b < 5; ++b) sgn[b] = ((lane >> b) & 1) ? -1.0f : 1.0f;
    }
};

// One key vector (a token of one KV head), lane l holding its elements l * D/32 ..: the literal sequence of fp32
// operations that defines the encoder.  Codes as bytes in element order, norm correction as fp16 bits.
template <int D, int FMT>
__device__ __forceinline__ void encode_key_token(const uint32_t (&raw)[D / 128], const DemoteLane<D, FMT>& K, float k_scale,
                                                 uint32_t (&packed)[D / 128], uint16_t& gcode)
{
    using CB = KeyCodebook<FMT>;
    constexpr int EPL = D / 32;
    const float c0sq = K.c0sq, c1sq = K.c1sq, c2sq = K.c2sq, c3sq = K.c3sq;
    const uint32_t (&flip)[EPL] = K.flip;
    const float (&sgn)[5] = K.sgn;
    float x[EPL], a[EPL];
#pragma unroll
    for (int r = 0; r < EPL; r += 2) {
        const float2 f = e4m3x2_to_f32((raw[r >> 2] >> (8 * (r & 3))) & 0xFFFFu);
        x[r] = f.x;
        x[r + 1] = f.y;
    }
    if (k_scale != 1.0f) {           // a product with 1 is the factor itself: the common case skips it
#pragma unroll
        for (int r = 0; r < EPL; ++r) x[r] = __fmul_rn(x[r], k_scale);
    }
#pragma unroll
    for (int r = 0; r < EPL; ++r) a[r] = __uint_as_float(__float_as_uint(x[r]) ^ flip[r]);
    // Walsh-Hadamard butterflies, strides ascending: inside the lane, then across lanes
    // (stride 1 pairs neighbours: scalar; from stride 2 on two butterflies share one packed instruction)
#pragma unroll
    for (int r = 0; r < EPL; r += 2) {
        const float u = a[r], w = a[r + 1];
        a[r] = __fadd_rn(u, w);
        a[r + 1] = __fsub_rn(u, w);
    }
    f32x2 ap[EPL / 2];
    const f32x2 minus1 = pack2(-1.0f, -1.0f);
#pragma unroll
    for (int r = 0; r < EPL / 2; ++r) ap[r] = pack2(a[2 * r], a[2 * r + 1]);
#pragma unroll
    for (int hh = 1; hh < EPL / 2; hh <<= 1)            // strides 2, 4 of the elements = 1, 2 of the pairs
#pragma unroll
        for (int r = 0; r < EPL / 2; ++r)
            if ((r & hh) == 0) {
                const f32x2 u = ap[r], w = ap[r + hh];
                ap[r] = add2(u, w);
                ap[r + hh] = fma2(w, minus1, u);        // u - w: the product with -1 is exact, one rounding
            }
#pragma unroll
    for (int b = 0; b < 5; ++b) {
        const f32x2 s2 = pack2(sgn[b], sgn[b]);
#pragma unroll
        for (int r = 0; r < EPL / 2; ++r) {
            // lower lane: o + a; upper lane: o - a.  The product with +-1 is exact, so the fused form rounds
            // once, exactly like the single addition it stands for (zero signs included)
            float lo, hi;
            unpack2(ap[r], lo, hi);
            const float olo = __shfl_xor_sync(0xffffffffu, lo, 1 << b), ohi = __shfl_xor_sync(0xffffffffu, hi, 1 << b);
            ap[r] = fma2(ap[r], s2, pack2(olo, ohi));
        }
    }
#pragma unroll
    for (int r = 0; r < EPL / 2; ++r) unpack2(ap[r], a[2 * r], a[2 * r + 1]);
    // |x|^2: pairwise tree in index order (every element of the butterfly ends equal)
    float e[EPL];
#pragma unroll
    for (int r = 0; r < EPL; r += 2) {
        const f32x2 xx = pack2(x[r], x[r + 1]);
        unpack2(mul2(xx, xx), e[r], e[r + 1]);
    }
#pragma unroll
    for (int hh = 1; hh < EPL; hh <<= 1)
#pragma unroll
        for (int r = 0; r < EPL; r += 2 * hh) e[r] = __fadd_rn(e[r], e[r + hh]);
    float n2 = e[0];
#pragma unroll
    for (int m = 1; m < 32; m <<= 1) n2 = __fadd_rn(n2, __shfl_xor_sync(0xffffffffu, n2, m));
    const float nx = __fsqrt_rn(n2);
    const float t1 = __fmul_rn(CB::B0, nx), t2 = __fmul_rn(CB::B1, nx), t3 = __fmul_rn(CB::B2, nx);
    float f[EPL];
    uint32_t sq64 = 4u * EPL;          // record format 2: 64 x the sum of this lane's squared levels (4, 36, 121, 324)
#pragma unroll
    for (int r = 0; r < EPL / 4; ++r) packed[r] = 0;
#pragma unroll
    for (int r = 0; r < EPL; ++r) {
        const float w = fabsf(a[r]);
        const bool g1 = w > t1, g2 = w > t2, g3 = w > t3;
        // sign bit of the code: a[r] < 0 (a zero of either sign is positive)
        uint32_t code = a[r] < 0.0f ? 4u : 0u;
        if (g1) code += 1u;
        if (g2) code += 1u;
        if (g3) code += 1u;
        packed[r >> 2] |= code << (8 * (r & 3));
        if constexpr (FMT == 2) {
            if (g1) sq64 += 32u;
            if (g2) sq64 += 85u;
            if (g3) sq64 += 203u;
        } else {
            f[r] = g2 ? (g3 ? c3sq : c2sq) : (g1 ? c1sq : c0sq);
        }
    }
    float nc2;
    if constexpr (FMT == 2) {
        // The squared levels of format 2 are multiples of 1/64 and d of them sum to at most 5.0625 d, so every
        // partial sum of the pairwise tree is exact in fp32: any order gives the same bits, and the sum can be
        // taken in integers (one warp reduction) instead.
        static_assert(324 * D < (1 << 24), "exact in fp32");
        nc2 = __fmul_rn((float)__reduce_add_sync(0xffffffffu, sq64), 0.015625f);
    } else {
#pragma unroll
        for (int hh = 1; hh < EPL; hh <<= 1)
#pragma unroll
            for (int r = 0; r < EPL; r += 2 * hh) f[r] = __fadd_rn(f[r], f[r + hh]);
        nc2 = f[0];
#pragma unroll
        for (int m = 1; m < 32; m <<= 1) nc2 = __fadd_rn(nc2, __shfl_xor_sync(0xffffffffu, nc2, m));
    }
    const float nc = __fsqrt_rn(nc2);
    gcode = (nx == 0.0f) ? (uint16_t)0 : f32_to_f16_sat_bits(__fdiv_rn(nx, nc));
}

// Minimum and maximum of a channel by strict comparison in token order (of equal values, +0 and -0, the earliest counts).
__device__ __forceinline__ void literal_min_max(const float (&val)[kPage], float& mn, float& mx)
{
    mn = mx = val[0];
#pragma unroll
    for (int t = 1; t < kPage; ++t) {
        if (val[t] < mn) mn = val[t];
        if (val[t] > mx) mx = val[t];
    }
}

// clamp(rint((val - zp) / sc), 0, 7) with the correctly rounded quotient, 0 when sc == 0 (and for a NaN)
__device__ __forceinline__ uint32_t literal_value_code(float val, float scf, float zpf)
{
    const float den = scf != 0.0f ? scf : 1.0f, num = __fsub_rn(val, zpf);
    float r = rintf(__fdiv_rn(num != 0.0f ? num : den, den));   // half to even
    r = r < 0.0f ? 0.0f : r;
    r = r > 7.0f ? 7.0f : r;
    return (num != 0.0f && scf != 0.0f) ? (uint32_t)(int)r : 0u;
}

// Encodes the 16 tokens of one FP8 record (rec8) into the record image img = [key codes | value codes | g |
// scale/zero] in shared memory; all D threads of the block call it.  OWN_META: the value scale and zero come
// from these 16 tokens (16-token pages); otherwise thread c passes the page's scale/zero of channel c.
template <int D, bool OWN_META, int FMT>
__device__ __forceinline__ void demote_tile(const uint8_t* rec8, uint8_t* img, uint8_t* kcode, uint8_t* vcode,
                                            const DemoteLane<D, FMT>& K, float k_scale, float v_scale, uint16_t sc_page,
                                            uint16_t zp_page)
{
    constexpr int EPL = D / 32, NJ = D / 64, KROW = D + 8, NT = D;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // ---- keys: warp w encodes tokens w, w + NT/32, ... ------------------------------------------
    for (int tok = warp; tok < kPage; tok += NT / 32) {
        uint32_t raw[EPL / 4], packed[EPL / 4];
        uint16_t gcode;
        if constexpr (EPL == 8) {
            const uint2 u = *reinterpret_cast<const uint2*>(rec8 + tok * D + lane * EPL);
            raw[0] = u.x;
            raw[1] = u.y;
        } else {
            raw[0] = *reinterpret_cast<const uint32_t*>(rec8 + tok * D + lane * EPL);
        }
        encode_key_token<D, FMT>(raw, K, k_scale, packed, gcode);
        if constexpr (EPL == 8)
            *reinterpret_cast<uint2*>(kcode + tok * KROW + lane * EPL) = make_uint2(packed[0], packed[1]);
        else
            *reinterpret_cast<uint32_t*>(kcode + tok * KROW + lane * EPL) = packed[0];
        if (lane == 0) *reinterpret_cast<uint16_t*>(img + 12 * D + 2 * tok) = gcode;
    }

    // ---- values: one thread per channel, 16 tokens of the page ------------------------------
    for (int c = tid; c < D; c += NT) {
        const uint4 raw = *reinterpret_cast<const uint4*>(rec8 + 16 * D + c * kPage);
        const uint32_t rw[4] = {raw.x, raw.y, raw.z, raw.w};
        float val[kPage];
#pragma unroll
        for (int t = 0; t < kPage; t += 2) {
            const float2 f = e4m3x2_to_f32((rw[t >> 2] >> (8 * (t & 3))) & 0xFFFFu);
            val[t] = f.x;
            val[t + 1] = f.y;
        }
        if (v_scale != 1.0f) {
#pragma unroll
            for (int t = 0; t < kPage; ++t) val[t] = __fmul_rn(val[t], v_scale);
        }
        // scale and zero of the channel: from this tile's 16 tokens (16-token pages), or the page's (given)
        uint16_t sc = sc_page, zp = zp_page;
        if constexpr (OWN_META) {
            // minimum and maximum by strict comparison in token order.  The min/max instructions give the same
            // value except for the sign of a zero extreme and a leading NaN; those cases take the literal loop
            float mn = val[0], mx = val[0];
#pragma unroll
            for (int t = 1; t < kPage; ++t) {
                mn = fminf(mn, val[t]);
                mx = fmaxf(mx, val[t]);
            }
            if (!(mn != 0.0f && mx != 0.0f) || val[0] != val[0]) literal_min_max(val, mn, mx);
            sc = f32_to_f16_sat_bits(__fdiv_rn(__fsub_rn(mx, mn), 7.0f));
            zp = f32_to_f16_sat_bits(mn);
        }
        const float scf = __half2float(__ushort_as_half(sc)), zpf = __half2float(__ushort_as_half(zp));
        {
            const int cb = c >> 4, row = c & 15;
            uint16_t* meta = reinterpret_cast<uint16_t*>(img + 12 * D + 32);
            const int hi = (cb >> 1) * 64 + (row & 7) * 8 + 4 * (cb & 1) + (row >> 3);
            meta[hi] = sc;
            meta[hi + 2] = zp;
        }
        // q = clamp(rint((val - zp) / sc), 0, 7), 0 when sc == 0, the division correctly rounded.
        // The correctly rounded quotient d = RN(num / sc) without the divider: with y = RN(1 / sc) (one correctly
        // rounded reciprocal per channel), q0 = RN(num y) is within 1.5 ulp of the quotient, one residual step
        // q1 = RN(q0 + (num - sc q0) y) makes it faithful, and for a faithful q1 the second step gives exactly d
        // (Markstein's theorem; the residuals are exact in an FMA).  No intermediate can overflow or underflow when
        // the value scale is between 2^-20 and 2^20 (numerators are 0 or at least 2^-52 and below 2^30, scales are
        // fp16 numbers); other scales take the divider.  A zero scale gives y = 0 and code 0, a zero numerator code 0,
        // a NaN input code 0, all as the quotient form does.
        const float den = scf != 0.0f ? scf : 1.0f;
        uint32_t q4[4] = {0u, 0u, 0u, 0u};
        if (v_scale >= 9.5367431640625e-07f && v_scale <= 1048576.0f) {
            const float y = scf != 0.0f ? __frcp_rn(scf) : 0.0f;
            // two tokens per instruction: the packed fp32 operations round each half like the scalar ones
            const f32x2 y2 = pack2(y, y), nden2 = pack2(-den, -den), nzp2 = pack2(-zpf, -zpf);
#pragma unroll
            for (int t = 0; t < kPage; t += 2) {
                const f32x2 num = add2(pack2(val[t], val[t + 1]), nzp2);           // val - zp (= val + (-zp), one rounding)
                const f32x2 q0 = mul2(num, y2);
                const f32x2 q1 = fma2(fma2(nden2, q0, num), y2, q0);
                const f32x2 d2 = fma2(fma2(nden2, q1, num), y2, q1);
                float d0, d1;
                unpack2(d2, d0, d1);
                const float r0 = fminf(fmaxf(rintf(d0), 0.0f), 7.0f);        // half to even; NaN -> 0
                const float r1 = fminf(fmaxf(rintf(d1), 0.0f), 7.0f);
                q4[t >> 2] |= ((uint32_t)(int)r0 << (8 * (t & 3))) | ((uint32_t)(int)r1 << (8 * ((t + 1) & 3)));
            }
        } else {
#pragma unroll
            for (int t = 0; t < kPage; ++t) q4[t >> 2] |= literal_value_code(val[t], scf, zpf) << (8 * (t & 3));
        }
        *reinterpret_cast<uint4*>(vcode + c * kPage) = make_uint4(q4[0], q4[1], q4[2], q4[3]);
    }
    __syncthreads();

    // ---- pack: one thread per (section, triple j, fragment lane L) --------------------------
    for (int item = tid; item < 2 * NJ * 32; item += NT) {
        const int L = item & 31, j = (item >> 5) % NJ, section = item / (32 * NJ);
        const int g = L >> 2, tq = L & 3;
        uint32_t w0 = 0, w1 = 0, w2 = 0;
        if (section == 0 && FMT == 2) {
            // record format 2: register e = 4 (step % 2) + 2 u + b of the triple holds, in its four nibbles, the
            // codes of token g + 8u at dims 32 step + 16 b + 4 tq .. + 3 (steps 2j, 2j+1).  A: registers 0,1 with
            // the signs of 4,5; B: registers 2,3 with the signs of 6,7; C: magnitudes of 4,5 (low pair), 6,7 (high).
            uint32_t x[8];
#pragma unroll
            for (int e = 0; e < 8; ++e)
                x[e] = *reinterpret_cast<const uint32_t*>(kcode + (g + 8 * ((e >> 1) & 1)) * KROW + 32 * (2 * j + (e >> 2)) +
                                                          16 * (e & 1) + 4 * tq);
            auto signs = [](uint32_t v) { return squeeze4((v >> 2) & 0x01010101u) << 3; };
            auto mags = [](uint32_t v) { return squeeze4(v & 0x03030303u); };
            w0 = squeeze4(x[0]) | (squeeze4(x[1]) << 16) | signs(x[4]) | (signs(x[5]) << 16);
            w1 = squeeze4(x[2]) | (squeeze4(x[3]) << 16) | signs(x[6]) | (signs(x[7]) << 16);
            w2 = mags(x[4]) | (mags(x[5]) << 16) | ((mags(x[6]) | (mags(x[7]) << 16)) << 2);
        } else if (section == 0) {
            // key codes: nibble n = 2r + half holds row g + 8(r&1), slot 2tq + 8(r>>1) + half.
            // A: block 4j with the signs of block 4j+2; B: block 4j+1 with the signs of 4j+3;
            // C: magnitudes of blocks 4j+2 (low pair) and 4j+3 (high pair).
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const uint8_t* at = kcode + (g + 8 * (r & 1)) * KROW + 64 * j + 2 * tq + 8 * (r >> 1);
                const uint32_t b0 = *reinterpret_cast<const uint16_t*>(at);        // (half 0, half 1)
                const uint32_t b1 = *reinterpret_cast<const uint16_t*>(at + 16);
                const uint32_t b2 = *reinterpret_cast<const uint16_t*>(at + 32);
                const uint32_t b3 = *reinterpret_cast<const uint16_t*>(at + 48);
                w0 |= squeeze_nibbles(b0 | ((b2 & 0x0404u) << 1)) << (8 * r);
                w1 |= squeeze_nibbles(b1 | ((b3 & 0x0404u) << 1)) << (8 * r);
                w2 |= squeeze_nibbles((b2 & 0x0303u) | ((b3 & 0x0303u) << 2)) << (8 * r);
            }
        } else {
            // value codes: four 24-bit streams (group, half) per triple; stream code k is
            // channel block 4j + 2 grp + (k>>2), row g + 8(k&1), token 2tq + 8((k>>1)&1) + half
            uint32_t S[2][2] = {{0u, 0u}, {0u, 0u}};
#pragma unroll
            for (int grp = 0; grp < 2; ++grp)
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int cb = 4 * j + 2 * grp + (k >> 2), r = k & 3;
                    const uint32_t two = *reinterpret_cast<const uint16_t*>(
                        vcode + (16 * cb + g + 8 * (r & 1)) * kPage + 2 * tq + 8 * (r >> 1));
                    S[grp][0] |= (two & 7u) << (3 * k);
                    S[grp][1] |= (two >> 8) << (3 * k);
                }
            w0 = (S[0][0] & 0xFFFFu) | (S[0][1] << 16);
            w1 = (S[0][0] >> 16) | ((S[1][0] & 0xFFu) << 8) | ((S[0][1] >> 16) << 16) | (S[1][1] << 24);
            w2 = (S[1][0] >> 8) | ((S[1][1] >> 8) << 16);
        }
        uint8_t* sec = img + section * 6 * D;
        *reinterpret_cast<uint32_t*>(sec + lane_word_offset(D, L, 3 * j)) = w0;
        *reinterpret_cast<uint32_t*>(sec + lane_word_offset(D, L, 3 * j + 1)) = w1;
        *reinterpret_cast<uint32_t*>(sec + lane_word_offset(D, L, 3 * j + 2)) = w2;
    }
    __syncthreads();
}

template <int D, bool BIG, int FMT>
__global__ void __launch_bounds__(D) demote_kernel(const uint8_t* fp8, uint8_t* __restrict__ tq3,
                                                      int fp8_pages, int tq3_pages, int hkv, int tiles, float k_scale,
                                                      float v_scale, SigmaBits sigma,
                                                      const int32_t* src_ids,
                                                      const int32_t* dst_ids, int32_t* block_table,
                                                      uint8_t* tier_tag, const int64_t* entry_index, int64_t n_entries,
                                                      uint32_t* __restrict__ status, uint32_t* page_tickets)
{
    constexpr int KROW = D + 8;          // padded row of the key-code tile
    constexpr int REC = 16 * D + 32;     // bytes of one TQ3 record
    constexpr int NT = D;                // threads: one per value channel, one per packed word triple
    __shared__ __align__(16) uint8_t kcode[kPage * KROW];
    __shared__ __align__(16) uint8_t vcode[D * kPage];
    __shared__ __align__(16) uint8_t image[2][REC];

    const int csize = (int)cluster_size(), crank = (int)cluster_rank();
    const int page = blockIdx.x / csize, tid = threadIdx.x, lane = tid & 31;
    pdl_wait();
    const int src = src_ids[page], dst = dst_ids[page];
    const bool valid = src >= 0 && src < fp8_pages && dst >= 0 && dst < tq3_pages;
    if (!valid && tid == 0 && crank == 0 && blockIdx.y == 0) atomicOr(status, kStBounds);
    DemoteLane<D, FMT> lane_consts;
    lane_consts.init(sigma, lane);

    int it = 0;
    for (int h = crank; valid && h < hkv; h += csize) {
        if constexpr (!BIG) {
            const uint8_t* rec8 = fp8 + ((size_t)src * hkv + h) * fp8_record_bytes(D);
            uint8_t* rec3 = tq3 + ((size_t)dst * hkv + h) * tq3_record_bytes(D);
            uint8_t* img = image[it++ & 1];
            demote_tile<D, true, FMT>(rec8, img, kcode, vcode, lane_consts, k_scale, v_scale, 0, 0);
            for (int i = tid; i < REC / 16; i += NT)
                reinterpret_cast<uint4*>(rec3)[i] = reinterpret_cast<const uint4*>(img)[i];
        } else {
            // pages of several tiles: the page's scale/zero were written by demote_minmax_kernel; the blocks of
            // grid row y take tiles y, y + gridDim.y, ... and write the tile part of the image only
            constexpr int TILE = 12 * D + 32;
            uint8_t* page3 = tq3 + ((size_t)dst * hkv + h) * tq3_page_bytes(D, tiles);
            const uint16_t* meta = reinterpret_cast<const uint16_t*>(page3 + (size_t)tiles * TILE);
            const int cb = tid >> 4, row = tid & 15;
            const int hi = (cb >> 1) * 64 + (row & 7) * 8 + 4 * (cb & 1) + (row >> 3);
            const uint16_t sc = meta[hi], zp = meta[hi + 2];
            for (int m = blockIdx.y; m < tiles; m += gridDim.y) {
                const uint8_t* rec8 = fp8 + (((size_t)src * hkv + h) * tiles + m) * fp8_record_bytes(D);
                uint8_t* img = image[it++ & 1];
                demote_tile<D, false, FMT>(rec8, img, kcode, vcode, lane_consts, k_scale, v_scale, sc, zp);
                uint4* out = reinterpret_cast<uint4*>(page3 + (size_t)m * TILE);
                for (int i = tid; i < TILE / 16; i += NT) out[i] = reinterpret_cast<const uint4*>(img)[i];
            }
        }
    }

    // copy-before-publish: every head's record is complete and visible before the id and tag appear.  The cluster
    // barrier (release / acquire) orders the record stores of every thread of the cluster before what the
    // publishing thread does next, and that thread's fence is cumulative: it orders them, device-wide, before its
    // own later stores.  (A fence in every thread would say the same and make each of them wait for its stores.)
    pdl_let_next_start();                   // (not sooner: see launch_pdl)
    cluster_barrier();
    if (valid && crank == 0 && tid == 0 && entry_index != nullptr && (__threadfence(), last_cluster_of_page(page_tickets, page))) {
        const int64_t e = entry_index[page];
        if (e >= n_entries) atomicOr(status, kStBounds);      // an entry beyond the tables: flagged, nothing published
        else if (e >= 0) {
            block_table[e] = dst;
            __threadfence();
            tier_tag[e] = (uint8_t)MKV_TAG_STALE;
        }
    }
}

// A lane's words of one code section to global memory, in the record's 16-byte chunks.
template <int D>
__device__ __forceinline__ void store_lane_words(uint8_t* sec, int lane, const uint32_t (&w)[3 * (D / 16) / 4])
{
    constexpr int LW = 3 * (D / 16) / 4;
#pragma unroll
    for (int c = 0; c < LW / 4; ++c)
        *reinterpret_cast<uint4*>(sec + c * 512 + lane * 16) = make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
    if constexpr (LW % 4 != 0)
        *reinterpret_cast<uint2*>(sec + (LW / 4) * 512 + lane * 8) = make_uint2(w[LW - 2], w[LW - 1]);
}

// squared level of a magnitude (a single fp32 product, as the record's norm correction defines it)
template <int FMT>
__device__ __forceinline__ float level_sq(uint32_t mag)
{
    using CB = KeyCodebook<FMT>;
    const float c0 = __fmul_rn(CB::C0, CB::C0), c1 = __fmul_rn(CB::C1, CB::C1), c2 = __fmul_rn(CB::C2, CB::C2),
                c3 = __fmul_rn(CB::C3, CB::C3);
    return mag & 2u ? (mag & 1u ? c3 : c2) : (mag & 1u ? c1 : c0);
}

#include "demote_warp.cuh"

// Pages of several tiles, first pass of Demote: the minimum and maximum of every value channel over all tokens
// of the page, then the page's scale and zero (same arithmetic and order of the halves as in the 16-token
// record).  One cluster per (page, KV head); block r of the cluster scans tiles r, r + cluster size, ... with one
// thread per channel, the partial extremes meet in the first block through distributed shared memory.
// The extremes are defined by a scan in token order with strict comparisons; min/max instructions give the same
// value except for the sign of a zero extreme and a leading NaN, and those channels (rare) are scanned again
// literally, by the thread that writes the result.
__device__ __forceinline__ float ld_cluster_f32(const float* local, uint32_t rank)
{
    uint32_t remote;
    float v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"((uint32_t)__cvta_generic_to_shared(local)), "r"(rank));
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(remote) : "memory");
    return v;
}

template <int D>
__global__ void __launch_bounds__(D) demote_minmax_kernel(const uint8_t* fp8, uint8_t* __restrict__ tq3,
                                                           int fp8_pages, int tq3_pages, int hkv, int tiles,
                                                           float v_scale, const int32_t* src_ids,
                                                           const int32_t* dst_ids)
{
    __shared__ float part[2][D];
    const int csize = (int)cluster_size(), crank = (int)cluster_rank();
    const int unit = blockIdx.x / csize, page = unit / hkv, h = unit % hkv, c = threadIdx.x;
    pdl_wait();
    const int src = src_ids[page], dst = dst_ids[page];
    const bool valid = src >= 0 && src < fp8_pages && dst >= 0 && dst < tq3_pages;      // flagged by demote_kernel
    const uint8_t* page8 = fp8 + ((size_t)(valid ? src : 0) * hkv + h) * fp8_page_bytes(D, tiles);
    auto value = [&](uint32_t two, int half) {
        const float2 f = e4m3x2_to_f32(two & 0xFFFFu);
        return __fmul_rn(half ? f.y : f.x, v_scale);
    };
    // every block starts from the page's first token, so that a block without tiles is neutral
    const float first = valid ? value(*reinterpret_cast<const uint32_t*>(page8 + 16 * D + c * kPage), 0) : 0.f;
    float mn = first, mx = first;
    constexpr int AHEAD = 4;        // tiles whose loads are issued together (a thread's tiles are 4 KB apart)
    for (int m0 = crank; valid && m0 < tiles; m0 += AHEAD * csize) {
        uint4 raw[AHEAD];
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
            const int m = m0 + u * csize;
            raw[u] = m < tiles ? *reinterpret_cast<const uint4*>(page8 + (size_t)m * fp8_record_bytes(D) + 16 * D + c * kPage)
                               : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int u = 0; u < AHEAD; ++u) {
            if (m0 + u * csize >= tiles) break;
            const uint32_t rw[4] = {raw[u].x, raw[u].y, raw[u].z, raw[u].w};
#pragma unroll
            for (int t = 0; t < kPage; t += 2) {
                const uint32_t two = rw[t >> 2] >> (8 * (t & 3));
                const float a = value(two, 0), b = value(two, 1);
                mn = fminf(mn, fminf(a, b));
                mx = fmaxf(mx, fmaxf(a, b));
            }
        }
    }
    part[0][c] = mn;
    part[1][c] = mx;
    pdl_let_next_start();                   // (not sooner: see launch_pdl)
    cluster_barrier();
    if (crank == 0 && valid) {
        for (int k = 1; k < csize; ++k) {
            mn = fminf(mn, ld_cluster_f32(&part[0][c], (uint32_t)k));
            mx = fmaxf(mx, ld_cluster_f32(&part[1][c], (uint32_t)k));
        }
        if (!(mn != 0.0f && mx != 0.0f) || first != first) {
            // the literal scan: of equal values (+0 and -0) the earliest token counts
            mn = mx = first;
            for (int m = 0; m < tiles; ++m) {
                const uint4 raw = *reinterpret_cast<const uint4*>(page8 + (size_t)m * fp8_record_bytes(D) + 16 * D + c * kPage);
                const uint32_t rw[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
                for (int t = 0; t < kPage; ++t) {
                    const float a = value(rw[t >> 2] >> (8 * (t & 2)), t & 1);
                    if (a < mn) mn = a;
                    if (a > mx) mx = a;
                }
            }
        }
        uint16_t* meta = reinterpret_cast<uint16_t*>(tq3 + ((size_t)dst * hkv + h) * tq3_page_bytes(D, tiles) +
                                                     (size_t)tiles * (12 * D + 32));
        const int cb = c >> 4, row = c & 15;
        const int hi = (cb >> 1) * 64 + (row & 7) * 8 + 4 * (cb & 1) + (row >> 3);
        meta[hi] = f32_to_f16_sat_bits(__fdiv_rn(__fsub_rn(mx, mn), 7.0f));
        meta[hi + 2] = f32_to_f16_sat_bits(mn);
    }
    cluster_barrier();              // the partial extremes stay readable until the first block has taken them
}

// Pages of several tiles, last pass of Demote / Promote: the kernels before it in the stream have written the
// whole page, so its id and tag may appear (copy-before-publish by stream order).
__global__ void publish_kernel(int n, const int32_t* src_ids, const int32_t* dst_ids,
                               int src_cap, int dst_cap, int32_t* block_table, uint8_t* tier_tag,
                               const int64_t* entry_index, int64_t n_entries, int tag, uint32_t* status)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    pdl_begin();
    if (i >= n) return;
    const int src = src_ids[i], dst = dst_ids[i];
    if (src < 0 || src >= src_cap || dst < 0 || dst >= dst_cap) return;
    const int64_t e = entry_index[i];
    if (e >= n_entries) atomicOr(status, kStBounds);
    else if (e >= 0) {
        block_table[e] = dst;
        __threadfence();
        tier_tag[e] = (uint8_t)tag;
    }
}

// Page tickets of the in-kernel publication: 48 counters in the pool's 256-byte status tail (word 0 is the status
// word, words 16..63 the tickets; the tail is zeroed with the arenas and every use leaves its counter at zero).
// Calls that convert more pages publish with a kernel of their own.
constexpr int kPageTickets = 48;
static uint32_t* page_tickets(mkv_pool* p) { return p->status_dev + 16; }

// grid rows of the tile-parallel passes: at least 16, and enough to fill the GPU when few pages are converted
static int tile_rows(int tiles, int n_pages, int hkv, int sms)
{
    int rows = (4 * sms + n_pages * hkv - 1) / (n_pages * hkv);
    if (rows < 16) rows = 16;
    return rows < tiles ? rows : tiles;
}

// blocks per page of the warp kernels: one, or a cluster that has a warp for every head when the call has few pages
static int warp_cluster(int hkv, int n_pages, int sms)
{
    const int c = (hkv + kDemoteWarps - 1) / kDemoteWarps;
    return n_pages > 2 * sms ? 1 : c < 8 ? c : 8;
}

// grid rows of the tile-parallel warp kernels: enough for 12 warps on every SM
static int warp_tile_rows(int tiles, int n_pages, int hkv, int sms)
{
    int rows = (12 * sms + n_pages * hkv - 1) / (n_pages * hkv);
    if (rows < 16) rows = 16;
    return rows < tiles ? rows : tiles;
}

template <int D, int FMT, bool BIG>
static cudaError_t launch_demote_warp(mkv_pool* p, const int32_t* src, const int32_t* dst, int n, int32_t* bt, uint8_t* tags,
                                      const int64_t* entry, int64_t n_entries, uint32_t* tickets, cudaStream_t s)
{
    const int warps = p->hkv < kDemoteWarps ? p->hkv : kDemoteWarps, c = warp_cluster(p->hkv, BIG ? 0 : n, p->dev.sm_count);
    const int smem = DemoteWarp<D>::OFF_WARPS + warps * DemoteWarp<D>::BYTES;
    static_assert(DemoteWarp<D>::OFF_WARPS + kDemoteWarps * DemoteWarp<D>::BYTES <= 48 * 1024, "no opt-in needed");
    return launch_pdl(demote_warp_kernel<D, FMT, BIG>, dim3((unsigned)n * c, BIG ? warp_tile_rows(p->tiles, n, p->hkv, p->dev.sm_count) : 1), 32 * warps,
                      (size_t)smem, c, s, (const uint8_t*)p->fp8, p->tq3, p->cfg.fp8_pages, p->cfg.tq3_pages, p->hkv,
                      p->tiles, p->sigma, src, dst, bt, tags, entry, n_entries, p->status_dev, tickets);
}

template <int D, int FMT>
static int32_t launch_demote_d(mkv_pool* p, const int32_t* src, const int32_t* dst, int n, int32_t* bt, uint8_t* tags,
                               const int64_t* entry, int64_t n_entries, cudaStream_t s)
{
    const bool unit_scales = p->cfg.k_scale == 1.0f && p->cfg.v_scale == 1.0f;      // what the warp kernel's exactness rests on
    // Few records at d = 256 take the general kernel: eight warps share a record and its code is a loop, where the warp
    // kernel runs 3,900 instructions in a row, which a call between two decode scans has to fetch anew.  Between decode
    // calls one page of 4 heads takes 9 us in the general kernel, 20 (format 1) and 17 us in the warp kernel, a page of
    // 1,792 tokens 22 against 29 and 23 against 25; the two meet at about 1,200 tile records in format 1 (24 us) and
    // 800 in the shorter code of format 2 (18.5 us).  At d = 128 they differ by less than 1.5 us.
    const bool few = D == 256 && (long long)n * p->hkv * p->tiles <= (FMT == 1 ? 8 : 5) * (long long)p->dev.sm_count;
    const bool warp_per_record = unit_scales && !few;
    if (p->tiles == 1 && warp_per_record) {
        MKV_CUDA((launch_demote_warp<D, FMT, false>(p, src, dst, n, bt, tags, entry, n_entries, nullptr, s)));
        return MKV_OK;
    }
    if (p->tiles == 1) {
        const int c = heads_cluster(p->hkv, n, p->dev.sm_count);
        MKV_CUDA(launch_pdl(demote_kernel<D, false, FMT>, dim3((unsigned)n * c), D, 0, c, s, (const uint8_t*)p->fp8, p->tq3, p->cfg.fp8_pages,
                                  p->cfg.tq3_pages, p->hkv, 1, p->cfg.k_scale, p->cfg.v_scale, p->sigma, src, dst, bt,
                                  tags, entry, n_entries, p->status_dev, (uint32_t*)nullptr));
        return MKV_OK;
    }
    // pages of several tiles: scale/zero of the page, then the tiles in parallel, then the publication (from inside
    // the tile kernel when the call is small enough for the pool's page tickets, else as a kernel of its own)
    const bool fused = entry != nullptr && n <= kPageTickets;
    {
        // blocks per (page, head): up to a portable cluster of 8, fewer when the call fills the GPU anyway
        int cs = 8;
        while (cs > 1 && (cs > p->tiles || (long long)n * p->hkv * cs > 8LL * p->dev.sm_count)) cs >>= 1;
        MKV_CUDA(launch_pdl(demote_minmax_kernel<D>, dim3((unsigned)n * p->hkv * cs), D, 0, cs, s, (const uint8_t*)p->fp8, p->tq3, p->cfg.fp8_pages,
                                  p->cfg.tq3_pages, p->hkv, p->tiles, p->cfg.v_scale, src, dst));
    }
    const int ch = heads_cluster(p->hkv, 0, p->dev.sm_count);
    if (warp_per_record)
        MKV_CUDA((launch_demote_warp<D, FMT, true>(p, src, dst, n, fused ? bt : nullptr, fused ? tags : nullptr,
                                                   fused ? entry : nullptr, fused ? n_entries : 0, fused ? page_tickets(p) : nullptr, s)));
    else
        MKV_CUDA(launch_pdl(demote_kernel<D, true, FMT>, dim3((unsigned)n * ch, tile_rows(p->tiles, n, p->hkv, p->dev.sm_count)), D, 0, ch, s,
                                   (const uint8_t*)p->fp8, p->tq3, p->cfg.fp8_pages, p->cfg.tq3_pages, p->hkv, p->tiles,
                                   p->cfg.k_scale, p->cfg.v_scale, p->sigma, src, dst, fused ? bt : (int32_t*)nullptr,
                                   fused ? tags : (uint8_t*)nullptr, fused ? entry : (const int64_t*)nullptr,
                                   fused ? n_entries : (int64_t)0, p->status_dev, fused ? page_tickets(p) : (uint32_t*)nullptr));
    if (entry && !fused) {
        MKV_CUDA(launch_pdl(publish_kernel, dim3((n + 127) / 128), 128, 0, 1, s, n, src, dst, p->cfg.fp8_pages, p->cfg.tq3_pages, bt, tags, entry,
                                                       n_entries, MKV_TAG_STALE, p->status_dev));
        MKV_CUDA(cudaGetLastError());
    }
    return MKV_OK;
}

int32_t launch_demote(mkv_pool* p, const int32_t* src, const int32_t* dst, int n, int32_t* bt, uint8_t* tags,
                      const int64_t* entry, int64_t n_entries, cudaStream_t s)
{
    if (p->fmt == 2)
        return p->d == 128 ? launch_demote_d<128, 2>(p, src, dst, n, bt, tags, entry, n_entries, s)
                           : launch_demote_d<256, 2>(p, src, dst, n, bt, tags, entry, n_entries, s);
    return p->d == 128 ? launch_demote_d<128, 1>(p, src, dst, n, bt, tags, entry, n_entries, s)
                       : launch_demote_d<256, 1>(p, src, dst, n, bt, tags, entry, n_entries, s);
}

// ------------------------------------------------------------------------------------------ promote
// Promote (Algorithm 1 step 3): reconstruct a Stale page into a newly allocated FP8 page, then publish it as Anchor.
#include "promote_warp.cuh"

template <int D, int FMT, bool BIG>
static cudaError_t launch_promote_warp(mkv_pool* p, const int32_t* src, const int32_t* dst, int n, int32_t* bt, uint8_t* tags,
                                       const int64_t* entry, int64_t n_entries, uint32_t* tickets, cudaStream_t s)
{
    const int warps = p->hkv < kDemoteWarps ? p->hkv : kDemoteWarps, c = warp_cluster(p->hkv, BIG ? 0 : n, p->dev.sm_count);
    const int smem = PromoteWarp<D>::OFF_WARPS + warps * PromoteWarp<D>::BYTES;
    static_assert(PromoteWarp<D>::OFF_WARPS + kDemoteWarps * PromoteWarp<D>::BYTES <= 48 * 1024, "no opt-in needed");
    const float ik = 1.0f / p->cfg.k_scale, iv = 1.0f / p->cfg.v_scale, rs = (float)(1.0 / sqrt((double)p->d));
    return launch_pdl(promote_warp_kernel<D, FMT, BIG>, dim3((unsigned)n * c, BIG ? warp_tile_rows(p->tiles, n, p->hkv, p->dev.sm_count) : 1),
                      32 * warps, (size_t)smem, c, s, (const uint8_t*)p->tq3, p->fp8, p->cfg.tq3_pages, p->cfg.fp8_pages,
                      p->hkv, p->tiles, ik, iv, rs, p->sigma, src, dst, bt, tags, entry, n_entries, p->status_dev, tickets);
}

template <int D, int FMT>
static int32_t launch_promote_d(mkv_pool* p, const int32_t* src, const int32_t* dst, int n, int32_t* bt, uint8_t* tags,
                                const int64_t* entry, int64_t n_entries, cudaStream_t s)
{
    if (p->tiles == 1) {
        MKV_CUDA((launch_promote_warp<D, FMT, false>(p, src, dst, n, bt, tags, entry, n_entries, nullptr, s)));
        return MKV_OK;
    }
    const bool fused = entry != nullptr && n <= kPageTickets;
    MKV_CUDA((launch_promote_warp<D, FMT, true>(p, src, dst, n, fused ? bt : nullptr, fused ? tags : nullptr,
                                                fused ? entry : nullptr, fused ? n_entries : 0, fused ? page_tickets(p) : nullptr, s)));
    if (entry && !fused) {
        MKV_CUDA(launch_pdl(publish_kernel, dim3((n + 127) / 128), 128, 0, 1, s, n, src, dst, p->cfg.tq3_pages,
                            p->cfg.fp8_pages, bt, tags, entry, n_entries, MKV_TAG_ANCHOR, p->status_dev));
    }
    return MKV_OK;
}

int32_t launch_promote(mkv_pool* p, const int32_t* src, const int32_t* dst, int n, int32_t* bt, uint8_t* tags,
                       const int64_t* entry, int64_t n_entries, cudaStream_t s)
{
    if (p->fmt == 2)
        return p->d == 128 ? launch_promote_d<128, 2>(p, src, dst, n, bt, tags, entry, n_entries, s)
                           : launch_promote_d<256, 2>(p, src, dst, n, bt, tags, entry, n_entries, s);
    return p->d == 128 ? launch_promote_d<128, 1>(p, src, dst, n, bt, tags, entry, n_entries, s)
                       : launch_promote_d<256, 1>(p, src, dst, n, bt, tags, entry, n_entries, s);
}

// ------------------------------------------------------------------------------------------ anchor
__global__ void set_anchor_kernel(uint8_t* tags, int64_t entry, int flag, uint32_t* status)
{
    pdl_begin();
    if (tags[entry] == MKV_TAG_STALE)
        atomicOr(status, kStState);
    else
        tags[entry] = flag ? MKV_TAG_ANCHOR : MKV_TAG_RECENT;
}

int32_t launch_set_anchor(mkv_pool* p, uint8_t* tags, int64_t entry, int flag, cudaStream_t s)
{
    MKV_CUDA(launch_pdl(set_anchor_kernel, dim3(1), 1, 0, 1, s, tags, entry, flag, p->status_dev));
    MKV_CUDA(cudaGetLastError());
    return MKV_OK;
}

}  // namespace mkv
