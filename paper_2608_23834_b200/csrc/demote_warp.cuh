// Demote with one warp per (page, KV head) or (tile, KV head), for pools whose FP8 scales are 1 (included by
// lifecycle_kernels.cu).
//
// The encoder is defined as a sequence of fp32 operations, and the records are those bit for bit; what changes is
// how the same numbers are reached (per page and head at d = 256, 8,760 -> 3,730 warp instructions):
//   * The Hadamard transform of an e4m3 vector is exact in fp32 as long as its coordinates are not huge: they are
//     multiples of 2^-9, and with |x|^2 < kExactNorm2 = 2^22 (checked on the norm that the encoder needs anyway) a signed
//     sum of n <= 256 of them is at most sqrt(n) |x| <= 2^15, that is 2^24 units of 2^-9: every partial sum is an integer
//     that fp32 holds, and every order of summation gives the same value (the sums of 16 inside an MMA are at most
//     2^22 units of products below 2^18).  Outlier channels of real keys stay far below; beyond are only records
//     whose coordinates average more than 128 of e4m3's 448.  H_d is then
//     taken as H_16 on the dims of a 16-dim block, by tensor-core products with a +-512 matrix (32 MMAs), times
//     butterflies over the blocks, which a lane has all to itself (packed additions, no shuffles; the 16 shuffle
//     stages per token were a quarter of the instructions).  The factor 512 makes every coordinate an integer, so a
//     threshold comparison is one saturating addition.
//   * The MMA's columns are ordered so that a lane ends with the codes of exactly the (token, dim) places that its
//     words of the record hold: key words are built in registers and stored.
//   * Value codes: coordinates and zero are multiples of 2^-9 and the fp16 scale of a range of such numbers leaves
//     every quotient either exactly on a half-integer or at least 2^-16 away from one, so an approximate quotient
//     rounded to 2^-18 decides like the correctly rounded one (checked over all ranges and values, tests): three packed
//     operations per two tokens instead of two divisions.
// Records with such keys or with NaNs take the literal sequence (per record for keys, per channel for values).

template <int D>
struct DemoteWarp {
    static constexpr int NBLK = D / 16, LW = 3 * NBLK / 4;
    static constexpr int KST = D + 16;               // padded token row of the staged keys (conflict-free ldmatrix)
    static constexpr int OFF_V = kPage * KST, OFF_META = OFF_V + kPage * D, BYTES = OFF_META + 4 * D;
    static constexpr int OFF_SIG = 0, OFF_WARPS = NBLK * 16;
    static_assert(kPage * KST >= kPage * D && OFF_V % 16 == 0 && OFF_META % 16 == 0, "value codes take the place of the keys");
};
constexpr int kDemoteWarps = 4;                      // warps per block, one head each
constexpr float kExactNorm2 = 4194304.0f;

__device__ __forceinline__ uint32_t e4m3x2_to_f16x2_bits(uint32_t two_bytes)
{
    const __half2_raw h = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)two_bytes, __NV_E4M3);
    return (uint32_t)h.x | ((uint32_t)h.y << 16);
}

__device__ __forceinline__ float2 f16x2_to_f32(uint32_t x) { return __half22float2(*reinterpret_cast<const __half2*>(&x)); }

// x * y + c of fp16 factors and an fp32 addend, rounded once: 1.1 cycles a warp and scheduler where a conversion alone takes
// 2.0 (3,500 pages of 4 heads, d 256, back to back: 91.2 -> 89.4 us)
__device__ __forceinline__ float fma_f16(uint16_t x, uint16_t y, float c)
{
    float r;
    asm("fma.rn.f32.f16 %0, %1, %2, %3;" : "=f"(r) : "h"(x), "h"(y), "f"(c));
    return r;
}
__device__ __forceinline__ uint16_t low_half(uint32_t x) { return (uint16_t)(x & 0xFFFFu); }
__device__ __forceinline__ uint16_t high_half(uint32_t x) { return (uint16_t)(x >> 16); }

__device__ __forceinline__ void hmma_zero(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

__device__ __forceinline__ float add_sat(float a, float b)
{
    float r;
    asm("add.sat.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4])
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}

// Bytes of 0xFF or 0x00 by the signs of two floats (selector nibbles 0xB: the first, 0xF: the second)
template <uint32_t SEL>
__device__ __forceinline__ uint32_t sign_bytes(float a, float b)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(__float_as_uint(a)), "r"(__float_as_uint(b)), "n"(SEL));
    return r;
}

// fp16 pair (+-512, +-512): (-1)^popc(k & n) 512 for two values of k
__device__ __forceinline__ uint32_t h16_pair(int k0, int k1, int n)
{
    return (0x6000u | ((__popc(k0 & n) & 1u) << 15)) | ((0x6000u | ((__popc(k1 & n) & 1u) << 15)) << 16);
}

// range / 7, correctly rounded (one reciprocal step from 1/7 rounded; Markstein's theorem; checked over all ranges)
__device__ __forceinline__ float div7(float x)
{
    const float y = 1.0f / 7.0f, q = __fmul_rn(x, y);
    return __fmaf_rn(__fmaf_rn(-7.0f, q, x), y, q);
}

// Magnitude |y| > t of an integer-valued y: saturate(|y| - floor(t)) is 1 or 0.  acc <- acc * step + number of the
// three thresholds that |y| exceeds.
__device__ __forceinline__ float push_magnitude(float acc, float step, float y, const float (&nt)[3])
{
    const float w = fabsf(y);
    return __fadd_rn(__fadd_rn(__fmaf_rn(acc, step, add_sat(w, nt[0])), add_sat(w, nt[1])), add_sat(w, nt[2]));
}

template <int D, int FMT, bool BIG>
__global__ void __launch_bounds__(32 * kDemoteWarps, D == 256 ? 3 : 4)
demote_warp_kernel(const uint8_t* fp8, uint8_t* __restrict__ tq3, int fp8_pages, int tq3_pages, int hkv, int tiles,
                   SigmaBits sigma, const int32_t* src_ids, const int32_t* dst_ids,
                   int32_t* block_table, uint8_t* tier_tag, const int64_t* entry_index, int64_t n_entries,
                   uint32_t* __restrict__ status, uint32_t* page_tickets)
{
    using G = DemoteWarp<D>;
    using CB = KeyCodebook<FMT>;
    constexpr uint32_t FULL = 0xffffffffu;
    constexpr int NBLK = G::NBLK, LW = G::LW, KST = G::KST, TILE = 12 * D + 32;
    extern __shared__ __align__(16) uint8_t dsm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, tq = lane & 3, n_warps = blockDim.x >> 5;
    uint32_t* sig = reinterpret_cast<uint32_t*>(dsm + G::OFF_SIG);         // [block][tq] sign bits of four bytes
    uint8_t* kbuf = dsm + G::OFF_WARPS + warp * G::BYTES;
    uint8_t* vbuf = kbuf + G::OFF_V;
    uint16_t* meta = reinterpret_cast<uint16_t*>(kbuf + G::OFF_META);
    const int csize = (int)cluster_size(), crank = (int)cluster_rank();
    const int page = blockIdx.x / csize;
    for (int i = tid; i < NBLK * 4; i += blockDim.x) {
        const int dim = 4 * i;
        const uint32_t n = (sigma.w[dim >> 5] >> (dim & 31)) & 0xFu;
        sig[i] = ((n * 0x00204081u) & 0x01010101u) << 7;
    }
    // B operands of H_16: K slot 2tq + e (and 8 + 2tq + e) is dim 4tq + e (4tq + 2 + e) of the block; column n = g of tile t
    // is the output dim that the record keeps in this place: 4 (n / 2) + 2t + n % 2 in format 2, 8t + n in format 1
    uint32_t hb[2][2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const int n = FMT == 2 ? 4 * (g >> 1) + 2 * t + (g & 1) : 8 * t + g;
        hb[t][0] = h16_pair(4 * tq, 4 * tq + 1, n);
        hb[t][1] = h16_pair(4 * tq + 2, 4 * tq + 3, n);
    }
    pdl_wait();
    __syncthreads();
    const int src = src_ids[page], dst = dst_ids[page];
    const bool valid = src >= 0 && src < fp8_pages && dst >= 0 && dst < tq3_pages;
    if (!valid && tid == 0 && crank == 0 && blockIdx.y == 0) atomicOr(status, kStBounds);

    const int m_first = BIG ? (int)blockIdx.y : 0, m_step = BIG ? (int)gridDim.y : 1, m_end = BIG ? tiles : 1;
    for (int h = crank * n_warps + warp; valid && h < hkv; h += csize * n_warps)
    for (int m = m_first; m < m_end; m += m_step) {
        const uint8_t* rec8 = fp8 + (((size_t)src * hkv + h) * tiles + m) * fp8_record_bytes(D);
        uint8_t* page3 = tq3 + ((size_t)dst * hkv + h) * tq3_page_bytes(D, tiles);
        uint8_t* out = page3 + (size_t)m * TILE;
        // ---- stage the record -----------------------------------------------------------------------------
        __syncwarp();
#pragma unroll
        for (int i = lane; i < D; i += 32) cp_async16(kbuf + (i / (D / 16)) * KST + 16 * (i % (D / 16)), rec8 + 16 * i);
#pragma unroll
        for (int i = lane; i < D; i += 32) cp_async16(vbuf + 16 * i, rec8 + 16 * D + 16 * i);
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncwarp();

        // ---- keys: tokens g and g + 8, dims 4tq .. 4tq + 3 of every block -----------------------------------
        uint32_t words[NBLK];               // format 2: [token half][block pair], format 1: [block]: eight codes each
        uint16_t gcode[2];
        {
            uint32_t a[NBLK][4];
            float e0[NBLK], e1[NBLK];
            const uint32_t row = (uint32_t)__cvta_generic_to_shared(kbuf) + (lane & 15) * KST + 16 * (lane >> 4);
#pragma unroll
            for (int b0 = 0; b0 < NBLK; b0 += 2) {
                uint32_t w[4];
                ldsm4(row + 16 * b0, w);
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    const uint32_t s = sig[(b0 + b) * 4 + tq], w0 = w[2 * b] ^ s, w1 = w[2 * b + 1] ^ s;
                    a[b0 + b][0] = e4m3x2_to_f16x2_bits(w0 & 0xFFFFu);
                    a[b0 + b][1] = e4m3x2_to_f16x2_bits(w1 & 0xFFFFu);
                    a[b0 + b][2] = e4m3x2_to_f16x2_bits(w0 >> 16);
                    a[b0 + b][3] = e4m3x2_to_f16x2_bits(w1 >> 16);
                    // first two levels of the pairwise tree of squares (a square is exact, so the fused form rounds once)
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        auto two_squares = [](uint32_t x) {
                            return fma_f16(high_half(x), high_half(x), fma_f16(low_half(x), low_half(x), 0.0f));
                        };
                        (u == 0 ? e0 : e1)[b0 + b] = __fadd_rn(two_squares(a[b0 + b][u]), two_squares(a[b0 + b][2 + u]));
                    }
                }
            }
#pragma unroll
            for (int o = 1; o <= 2; o <<= 1)
#pragma unroll
                for (int b = 0; b < NBLK; ++b) {
                    e0[b] = __fadd_rn(e0[b], __shfl_xor_sync(FULL, e0[b], o));
                    e1[b] = __fadd_rn(e1[b], __shfl_xor_sync(FULL, e1[b], o));
                }
#pragma unroll
            for (int o = 1; o < NBLK; o <<= 1)
#pragma unroll
                for (int b = 0; b < NBLK; b += 2 * o) {
                    e0[b] = __fadd_rn(e0[b], e0[b + o]);
                    e1[b] = __fadd_rn(e1[b], e1[b + o]);
                }
            if (__all_sync(FULL, e0[0] < kExactNorm2 && e1[0] < kExactNorm2)) {
                const float nx[2] = {__fsqrt_rn(e0[0]), __fsqrt_rn(e1[0])};
                float nt[2][3];             // minus the thresholds, in units of 2^-9, rounded down
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    nt[u][0] = -floorf(__fmul_rn(CB::B0, nx[u]) * 512.0f);
                    nt[u][1] = -floorf(__fmul_rn(CB::B1, nx[u]) * 512.0f);
                    nt[u][2] = -floorf(__fmul_rn(CB::B2, nx[u]) * 512.0f);
                }
                float f0[FMT == 1 ? NBLK : 1], f1[FMT == 1 ? NBLK : 1];     // format 1: 16-dim sums of squared levels
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    float c[NBLK][4];
#pragma unroll
                    for (int b = 0; b < NBLK; ++b) hmma_zero(c[b], a[b], hb[t][0], hb[t][1]);
                    f32x2 v[NBLK][2];
                    const f32x2 minus1 = pack2(-1.0f, -1.0f);
#pragma unroll
                    for (int b = 0; b < NBLK; ++b) {
                        v[b][0] = pack2(c[b][0], c[b][1]);
                        v[b][1] = pack2(c[b][2], c[b][3]);
                    }
#pragma unroll
                    for (int o = 1; o < NBLK; o <<= 1)
#pragma unroll
                        for (int b = 0; b < NBLK; ++b)
                            if ((b & o) == 0)
#pragma unroll
                                for (int u = 0; u < 2; ++u) {
                                    const f32x2 x = v[b][u], y = v[b + o][u];
                                    v[b][u] = add2(x, y);
                                    v[b + o][u] = fma2(y, minus1, x);
                                }
#pragma unroll
                    for (int b = 0; b < NBLK; ++b) {
                        unpack2(v[b][0], c[b][0], c[b][1]);
                        unpack2(v[b][1], c[b][2], c[b][3]);
                    }
                    // codes: eight nibbles per word; the magnitudes of four places gather in one float (below 2^23),
                    // the signs come from the top bytes
                    if constexpr (FMT == 2) {
#pragma unroll
                        for (int u = 0; u < 2; ++u)
#pragma unroll
                            for (int kp = 0; kp < NBLK / 2; ++kp) {
                                const float y00 = c[2 * kp][2 * u], y01 = c[2 * kp][2 * u + 1], y10 = c[2 * kp + 1][2 * u],
                                            y11 = c[2 * kp + 1][2 * u + 1];
                                float acc = push_magnitude(0.0f, 1.0f, y11, nt[u]);
                                acc = push_magnitude(acc, 16.0f, y10, nt[u]);
                                acc = push_magnitude(acc, 4096.0f, y01, nt[u]);
                                acc = push_magnitude(acc, 16.0f, y00, nt[u]);
                                const uint32_t bits = __float_as_uint(__fadd_rn(acc, 8388608.0f));
                                const uint32_t s0 = sign_bytes<0xFFBB>(y00, y10), s1 = sign_bytes<0xFFBB>(y01, y11);
                                uint32_t& w = words[u * (NBLK / 2) + kp];
                                w = t == 0 ? bits - 0x4B000000u : w + (bits << 8);
                                w |= (s0 & (0x00040004u << (8 * t))) | (s1 & (0x00400040u << (8 * t)));
                            }
                    } else {
#pragma unroll
                        for (int b = 0; b < NBLK; ++b) {
                            float acc = push_magnitude(0.0f, 1.0f, c[b][3], nt[1]);
                            acc = push_magnitude(acc, 16.0f, c[b][2], nt[1]);
                            acc = push_magnitude(acc, 16.0f, c[b][1], nt[0]);
                            acc = push_magnitude(acc, 16.0f, c[b][0], nt[0]);
                            const uint32_t bits = __float_as_uint(__fadd_rn(acc, 8388608.0f));
                            const uint32_t s0 = sign_bytes<0xFBFB>(c[b][0], c[b][2]), s1 = sign_bytes<0xFBFB>(c[b][1], c[b][3]);
                            words[b] = t == 0 ? bits - 0x4B000000u : words[b] + (bits << 16);
                            words[b] |= (s0 & (0x00000404u << (16 * t))) | (s1 & (0x00004040u << (16 * t)));
                            // squared levels of the pair, then the tree over the tq lanes (dims 8t .. 8t + 7 of the block)
                            const uint32_t two = (words[b] >> (16 * t)) & 0x3333u;
                            float p0 = __fadd_rn(level_sq<FMT>(two & 3u), level_sq<FMT>((two >> 4) & 3u));
                            float p1 = __fadd_rn(level_sq<FMT>((two >> 8) & 3u), level_sq<FMT>(two >> 12));
#pragma unroll
                            for (int o = 1; o <= 2; o <<= 1) {
                                p0 = __fadd_rn(p0, __shfl_xor_sync(FULL, p0, o));
                                p1 = __fadd_rn(p1, __shfl_xor_sync(FULL, p1, o));
                            }
                            f0[b] = t == 0 ? p0 : __fadd_rn(f0[b], p0);
                            f1[b] = t == 0 ? p1 : __fadd_rn(f1[b], p1);
                        }
                    }
                }
                float nc2[2];
                if constexpr (FMT == 2) {
                    // 64 x the sum of squared levels: 4, 36, 121, 324 for magnitudes 0..3 = 4 + 32 lo + 117 hi + 171 lo hi
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        uint32_t lo = 0, hi = 0, both = 0;       // nibble counters over at most eight words
#pragma unroll
                        for (int kp = 0; kp < NBLK / 2; ++kp) {
                            const uint32_t w = words[u * (NBLK / 2) + kp], r = w >> 1;
                            lo += w & 0x11111111u;
                            hi += r & 0x11111111u;
                            both += w & r & 0x11111111u;
                        }
                        auto total = [](uint32_t x) { return (((x & 0x0F0F0F0Fu) + ((x >> 4) & 0x0F0F0F0Fu)) * 0x01010101u) >> 24; };
                        uint32_t sq64 = 4u * (4 * NBLK) + 32u * total(lo) + 117u * total(hi) + 171u * total(both);
                        sq64 += __shfl_xor_sync(FULL, sq64, 1);
                        sq64 += __shfl_xor_sync(FULL, sq64, 2);
                        nc2[u] = __fmul_rn((float)sq64, 0.015625f);
                    }
                } else {
#pragma unroll
                    for (int o = 1; o < NBLK; o <<= 1)
#pragma unroll
                        for (int b = 0; b < NBLK; b += 2 * o) {
                            f0[b] = __fadd_rn(f0[b], f0[b + o]);
                            f1[b] = __fadd_rn(f1[b], f1[b + o]);
                        }
                    nc2[0] = f0[0];
                    nc2[1] = f1[0];
                }
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    gcode[u] = nx[u] == 0.0f ? (uint16_t)0 : f32_to_f16_sat_bits(__fdiv_rn(nx[u], __fsqrt_rn(nc2[u])));
            } else {
                // the literal sequence, token by token; the code bytes take the place of the token's own bytes
                constexpr int EPL = D / 32;
                DemoteLane<D, FMT> lc;
                lc.init(sigma, lane);
#pragma unroll 1
                for (int tok = 0; tok < kPage; ++tok) {
                    uint32_t raw[EPL / 4], packed[EPL / 4];
                    uint16_t gc;
                    uint32_t* at = reinterpret_cast<uint32_t*>(kbuf + tok * KST + lane * EPL);
#pragma unroll
                    for (int i = 0; i < EPL / 4; ++i) raw[i] = at[i];
                    encode_key_token<D, FMT>(raw, lc, 1.0f, packed, gc);
#pragma unroll
                    for (int i = 0; i < EPL / 4; ++i) at[i] = packed[i];
                    if (tok == g) gcode[0] = gc;
                    if (tok == g + 8) gcode[1] = gc;
                }
                __syncwarp();
                if constexpr (FMT == 2) {
#pragma unroll
                    for (int u = 0; u < 2; ++u)
#pragma unroll
                        for (int kp = 0; kp < NBLK / 2; ++kp) {
                            const uint8_t* at = kbuf + (g + 8 * u) * KST + 32 * kp + 4 * tq;
                            words[u * (NBLK / 2) + kp] = squeeze4(*reinterpret_cast<const uint32_t*>(at)) |
                                                         (squeeze4(*reinterpret_cast<const uint32_t*>(at + 16)) << 16);
                        }
                } else {
#pragma unroll
                    for (int b = 0; b < NBLK; ++b) {
                        words[b] = 0;
#pragma unroll
                        for (int r = 0; r < 4; ++r)
                            words[b] |= squeeze_nibbles(*reinterpret_cast<const uint16_t*>(
                                            kbuf + (g + 8 * (r & 1)) * KST + 16 * b + 2 * tq + 8 * (r >> 1))) << (8 * r);
                    }
                }
            }
        }
        {
            // word triples (A, B, C) of 64 dims: eight codes and the signs of eight others, twice, and their magnitudes
            uint32_t o[LW];
#pragma unroll
            for (int j = 0; j < NBLK / 4; ++j) {
                const uint32_t p0 = FMT == 2 ? words[2 * j] : words[4 * j];
                const uint32_t p1 = FMT == 2 ? words[2 * j + 1] : words[4 * j + 2];
                const uint32_t p2 = FMT == 2 ? words[NBLK / 2 + 2 * j] : words[4 * j + 1];
                const uint32_t p3 = FMT == 2 ? words[NBLK / 2 + 2 * j + 1] : words[4 * j + 3];
                o[3 * j] = p0 | ((p1 & 0x44444444u) << 1);
                o[3 * j + 1] = p2 | ((p3 & 0x44444444u) << 1);
                o[3 * j + 2] = (p1 & 0x33333333u) | ((p3 & 0x33333333u) << 2);
            }
            store_lane_words<D>(out, lane, o);
            if (tq == 0) {
                reinterpret_cast<uint16_t*>(out + 12 * D)[g] = gcode[0];
                reinterpret_cast<uint16_t*>(out + 12 * D)[g + 8] = gcode[1];
            }
        }
        __syncwarp();                       // value codes go where the keys were

        // ---- values: a lane per channel ---------------------------------------------------------------------
        uint4* vcode = reinterpret_cast<uint4*>(kbuf);      // [channel]: per tq, tokens 2tq | 2tq+8 << 6 | (2tq+1 | 2tq+9 << 6) << 16
#pragma unroll 2
        for (int i = 0; i < D / 32; ++i) {
            const int ch = lane + 32 * i;
            const uint4 raw = *reinterpret_cast<const uint4*>(vbuf + 16 * ch);
            const uint32_t rw[4] = {raw.x, raw.y, raw.z, raw.w};
            __half2 hv[kPage / 2];
#pragma unroll
            for (int t = 0; t < kPage; t += 2) {
                const uint32_t two = e4m3x2_to_f16x2_bits((rw[t >> 2] >> (8 * (t & 3))) & 0xFFFFu);
                hv[t / 2] = *reinterpret_cast<const __half2*>(&two);
            }
            auto values = [&](float (&val)[kPage]) {         // the literal sequences want them in fp32
#pragma unroll
                for (int t = 0; t < kPage; t += 2) {
                    const float2 f = __half22float2(hv[t / 2]);
                    val[t] = f.x;
                    val[t + 1] = f.y;
                }
            };
            const int cb = ch >> 4, row = ch & 15;
            const int hi = (cb >> 1) * 64 + (row & 7) * 8 + 4 * (cb & 1) + (row >> 3);
            uint16_t sc, zp;
            if constexpr (!BIG) {
                __half2 mn2 = hv[0], mx2 = hv[0];
#pragma unroll
                for (int t = 1; t < kPage / 2; ++t) {
                    mn2 = __hmin2(mn2, hv[t]);
                    mx2 = __hmax2(mx2, hv[t]);
                }
                float mn = fminf(__low2float(mn2), __high2float(mn2)), mx = fmaxf(__low2float(mx2), __high2float(mx2));
                // (the sign of a zero extreme and a leading NaN follow the literal scan)
                if (!(mn != 0.0f && mx != 0.0f) || __hisnan(__low2half(hv[0]))) {
                    float val[kPage];
                    values(val);
                    literal_min_max(val, mn, mx);
                }
                sc = f32_to_f16_sat_bits(div7(__fsub_rn(mx, mn)));
                zp = f32_to_f16_sat_bits(mn);
                meta[hi] = sc;
                meta[hi + 2] = zp;
            } else {
                const uint16_t* pm = reinterpret_cast<const uint16_t*>(page3 + (size_t)tiles * TILE);
                sc = pm[hi];
                zp = pm[hi + 2];
            }
            const float scf = __half2float(__ushort_as_half(sc)), zpf = __half2float(__ushort_as_half(zp));
            float y;
            asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(scf));
            if (scf == 0.0f) y = 0.0f;
            const f32x2 y2 = pack2(y, y), snap2 = pack2(40.0f, 40.0f),
                        magic2 = pack2(12582912.0f - 40.0f, 12582912.0f - 40.0f);
            uint32_t q[kPage], any = 0;
#pragma unroll
            for (int t = 0; t < kPage; t += 2) {
                // quotient rounded to a multiple of 2^-18 (40 + quotient), then to an integer, half to even
                const uint32_t two = *reinterpret_cast<const uint32_t*>(&hv[t / 2]);
                const f32x2 snapped = fma2(pack2(fma_f16(low_half(two), 0x3C00u, -zpf), fma_f16(high_half(two), 0x3C00u, -zpf)), y2, snap2);
                float r0, r1;
                unpack2(add2(snapped, magic2), r0, r1);
                q[t] = __float_as_uint(r0);
                q[t + 1] = __float_as_uint(r1);
                any |= q[t] | q[t + 1];
            }
            constexpr uint32_t kBase = 0x4B400000u;          // 12582912.0f: the code is in the low bits
            if ((any & ~7u) != kBase) {                      // a NaN, or an odd page scale: the literal quotients
                float val[kPage];
                values(val);
#pragma unroll
                for (int t = 0; t < kPage; ++t) q[t] = kBase + literal_value_code(val[t], scf, zpf);
            }
            uint32_t x[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                x[k] = q[2 * k] + (q[2 * k + 8] << 6) + (q[2 * k + 1] << 16) + (q[2 * k + 9] << 22) -
                       (kBase + (kBase << 6) + (kBase << 16) + (kBase << 22));
            vcode[ch] = make_uint4(x[0], x[1], x[2], x[3]);
        }
        __syncwarp();
        {
            // value words: four 24-bit streams per triple, the even tokens in the low half-words, the odd in the high
            const uint32_t* vc = reinterpret_cast<const uint32_t*>(kbuf) + g * 4 + tq;
            uint32_t o[LW];
#pragma unroll
            for (int j = 0; j < NBLK / 4; ++j) {
                uint32_t lo[2], hi[2];
#pragma unroll
                for (int grp = 0; grp < 2; ++grp) {
                    const uint32_t* at = vc + (4 * j + 2 * grp) * 64;
                    const uint32_t y = at[0] + (at[32] << 3), z = at[64] + (at[96] << 3);      // rows g, g + 8 of two blocks
                    lo[grp] = y | ((z & 0x000F000Fu) << 12);
                    hi[grp] = (z >> 4) & 0x00FF00FFu;
                }
                o[3 * j] = lo[0];
                o[3 * j + 1] = hi[0] | ((lo[1] & 0x00FF00FFu) << 8);
                o[3 * j + 2] = ((lo[1] >> 8) & 0x00FF00FFu) | (hi[1] << 8);
            }
            store_lane_words<D>(out + 6 * D, lane, o);
            if constexpr (!BIG)
                for (int i = lane; i < 4 * D / 16; i += 32)
                    reinterpret_cast<uint4*>(out + TILE)[i] = reinterpret_cast<const uint4*>(meta)[i];
        }
    }

    pdl_let_next_start();                   // (not sooner: see launch_pdl)
    // copy-before-publish, as in demote_kernel
    cluster_barrier();
    if (valid && crank == 0 && tid == 0 && entry_index != nullptr && (__threadfence(), last_cluster_of_page(page_tickets, page))) {
        const int64_t e = entry_index[page];
        if (e >= n_entries) atomicOr(status, kStBounds);
        else if (e >= 0) {
            block_table[e] = dst;
            __threadfence();
            tier_tag[e] = (uint8_t)MKV_TAG_STALE;
        }
    }
}
