// Promote with one warp per (page, KV head) or (tile, KV head) (included by lifecycle_kernels.cu).
//
// The reconstruction is defined as fp32 operations in a fixed order, and the bytes are those; how they are reached:
//   * Keys: the levels of both formats are multiples of 2^-10 below 2.26, so every partial sum of a token's Hadamard
//     transform is a multiple of 2^-10 below 2^10 and exact in fp32: any order gives the same value.  H_d is H_16 on the dims of a
//     16-dim block, a tensor-core product of the levels (fp16, the record's key section is the A fragment after a byte
//     lookup) with a +-1 matrix, times packed butterflies over the blocks, which a lane has all to itself.  No
//     shuffles, 2 D / 16 MMAs for 16 tokens (before: per-token shuffle butterflies in format 1, a full D x D integer
//     product in format 2).
//   * The matrix columns are ordered so that a lane ends with four consecutive dims of its tokens.
//   * Values: the eight possible output bytes of a channel are computed once; a byte lookup turns a lane's four codes
//     of a channel into four bytes.
// Nothing of the record passes through shared memory: a lane's words are loaded as they stand.  Only the output rows,
// which lanes have in fragments, are put together there and leave as 16-byte stores.

template <int D>
struct PromoteWarp {
    static constexpr int NBLK = D / 16, LW = 3 * NBLK / 4;
    static constexpr int KST = D + 16;               // padded token row of the output keys
    static constexpr int OFF_LUT = kPage * KST, BYTES = OFF_LUT + 8 * D;
    static constexpr int OFF_WARPS = NBLK * 16;
};

// +-1 in fp16 for two values of k: (-1)^popc(k & n)
__device__ __forceinline__ uint32_t h16_unit_pair(int k0, int k1, int n)
{
    return (0x3C00u | ((__popc(k0 & n) & 1u) << 15)) | ((0x3C00u | ((__popc(k1 & n) & 1u) << 15)) << 16);
}

// byte lookup by the four low nibbles of sel (each below 8: the intrinsic would mask them once more)
__device__ __forceinline__ uint32_t lookup4(uint32_t lo, uint32_t hi, uint32_t sel)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(lo), "r"(hi), "r"(sel));
    return r;
}

// Four 3-bit key codes in the low nibbles of sel -> two fp16 pairs of signed levels (high and low bytes looked up)
template <int FMT>
__device__ __forceinline__ void key_levels(uint32_t sel, uint32_t& r0, uint32_t& r1)
{
    const uint32_t hi = FMT == 2 ? lookup4(0x403D3A34u, 0xC0BDBAB4u, sel) : lookup4(0x403D3A33u, 0xC0BDBAB3u, sel);
    const uint32_t lo = FMT == 2 ? lookup4(0x80800000u, 0x80800000u, sel) : lookup4(0x4E600CD8u, 0x4E600CD8u, sel);
    r0 = __byte_perm(lo, hi, 0x5140u);
    r1 = __byte_perm(lo, hi, 0x7362u);
}

template <int D>
__device__ __forceinline__ void fetch_lane_words(const uint8_t* sec, int lane, uint32_t (&w)[3 * (D / 16) / 4])
{
    constexpr int LW = 3 * (D / 16) / 4;
#pragma unroll
    for (int c = 0; c < LW / 4; ++c) {
        const uint4 v = *reinterpret_cast<const uint4*>(sec + c * 512 + lane * 16);
        w[4 * c] = v.x; w[4 * c + 1] = v.y; w[4 * c + 2] = v.z; w[4 * c + 3] = v.w;
    }
    if constexpr (LW % 4 != 0) {
        const uint2 v = *reinterpret_cast<const uint2*>(sec + (LW / 4) * 512 + lane * 8);
        w[LW - 2] = v.x; w[LW - 1] = v.y;
    }
}

__device__ __forceinline__ uint32_t e4m3_pair(float lo, float hi)
{
    return (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(lo, hi), __NV_SATFINITE, __NV_E4M3);
}

// the four codes of one channel row: x holds tokens 2tq (low half), 2tq + 1 (high) at bit P0, y tokens 2tq + 8, + 9 at bit
// P1 -> byte-lookup selector with the codes in that order
template <int P0, int P1>
__device__ __forceinline__ uint32_t code_selector(uint32_t x, uint32_t y)
{
    const uint32_t far = P1 <= 8 ? y << (8 - P1) : y >> (P1 - 8);
    const uint32_t s = ((x >> P0) & 0x00070007u) | (far & 0x07000700u);
    return s | (s >> 12);
}

template <int D, int FMT, bool BIG>
__global__ void __launch_bounds__(32 * kDemoteWarps, D == 256 ? 3 : 4)
promote_warp_kernel(const uint8_t* tq3, uint8_t* __restrict__ fp8, int tq3_pages, int fp8_pages, int hkv, int tiles,
                    float inv_k_scale, float inv_v_scale, float rs, SigmaBits sigma, const int32_t* src_ids,
                    const int32_t* dst_ids, int32_t* block_table, uint8_t* tier_tag, const int64_t* entry_index,
                    int64_t n_entries, uint32_t* __restrict__ status, uint32_t* page_tickets)
{
    using G = PromoteWarp<D>;
    constexpr uint32_t FULL = 0xffffffffu;
    constexpr int NBLK = G::NBLK, LW = G::LW, KST = G::KST, TILE = 12 * D + 32;
    extern __shared__ __align__(16) uint8_t psm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, tq = lane & 3, n_warps = blockDim.x >> 5;
    uint32_t* sig = reinterpret_cast<uint32_t*>(psm);                // sign bits of four bytes
    uint8_t* tile = psm + G::OFF_WARPS + warp * G::BYTES;
    uint2* lut = reinterpret_cast<uint2*>(tile + G::OFF_LUT);        // [channel] output bytes of codes 0 .. 7
    const int csize = (int)cluster_size(), crank = (int)cluster_rank();
    const int page = blockIdx.x / csize;
    for (int i = tid; i < NBLK * 4; i += blockDim.x) {
        const int dim = 4 * i;
        const uint32_t n = (sigma.w[dim >> 5] >> (dim & 31)) & 0xFu;
        sig[i] = ((n * 0x00204081u) & 0x01010101u) << 7;
    }
    // B operands of H_16.  K slots 2tq + e, 8 + 2tq + e are dims 4tq + e, 4tq + 2 + e of the block in format 2 and themselves
    // in format 1; column n = g of matrix t is dim 4 (n / 2) + 2t + n % 2, so that a lane's columns 2tq, 2tq + 1 of the two
    // matrices are dims 4tq .. 4tq + 3
    uint32_t hb[2][2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const int n = 4 * (g >> 1) + 2 * t + (g & 1);
        hb[t][0] = FMT == 2 ? h16_unit_pair(4 * tq, 4 * tq + 1, n) : h16_unit_pair(2 * tq, 2 * tq + 1, n);
        hb[t][1] = FMT == 2 ? h16_unit_pair(4 * tq + 2, 4 * tq + 3, n) : h16_unit_pair(2 * tq + 8, 2 * tq + 9, n);
    }
    pdl_wait();
    __syncthreads();
    const int src = src_ids[page], dst = dst_ids[page];
    const bool valid = src >= 0 && src < tq3_pages && dst >= 0 && dst < fp8_pages;
    if (!valid && tid == 0 && crank == 0 && blockIdx.y == 0) atomicOr(status, kStBounds);
    const bool unit_k = inv_k_scale == 1.0f, unit_v = inv_v_scale == 1.0f;   // a product with 1 is skipped

    const int m_first = BIG ? (int)blockIdx.y : 0, m_step = BIG ? (int)gridDim.y : 1, m_end = BIG ? tiles : 1;
    const int h_first = crank * n_warps + warp, h_step = csize * n_warps;
    auto page_of = [&](int h) { return tq3 + ((size_t)src * hkv + h) * tq3_page_bytes(D, tiles); };
    // What a lane needs of a record.  At d = 128 each part of the next record is asked for as soon as this record's is used
    // up: the loads then fly under the work on this one, in the registers that have just become free (d = 256 has none).
    constexpr bool AHEAD = D == 128;
    uint32_t kw[LW], vw[LW];
    uint4 mt[D / 128];
    uint16_t g0 = 0, g1 = 0;
    auto fetch_keys = [&](const uint8_t* rec3) {
        fetch_lane_words<D>(rec3, lane, kw);
        g0 = reinterpret_cast<const uint16_t*>(rec3 + 12 * D)[g];
        g1 = reinterpret_cast<const uint16_t*>(rec3 + 12 * D)[g + 8];
    };
    auto fetch_meta = [&](const uint8_t* page3) {    // (16-token pages: right behind the one tile)
#pragma unroll
        for (int i = 0; i < D / 128; ++i) mt[i] = reinterpret_cast<const uint4*>(page3 + (size_t)tiles * TILE)[lane + 32 * i];
    };
    auto fetch_record = [&](int h, int m) {
        const uint8_t* page3 = page_of(h);
        fetch_keys(page3 + (size_t)m * TILE);
        fetch_meta(page3);
        fetch_lane_words<D>(page3 + (size_t)m * TILE + 6 * D, lane, vw);
    };
    if (AHEAD && valid && h_first < hkv && m_first < m_end) fetch_record(h_first, m_first);
    for (int h = h_first; valid && h < hkv; h += h_step)
    for (int m = m_first; m < m_end; m += m_step) {
        uint8_t* rec8 = fp8 + (((size_t)dst * hkv + h) * tiles + m) * fp8_record_bytes(D);
        const int next_m = m + m_step < m_end ? m + m_step : m_first, next_h = m + m_step < m_end ? h : h + h_step;
        const bool more = AHEAD && next_h < hkv;
        if constexpr (!AHEAD) fetch_record(h, m);
        const uint8_t* next_page = page_of(more ? next_h : h);
        const uint8_t* next = next_page + (size_t)next_m * TILE;

        // ---- keys
        {
            uint32_t a[NBLK][4];
#pragma unroll
            for (int j = 0; j < NBLK / 4; ++j) {
                const uint32_t A = kw[3 * j], Bw = kw[3 * j + 1], Cw = kw[3 * j + 2];
                uint32_t sel[4];
                sel[0] = A & 0x77777777u;
                sel[1] = Bw & 0x77777777u;
                sel[2] = ((A >> 1) & 0x44444444u) | (Cw & 0x33333333u);
                sel[3] = ((Bw >> 1) & 0x44444444u) | ((Cw >> 2) & 0x33333333u);
                if constexpr (FMT == 2) {            // a word holds one token (g or g + 8) of two blocks
#pragma unroll
                    for (int b = 0; b < 4; ++b)
#pragma unroll
                        for (int u = 0; u < 2; ++u) {
                            const uint32_t s = sel[2 * (b >> 1) + u];
                            key_levels<2>((b & 1) ? s >> 16 : s, a[4 * j + b][u], a[4 * j + b][2 + u]);
                        }
                } else {                             // a word holds a block
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        key_levels<1>(sel[b], a[4 * j + b][0], a[4 * j + b][1]);
                        key_levels<1>(sel[b] >> 16, a[4 * j + b][2], a[4 * j + b][3]);
                    }
                }
            }
            const float gr0 = __fmul_rn(__half2float(__ushort_as_half(g0)), rs), gr1 = __fmul_rn(__half2float(__ushort_as_half(g1)), rs);
            if (more) fetch_keys(next);
            __syncwarp();                            // the tile of the round before has been read
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                f32x2 v[NBLK][2];
                const f32x2 minus1 = pack2(-1.0f, -1.0f);
#pragma unroll
                for (int b = 0; b < NBLK; ++b) {
                    float c[4];
                    hmma_zero(c, a[b], hb[t][0], hb[t][1]);
                    v[b][0] = pack2(c[0], c[1]);
                    v[b][1] = pack2(c[2], c[3]);
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
                const f32x2 gs[2] = {pack2(gr0, gr0), pack2(gr1, gr1)};
#pragma unroll
                for (int b = 0; b < NBLK; ++b)
#pragma unroll
                    for (int u = 0; u < 2; ++u) v[b][u] = mul2(gs[u], v[b][u]);
                if (!unit_k) {                       // (a branch, not predicated products)
                    const f32x2 ik = pack2(inv_k_scale, inv_k_scale);
#pragma unroll
                    for (int b = 0; b < NBLK; ++b)
#pragma unroll
                        for (int u = 0; u < 2; ++u) v[b][u] = mul2(v[b][u], ik);
                }
#pragma unroll
                for (int b = 0; b < NBLK; ++b)
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        float lo, hi;
                        unpack2(v[b][u], lo, hi);
                        *reinterpret_cast<uint16_t*>(tile + (g + 8 * u) * KST + 16 * b + 4 * tq + 2 * t) = (uint16_t)e4m3_pair(lo, hi);
                    }
            }
            // rotation signs on the bytes: the conversion is symmetric, but a NaN (of a norm correction that is none) stays as it is
            const bool odd = __any_sync(FULL, !(fabsf(gr0) < CUDART_INF_F && fabsf(gr1) < CUDART_INF_F));
            __syncwarp();
#pragma unroll
            for (int i = lane; i < D; i += 32) {
                const int tok = i / NBLK, b = i % NBLK;
                uint4 w = *reinterpret_cast<const uint4*>(tile + tok * KST + 16 * b);
                uint4 s = *reinterpret_cast<const uint4*>(sig + 4 * b);
                if (odd) {
                    s.x &= ~__vcmpeq4(w.x, 0x7F7F7F7Fu); s.y &= ~__vcmpeq4(w.y, 0x7F7F7F7Fu);
                    s.z &= ~__vcmpeq4(w.z, 0x7F7F7F7Fu); s.w &= ~__vcmpeq4(w.w, 0x7F7F7F7Fu);
                }
                w.x ^= s.x; w.y ^= s.y; w.z ^= s.z; w.w ^= s.w;
                reinterpret_cast<uint4*>(rec8)[i] = w;
            }
        }
        // ---- values: output bytes of the eight codes, four channels per chunk of scales and zeros
#pragma unroll
        for (int i = 0; i < D / 128; ++i) {
            const int c = lane + 32 * i, ch0 = (c >> 3) * 32 + (c & 7);
            const float2 sc[2] = {f16x2_to_f32(mt[i].x), f16x2_to_f32(mt[i].z)}, zp[2] = {f16x2_to_f32(mt[i].y), f16x2_to_f32(mt[i].w)};
            f32x2 lv[4][4];                          // [block e / 2, row half e % 2][codes 2 k, 2 k + 1]
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float s = e & 1 ? sc[e >> 1].y : sc[e >> 1].x, z = e & 1 ? zp[e >> 1].y : zp[e >> 1].x;
                const f32x2 s2 = pack2(s, s), z2 = pack2(z, z);
#pragma unroll
                for (int k = 0; k < 4; ++k) lv[e][k] = add2(mul2(s2, pack2((float)(2 * k), (float)(2 * k + 1))), z2);
            }
            if (!unit_v) {
                const f32x2 iv = pack2(inv_v_scale, inv_v_scale);
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int k = 0; k < 4; ++k) lv[e][k] = mul2(lv[e][k], iv);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                uint32_t pr[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float lo, hi;
                    unpack2(lv[e][k], lo, hi);
                    pr[k] = e4m3_pair(lo, hi);
                }
                lut[ch0 + 16 * (e >> 1) + 8 * (e & 1)] = make_uint2(pr[0] | (pr[1] << 16), pr[2] | (pr[3] << 16));
            }
        }
        if (more && (!BIG || next_h != h)) fetch_meta(next_page);
        __syncwarp();                                // tables complete, key rows read: the tile takes the value rows
        uint32_t* vrow = reinterpret_cast<uint32_t*>(tile);          // [channel][tq]: tokens 2tq, 2tq+1, 2tq+8, 2tq+9
        auto put = [&](int ch, uint32_t sel) {
            const uint2 l = lut[ch];
            vrow[ch * 4 + tq] = lookup4(l.x, l.y, sel);
        };
#pragma unroll
        for (int j = 0; j < NBLK / 4; ++j) {
            const uint32_t W0 = vw[3 * j], W1 = vw[3 * j + 1], W2 = vw[3 * j + 2];
            const uint32_t X = __byte_perm(W0, W1, 0x6341), Y = __byte_perm(W1, W2, 0x6341);
            const int ch = 64 * j + g;
            put(ch, code_selector<0, 6>(W0, W0));
            put(ch + 8, code_selector<3, 1>(W0, X));
            put(ch + 16, code_selector<4, 2>(X, W1));
            put(ch + 24, code_selector<7, 5>(X, W1));
            put(ch + 32, code_selector<0, 6>(Y, Y));
            put(ch + 40, code_selector<3, 1>(Y, W2));
            put(ch + 48, code_selector<4, 10>(W2, W2));
            put(ch + 56, code_selector<7, 13>(W2, W2));
        }
        if (more) fetch_lane_words<D>(next + 6 * D, lane, vw);
        __syncwarp();
#pragma unroll
        for (int i = lane; i < D; i += 32) {
            const uint4 w = *reinterpret_cast<const uint4*>(vrow + 4 * i);
            reinterpret_cast<uint4*>(rec8 + 16 * D)[i] = make_uint4(__byte_perm(w.x, w.y, 0x5410), __byte_perm(w.z, w.w, 0x5410),
                                                                    __byte_perm(w.x, w.y, 0x7632), __byte_perm(w.z, w.w, 0x7632));
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
            tier_tag[e] = (uint8_t)MKV_TAG_ANCHOR;
        }
    }
}
