// Tensor-core decode attention (MKV_DECODE_TENSOR): one-pass mixed-format split-KV scan.
//
// Section 3.3 / 4.1: every page of a request row is read in its own physical format (FP8 for
// Recent/Anchor, TQ3 for Stale), all tokens share one softmax, the whole GQA group reuses each
// unpacked tile, and split partials (m, l, O) are merged with Eq. (softmax-merge).
//
// Mapping to the hardware
//   * work = (request, KV head, page) triples in row-major order (several layers: end to end), cut into
//     contiguous ranges, one per block (persistent grid, one or two blocks per SM); a block processes the
//     (request, KV head) segments of its range one after another, its warps taking contiguous runs of pages.
//   * each warp streams its pages through a private ring of shared-memory slots filled by bulk
//     asynchronous copies (cp.async.bulk + mbarrier), several pages ahead of the arithmetic.
//   * a 16-token page x d dims is exactly the A operand of m16n8k16 MMAs whose B operand is the
//     (rotated) query of the 8-column head group: S[16 tokens][8 heads] = K q^T.  TQ3 keys stay in
//     the rotated domain; the query is rotated instead (q' = d^-1/2 H (sigma . q)).  The packed
//     3-bit codes are stored in the register layout of that A fragment, so unpacking is a byte
//     table lookup (PRMT) per four codes for keys and one mask per two codes for values -- no
//     shared-memory round trip, no dequantised tile.
//   * P = exp2(S - m) is transposed in registers (movmatrix) into the B operand of
//     O^T[16 channels][8 heads] += V^T P, one MMA per 16 channels; the row sums come from one more
//     MMA against a matrix of ones.  TQ3 values enter that MMA as their integer codes; the
//     per-channel fp16 scale and zero of the page are applied to the 16x8 result in fp32.
//   * partial results of a block that covers only part of a (request, KV head) row go to the
//     workspace; every such block then takes a ticket of its row, and the block that draws the last
//     ticket combines the row's partials (Eq. softmax-merge) and writes the output.  No block ever
//     waits for another, and there is no second launch.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <math_constants.h>

#include <cstdlib>
#include <mutex>

#include "decode_cut.cuh"
#include "mkv_internal.cuh"

namespace mkv {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kRescaleSlack = 8.0f;                        // the running maximum is only raised when exceeded by 2^8
constexpr unsigned long long kDefaultWaitNs = 20000000ull;   // 20 ms: far beyond any copy that is going to arrive

size_t decode_ws_tensor_bytes(int, int, int, int d)
{
    return (size_t)2 * kMaxCtas * (8 * d + 16) * sizeof(float);
}

struct DecodeParams {
    const uint8_t* fp8;
    const uint8_t* tq3;
    int fp8_pages, tq3_pages, hkv, group;
    float k_scale, v_scale;
    SigmaBits sigma;
    const __nv_bfloat16* q;
    const int32_t* bt;
    const uint8_t* tags;
    const int32_t* lens;
    int B, max_pages;
    int tiles;             // 16-token tiles per page (page = 16 * tiles tokens); table entries are per page
    float scale;
    float* out;
    float* lse;
    float* partials;       // [2 * grid][8*D + 16]
    uint32_t* tickets;     // [max_blocks] arrival counters of split rows, indexed by the row's first block; zero between calls
    int max_blocks;        // the partial area holds 2 * max_blocks slots
    float* mass;           // scored variant: [B][hq][max_pages], log2-domain page sums from the scan (else unused)
    uint32_t* status;
    unsigned long long wait_ns;   // wall-time limit of a wait for a page copy (kDefaultWaitNs unless the pool says otherwise)
};

// One launch can scan the pools of several layers (Section 4.1 runs the decode step of all full-attention
// layers from one CUDA graph): the layers share the requests (lengths, batch, geometry) and differ in
// their arenas, tables, queries, outputs and workspaces.  A block walks its share of layer 0, then of
// layer 1, ... without waiting for the other blocks, so the start-up and the merge tail of one layer
// overlap the page loops of its neighbours.
constexpr int kMaxLayers = 32;
//
// Two cuts of the work.  Up to 3 layers: every layer is cut over the whole grid like a call of its own (results
// are bit for bit those of single calls), and every block visits every layer.  From kMinFlatLayers layers on
// (template parameter FLAT) the layers are laid end to end and the grid cuts the whole list once: a block then meets one or two
// rows instead of one per layer, and pays the set-up of a row (table entries, first pages, query rotation:
// 3 us) and its tail (reduction, partial, ticket: 3 us, warps waiting for the last one: 2 us) that much less often.
constexpr int kMinFlatLayers = 4;
template <int MAXL>
struct LayerSet {
    int n;
    DecodeParams layer[MAXL];
};

// ------------------------------------------------------------------------------------------------
// small PTX wrappers
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t s)
{
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(s));
    return r;
}

// (a & b) | c in one LOP3
__device__ __forceinline__ uint32_t lop3_and_or(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}

__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// same product with a zero accumulator: d = A B
__device__ __forceinline__ void mma16816_zero(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

// D += A B with signed 8-bit integer operands and 32-bit integer accumulators: A 16 x 32 (row-major fragment),
// B 32 x 8.  (Measured on B200: this legacy integer MMA is one native instruction at the rate of the fp16
// m16n8k16 one, i.e. twice its products per instruction; the e4m3 form of mma.sync is expanded by the compiler
// into conversions and fp16 MMAs and is slower than the fp16 path it was meant to replace.)
__device__ __forceinline__ void mma16832_s8(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// the same product with a zero accumulator
__device__ __forceinline__ void mma16832_s8_zero(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                 : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "r"(0));
}

__device__ __forceinline__ uint32_t lds32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

__device__ __forceinline__ uint32_t movmatrix_trans(uint32_t x)
{
    uint32_t r;
    asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(r) : "r"(x));
    return r;
}

__device__ __forceinline__ uint32_t pack_f16x2(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

__device__ __forceinline__ uint32_t e4m3x2_to_f16x2(uint16_t v)
{
    uint32_t r;
    asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(r) : "h"(v));
    return r;
}

__device__ __forceinline__ float fast_exp2(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ uint32_t hfma2_u32(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t r;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}

__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}

// Arrival on a row's ticket: what this block has stored (before a block barrier) is released, what the others have is acquired
__device__ __forceinline__ uint32_t ticket_add(uint32_t* p, uint32_t v)
{
    uint32_t old;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

__device__ __forceinline__ uint32_t ticket_or(uint32_t* p, uint32_t v)
{
    uint32_t old;
    asm volatile("atom.or.acq_rel.gpu.global.b32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

// bulk asynchronous copy global -> this block's shared memory, completion counted on an mbarrier
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

__device__ __forceinline__ uint4 lds128(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}

__device__ __forceinline__ uint2 lds64(uint32_t addr)
{
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
    return v;
}

__device__ __forceinline__ uint16_t lds16(uint32_t addr)
{
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
    return v;
}

// ------------------------------------------------------------------------------------------------
// TQ3 unpack
// ------------------------------------------------------------------------------------------------
// Four 3-bit key codes in the four low nibbles of `sel` (bit 3 of each nibble clear) -> two half2
// registers holding the signed fp16 codebook levels.  The two byte tables hold the high and the low
// bytes of {+C0,+C1,+C2,+C3,-C0,-C1,-C2,-C3} = fp16 {33D8, 3A0C, 3D60, 404E | sign}.
__device__ __forceinline__ void key_lut4(uint32_t sel, uint32_t& r0, uint32_t& r1)
{
    const uint32_t hi = prmt(0x403D3A33u, 0xC0BDBAB3u, sel);
    const uint32_t lo = prmt(0x4E600CD8u, 0x4E600CD8u, sel);
    r0 = prmt(lo, hi, 0x5140u);
    r1 = prmt(lo, hi, 0x7362u);
}

// Two 3-bit value codes sitting at bit POS of each 16-bit half of x -> half2 of the integer codes.
// (x & mask) | 0x6400 is the fp16 number 1024 + code * 2^POS; one FMA recovers the code exactly.
// (The masked bits alone are the exact operand code * 2^(POS - 24), a subnormal, and save the FMA: 2 x 59,008 tokens in
// 16 layers 554 -> 592 us with it.  But the tensor core aligns the products of an MMA by the exponents of their factors,
// and a subnormal has the exponent of the first binade: every bit that a code stands below bit 10 is a bit less of the
// sum.  Rows of 30,000 equally weighted tokens came out 3 to 4 times as far from the fp64 result, 3e-6 to 5e-6 against
// 1e-6, with codes at bits 5 to 8, and 100 times with codes left where they are.)
template <int POS>
__device__ __forceinline__ uint32_t value_code(uint32_t x)
{
    constexpr uint32_t mask = 0x00070007u << POS;
    const uint32_t u = lop3_and_or(x, mask, 0x64006400u);
    // 2^-POS and -1024 * 2^-POS as fp16 pairs (exponent arithmetic on 1.0 = 0x3C00, -1024 = 0xE400)
    constexpr uint32_t mul = (0x3C00u - (POS << 10)) * 0x00010001u;
    constexpr uint32_t add = (0xE400u - (POS << 10)) * 0x00010001u;
    return hfma2_u32(u, mul, add);
}

// A operands of the four channel blocks of a word triple
template <int BLOCK>
__device__ __forceinline__ void value_operands(uint32_t (&a)[4], uint32_t W0, uint32_t W1, uint32_t W2, uint32_t X)
{
    if constexpr (BLOCK == 0) {          // X = bytes of W0, W1 between the two
        a[0] = value_code<0>(W0); a[1] = value_code<3>(W0); a[2] = value_code<6>(W0); a[3] = value_code<1>(X);
    } else if constexpr (BLOCK == 1) {
        a[0] = value_code<4>(X); a[1] = value_code<7>(X); a[2] = value_code<2>(W1); a[3] = value_code<5>(W1);
    } else if constexpr (BLOCK == 2) {   // X = bytes of W1, W2
        a[0] = value_code<0>(X); a[1] = value_code<3>(X); a[2] = value_code<6>(X); a[3] = value_code<1>(W2);
    } else {
        const uint32_t X2 = W2 >> 8;
        a[0] = value_code<4>(W2); a[1] = value_code<7>(W2); a[2] = value_code<2>(X2); a[3] = value_code<5>(X2);
    }
}

__device__ __forceinline__ float2 half2_to_float2(uint32_t x)
{
    return __half22float2(*reinterpret_cast<const __half2*>(&x));
}

// acc[channel rows g, g+8][heads] += scale_row * t + zero_row * psum_head
__device__ __forceinline__ void affine_accumulate(float (&acc)[4], const float (&t)[4], uint32_t sc_pair, uint32_t zp_pair,
                                                  float ps0, float ps1)
{
    const float2 sc = half2_to_float2(sc_pair), zp = half2_to_float2(zp_pair);
    acc[0] = fmaf(sc.x, t[0], fmaf(zp.x, ps0, acc[0]));
    acc[1] = fmaf(sc.x, t[1], fmaf(zp.x, ps1, acc[1]));
    acc[2] = fmaf(sc.y, t[2], fmaf(zp.y, ps0, acc[2]));
    acc[3] = fmaf(sc.y, t[3], fmaf(zp.y, ps1, acc[3]));
}

// ------------------------------------------------------------------------------------------------
// kernel
// ------------------------------------------------------------------------------------------------

template <int D, int NW, int NSTAGE, bool SHORT_ROUNDS = false>
struct Geo {
    static constexpr int NB = D / 16;                       // 16-wide blocks along d
    static constexpr int LW = 3 * NB / 4;                   // packed words per lane and code section
    static constexpr int TQ3_REC = 16 * D + 32;
    static constexpr int FP8_HALF = 16 * D;
    static constexpr int SLOT = (TQ3_REC + 127) / 128 * 128;
    // pages of one warp whose table entries are compacted at a time (fewer where the ring leaves little room)
    static constexpr int ROUND = SHORT_ROUNDS ? 64 : 128;
    // The ring is used in pairs of slots with one barrier each: a pair holds two Stale records, or the keys and values of one
    // FP8 page, asked for together and waited for once.
    static constexpr int NP = NSTAGE / 2, PAIR = 2 * SLOT;
    static constexpr int RING = NW * NSTAGE * SLOT;
    static constexpr int QROT = NB * 32 * 16;               // rotated query B fragments, hi and lo interleaved
    static constexpr int QPLAIN = NB * 32 * 8;              // plain query B fragments (FP8 pages)
    static constexpr int OFF_QT = RING;
    static constexpr int OFF_QF = OFF_QT + QROT;
    static constexpr int OFF_BAR = OFF_QF + QPLAIN;
    static constexpr int OFF_LIST = (OFF_BAR + NW * NP * 8 + 15) / 16 * 16;   // [warp][2 formats][ROUND] page ids, then [warp][2][ROUND] logical pages
    static constexpr int OFF_CUM = OFF_LIST + NW * 4 * ROUND * 4;
    static constexpr int OFF_LENS = OFF_CUM + (kMaxBatch + 1) * 4;
    static constexpr int OFF_M = OFF_LENS + kMaxBatch * 4;
    static constexpr int OFF_L = OFF_M + NW * 8 * 4;
    static constexpr int OFF_PART = (OFF_L + NW * 8 * 4 + 15) / 16 * 16;    // holds 64-bit fields
    static constexpr int OFF_LAST = OFF_PART + ((int)sizeof(Partition) + 15) / 16 * 16;
    static constexpr int OFF_QS = OFF_LAST + 16;             // record format 2: digit unit of the rotated query, per head
    static constexpr int SMEM = OFF_QS + 32;
    static_assert(SLOT % 128 == 0 && OFF_QT % 16 == 0 && OFF_QF % 16 == 0 && OFF_BAR % 8 == 0,
                  "slots are bulk-copy destinations; query fragments are read with 16- and 8-byte loads");
    static_assert(OFF_PART % alignof(Partition) == 0 && OFF_LAST % 16 == 0, "alignment of the partition record");
    static_assert(NW >= 4, "a warp builds the query fragments of at most two columns of the 8-wide head group");
    static_assert(NSTAGE >= 4 && NSTAGE % 2 == 0 && NSTAGE <= 16, "an FP8 page takes a pair of slots; one phase bit per pair");
    static_assert(NSTAGE * SLOT >= 8 * D * 4, "ring doubles as the cross-warp reduction buffer");
    static_assert(FP8_HALF <= SLOT, "half an FP8 record fits a slot");
};


// Running state of one warp for one (request, KV head) segment: O^T accumulators [d channels x 8
// heads] in the MMA C layout, row sums and the (lazily raised) running maximum of the two head
// columns this lane owns, all in log2 units.
template <int NB>
struct WarpAcc {
    float o[NB][4];
    float l[2];
    float m[2];
    // pages of several tiles only: while the tiles of one Stale page are scanned, o holds sum p * code of
    // that page (the page's scale/zero are applied once, when the page is left), lp its row sums, and the
    // output accumulated before sits in shared memory, to be multiplied by pk (the rescales since then)
    float lp[2];
    float pk[2];
    // record format 2: its score tile has the heads in the rows, so the lane also keeps the running maximum
    // of head g (`mr`); m[] (heads 2tq, 2tq+1: the columns of the output tile) stays the master copy that the
    // Recent/Anchor pages, the page mass and the reduction use, and the two are brought in line on every change
    float mr;
};

// Scores of one page -> probabilities.  s[0..1] = token g, s[2..3] = token g+8 (heads 2tq, 2tq+1).
// Updates the running maximum (only when it is exceeded by more than 2^kRescaleSlack, so that
// accumulators are rarely rescaled), and returns P^T as MMA B fragments split into an fp16 pair
// hi (pb) + lo (pc), plus the page's row sums ps[0..1].
//
// SPLIT (groups of at most four query heads, kernel template parameter): the head columns 4-7 of the MMAs, which would
// stand idle, carry the low halves of heads 0-3, so that ONE MMA does the work of the pair hi + lo: scores, maxima and
// probabilities of heads 0-3 are present twice (columns or rows h and h + 4), b0, b1 hold the high halves in columns
// 0-3 and the low halves in columns 4-7, and the two column halves of the output tile are added when the block
// reduces it.  The same products and sums, half the tensor-core instructions (17 instead of 34 per Stale page at
// d = 128): each of them holds up the issue of everything else for about five cycles.
struct PFrag {
    uint32_t b0, b1, c0, c1;
    float ps0, ps1;
};

// First half: raise the running maximum (and rescale the accumulators) if the page asks for it.
template <int NB, bool TILED = false>
__device__ __forceinline__ void softmax_rescale(WarpAcc<NB>& acc, const float (&s)[4])
{
    constexpr uint32_t FULL = 0xffffffffu;
    float mx0 = fmaxf(s[0], s[2]), mx1 = fmaxf(s[1], s[3]);
    // the page maximum is only needed when some score exceeds the running maximum by more than the slack
    if (__any_sync(FULL, mx0 > acc.m[0] + kRescaleSlack || mx1 > acc.m[1] + kRescaleSlack)) {
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
            mx0 = fmaxf(mx0, __shfl_xor_sync(FULL, mx0, o));
            mx1 = fmaxf(mx1, __shfl_xor_sync(FULL, mx1, o));
        }
        const bool up0 = mx0 > acc.m[0] + kRescaleSlack, up1 = mx1 > acc.m[1] + kRescaleSlack;
        const float f0 = up0 ? fast_exp2(acc.m[0] - mx0) : 1.f, f1 = up1 ? fast_exp2(acc.m[1] - mx1) : 1.f;
        if (up0) acc.m[0] = mx0;
        if (up1) acc.m[1] = mx1;
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            acc.o[i][0] *= f0; acc.o[i][2] *= f0;
            acc.o[i][1] *= f1; acc.o[i][3] *= f1;
        }
        acc.l[0] *= f0;
        acc.l[1] *= f1;
        if constexpr (TILED) {
            acc.lp[0] *= f0; acc.lp[1] *= f1;
            acc.pk[0] *= f0; acc.pk[1] *= f1;
        }
    }
}

// Second half, branch-free (so that it can be scheduled into the unpack work of the next page): P and its row sums.
template <int NB, bool SPLIT>
__device__ __forceinline__ void softmax_probs(WarpAcc<NB>& acc, const float (&s)[4], PFrag& pf, int lane)
{
    const float p0 = fast_exp2(s[0] - acc.m[0]), p1 = fast_exp2(s[1] - acc.m[1]);
    const float p2 = fast_exp2(s[2] - acc.m[0]), p3 = fast_exp2(s[3] - acc.m[1]);
    const uint32_t ph01 = pack_f16x2(p0, p1), ph23 = pack_f16x2(p2, p3);
    const float2 h01 = half2_to_float2(ph01), h23 = half2_to_float2(ph23);
    const uint32_t pl01 = pack_f16x2(p0 - h01.x, p1 - h01.y), pl23 = pack_f16x2(p2 - h23.x, p3 - h23.y);
    if constexpr (SPLIT) {                   // columns 2tq, 2tq + 1 of lanes with tq >= 2 carry the low halves
        pf.b0 = movmatrix_trans(lane & 2 ? pl01 : ph01);
        pf.b1 = movmatrix_trans(lane & 2 ? pl23 : ph23);
    } else {
        pf.b0 = movmatrix_trans(ph01);
        pf.b1 = movmatrix_trans(ph23);
        pf.c0 = movmatrix_trans(pl01);
        pf.c1 = movmatrix_trans(pl23);
    }
    // row sums through the tensor core: the same P that multiplies V
    const uint32_t ones[4] = {0x3C003C00u, 0x3C003C00u, 0x3C003C00u, 0x3C003C00u};
    float ps[4];
    mma16816_zero(ps, ones, pf.b0, pf.b1);
    if constexpr (!SPLIT) mma16816(ps, ones, pf.c0, pf.c1);
    pf.ps0 = ps[0];
    pf.ps1 = ps[1];
    acc.l[0] += ps[0];
    acc.l[1] += ps[1];
}

template <int NB, bool SPLIT>
__device__ __forceinline__ void softmax_page(WarpAcc<NB>& acc, const float (&s)[4], PFrag& pf, int lane)
{
    softmax_rescale<NB>(acc, s);
    softmax_probs<NB, SPLIT>(acc, s, pf, lane);
}

// Scored variant (Section 3.1): log2 of the page's exponential sum, referred to an absolute origin
// (row sum relative to the running maximum, plus that maximum), for the two heads this lane owns.
// mass_pg points at (request, first head of the group, this page); heads are mass_stride apart.
// The finishing kernel turns it into the globally normalised mass with the row's log-sum-exp.
// *addr <- log2(2^*addr + 2^v): several warps add their parts of one page's exponential sum (pages of several
// tiles); the entries start at -inf.
__device__ __forceinline__ void atomic_log2_add(float* addr, float v)
{
    int* ia = reinterpret_cast<int*>(addr);
    int old = *reinterpret_cast<volatile int*>(ia), assumed;
    do {
        assumed = old;
        const float a = __int_as_float(assumed);
        const float hi = fmaxf(a, v), lo = fminf(a, v);
        const float nv = lo == -CUDART_INF_F ? hi : hi + __log2f(1.f + fast_exp2(lo - hi));
        old = atomicCAS(ia, assumed, __float_as_int(nv));
    } while (old != assumed);
}

// ACCUMULATE: the entry receives a part of the page (a tile, or a run of tiles) and is added to, not stored.
template <int NB, bool SPLIT, bool ACCUMULATE = false>
__device__ __forceinline__ void store_page_mass(const WarpAcc<NB>& acc, float ps0, float ps1, float* mass_pg, int mass_stride,
                                                int GQ, int lane)
{
    if constexpr (SPLIT) {
        ps0 += __shfl_xor_sync(0xffffffffu, ps0, 2);
        ps1 += __shfl_xor_sync(0xffffffffu, ps1, 2);
    }
    if (lane < 4) {                  // g == 0: one lane per head pair
        const int h0 = 2 * lane;
        const float v0 = __log2f(ps0) + acc.m[0], v1 = __log2f(ps1) + acc.m[1];
        if constexpr (ACCUMULATE) {
            if (h0 < GQ) atomic_log2_add(mass_pg + (size_t)h0 * mass_stride, v0);
            if (h0 + 1 < GQ) atomic_log2_add(mass_pg + (size_t)(h0 + 1) * mass_stride, v1);
        } else {
            if (h0 < GQ) mass_pg[(size_t)h0 * mass_stride] = v0;
            if (h0 + 1 < GQ) mass_pg[(size_t)(h0 + 1) * mass_stride] = v1;
        }
    }
}

// All packed words of one lane for one code section.
template <int D>
__device__ __forceinline__ void load_lane_words(uint32_t sec, int lane, uint32_t (&w)[3 * (D / 16) / 4])
{
    constexpr int LW = 3 * (D / 16) / 4;
#pragma unroll
    for (int c = 0; c < LW / 4; ++c) {
        const uint4 v = lds128(sec + c * 512 + lane * 16);
        w[4 * c] = v.x; w[4 * c + 1] = v.y; w[4 * c + 2] = v.z; w[4 * c + 3] = v.w;
    }
    if constexpr (LW % 4 != 0) {
        const uint2 v = lds64(sec + (LW / 4) * 512 + lane * 8);
        w[LW - 2] = v.x; w[LW - 1] = v.y;
    }
}

// Scores of the four key blocks 4j..4j+3 of a Stale page: 12 byte-table lookups per block pair and two
// MMAs per block (query hi and lo).
template <bool SPLIT>
__device__ __forceinline__ void tq3_key_quad(float (&S0)[4], float (&S1)[4], uint32_t A, uint32_t Bw, uint32_t Cw,
                                             uint32_t q_quad)
{
    uint32_t sel[4];
    sel[0] = A & 0x77777777u;
    sel[1] = Bw & 0x77777777u;
    sel[2] = lop3_and_or(A >> 1, 0x44444444u, Cw & 0x33333333u);
    sel[3] = lop3_and_or(Bw >> 1, 0x44444444u, (Cw >> 2) & 0x33333333u);
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        uint32_t a[4];
        key_lut4(sel[w], a[0], a[1]);
        key_lut4(sel[w] >> 16, a[2], a[3]);
        if constexpr (SPLIT) {                             // {b0, b1}: hi in columns 0-3, lo in columns 4-7
            const uint2 q = lds64(q_quad + w * 256);
            if (w & 1) mma16816(S1, a, q.x, q.y);
            else       mma16816(S0, a, q.x, q.y);
            continue;
        }
        const uint4 q = lds128(q_quad + w * 512);          // {hi b0, hi b1, lo b0, lo b1}
        if (w & 1) { mma16816(S1, a, q.x, q.y); mma16816(S1, a, q.z, q.w); }
        else       { mma16816(S0, a, q.x, q.y); mma16816(S0, a, q.z, q.w); }
    }
}

// Output update of the four channel blocks 4j..4j+3 of a Stale page: integer codes through the tensor
// core, then the fp16 scale and zero of every channel applied to the 16x8 result in fp32.
// DEFER (long pages): sum p * code only, the accumulators are in code units until the page is left.
template <bool DEFER, bool SPLIT>
__device__ __forceinline__ void tq3_value_quad(float (&o0)[4], float (&o1)[4], float (&o2)[4], float (&o3)[4],
                                               uint32_t W0, uint32_t W1, uint32_t W2, uint32_t meta_quad, const PFrag& pf)
{
    float t[4];
    uint32_t a[4];
    auto product = [&](float (&o)[4]) {
        if constexpr (DEFER) mma16816(o, a, pf.b0, pf.b1);
        else mma16816_zero(o, a, pf.b0, pf.b1);
        if constexpr (!SPLIT) mma16816(o, a, pf.c0, pf.c1);
    };
    uint4 mt;
    {   // blocks 4j, 4j+1
        if constexpr (!DEFER) mt = lds128(meta_quad);
        const uint32_t X = prmt(W0, W1, 0x6341u);
        value_operands<0>(a, W0, W1, W2, X);
        product(DEFER ? o0 : t);
        if constexpr (!DEFER) affine_accumulate(o0, t, mt.x, mt.y, pf.ps0, pf.ps1);
        value_operands<1>(a, W0, W1, W2, X);
        product(DEFER ? o1 : t);
        if constexpr (!DEFER) affine_accumulate(o1, t, mt.z, mt.w, pf.ps0, pf.ps1);
    }
    {   // blocks 4j+2, 4j+3
        if constexpr (!DEFER) mt = lds128(meta_quad + 128);
        const uint32_t X = prmt(W1, W2, 0x6341u);
        value_operands<2>(a, W0, W1, W2, X);
        product(DEFER ? o2 : t);
        if constexpr (!DEFER) affine_accumulate(o2, t, mt.x, mt.y, pf.ps0, pf.ps1);
        value_operands<3>(a, W0, W1, W2, X);
        product(DEFER ? o3 : t);
        if constexpr (!DEFER) affine_accumulate(o3, t, mt.z, mt.w, pf.ps0, pf.ps1);
    }
}

// ---- record format 2 ---------------------------------------------------------------------------------
// The key levels of format 2 are eighths of small integers (2, 6, 11, 18), and four consecutive dims of a
// token are the four nibbles of one half-word: one byte-table lookup turns four codes into four signed bytes,
// and the products run as integer MMAs with the roles swapped: A = the rotated query (16 rows = 8 heads x 2
// of its 3 digits per MMA), B = the keys of eight tokens (32 dims per step).  S[head g][tokens 2tq, 2tq+1]
// then sits in the lane that needs exactly these probabilities as the B fragment of the value product: no
// transposition.
//
// Rotated query of head h: q' = delta_h (2^14 t0 + 2^7 t1 + t2), digits in [-64, 63], delta_h = max|q'| / (63 2^14):
// 21 bits below the largest coordinate (one fp16, 11 bits, is not enough for the 2e-3 bound; two int8 digits,
// 15 bits, fail it on short peaked rows by simulation).  The integer sums are exact.

// Two 32-dim steps (2j, 2j+1) of a Stale page: word triple (A, B, C) of the lane -> eight operand registers
// (step, token half, K half), tokens g and g + 8.  They are an A fragment (16 tokens x 32 dims) as well as two B
// fragments (32 dims x 8 tokens):
//   more than four heads: A = keys, B = one query digit of eight heads: three MMAs per step give S_d[token][head],
//     d = 0, 1, 2 (with the query as A its digits fill one and a half fragments: four MMAs for 16 tokens; 2 x 59,008
//     tokens in 16 layers: 558 -> 540 us);
//   SPLIT: A = query, rows 0-3 digit 0, 4-7 digit 1, 8-11 and 12-15 digit 2 of heads 0-3: one MMA per token half.
// q_pair: shared-memory address of this lane's query fragments of step 2j; a step has 512 bytes (SPLIT), or
// digits 0 and 1 (16 bytes a lane), then digit 2 (8 bytes a lane; `q2_pair`) 512 bytes behind, 768 in all.
template <bool FIRST, bool SPLIT>      // FIRST: the page's first two steps start the sums
__device__ __forceinline__ void tq3_key_pair_v2(int (&S0)[4], int (&S1)[4], int (&S2)[4],
                                                uint32_t A, uint32_t Bw, uint32_t Cw, uint32_t q_pair, uint32_t q2_pair)
{
    // signed levels +-{2, 6, 11, 18} (eight times the codebook) as bytes, indexed by code = magnitude | sign << 2
    constexpr uint32_t T0 = 0x120B0602u, T1 = 0xEEF5FAFEu;
    uint32_t sel[4], r[8];
    sel[0] = A & 0x77777777u;
    sel[1] = Bw & 0x77777777u;
    sel[2] = lop3_and_or(A >> 1, 0x44444444u, Cw & 0x33333333u);
    sel[3] = lop3_and_or(Bw >> 1, 0x44444444u, (Cw >> 2) & 0x33333333u);
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        r[2 * w] = prmt(T0, T1, sel[w]);
        r[2 * w + 1] = prmt(T0, T1, sel[w] >> 16);
    }
#pragma unroll
    for (int st = 0; st < 2; ++st) {
        const uint32_t k0 = r[4 * st], k1 = r[4 * st + 1], k2 = r[4 * st + 2], k3 = r[4 * st + 3];
        if constexpr (SPLIT) {
            const uint4 q = lds128(q_pair + st * 512);
            if (FIRST && st == 0) {
                mma16832_s8_zero(S0, q.x, q.y, q.z, q.w, k0, k1);
                mma16832_s8_zero(S1, q.x, q.y, q.z, q.w, k2, k3);
            } else {
                mma16832_s8(S0, q.x, q.y, q.z, q.w, k0, k1);
                mma16832_s8(S1, q.x, q.y, q.z, q.w, k2, k3);
            }
        } else {
            const uint4 q = lds128(q_pair + st * 768);
            const uint2 q2 = lds64(q2_pair + st * 768);
            if (FIRST && st == 0) {
                mma16832_s8_zero(S0, k0, k2, k1, k3, q.x, q.y);
                mma16832_s8_zero(S1, k0, k2, k1, k3, q.z, q.w);
                mma16832_s8_zero(S2, k0, k2, k1, k3, q2.x, q2.y);
            } else {
                mma16832_s8(S0, k0, k2, k1, k3, q.x, q.y);
                mma16832_s8(S1, k0, k2, k1, k3, q.z, q.w);
                mma16832_s8(S2, k0, k2, k1, k3, q2.x, q2.y);
            }
        }
    }
}

// head g, one token: exact integer sums of the three digits -> the score in units of delta_h / 8
__device__ __forceinline__ float digits_to_score(int hi, int mid, int lo)
{
    return fmaf((float)hi, 16384.f, (float)(mid * 128 + lo));
}

// row form of the maximum from the column form and back (lanes 4h .. 4h+3 hold head h's row value; lane
// (g, tq) holds the column values of heads 2tq, 2tq+1)
template <int NB>
__device__ __forceinline__ void max_rows_from_columns(WarpAcc<NB>& acc, int lane)
{
    const int g = lane >> 2;
    const float a = __shfl_sync(0xffffffffu, acc.m[0], g >> 1), b = __shfl_sync(0xffffffffu, acc.m[1], g >> 1);
    acc.mr = (g & 1) ? b : a;
}

// Scores s[0..1] = tokens 2tq, 2tq+1, s[2..3] = tokens 2tq+8, 2tq+9, all of head g.  Raises the running
// maximum of head g when it is exceeded by more than the slack and rescales the accumulator columns.
template <int NB, bool TILED = false>
__device__ __forceinline__ void softmax_rescale_v2(WarpAcc<NB>& acc, const float (&s)[4], int lane)
{
    constexpr uint32_t FULL = 0xffffffffu;
    float mx = fmaxf(fmaxf(s[0], s[1]), fmaxf(s[2], s[3]));
    if (__any_sync(FULL, mx > acc.mr + kRescaleSlack)) {
        mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, 2));
        const bool up = mx > acc.mr + kRescaleSlack;
        const float f = up ? fast_exp2(acc.mr - mx) : 1.f;
        if (up) acc.mr = mx;
        const int tq = lane & 3;
        const float f0 = __shfl_sync(FULL, f, 8 * tq), f1 = __shfl_sync(FULL, f, 8 * tq + 4);
        acc.m[0] = __shfl_sync(FULL, acc.mr, 8 * tq);
        acc.m[1] = __shfl_sync(FULL, acc.mr, 8 * tq + 4);
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            acc.o[i][0] *= f0; acc.o[i][2] *= f0;
            acc.o[i][1] *= f1; acc.o[i][3] *= f1;
        }
        acc.l[0] *= f0;
        acc.l[1] *= f1;
        if constexpr (TILED) {
            acc.lp[0] *= f0; acc.lp[1] *= f1;
            acc.pk[0] *= f0; acc.pk[1] *= f1;
        }
    }
}

// P of head g for the lane's four tokens is the B fragment of the value product as it stands.
template <int NB>
__device__ __forceinline__ void softmax_probs_v2(WarpAcc<NB>& acc, const float (&s)[4], PFrag& pf, int lane)
{
    const float p0 = fast_exp2(s[0] - acc.mr), p1 = fast_exp2(s[1] - acc.mr);
    const float p2 = fast_exp2(s[2] - acc.mr), p3 = fast_exp2(s[3] - acc.mr);
    pf.b0 = pack_f16x2(p0, p1);
    pf.b1 = pack_f16x2(p2, p3);
    const float2 h01 = half2_to_float2(pf.b0), h23 = half2_to_float2(pf.b1);
    pf.c0 = pack_f16x2(p0 - h01.x, p1 - h01.y);
    pf.c1 = pack_f16x2(p2 - h23.x, p3 - h23.y);
    pf.b0 = lane & 16 ? pf.c0 : pf.b0;       // rows 4-7 carry the low halves of heads 0-3
    pf.b1 = lane & 16 ? pf.c1 : pf.b1;
    const uint32_t ones[4] = {0x3C003C00u, 0x3C003C00u, 0x3C003C00u, 0x3C003C00u};
    float ps[4];
    mma16816_zero(ps, ones, pf.b0, pf.b1);
    pf.ps0 = ps[0];
    pf.ps1 = ps[1];
    acc.l[0] += ps[0];
    acc.l[1] += ps[1];
}

// Software-pipelined step over Stale pages: the value phase of the current page (record rec_v, its
// probabilities pf) and the score phase of the next page (record rec_k) are issued quad by quad in
// one instruction stream, so that table lookups, half-precision FMAs, fp32 FMAs and MMAs of the two
// phases overlap.  DO_V / DO_K switch the halves off for the first and the last page.
template <int D, bool DO_V, bool DO_K, bool DEFER, int FMT, bool SPLIT>
__device__ __forceinline__ void tq3_step(WarpAcc<D / 16>& acc, uint32_t rec_v, const float (&s_cur)[4], PFrag& pf, uint32_t rec_k,
                                         uint32_t qt_lane, float sc2, float sc2b, int lane, float (&s_next)[4])
{
    constexpr int NB = D / 16, LW = 3 * NB / 4;
    const int g = lane >> 2;
    uint32_t kw[LW], vw[LW];
    float S0[4] = {0.f, 0.f, 0.f, 0.f}, S1[4] = {0.f, 0.f, 0.f, 0.f};
    int I0[4], I1[4], I2[4];            // format 2: digits 0, 1, 2; SPLIT: tokens g, g + 8; started by the first pair of steps
    if constexpr (DO_K) load_lane_words<D>(rec_k, lane, kw);
    if constexpr (DO_V) load_lane_words<D>(rec_v + 6 * D, lane, vw);
    if constexpr (DO_V) {      // in one block with the key unpack of the next page
        if constexpr (FMT == 2 && SPLIT) softmax_probs_v2<NB>(acc, s_cur, pf, lane);
        else softmax_probs<NB, SPLIT>(acc, s_cur, pf, lane);
    }
    if constexpr (DO_V && DEFER) {
        acc.lp[0] += pf.ps0;
        acc.lp[1] += pf.ps1;
    }
    const uint32_t meta = rec_v + 12 * D + 32 + g * 16;
#pragma unroll
    for (int j = 0; j < NB / 4; ++j) {
        if constexpr (DO_K) {
            if constexpr (FMT == 2) {
                const uint32_t q = qt_lane + j * (SPLIT ? 1024 : 1536), q2 = q - lane * 8 + 512;
                if (j == 0) tq3_key_pair_v2<true, SPLIT>(I0, I1, I2, kw[0], kw[1], kw[2], q, q2);
                else tq3_key_pair_v2<false, SPLIT>(I0, I1, I2, kw[3 * j], kw[3 * j + 1], kw[3 * j + 2], q, q2);
            }
            else tq3_key_quad<SPLIT>(S0, S1, kw[3 * j], kw[3 * j + 1], kw[3 * j + 2], qt_lane + j * (SPLIT ? 1024 : 2048));
        }
        if constexpr (DO_V)
            tq3_value_quad<DEFER, SPLIT>(acc.o[4 * j], acc.o[4 * j + 1], acc.o[4 * j + 2], acc.o[4 * j + 3], vw[3 * j], vw[3 * j + 1],
                                         vw[3 * j + 2], meta + j * 256, pf);
    }
    if constexpr (DO_K && FMT == 2 && SPLIT) {
        // head g % 4, tokens 2tq, 2tq+1 (I0) and 2tq+8, 2tq+9 (I1): the three query digits, then the token's norm
        // correction (sc2 carries the head's digit unit delta_h / 8 here)
        const int tq = lane & 3;
        const uint32_t gaddr = rec_k + 12 * D + 4 * tq;
        const float2 ga = half2_to_float2(lds32(gaddr)), gb = half2_to_float2(lds32(gaddr + 16));
        // This lane has digit 0 (g < 4) or 1 (g >= 4) and digit 2 of head g % 4, the lane 16 away the other one.  Both put
        // the score together in the same order: rows h and h + 4 supply the high and the low halves of the same
        // probabilities, so their scores have to be the same bits.
        float d[4];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int o0 = __shfl_xor_sync(0xffffffffu, I0[e], 16), o1 = __shfl_xor_sync(0xffffffffu, I1[e], 16);
            d[e] = lane & 16 ? digits_to_score(o0, I0[e], I0[2 + e]) : digits_to_score(I0[e], o0, I0[2 + e]);
            d[2 + e] = lane & 16 ? digits_to_score(o1, I1[e], I1[2 + e]) : digits_to_score(I1[e], o1, I1[2 + e]);
        }
        s_next[0] = d[0] * (ga.x * sc2);
        s_next[1] = d[1] * (ga.y * sc2);
        s_next[2] = d[2] * (gb.x * sc2);
        s_next[3] = d[3] * (gb.y * sc2);
    }
    if constexpr (DO_K && FMT == 2 && !SPLIT) {
        // tokens g, g + 8 of heads 2tq, 2tq + 1 (digit units in sc2, sc2b)
        const uint32_t gaddr = rec_k + 12 * D;
        const float r0 = __half2float(__ushort_as_half(lds16(gaddr + 2 * g))), r1 = __half2float(__ushort_as_half(lds16(gaddr + 2 * g + 16)));
        s_next[0] = digits_to_score(I0[0], I1[0], I2[0]) * (r0 * sc2);
        s_next[1] = digits_to_score(I0[1], I1[1], I2[1]) * (r0 * sc2b);
        s_next[2] = digits_to_score(I0[2], I1[2], I2[2]) * (r1 * sc2);
        s_next[3] = digits_to_score(I0[3], I1[3], I2[3]) * (r1 * sc2b);
    }
    if constexpr (DO_K && FMT == 1) {
        const uint32_t gaddr = rec_k + 12 * D;
        const float r0 = __half2float(__ushort_as_half(lds16(gaddr + 2 * g))) * sc2;
        const float r1 = __half2float(__ushort_as_half(lds16(gaddr + 2 * g + 16))) * sc2;
        s_next[0] = (S0[0] + S1[0]) * r0;
        s_next[1] = (S0[1] + S1[1]) * r0;
        s_next[2] = (S0[2] + S1[2]) * r1;
        s_next[3] = (S0[3] + S1[3]) * r1;
        if constexpr (SPLIT) {               // products with the high and the low half of the query
#pragma unroll
            for (int e = 0; e < 4; ++e) s_next[e] += __shfl_xor_sync(0xffffffffu, s_next[e], 2);
        }
    }
}

// Four 8x8 matrices of 16-bit elements from shared memory in the MMA fragment layout: lane l supplies the
// address of row l % 8 of matrix l / 8; every lane receives, per matrix, the 32 bits at (row lane / 4,
// 16-bit columns 2 (lane % 4), 2 (lane % 4) + 1).
__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}

// One Recent/Anchor page: keys [16 tokens][d] e4m3 at kaddr, values [d channels][16 tokens] at vaddr.
// MMA row r of the score tile holds token pi(r) = 4 (r % 8 / 2) + r % 2 + 2 (r / 8), so that the value
// fragments can be fetched with ldmatrix: a lane then holds the four consecutive tokens 4tq .. 4tq+3 of
// its two channel rows, which is the order P^T has after the transposition of a score tile whose rows
// are permuted this way.
template <int D, bool SCORED, bool ACCUMULATE, bool SPLIT>
__device__ __forceinline__ void fp8_page(WarpAcc<D / 16>& acc, uint32_t kaddr, uint32_t vaddr, uint32_t qf_lane,
                                         float score_scale, float v_scale, int valid, int lane, float* mass_pg,
                                         int mass_stride, int GQ)
{
    constexpr int NB = D / 16;
    const int g = lane >> 2, tq = lane & 3;
    const int tok0 = 4 * (g >> 1) + (g & 1), tok1 = tok0 + 2;       // tokens of the lane's two score rows
    float S0[4] = {0.f, 0.f, 0.f, 0.f}, S1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int j = 0; j < D / 64; ++j) {
        const uint4 r0 = lds128(kaddr + tok0 * D + 64 * j + 16 * tq);
        const uint4 r1 = lds128(kaddr + tok1 * D + 64 * j + 16 * tq);
        const uint32_t w0[4] = {r0.x, r0.y, r0.z, r0.w}, w1[4] = {r1.x, r1.y, r1.z, r1.w};
#pragma unroll
        for (int w = 0; w < 4; ++w) {
            uint32_t a[4];
            a[0] = e4m3x2_to_f16x2((uint16_t)(w0[w] & 0xFFFFu));
            a[1] = e4m3x2_to_f16x2((uint16_t)(w1[w] & 0xFFFFu));
            a[2] = e4m3x2_to_f16x2((uint16_t)(w0[w] >> 16));
            a[3] = e4m3x2_to_f16x2((uint16_t)(w1[w] >> 16));
            const uint2 qv = lds64(qf_lane + (4 * j + w) * 256);
            if (w & 1) mma16816(S1, a, qv.x, qv.y);
            else       mma16816(S0, a, qv.x, qv.y);
        }
    }
    float s[4] = {(S0[0] + S1[0]) * score_scale, (S0[1] + S1[1]) * score_scale, (S0[2] + S1[2]) * score_scale,
                  (S0[3] + S1[3]) * score_scale};
    // bytes of tokens beyond the sequence end are cleared so that stale NaN patterns cannot leak
    uint32_t keep = 0xFFFFFFFFu;                     // byte mask for the tokens 4tq .. 4tq+3 of a value word
    if (valid < kPage) {
        if (tok0 >= valid) s[0] = s[1] = -CUDART_INF_F;
        if (tok1 >= valid) s[2] = s[3] = -CUDART_INF_F;
        keep = (4 * tq < valid ? 0x000000FFu : 0u) | (4 * tq + 1 < valid ? 0x0000FF00u : 0u) |
               (4 * tq + 2 < valid ? 0x00FF0000u : 0u) | (4 * tq + 3 < valid ? 0xFF000000u : 0u);
    }
    PFrag pf;
    softmax_page<NB, SPLIT>(acc, s, pf, lane);
    if constexpr (SCORED) store_page_mass<NB, SPLIT, ACCUMULATE>(acc, pf.ps0, pf.ps1, mass_pg, mass_stride, GQ, lane);
    const bool scale_v = v_scale != 1.0f;
#pragma unroll
    for (int cb = 0; cb < NB; cb += 2) {
        // channels 16cb .. 16cb+31: rows of 16 bytes, lane l addresses row l
        uint32_t v[4];
        ldmatrix_x4(vaddr + cb * 256 + lane * 16, v[0], v[1], v[2], v[3]);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const uint32_t lo = v[2 * e] & keep, hi = v[2 * e + 1] & keep;      // channel rows g and g + 8 of block cb + e
            uint32_t a[4];
            a[0] = e4m3x2_to_f16x2((uint16_t)(lo & 0xFFFFu));
            a[1] = e4m3x2_to_f16x2((uint16_t)(hi & 0xFFFFu));
            a[2] = e4m3x2_to_f16x2((uint16_t)(lo >> 16));
            a[3] = e4m3x2_to_f16x2((uint16_t)(hi >> 16));
            if (scale_v) {
                float t[4];
                mma16816_zero(t, a, pf.b0, pf.b1);
                if constexpr (!SPLIT) mma16816(t, a, pf.c0, pf.c1);
#pragma unroll
                for (int i = 0; i < 4; ++i) acc.o[cb + e][i] = fmaf(v_scale, t[i], acc.o[cb + e][i]);
            } else {
                mma16816(acc.o[cb + e], a, pf.b0, pf.b1);
                if constexpr (!SPLIT) mma16816(acc.o[cb + e], a, pf.c0, pf.c1);
            }
        }
    }
}

// Eq. (softmax-merge) of one (request, KV head) row that was split over n_parts blocks.  Part 0 sits
// in slot first_slot, part j > 0 in slot even_base + 2j.  Called by all NT threads of the block that
// drew the row's last ticket; `buf` is idle shared memory.  Warp hd < 8 reduces the maxima and row sums of head hd
// (one trip to L2: both are loaded together and kept in shared memory); a thread owns float4 groups (one channel,
// four heads) of the [channel][8 heads] tile.  With twice as many threads as groups (16 warps at d = 128) every
// other part goes to the second half of the threads.  KP loads per thread are in flight, issued before the weights
// are worked out.
template <int D, int NT, int KPMAX>
__device__ __forceinline__ void merge_row(const DecodeParams& P, int first_slot, int even_base, int n_parts,
                                          float* buf, int b, int h)
{
    constexpr uint32_t FULL = 0xffffffffu;
    constexpr int STRIDE = 8 * D + 16, GROUPS = 2 * D, GPT = (GROUPS + NT - 1) / NT, S = NT >= 2 * GROUPS ? 2 : 1;
    constexpr int KP = KPMAX / GPT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int GQ = P.group, hq = P.hkv * GQ;
    float* w_s = buf;                        // [n_parts][8] maxima, then weights e^{m_j - m}
    float* l_s = buf + n_parts * 8;          // [n_parts][8] row sums
    float* ml_s = buf + n_parts * 16;        // [8] m, [8] l of the row
    auto slot_of = [&](int j) -> const float* {
        return P.partials + (size_t)(j == 0 ? first_slot : even_base + 2 * j) * STRIDE;
    };
    __syncthreads();
    float4 acc[GPT], v[KP][GPT];
#pragma unroll
    for (int k = 0; k < GPT; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int first = S > 1 ? tid / GROUPS : 0, grp0 = S > 1 ? tid % GROUPS : tid;     // parts first, first + S, ...
    const int head0 = (tid & 1) * 4;         // NT is even: every group of this thread covers the same four heads
    auto load_round = [&](int j0) {
#pragma unroll
        for (int p = 0; p < KP; ++p) {
            const float* ps = slot_of(min(j0 + p * S, n_parts - 1));
#pragma unroll
            for (int k = 0; k < GPT; ++k)
                v[p][k] = __ldcg(reinterpret_cast<const float4*>(ps) + min(grp0 + k * NT, GROUPS - 1));
        }
    };
    auto use_round = [&](int j0) {
#pragma unroll
        for (int p = 0; p < KP; ++p)
            if (j0 + p * S < n_parts) {
                const float4 w = *reinterpret_cast<const float4*>(w_s + (j0 + p * S) * 8 + head0);
#pragma unroll
                for (int k = 0; k < GPT; ++k) {
                    acc[k].x = fmaf(w.x, v[p][k].x, acc[k].x);
                    acc[k].y = fmaf(w.y, v[p][k].y, acc[k].y);
                    acc[k].z = fmaf(w.z, v[p][k].z, acc[k].z);
                    acc[k].w = fmaf(w.w, v[p][k].w, acc[k].w);
                }
            }
    };
    load_round(first);                       // in flight while the weights are worked out
    for (int hd = warp; hd < 8; hd += NT / 32) {
        float M = -CUDART_INF_F;
        for (int j = lane; j < n_parts; j += 32) {
            const float* ps = slot_of(j) + 8 * D;
            const float lj = __ldcg(ps + 8 + hd), mj = __ldcg(ps + hd);
            l_s[j * 8 + hd] = lj;
            w_s[j * 8 + hd] = mj;
            if (lj > 0.f) M = fmaxf(M, mj);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(FULL, M, o));
        float L = 0.f;
        for (int j = lane; j < n_parts; j += 32) {      // re-reads this lane's own entries
            const float lj = l_s[j * 8 + hd];
            const float w = lj > 0.f ? fast_exp2(w_s[j * 8 + hd] - M) : 0.f;
            w_s[j * 8 + hd] = w;
            L = fmaf(w, lj, L);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) L += __shfl_xor_sync(FULL, L, o);
        if (lane == 0) {
            ml_s[hd] = M;
            ml_s[8 + hd] = L;
        }
    }
    __syncthreads();
    use_round(first);
    for (int j0 = first + KP * S; j0 < n_parts; j0 += KP * S) {
        load_round(j0);
        use_round(j0);
    }
    if constexpr (S > 1) {                   // the second half of the threads hands its sums over
        float4* half = reinterpret_cast<float4*>(buf + n_parts * 16 + 16);
        if (first == 1) half[grp0] = acc[0];
        __syncthreads();
        if (first == 0) {
            const float4 o = half[grp0];
            acc[0].x += o.x; acc[0].y += o.y; acc[0].z += o.z; acc[0].w += o.w;
        }
    }
#pragma unroll
    for (int k = 0; k < GPT; ++k) {
        const int grp = grp0 + k * NT, ch = grp >> 1;
        if (grp >= GROUPS || first > 0) continue;
        const float av[4] = {acc[k].x, acc[k].y, acc[k].z, acc[k].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int head = head0 + e;
            if (head < GQ) {
                const float L = ml_s[8 + head];
                P.out[((size_t)b * hq + h * GQ + head) * D + ch] = L > 0.f ? av[e] / L : 0.f;
            }
        }
    }
    if (P.lse && tid < GQ)
        P.lse[(size_t)b * hq + h * GQ + tid] = ml_s[8 + tid] > 0.f ? (ml_s[tid] + log2f(ml_s[8 + tid])) * kLn2 : -CUDART_INF_F;
}

template <int D, int NW, int NSTAGE, int MINB, bool SCORED, bool TILED, int MAXL, int FMT, bool FLAT, bool SPLIT>
__global__ void __launch_bounds__(NW * 32, MINB) decode_tensor_kernel(const LayerSet<MAXL> LS)
{
    const DecodeParams& P0 = LS.layer[0];    // requests and geometry are common to all layers
    // 16-byte loads that a thread of the merge keeps in flight.  (d 256: 20 and 40 are alike also for rows of many parts, 37:
    // 1 x 59,008 tokens 31.1 / 30.6 us a call, 1 x 131,072 53.4 / 53.1; 74: 33.2 / 33.1; 40 cost registers elsewhere.)
    constexpr int MERGE_LOADS = NW * MINB <= 8 ? 20 : 16;
    constexpr int ROW_COST = cut_row_cost(NW, TILED), MIN_PAGES = cut_min_pages(NW, MINB);
    using G = Geo<D, NW, NSTAGE, TILED>;     // pages of several tiles: short rounds leave room for the parked rows
    constexpr int NB = G::NB;
    constexpr uint32_t FULL = 0xffffffffu;
    extern __shared__ __align__(128) uint8_t smem[];
    const uint32_t sbase = smem_u32(smem);
    int* cum = reinterpret_cast<int*>(smem + G::OFF_CUM);
    int* lens_s = reinterpret_cast<int*>(smem + G::OFF_LENS);
    float* sm_m = reinterpret_cast<float*>(smem + G::OFF_M);
    float* sm_l = reinterpret_cast<float*>(smem + G::OFF_L);
    Partition* pt = reinterpret_cast<Partition*>(smem + G::OFF_PART);
    int* last_s = reinterpret_cast<int*>(smem + G::OFF_LAST);
    float* red = reinterpret_cast<float*>(smem);            // [NW][D][8] over the ring, between segments

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, tq = lane & 3;
    const int hkv = P0.hkv, GQ = P0.group, hq = hkv * GQ;
    const int n_layers = MAXL == 1 ? 1 : LS.n;
    // a length beyond the table row is cut to the row (and flagged), so that no entry past it is ever read
    const int len_cap = P0.max_pages * P0.tiles * kPage;
    auto length_of = [&](int b) -> int {
        const int len = P0.lens[b];
        if (len > len_cap) {
            atomicOr(P0.status, kStBounds);
            return len_cap;
        }
        return len < 0 ? 0 : len;
    };

    // ---- prologue: barriers, lengths, prefix of pages, this block's share ---------------------------------------
    if (tid == 0) {
        for (int i = 0; i < NW * G::NP; ++i) mbar_init(sbase + G::OFF_BAR + 8 * i, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        last_s[1] = 0;
    }
    pdl_wait();
    if (warp == 0) {
        RowSums sum = {0, 0};
        for (int b0 = 0; b0 < P0.B; b0 += 32) {
            const int b = b0 + lane;
            int n = 0;
            if (b < P0.B) {
                const int len = length_of(b);
                lens_s[b] = len;
                n = positions_of(len, hkv, ROW_COST);
            }
            add_requests(sum, cum, P0.B, b0, n, lane);
        }
        if (lane == 0) cum[P0.B] = sum.positions;
        __syncwarp();
        const int pages = sum.positions - sum.requests * hkv * ROW_COST;
        if constexpr (!FLAT || TILED)
            build_partition(pt, cum, lens_s, P0.B, hkv, gridDim.x, pages, ROW_COST, MIN_PAGES, cut_straddle(NW), blockIdx.x, lane);
        if constexpr (FLAT) build_flat_partition(pt, cum, sum.positions, P0.B, n_layers, gridDim.x, pages, MIN_PAGES, blockIdx.x, lane);
    }
    __syncthreads();
    int my_start = 0, my_end = 0;                          // more blocks than work: an empty range
    int layer_first = 0, layer_end = n_layers;
    if constexpr (FLAT) {
        layer_first = pt->first_layer;
        layer_end = pt->end_layer;
    } else {
        my_start = pt->start;
        my_end = pt->end;
    }

    // per-warp ring of NP slot pairs; one bit per pair holds the mbarrier phase the next wait must see
    uint32_t phase = 0;
    bool failed = false;
    const uint32_t ring = sbase + warp * NSTAGE * G::SLOT;
    const uint32_t bars = sbase + G::OFF_BAR + warp * G::NP * 8;
    const uint32_t qt_lane = sbase + G::OFF_QT + lane * (SPLIT && FMT == 1 ? 8 : 16), qf_lane = sbase + G::OFF_QF + lane * 8;
    int* list3 = reinterpret_cast<int*>(smem + G::OFF_LIST) + warp * 2 * G::ROUND;   // Stale page ids of the round
    int* list8 = list3 + G::ROUND;                                                   // FP8 page ids | valid << 27
    int* lpg3 = reinterpret_cast<int*>(smem + G::OFF_LIST) + (NW + warp) * 2 * G::ROUND;   // their logical pages (scored variant)
    int* lpg8 = lpg3 + G::ROUND;
    const float sc2 = P0.scale * kLog2e;     // scores are kept in log2 units
    uint32_t pending = 0;                    // slot pairs with copies in flight that nobody has waited for yet
    // Bounded wait for slot pair s, then flip its expected phase.  `limit_ns` of wall time (the pool's wait
    // limit, 20 ms by default); returns false when it ran out.
    auto wait_bounded = [&](uint32_t s, unsigned long long limit_ns) -> bool {
        const uint32_t bar = bars + 8 * s, parity = (phase >> s) & 1u;
        // (limit 0, diagnostic: a copy that this first look does not find counts as late; the first copies of a row are looked
        // at as soon as they are issued)
        bool ok = mbar_try_wait(bar, parity);
        if (!ok && limit_ns != 0) {
            unsigned long long t0, t1;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
            for (int spins = 1; !ok; ++spins) {
                ok = mbar_try_wait(bar, parity);
                if (!ok && (spins & 255) == 0) {
                    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
                    if (t1 - t0 >= limit_ns) break;
                }
            }
        }
        ok = __all_sync(FULL, ok);           // the copy has landed for every lane, or the warp gives up as one
        if (ok) {
            phase ^= 1u << s;
            pending &= ~(1u << s);
        }
        return ok;
    };
    // After a wait has run out the warp stops scanning; before anybody reuses the ring (as the reduction
    // buffer) or the block leaves, every copy this warp still has in flight is waited for with the
    // default limit, so that nothing lands in memory that has changed hands.
    auto drain = [&]() {
        bool lost = false;
#pragma unroll 1
        for (uint32_t s = 0; s < (uint32_t)G::NP; ++s)
            if (pending & (1u << s)) lost |= !wait_bounded(s, kDefaultWaitNs);
        return lost;
    };

    // rows of empty requests
    for (int i0 = blockIdx.x; i0 < P0.B * n_layers; i0 += gridDim.x) {
        const int b = i0 % P0.B;
        if (lens_s[b] > 0) continue;
        const DecodeParams& P = LS.layer[MAXL == 1 ? 0 : i0 / P0.B];
        for (int i = tid; i < hq * D; i += NW * 32) P.out[(size_t)b * hq * D + i] = 0.f;
        if (P.lse)
            for (int i = tid; i < hq; i += NW * 32) P.lse[(size_t)b * hq + i] = -CUDART_INF_F;
    }

    for (int layer = layer_first; layer < layer_end; ++layer) {
    const DecodeParams& P = LS.layer[MAXL == 1 ? 0 : layer];
    if constexpr (FLAT) range_in_layer(pt, cum[P0.B], layer, blockIdx.x, my_start, my_end);
    auto wait_slot = [&](uint32_t s) -> bool {
        if (wait_bounded(s, P.wait_ns)) return true;
        failed = true;
        atomicOr(P.status, kStTimeout);
        return false;
    };
    int pos = my_start;
    int b = FLAT && layer > layer_first ? 0 : pt->first_b;
    while (pos < my_end) {
        // ---- locate the segment: request b, KV head h, positions [pg0, pg0 + n_seg) of the row ------
        const Segment sg = segment_at(cum, lens_s, ROW_COST, pos, my_end, b);
        const int len = lens_s[b], h = sg.h, n_pages = sg.n_pages, pg0 = sg.pg0, n_seg = sg.n;
        if (n_seg <= 0) {                          // the block's range ends before the row's first page
            pos = sg.end;
            continue;
        }
        const int32_t* bt_row = P.bt + (size_t)b * P.max_pages;
        const uint8_t* tag_row = P.tags + (size_t)b * P.max_pages;
        // this warp's pages: a contiguous run of positions (which holds FP8 and TQ3 pages in the row's proportion,
        // see page_at, so the warps of a block finish together)
        const int warp_first = (int)(((unsigned)n_seg * (unsigned)warp) / NW);
        const int n_my = (int)(((unsigned)n_seg * (unsigned)(warp + 1)) / NW) - warp_first;
        constexpr int EPL = D / 32;
        constexpr int HPW = (8 + NW - 1) / NW;      // query heads a warp prepares (head warp, warp + NW, ...)
        float qx[HPW][EPL];       // loaded before anything else waits
#pragma unroll
        for (int k = 0; k < HPW; ++k) {
            const int hd = warp + k * NW;
            uint2 raw[EPL / 4];                     // (the entry points take queries on 16-byte boundaries)
#pragma unroll
            for (int r = 0; r < EPL / 4; ++r)
                raw[r] = hd < GQ ? reinterpret_cast<const uint2*>(P.q + ((size_t)b * hq + h * GQ + hd) * D + lane * EPL)[r]
                                 : make_uint2(0u, 0u);
#pragma unroll
            for (int r = 0; r < EPL; r += 2) {
                const uint32_t w = r & 2 ? raw[r / 4].y : raw[r / 4].x;
                qx[k][r] = __uint_as_float(w << 16);
                qx[k][r + 1] = __uint_as_float(w & 0xFFFF0000u);
            }
        }
        float* mass_row = SCORED ? P.mass + ((size_t)b * hq + (size_t)h * GQ) * P.max_pages : nullptr;
        const uint8_t* tq3_base = P.tq3 + (size_t)h * G::TQ3_REC;
        const uint8_t* fp8_base = P.fp8 + (size_t)h * (2 * G::FP8_HALF);
        // pages of several tiles: a TQ3 page is tiles * (12 D + 32) bytes of tiles, then 4 D bytes of value
        // scale/zero shared by its tiles; an FP8 page is `tiles` consecutive 16-token records
        constexpr int TQ3_TILE = 12 * D + 32, TQ3_META = 4 * D;
        const size_t tq3_page = (size_t)P.tiles * TQ3_TILE + TQ3_META;

        // Table entries of up to G::ROUND of the warp's pages are compacted into two id lists, one per
        // format (entry i of a 32-page chunk is read by lane i, all chunks before the first is looked at; ballots give the
        // positions).
        // Returns how many of the warp's pages (from `first` on) the lists cover.  Long pages in the flat cut: a Stale
        // tile that opens a warp's run of the per-layer cut is marked (kOpens); the scan leaves the page there, and
        // a round ends at the last such tile, so that code sums are gathered over the same runs of tiles as there
        // (their rounding inside the tensor core grows with the length of a run).
        int n3 = 0, n8 = 0;
        constexpr int kOpens = 0x8000;
        auto build_lists = [&](int first) -> int {
            n3 = n8 = 0;
            int covered = min(G::ROUND, n_my - first), cut3 = 0, cut8 = 0, cut = 0;
            constexpr int CH = G::ROUND / 32;
            int ids[CH], tg[CH], pgs[CH];
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int i = first + c * 32 + lane;
                ids[c] = -1;
                tg[c] = pgs[c] = 0;
                if (i < n_my) {
                    // `pg` counts 16-token tiles of the row (long pages: in their order, so that a warp's run stays inside one or
                    // two pages); the table has one entry per page of P.tiles tiles
                    const int pg = TILED ? pg0 + warp_first + i : page_at(pg0 + warp_first + i, n_pages);
                    const int entry = TILED ? pg / P.tiles : pg;
                    pgs[c] = pg;
                    ids[c] = bt_row[entry];
                    tg[c] = tag_row[entry];
                }
            }
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const int i = first + c * 32 + lane;
                if (first + c * 32 >= n_my) break;
                int kind = 0, id = ids[c], valid = kPage, pg = pgs[c];
                if (i < n_my) {
                    valid = min(kPage, len - pg * kPage);
                    if (tg[c] == MKV_TAG_STALE)
                        kind = (id >= 0 && id < P.tq3_pages && valid == kPage) ? 1 : 0;
                    else
                        kind = (tg[c] <= MKV_TAG_ANCHOR && id >= 0 && id < P.fp8_pages) ? 2 : 0;
                    if (kind == 0) atomicOr(P.status, kStBounds);     // never dereferenced
                    if constexpr (TILED) {   // second list: tile inside its page | logical page << 16
                        const int entry = pg / P.tiles;
                        const bool opens = FLAT && opens_warp_run(pt, b * hkv + h, sg.row_start, sg.row_end, sg.row_start + pg, NW);
                        pg = (pg - entry * P.tiles) | (entry << 16) | (opens ? kOpens : 0);
                    }
                }
                const uint32_t m3 = __ballot_sync(FULL, kind == 1), m8 = __ballot_sync(FULL, kind == 2);
                const uint32_t lt = (1u << lane) - 1u;
                if (kind == 1) list3[n3 + __popc(m3 & lt)] = id;
                if (kind == 2) list8[n8 + __popc(m8 & lt)] = id | ((valid & 15) << 27);
                if constexpr (SCORED || TILED) {     // logical page (scored output) or tile inside the page (pages of several tiles)
                    if (kind == 1) lpg3[n3 + __popc(m3 & lt)] = pg;
                    if (kind == 2) lpg8[n8 + __popc(m8 & lt)] = pg;
                }
                if constexpr (TILED && FLAT) {
                    const uint32_t mo = __ballot_sync(FULL, i < n_my && (pg & kOpens));
                    if (mo) {
                        const int at = 31 - __clz(mo);
                        cut = c * 32 + at;
                        cut3 = n3 + __popc(m3 & ((1u << at) - 1u));
                        cut8 = n8 + __popc(m8 & ((1u << at) - 1u));
                    }
                }
                n3 += __popc(m3);
                n8 += __popc(m8);
            }
            if (TILED && FLAT && cut > 0 && first + covered < n_my) {
                covered = cut;
                n3 = cut3;
                n8 = cut8;
            }
            __syncwarp();
            return covered;
        };
        // Copy Stale pages 2j, 2j + 1 of the round (the second if there is one) into slot pair j % NP, a lane each.
        auto issue_tq3 = [&](int j) {
            const uint32_t s = (uint32_t)j % G::NP;
            const int n = min(n3 - 2 * j, 2);
            pending |= 1u << s;
            if (lane < n) {
                constexpr uint32_t BYTES = TILED ? TQ3_TILE : G::TQ3_REC;    // long pages: the tile only, their scale/zero are applied once
                const int i = 2 * j + lane, page = list3[i];
                const uint8_t* src = TILED ? P.tq3 + ((size_t)page * hkv + h) * tq3_page + (size_t)(lpg3[i] & 0x7FFF) * TQ3_TILE
                                           : tq3_base + (size_t)page * hkv * G::TQ3_REC;
                if (lane == 0) mbar_expect_tx(bars + 8 * s, n * BYTES);
                bulk_load(ring + s * G::PAIR + lane * G::SLOT, src, BYTES, bars + 8 * s);
            }
        };
        // FP8 page i of the round goes into slot pair (first8 + i) % NP: the first pair is one that the round's last Stale
        // page does not occupy, so that the FP8 copies start before that page is finished
        uint32_t first8 = 0;
        auto issue_fp8 = [&](int i) {
            const uint32_t s = (first8 + (uint32_t)i) % G::NP;
            pending |= 1u << s;
            if (lane == 0) {
                const int e8 = list8[i] & 0x7FFFFFF;
                const uint8_t* rec;
                if constexpr (!TILED) {
                    rec = fp8_base + (size_t)e8 * hkv * (2 * G::FP8_HALF);
                } else {
                    rec = P.fp8 + (((size_t)e8 * hkv + h) * P.tiles + (lpg8[i] & 0x7FFF)) * (2 * G::FP8_HALF);
                }
                mbar_expect_tx(bars + 8 * s, 2 * G::FP8_HALF);
                bulk_load(ring + s * G::PAIR, rec, 2 * G::FP8_HALF, bars + 8 * s);
            }
        };
        auto start_round = [&]() {         // the first copies of a round
            first8 = n3 > 0 ? ((uint32_t)(n3 - 1) / 2 + 1) % G::NP : 0u;
            for (int j = 0; j < min((n3 + 1) / 2, G::NP); ++j) issue_tq3(j);
            if (n3 == 0)
                for (int i = 0; i < min(n8, G::NP); ++i) issue_fp8(i);
        };

        WarpAcc<NB> acc;
        // Pages of several tiles.  While the scan is inside a Stale page, acc.o holds sum p * code and the
        // output gathered before waits in this warp's shared-memory rows ("parked"); leaving the page adds
        // scale * acc.o + zero * acc.lp to it (fold).  The scale/zero halves come straight from the page's
        // metadata in global memory, in the order of the 16-token record.
        float* park = reinterpret_cast<float*>(smem + G::SMEM) + (size_t)warp * NB * 128;
        auto park_store = [&]() {
#pragma unroll
            for (int i = 0; i < NB; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    park[(i * 4 + e) * 32 + lane] = acc.o[i][e];
                    acc.o[i][e] = 0.f;
                }
            acc.pk[0] = acc.pk[1] = 1.f;
            acc.lp[0] = acc.lp[1] = 0.f;
        };
        auto fold = [&](int page, bool to_regs, int logical_page) {
            if constexpr (SCORED)      // this warp's part of the page's exponential sum
                store_page_mass<NB, SPLIT, true>(acc, acc.lp[0], acc.lp[1], mass_row + logical_page, P.max_pages, GQ, lane);
            const uint4* meta = reinterpret_cast<const uint4*>(P.tq3 + ((size_t)page * hkv + h) * tq3_page +
                                                                (size_t)P.tiles * TQ3_TILE + g * 16);
#pragma unroll
            for (int j = 0; j < NB / 4; ++j) {
                const uint4 m01 = meta[j * 16], m23 = meta[j * 16 + 8];
                const uint32_t scp[4] = {m01.x, m01.z, m23.x, m23.z}, zpp[4] = {m01.y, m01.w, m23.y, m23.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int i = 4 * j + q;
                    const float2 sc = half2_to_float2(scp[q]), zp = half2_to_float2(zpp[q]);
                    float r[4];
                    r[0] = fmaf(park[(i * 4 + 0) * 32 + lane], acc.pk[0], fmaf(sc.x, acc.o[i][0], zp.x * acc.lp[0]));
                    r[1] = fmaf(park[(i * 4 + 1) * 32 + lane], acc.pk[1], fmaf(sc.x, acc.o[i][1], zp.x * acc.lp[1]));
                    r[2] = fmaf(park[(i * 4 + 2) * 32 + lane], acc.pk[0], fmaf(sc.y, acc.o[i][2], zp.y * acc.lp[0]));
                    r[3] = fmaf(park[(i * 4 + 3) * 32 + lane], acc.pk[1], fmaf(sc.y, acc.o[i][3], zp.y * acc.lp[1]));
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        if (to_regs) acc.o[i][e] = r[e];
                        else { park[(i * 4 + e) * 32 + lane] = r[e]; acc.o[i][e] = 0.f; }
                    }
                }
            }
            acc.pk[0] = acc.pk[1] = 1.f;
            acc.lp[0] = acc.lp[1] = 0.f;
        };
        (void)park_store; (void)fold;
#pragma unroll
        for (int i = 0; i < NB; ++i) acc.o[i][0] = acc.o[i][1] = acc.o[i][2] = acc.o[i][3] = 0.f;
        acc.l[0] = acc.l[1] = 0.f;
        acc.m[0] = acc.m[1] = -CUDART_INF_F;
        acc.mr = -CUDART_INF_F;

        // first round: start the copies, then build the query fragments while they fly
        int done = 0;
        if (n_my > 0) {
            done = build_lists(0);
            // The ring was the reduction buffer: the copies come after those stores.  (Slots that are used again inside a
            // segment were only read since, and the reads are over: no fence per page.)
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            start_round();
            // limit 0 (diagnostic): the first look comes before the query is prepared, while the copy is still in flight
            if (P.wait_ns == 0 && n3 + n8 > 0 && !__all_sync(FULL, mbar_test_wait(bars, phase & 1u))) {
                failed = true;
                atomicOr(P.status, kStTimeout);
            }
        }

        // query fragments: a warp rotates head `warp` (and `warp + NW`); loads were issued before the copies started
#pragma unroll
        for (int k = 0; k < HPW; ++k) {
            const int hd = warp + k * NW;
            if (hd >= (SPLIT ? 4 : 8)) break;
            float a[EPL];
#pragma unroll
            for (int r = 0; r < EPL; ++r) {
                const int i = lane * EPL + r;
                a[r] = ((P.sigma.w[i >> 5] >> (i & 31)) & 1u) ? -qx[k][r] : qx[k][r];
            }
#pragma unroll
            for (int hh = 1; hh < EPL; hh <<= 1)
#pragma unroll
                for (int r = 0; r < EPL; ++r)
                    if ((r & hh) == 0) {
                        const float u = a[r], w = a[r + hh];
                        a[r] = u + w;
                        a[r + hh] = u - w;
                    }
#pragma unroll
            for (int m = 1; m < 32; m <<= 1)
#pragma unroll
                for (int r = 0; r < EPL; ++r) {
                    const float o = __shfl_xor_sync(FULL, a[r], m);
                    a[r] = (lane & m) ? o - a[r] : a[r] + o;
                }
            const float rs = rsqrtf((float)D);
            __half* qt = reinterpret_cast<__half*>(smem + G::OFF_QT);
            __half* qf = reinterpret_cast<__half*>(smem + G::OFF_QF);
            if constexpr (FMT == 2) {
                // rotated query as three balanced base-128 digits in the fragment order of the integer key
                // products: dim i sits in step i/32 at K slot k = i%32 of fragment lane 4 hd + (k%16)/4, byte k%4 of
                // register k/16 of its digit (see tq3_key_pair_v2)
                uint8_t* qt8 = smem + G::OFF_QT;
                float amax = 0.f;
#pragma unroll
                for (int r = 0; r < EPL; ++r) amax = fmaxf(amax, fabsf(a[r] * rs));
#pragma unroll
                for (int m = 16; m > 0; m >>= 1) amax = fmaxf(amax, __shfl_xor_sync(FULL, amax, m));
                const float delta = amax > 0.f ? amax * (1.f / (63.f * 16384.f)) : 1.f, inv_delta = 1.f / delta;
                if (lane == 0) reinterpret_cast<float*>(smem + G::OFF_QS)[hd] = delta * 0.125f;   // key levels are eighths
#pragma unroll
                for (int r0 = 0; r0 < EPL; r0 += 4) {
                    uint32_t word[3] = {0u, 0u, 0u};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int Q = __float2int_rn(a[r0 + e] * rs * inv_delta);
                        const int t2 = ((Q + 64) & 127) - 64, Q1 = (Q - t2) >> 7;
                        const int t1 = ((Q1 + 64) & 127) - 64, t0 = (Q1 - t1) >> 7;
                        word[0] |= (uint32_t)(t0 & 0xFF) << (8 * e);
                        word[1] |= (uint32_t)(t1 & 0xFF) << (8 * e);
                        word[2] |= (uint32_t)(t2 & 0xFF) << (8 * e);
                    }
                    const int i0 = lane * EPL + r0, st = i0 >> 5, k = i0 & 31;
                    const int L = 4 * hd + ((k & 15) >> 2);
                    if constexpr (SPLIT) {      // one fragment per step: rows hd, hd + 4, hd + 8, hd + 12
                        uint8_t* at = qt8 + (st * 32 + L) * 16 + (k >> 4) * 8;
                        *reinterpret_cast<uint2*>(at) = make_uint2(word[0], word[2]);
                        *reinterpret_cast<uint2*>(at + 256) = make_uint2(word[1], word[2]);
                        continue;
                    }
                    uint32_t* at = reinterpret_cast<uint32_t*>(qt8 + st * 768 + L * 16) + (k >> 4);
                    at[0] = word[0];
                    at[2] = word[1];
                    reinterpret_cast<uint32_t*>(qt8 + st * 768 + 512 + L * 8)[k >> 4] = word[2];
                }
            }
            if constexpr (FMT == 1) {       // rotated query, natural slot order: block i/16, slot s = i%16; per lane {hi b0, hi b1, lo b0, lo b1}
#pragma unroll
                for (int r = 0; r < EPL; r += 2) {
                    const int i = lane * EPL + r, kb = i >> 4, s = i & 15;
                    const int at = (kb * 32 + 4 * hd + ((s & 7) >> 1)) * (SPLIT ? 4 : 8) + (s >> 3) * 2;
                    // fp16 pair hi + lo carries the rotated query to ~2^-22
                    const float v0 = a[r] * rs, v1 = a[r + 1] * rs;
                    const __half2 vh = __floats2half2_rn(v0, v1);
                    *reinterpret_cast<__half2*>(qt + at) = vh;
                    *reinterpret_cast<__half2*>(qt + at + (SPLIT ? 64 : 4)) =           // SPLIT: column hd + 4
                        __floats2half2_rn(v0 - __low2float(vh), v1 - __high2float(vh));
                }
            }
            // plain query in the slot order of the FP8 key loads: 16 consecutive dims per lane
#pragma unroll
            for (int r = 0; r < EPL; r += 4) {
                const int i = lane * EPL + r, j = i >> 6, t4 = (i & 63) >> 4, wv = (i & 15) >> 2;
                __half* at = qf + ((4 * j + wv) * 32 + 4 * hd + t4) * 4;
                const uint2 four = make_uint2(pack_f16x2(qx[k][r], qx[k][r + 1]), pack_f16x2(qx[k][r + 2], qx[k][r + 3]));
                *reinterpret_cast<uint2*>(at) = four;
                if constexpr (SPLIT) *reinterpret_cast<uint2*>(at + 64) = four;         // column hd + 4: the same scores
            }
        }
        __syncthreads();
        // score units of the Stale pages: record format 2 counts in digit units of this lane's head(s)
        const float* digit_unit = reinterpret_cast<const float*>(smem + G::OFF_QS);
        const float sc2k = FMT == 2 ? sc2 * digit_unit[SPLIT ? g & 3 : 2 * tq] : sc2;
        const float sc2k1 = FMT == 2 && !SPLIT ? sc2 * digit_unit[2 * tq + 1] : sc2;

        for (bool more = n_my > 0; more && !failed;) {
            // ---- Stale pages: scores of page i+1 are computed together with the output update of page i
            if (n3 > 0) {
                float s_cur[4], s_next[4];
                PFrag pf;
                int cur_page = 0, cur_lp = 0;             // physical id and logical index of the Stale page being scanned
                if constexpr (TILED) {
                    park_store();
                    cur_page = list3[0];
                    cur_lp = lpg3[0] >> 16;
                }
                wait_slot(0);
                if (failed) break;
                tq3_step<D, false, true, TILED, FMT, SPLIT>(acc, 0, s_cur, pf, ring, qt_lane, sc2k, sc2k1, lane, s_cur);
                // (twice in the code where that was faster: 64 ragged requests 542 -> 534 us; long pages and several layers, whose
                // loop is larger, lose by it: 634 -> 726 us)
                constexpr int UNROLL = SPLIT && !TILED && !FLAT ? 2 : 1;
#pragma unroll UNROLL
                for (int i = 0; i + 1 < n3; ++i) {
                    const uint32_t cur = (uint32_t)i % NSTAGE, nxt = (uint32_t)(i + 1) % NSTAGE;
                    if ((i & 1) && !wait_slot(nxt / 2)) break;       // the next page opens a slot pair
                    if constexpr (FMT == 2 && SPLIT) softmax_rescale_v2<NB, TILED>(acc, s_cur, lane);
                    else softmax_rescale<NB, TILED>(acc, s_cur);
                    if constexpr (TILED) {
                        const int pg_i = list3[i];
                        if (pg_i != cur_page || (FLAT && i > 0 && (lpg3[i] & kOpens))) {
                            fold(cur_page, false, cur_lp);
                            cur_page = pg_i;
                            cur_lp = lpg3[i] >> 16;
                        }
                    }
                    tq3_step<D, true, true, TILED, FMT, SPLIT>(acc, ring + cur * G::SLOT, s_cur, pf, ring + nxt * G::SLOT, qt_lane, sc2k, sc2k1, lane, s_next);
                    if constexpr (SCORED && !TILED) store_page_mass<NB, SPLIT>(acc, pf.ps0, pf.ps1, mass_row + lpg3[i], P.max_pages, GQ, lane);
#pragma unroll
                    for (int e = 0; e < 4; ++e) s_cur[e] = s_next[e];
                    __syncwarp();
                    if ((i & 1) && i + 2 * G::NP - 1 < n3) issue_tq3(i / 2 + G::NP);    // the pair of pages i - 1, i is free
                }
                if (!failed) {
                    if (n8 > 0) issue_fp8(0);
                    if constexpr (FMT == 2 && SPLIT) softmax_rescale_v2<NB, TILED>(acc, s_cur, lane);
                    else softmax_rescale<NB, TILED>(acc, s_cur);
                    if constexpr (TILED) {
                        const int pg_i = list3[n3 - 1];
                        if (pg_i != cur_page || (FLAT && n3 > 1 && (lpg3[n3 - 1] & kOpens))) {
                            fold(cur_page, false, cur_lp);
                            cur_page = pg_i;
                            cur_lp = lpg3[n3 - 1] >> 16;
                        }
                    }
                    tq3_step<D, true, false, TILED, FMT, SPLIT>(acc, ring + ((uint32_t)(n3 - 1) % NSTAGE) * G::SLOT, s_cur, pf, 0, qt_lane, sc2k, sc2k1, lane, s_next);
                    if constexpr (SCORED && !TILED) store_page_mass<NB, SPLIT>(acc, pf.ps0, pf.ps1, mass_row + lpg3[n3 - 1], P.max_pages, GQ, lane);
                    if constexpr (TILED) fold(cur_page, true, cur_lp);   // back to output units for the FP8 pages and the reduction
                }
                __syncwarp();
                if (!failed)
                    for (int i = 1; i < min(n8, G::NP); ++i) issue_fp8(i);
            }
            // ---- Recent/Anchor pages: two slots per page (keys, values)
            if (n8 > 0 && !failed) {
                for (int i = 0; i < n8; ++i) {
                    const uint32_t s = (first8 + (uint32_t)i) % G::NP;
                    if (!wait_slot(s)) break;
                    const int e = list8[i];
                    const int valid = (e >> 27) & 15;
                    fp8_page<D, SCORED, TILED, SPLIT>(acc, ring + s * G::PAIR, ring + s * G::PAIR + G::FP8_HALF, qf_lane, sc2 * P.k_scale, P.v_scale,
                                               valid ? valid : kPage, lane,
                                               SCORED ? mass_row + (TILED ? (lpg8[i] >> 16) : lpg8[i]) : nullptr, P.max_pages, GQ);
                    if constexpr (FMT == 2 && SPLIT) max_rows_from_columns<NB>(acc, lane);     // the page may have raised the maxima
                    __syncwarp();
                    if (i + G::NP < n8) issue_fp8(i + G::NP);
                }
            }
            more = done < n_my;
            if (more && !failed) {
                done += build_lists(done);
                start_round();
            }
        }
        const bool last_segment = sg.end == my_end && layer + 1 == layer_end;
        float (&oacc)[NB][4] = acc.o;
        float (&lacc)[2] = acc.l;
        float (&m_run)[2] = acc.m;

        // ---- combine the warps of the block (ring memory is idle now) ---------------------------
        if (failed && drain()) last_s[1] = 1;      // a copy never arrived at all: the block must not touch the ring
        __syncthreads();
        if (last_s[1]) return;                     // (the call has failed; its workspace needs mkv_workspace_init again)
        if (g == 0) {
            sm_m[warp * 8 + 2 * tq] = m_run[0];
            sm_m[warp * 8 + 2 * tq + 1] = m_run[1];
        }
        __syncthreads();
        float M0 = -CUDART_INF_F, M1 = -CUDART_INF_F;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            M0 = fmaxf(M0, sm_m[w * 8 + 2 * tq]);
            M1 = fmaxf(M1, sm_m[w * 8 + 2 * tq + 1]);
        }
        {
            const float f0 = m_run[0] == -CUDART_INF_F ? 0.f : fast_exp2(m_run[0] - M0);
            const float f1 = m_run[1] == -CUDART_INF_F ? 0.f : fast_exp2(m_run[1] - M1);
            float* mine = red + (size_t)warp * D * 8;
#pragma unroll
            for (int i = 0; i < NB; ++i) {
                // element (channel 16i + g + 8*(e>>1), head 2tq + (e&1)) at [channel][8 heads]
                *reinterpret_cast<float2*>(mine + (16 * i + g) * 8 + 2 * tq) = make_float2(oacc[i][0] * f0, oacc[i][1] * f1);
                *reinterpret_cast<float2*>(mine + (16 * i + g + 8) * 8 + 2 * tq) = make_float2(oacc[i][2] * f0, oacc[i][3] * f1);
            }
            if (g == 0) {
                sm_l[warp * 8 + 2 * tq] = lacc[0] * f0;
                sm_l[warp * 8 + 2 * tq + 1] = lacc[1] * f1;
            }
        }
        __syncthreads();

        const bool whole_row = n_seg == n_pages;
        // sum of the warps for one channel (item e4 / 2) and four heads (first: 4 (e4 % 2)); SPLIT: columns 4 - 7 are the low
        // halves of heads 0 - 3
        auto sum_of_warps = [&](int e4) -> float4 {
            float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                const float4* row = reinterpret_cast<const float4*>(red + (size_t)w * D * 8);
                const float4 hi = row[e4];
                s.x += hi.x; s.y += hi.y; s.z += hi.z; s.w += hi.w;
                if constexpr (SPLIT) {
                    const float4 lo = row[e4 + 1];
                    s.x += lo.x; s.y += lo.y; s.z += lo.z; s.w += lo.w;
                }
            }
            return s;
        };
        constexpr int ITEMS = SPLIT ? D : 2 * D, PER_THREAD = (ITEMS + NW * 32 - 1) / (NW * 32);
        if (whole_row) {
#pragma unroll
            for (int k = 0; k < PER_THREAD; ++k) {
                const int i = tid + k * NW * 32, e4 = SPLIT ? 2 * i : i, ch = e4 >> 1;
                if (i >= ITEMS) break;
                const float4 s = sum_of_warps(e4);
                const float v[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int head = 4 * (e4 & 1) + e;
                    if (head >= GQ) continue;
                    float l = 0.f;
#pragma unroll
                    for (int w = 0; w < NW; ++w) {
                        l += sm_l[w * 8 + head];
                        if constexpr (SPLIT) l += sm_l[w * 8 + head + 4];
                    }
                    P.out[((size_t)b * hq + h * GQ + head) * D + ch] = l > 0.f ? v[e] / l : 0.f;
                }
            }
            if (P.lse && tid < GQ) {
                float l = 0.f, M = -CUDART_INF_F;
                for (int w = 0; w < NW; ++w) {
                    l += sm_l[w * 8 + tid];
                    if constexpr (SPLIT) l += sm_l[w * 8 + tid + 4];
                    M = fmaxf(M, sm_m[w * 8 + tid]);
                }
                P.lse[(size_t)b * hq + h * GQ + tid] = l > 0.f ? (M + log2f(l)) * kLn2 : -CUDART_INF_F;
            }
        } else {
            // partial (m, l, O) of this block for the row
            float* slot = P.partials + (size_t)partial_slot(blockIdx.x, pos, my_start) * (8 * D + 16);
#pragma unroll
            for (int k = 0; k < PER_THREAD; ++k) {
                const int i = tid + k * NW * 32, e4 = SPLIT ? 2 * i : i;
                if (i >= ITEMS) break;
                reinterpret_cast<float4*>(slot)[e4] = sum_of_warps(e4);
                if constexpr (SPLIT) reinterpret_cast<float4*>(slot)[e4 + 1] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
            if (tid < 8) {
                float l = 0.f, M = -CUDART_INF_F;
                for (int w = 0; w < NW; ++w) {
                    l += sm_l[w * 8 + tid];
                    if constexpr (SPLIT) l += tid < 4 ? sm_l[w * 8 + tid + 4] : 0.f;
                    M = fmaxf(M, sm_m[w * 8 + tid]);
                }
                slot[8 * D + tid] = M;
                slot[8 * D + 8 + tid] = l;
            }
            // Ticket of the row (all threads' stores, block barrier, releasing ticket on the writers' side; acquiring ticket, block
            // barrier, loads on the merger's).  Who merges?  In the last layer of the launch the block that draws the row's last
            // ticket.  In an earlier layer the row is left to the block that is FIRST to finish the same row in
            // the next layer -- the one that is ahead of the others, so that the merges do not keep falling on
            // the block that is already late.  That block finds the row complete and merges it, or it leaves a
            // request (the counter's top bit) and the row's last arrival, seeing the request, merges after all.
            // Either way exactly one block merges, and it leaves the counter at zero for the next call.
            int c0, c1;                                // (flat cut: the row's last arrival merges, no block is ahead of the others)
            blocks_of_row<FLAT>(pt, cum[P0.B], layer, b * hkv + h, sg.row_start + ROW_COST, sg.row_end, c0, c1);
            const int n_parts = c1 - c0 + 1;
            constexpr uint32_t kRequest = 0x80000000u;
            __syncthreads();
            if (tid == 0) {
                const uint32_t prev = ticket_add(P.tickets + c0, 1u);
                int todo = 0;                          // 1: merge this layer's row, 2: merge the row of the layer before
                if ((prev & ~kRequest) == (uint32_t)(n_parts - 1) && (FLAT || layer == n_layers - 1 || (prev & kRequest))) todo |= 1;
                if (MAXL > 1 && !FLAT && layer > 0 && (prev & ~kRequest) == 0u) {
                    const uint32_t old = ticket_or(LS.layer[layer - 1].tickets + c0, kRequest);
                    if (old == (uint32_t)n_parts) todo |= 2;
                }
                *last_s = todo;
            }
            __syncthreads();
            const int todo = *last_s;
            if (last_segment) pdl_let_next_start();    // what is left of the block is at most a merge
            if (todo) {
                const int first_slot = first_partial_slot<FLAT>(pt, cum[P0.B], layer, c0, sg.row_start);
                if constexpr (MAXL > 1 && !FLAT) {
                    if (todo & 2) {
                        const DecodeParams& Q = LS.layer[layer - 1];
                        merge_row<D, NW * 32, MERGE_LOADS>(Q, first_slot, 2 * c0, n_parts, red, b, h);
                        if (tid == 0) Q.tickets[c0] = 0;
                    }
                }
                if (todo & 1) {
                    merge_row<D, NW * 32, MERGE_LOADS>(P, first_slot, 2 * c0, n_parts, red, b, h);
                    if (tid == 0) P.tickets[c0] = 0;
                }
            }
        }
        __syncthreads();
        pos = sg.end;
    }
    }   // layers
}

#include "decode_tmem.cuh"

// Per-device launch state of one kernel instantiation (dynamic shared memory opt-in, persistent grid size).
constexpr int kMaxDevices = 64;
struct LaunchCache {
    std::mutex mu;
    int grid[kMaxDevices] = {};
};

template <int D>
static int32_t run_tmem(mkv_pool* p, DecodeParams& prm, cudaStream_t s)
{
    using G = tm::TG<D>;
    auto kern = decode_tmem_kernel<D>;
    static LaunchCache cache;
    const int dev = p->device;
    if (dev < 0 || dev >= kMaxDevices) {
        set_last_error("decode attention: device index beyond the 64 this library keeps launch state for");
        return MKV_E_INVALID;
    }
    int grid;
    {
        std::lock_guard<std::mutex> lk(cache.mu);
        if (cache.grid[dev] == 0) {
            MKV_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, G::SMEM));
            cache.grid[dev] = p->dev.sm_count > kMaxCtas ? kMaxCtas : p->dev.sm_count;   // one block per SM: it takes all the tensor memory
        }
        grid = cache.grid[dev];
    }
    if (grid > prm.max_blocks) {
        set_last_error("decode attention: the scan launches more blocks on this GPU than the partial area has slots for");
        return MKV_E_INVALID;
    }
    kern<<<grid, tm::kThreads, G::SMEM, s>>>(prm);
    MKV_CUDA(cudaGetLastError());
    return MKV_OK;
}

template <int D, int NW, int NSTAGE, int MINB, bool SCORED, bool TILED, int MAXL, int FMT, bool FLAT, bool SPLIT>
static int32_t run_tensor_fmt(mkv_pool* p, const LayerSet<MAXL>& ls, cudaStream_t s)
{
    using G = Geo<D, NW, NSTAGE, TILED>;
    auto kern = decode_tensor_kernel<D, NW, NSTAGE, MINB, SCORED, TILED, MAXL, FMT, FLAT, SPLIT>;
    // pages of several tiles: one row of parked accumulators (8 D floats) per warp behind the usual layout
    constexpr int SMEM = G::SMEM + (TILED ? NW * 8 * D * 4 : 0);
    static_assert(SMEM <= 232448, "dynamic shared memory of one block");
    static LaunchCache cache;
    const int dev = p->device;
    if (dev < 0 || dev >= kMaxDevices) {
        set_last_error("decode attention: device index beyond the 64 this library keeps launch state for");
        return MKV_E_INVALID;
    }
    int grid;
    {
        std::lock_guard<std::mutex> lk(cache.mu);
        if (cache.grid[dev] == 0) {
            MKV_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM));
            int per_sm = 0;
            MKV_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NW * 32, SMEM));
            if (per_sm < 1) return MKV_E_INVALID;
            const int g = p->dev.sm_count * per_sm;
            cache.grid[dev] = g > kMaxCtas ? kMaxCtas : g;
        }
        grid = cache.grid[dev];
    }
    if (grid > ls.layer[0].max_blocks) {
        set_last_error("decode attention: the scan launches more blocks on this GPU than the partial area has slots for");
        return MKV_E_INVALID;
    }
    MKV_CUDA(launch_pdl(kern, dim3((unsigned)grid), NW * 32, SMEM, 1, s, ls));
    return MKV_OK;
}

// The pool's record format selects the instantiation, and for 16-token pages its group: groups of at most four query
// heads use two column halves (see PFrag).  Not for long pages: their code sums stay in the tensor core's accumulators
// over many tiles, and the split changes their rounding there.  GROUPS: which groups the caller sends here.
enum Groups { kAnyGroup, kMoreThanFour };
template <int D, int NW, int NSTAGE, int MINB, bool SCORED = false, bool TILED = false, int MAXL = 1, bool FLAT = false, Groups GROUPS = kAnyGroup>
static int32_t run_tensor(mkv_pool* p, const LayerSet<MAXL>& ls, cudaStream_t s)
{
    if constexpr (!TILED && GROUPS != kMoreThanFour)
        if (p->group <= 4)
            return p->fmt == 2 ? run_tensor_fmt<D, NW, NSTAGE, MINB, SCORED, TILED, MAXL, 2, FLAT, true>(p, ls, s)
                               : run_tensor_fmt<D, NW, NSTAGE, MINB, SCORED, TILED, MAXL, 1, FLAT, true>(p, ls, s);
    return p->fmt == 2 ? run_tensor_fmt<D, NW, NSTAGE, MINB, SCORED, TILED, MAXL, 2, FLAT, false>(p, ls, s)
                       : run_tensor_fmt<D, NW, NSTAGE, MINB, SCORED, TILED, MAXL, 1, FLAT, false>(p, ls, s);
}

template <int D, int NW, int NSTAGE, int MINB, bool SCORED = false, bool TILED = false>
static int32_t run_tensor1(mkv_pool* p, const DecodeParams& prm, cudaStream_t s)
{
    LayerSet<1> ls;
    ls.n = 1;
    ls.layer[0] = prm;
    return run_tensor<D, NW, NSTAGE, MINB, SCORED, TILED, 1>(p, ls, s);
}

int32_t launch_decode_tensor(mkv_pool* p, const void* q, const int32_t* bt, const uint8_t* tags,
                             const int32_t* lens, int B, int max_pages, float scale, float* out, float* lse,
                             void* ws, size_t, cudaStream_t s)
{
    // header: 256 reserved bytes, then kMaxCtas ticket words (cleared by mkv_workspace_init, left clear by every call)
    uint32_t* tickets = reinterpret_cast<uint32_t*>(static_cast<uint8_t*>(ws) + 256);
    float* partials = reinterpret_cast<float*>(static_cast<uint8_t*>(ws) + decode_ws_header_bytes(B, p->hkv));
    return launch_decode_tensor_at(p, q, bt, tags, lens, B, max_pages, scale, out, lse, partials, tickets, kMaxCtas,
                                   nullptr, s);
}

int decode_tensor_partial_floats(int d) { return 8 * d + 16; }

// Second step of the scored variant: mass[b][hq][p] holds log2 of page p's exponential sum on an
// absolute origin; with the row's log-sum-exp it becomes q_p = 2^(that - lse2), and q~_p = q_p / sum q_p
// (Eq. score-global-weight and the normalisation over page-addressable mass that follows it).
// One block per (query head, request); entries beyond the request's pages are set to zero.  The first 4,096 pages of a row
// are loaded at once and stay in registers between the two steps; what is beyond is read twice.  (Bound by the trips to
// memory: with one load at a time and a second reading, the score update behind it likewise, a scored step over four rows
// of 2,501 pages x 24 heads took 69.6 us, so 65.)
__global__ void __launch_bounds__(512) page_mass_finish_kernel(float* mass, const float* lse, const int32_t* lens,
                                                              int hq, int max_pages, int page_tokens)
{
    constexpr int NT = 512, KEEP = 8;
    __shared__ float red[NT / 32];
    pdl_begin();
    const int b = blockIdx.y, h = blockIdx.x, tid = threadIdx.x;
    const int len = lens[b], n_pages = len > 0 ? min((len + page_tokens - 1) / page_tokens, max_pages) : 0;
    float* row = mass + ((size_t)b * hq + h) * max_pages;
    const float lse2 = n_pages > 0 ? lse[(size_t)b * hq + h] * kLog2e : 0.f;
    float kept[KEEP], sum = 0.f;
#pragma unroll
    for (int k = 0; k < KEEP; ++k) kept[k] = tid + k * NT < n_pages ? row[tid + k * NT] : -CUDART_INF_F;
#pragma unroll
    for (int k = 0; k < KEEP; ++k) {
        kept[k] = tid + k * NT < n_pages ? fast_exp2(kept[k] - lse2) : 0.f;
        sum += kept[k];
    }
    for (int p = tid + KEEP * NT; p < n_pages; p += NT) {
        const float qv = fast_exp2(row[p] - lse2);
        row[p] = qv;
        sum += qv;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if ((tid & 31) == 0) red[tid >> 5] = sum;
    __syncthreads();
    float total = 0.f;
#pragma unroll
    for (int w = 0; w < NT / 32; ++w) total += red[w];
    const float inv = total > 0.f ? 1.f / total : 0.f;
#pragma unroll
    for (int k = 0; k < KEEP; ++k)
        if (tid + k * NT < max_pages) row[tid + k * NT] = kept[k] * inv;
    for (int p = tid + KEEP * NT; p < max_pages; p += NT) row[p] = p < n_pages ? row[p] * inv : 0.f;
}

// Eq. (attention-score): r_p = mean over the sampled heads of q~_{h,p}; a_p <- beta a_p + (1 - beta) r_p.
__global__ void __launch_bounds__(256) page_score_kernel(const float* mass, const int32_t* lens, int hq, int max_pages,
                                                         unsigned long long head_mask, float beta, float inv_heads,
                                                         float* score, int page_tokens)
{
    pdl_begin();
    const int b = blockIdx.y, p = blockIdx.x * 256 + threadIdx.x;
    const int len = lens[b], n_pages = len > 0 ? min((len + page_tokens - 1) / page_tokens, max_pages) : 0;
    if (p >= n_pages) return;
    float r = 0.f;
#pragma unroll 16
    for (int h = 0; h < hq; ++h)            // many loads in flight
        r += (head_mask >> h) & 1ull ? mass[((size_t)b * hq + h) * max_pages + p] : 0.f;
    float* a = score + (size_t)b * max_pages + p;
    *a = beta * *a + (1.f - beta) * (r * inv_heads);
}

// pages of several tiles: the scan adds parts of a page's sum to its entry, which therefore starts at -inf
__global__ void page_mass_clear_kernel(float* mass, size_t n)
{
    pdl_begin();
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) mass[i] = -CUDART_INF_F;
}

int32_t launch_page_mass_finish(float* mass, const float* lse, const int32_t* lens, int B, int hq, int max_pages,
                                int page_tokens, cudaStream_t s)
{
    MKV_CUDA(launch_pdl(page_mass_finish_kernel, dim3(hq, B), 512, 0, 1, s, mass, lse, lens, hq, max_pages, page_tokens));
    return MKV_OK;
}

int32_t launch_page_score(const float* mass, const int32_t* lens, int B, int hq, int max_pages, uint64_t head_mask,
                          float beta, float* score, int page_tokens, cudaStream_t s)
{
    int n = 0;
    for (int h = 0; h < hq; ++h) n += (int)((head_mask >> h) & 1ull);
    if (n == 0) return MKV_E_INVALID;
    MKV_CUDA(launch_pdl(page_score_kernel, dim3((max_pages + 255) / 256, B), 256, 0, 1, s, mass, lens, hq, max_pages,
                        (unsigned long long)head_mask, beta, 1.f / (float)n, score, page_tokens));
    return MKV_OK;
}

static DecodeParams make_params(mkv_pool* p, const void* q, const int32_t* bt, const uint8_t* tags, const int32_t* lens,
                                int B, int max_pages, float scale, float* out, float* lse, float* partials,
                                uint32_t* tickets, int max_blocks, float* mass)
{
    DecodeParams prm;
    prm.tiles = p->tiles;
    prm.fp8 = p->fp8; prm.tq3 = p->tq3;
    prm.fp8_pages = p->cfg.fp8_pages; prm.tq3_pages = p->cfg.tq3_pages;
    prm.hkv = p->hkv; prm.group = p->group;
    prm.k_scale = p->cfg.k_scale; prm.v_scale = p->cfg.v_scale;
    prm.sigma = p->sigma;
    prm.q = static_cast<const __nv_bfloat16*>(q);
    prm.bt = bt; prm.tags = tags; prm.lens = lens;
    prm.B = B; prm.max_pages = max_pages; prm.scale = scale;
    prm.out = out; prm.lse = lse;
    prm.partials = partials;
    prm.tickets = tickets;
    prm.max_blocks = max_blocks;
    prm.mass = mass;
    prm.status = p->status_dev;
    prm.wait_ns = p->wait_ns;
    return prm;
}

// Two blocks of half the warps per SM instead of one: the set-up, reduction and merge of one overlap the pages of the
// other, which pays the more rows a block meets (d 128, 8 x 4 heads: 64 ragged requests 632 -> 579 us, 8 x 4,096 tokens
// 30.7 -> 23.6 us).  At d = 256 a merge by four warps costs more, and few rows have many partials: from 32 rows (8 x
// 32,768 tokens, 4 heads: 78 -> 70 us; 16 rows of 8,000 and 30,000: 20.9 -> 24.4, 47.6 -> 49.4).  Partial areas for one
// block per SM only take one.
static bool two_blocks(const mkv_pool* p, int B, int max_blocks)
{
    return max_blocks >= 2 * p->dev.sm_count && (p->d == 128 || B * p->hkv >= 32);
}

constexpr int kRowsOfTwoBlocks = 64;     // several layers laid end to end

// Decode attention of several layers in one launch: layer i reads pool[i], q[i], bt[i], tags[i] and writes
// out[i], lse[i] (or none), with its own workspace ws[i]; the requests (lens, B, max_pages, scale) are common.
int32_t launch_decode_tensor_layers(mkv_pool* const* pools, const void* const* q, const int32_t* const* bt,
                                    const uint8_t* const* tags, const int32_t* lens, int B, int max_pages, float scale,
                                    float* const* out, float* const* lse, void* const* ws, int n_layers, cudaStream_t s)
{
    mkv_pool* p0 = pools[0];
    if (B > kMaxBatch || n_layers > kMaxLayers) return MKV_E_INVALID;
    if ((int64_t)max_pages * p0->tiles > 65535) {
        set_last_error("mkv_decode_attention_layers: more than 65535 16-token tiles per table row (1,048,560 tokens per request)");
        return MKV_E_INVALID;
    }
    // more positions than a launch counts: one launch after the other, on the same workspaces
    if (const int most = requests_per_launch(p0->hkv, max_pages * p0->tiles); B > most) {
        for (int b0 = 0; b0 < B; b0 += most) {
            const size_t row = (size_t)b0 * max_pages, head = (size_t)b0 * p0->hkv * p0->group, vec = head * p0->d;
            const void* qs[kMaxLayers];
            const int32_t* bts[kMaxLayers];
            const uint8_t* tagss[kMaxLayers];
            float *outs[kMaxLayers], *lses[kMaxLayers];
            for (int i = 0; i < n_layers; ++i) {
                qs[i] = static_cast<const __nv_bfloat16*>(q[i]) + vec;
                bts[i] = bt[i] + row;
                tagss[i] = tags[i] + row;
                outs[i] = out[i] + vec;
                lses[i] = lse && lse[i] ? lse[i] + head : nullptr;
            }
            const int32_t rc = launch_decode_tensor_layers(pools, qs, bts, tagss, lens + b0, B - b0 < most ? B - b0 : most, max_pages,
                                                           scale, outs, lse ? lses : nullptr, ws, n_layers, s);
            if (rc != MKV_OK) return rc;
        }
        return MKV_OK;
    }
    LayerSet<kMaxLayers> ls;
    ls.n = n_layers;
    for (int i = 0; i < n_layers; ++i) {
        uint32_t* tickets = reinterpret_cast<uint32_t*>(static_cast<uint8_t*>(ws[i]) + 256);
        float* partials = reinterpret_cast<float*>(static_cast<uint8_t*>(ws[i]) + decode_ws_header_bytes(B, p0->hkv));
        ls.layer[i] = make_params(pools[i], q[i], bt[i], tags[i], lens, B, max_pages, scale, out[i], lse ? lse[i] : nullptr,
                                  partials, tickets, kMaxCtas, nullptr);
    }
    if (p0->tiles > 1 && n_layers >= kMinFlatLayers)   // pages of several tiles (all pools of the call have the same page size)
        return p0->d == 128 ? run_tensor<128, 12, 4, 1, false, true, kMaxLayers, true>(p0, ls, s)
                            : run_tensor<256, 8, 4, 1, false, true, kMaxLayers, true>(p0, ls, s);
    if (p0->tiles > 1)
        return p0->d == 128 ? run_tensor<128, 12, 4, 1, false, true, kMaxLayers>(p0, ls, s)
                            : run_tensor<256, 8, 4, 1, false, true, kMaxLayers>(p0, ls, s);
    // Two blocks of half the warps per SM from 64 rows on: one's set-up, reduction and merge overlap the other's pages, but
    // few rows have partials that four warps take longer to merge.  us with one block and with two (layers x requests x
    // tokens): d 256, 16 x 2 x 59,008 540 / 510, 4 x 4 x 20,000 (64 rows) 109.0 / 102.7, 16 x 1 x 30,000 (64) 155 / 143.5,
    // 16 x 1 x 4,000 (64) both 33.6, 4 x 1 x 3,000 (16) 17.7 / 21.2; d 128, eight query heads, 16 x 8 x 512..16,384 (512)
    // 132 / 127.6, 16 x 2 x 2,000 (128) 24.5 / 23.3, 4 x 2 x 8,000 (8) 15.1 / 17.1.  Up to four query heads at d = 128 two
    // blocks are better at any size.  (Long pages: 16 x 1 x 4,000 45.8 / 43.0, but 16 x 2 x 59,008 552 / 592: two blocks
    // leave room for rounds of 32 tiles only.)
    if (n_layers >= kMinFlatLayers) {
        const bool two = n_layers * B * p0->hkv >= kRowsOfTwoBlocks;
        if (p0->d == 256)
            return two ? run_tensor<256, 4, 4, 2, false, false, kMaxLayers, true>(p0, ls, s)
                       : run_tensor<256, 8, 4, 1, false, false, kMaxLayers, true>(p0, ls, s);
        if (two || p0->group <= 4) return run_tensor<128, 8, 4, 2, false, false, kMaxLayers, true>(p0, ls, s);
        return run_tensor<128, 16, 4, 1, false, false, kMaxLayers, true, kMoreThanFour>(p0, ls, s);
    }
    // as a call of one layer (the results are the same bits); a workspace has room for two blocks per SM
    if (p0->d == 128) return run_tensor<128, 8, 4, 2, false, false, kMaxLayers>(p0, ls, s);
    return two_blocks(p0, B, kMaxCtas) ? run_tensor<256, 4, 4, 2, false, false, kMaxLayers>(p0, ls, s)
                                       : run_tensor<256, 8, 4, 1, false, false, kMaxLayers>(p0, ls, s);
}

int32_t launch_decode_tensor_at(mkv_pool* p, const void* q, const int32_t* bt, const uint8_t* tags,
                                const int32_t* lens, int B, int max_pages, float scale, float* out, float* lse,
                                float* partials, uint32_t* tickets, int max_blocks, float* mass, cudaStream_t s)
{
    if (B > kMaxBatch) return MKV_E_INVALID;
    if ((int64_t)max_pages * p->tiles > 65535) {   // tile counts: small_div takes up to 2^20, the lists of long pages 16 bits
        set_last_error("mkv_decode_attention: more than 65535 16-token tiles per table row (1,048,560 tokens per request)");
        return MKV_E_INVALID;
    }
    if (p->tiles > 1 && p->variant == MKV_DECODE_TMEM) {
        set_last_error("mkv_decode_attention: pages of several tiles are served by the tensor-core kernel");
        return MKV_E_INVALID;
    }
    if (p->fmt == 2 && p->variant == MKV_DECODE_TMEM) {
        set_last_error("mkv_decode_attention: record format 2 is served by the tensor-core and the CUDA-core kernels");
        return MKV_E_INVALID;
    }
    // more positions than a launch counts: one launch after the other, on the same workspace
    if (const int most = requests_per_launch(p->hkv, max_pages * p->tiles); B > most) {
        for (int b0 = 0; b0 < B; b0 += most) {
            const size_t row = (size_t)b0 * max_pages, head = (size_t)b0 * p->hkv * p->group, vec = head * p->d;
            const int32_t rc = launch_decode_tensor_at(p, static_cast<const __nv_bfloat16*>(q) + vec, bt + row, tags + row, lens + b0,
                                                       B - b0 < most ? B - b0 : most, max_pages, scale, out + vec, lse ? lse + head : nullptr,
                                                       partials, tickets, max_blocks, mass ? mass + head * max_pages : nullptr, s);
            if (rc != MKV_OK) return rc;
        }
        return MKV_OK;
    }
    DecodeParams prm = make_params(p, q, bt, tags, lens, B, max_pages, scale, out, lse, partials, tickets, max_blocks, mass);
    if (mass) {                          // scored variant: the default launch shapes only
        int32_t rc;
        if (p->tiles > 1) {
            const size_t n = (size_t)B * p->hkv * p->group * max_pages;
            MKV_CUDA(launch_pdl(page_mass_clear_kernel, dim3((unsigned)((n + 255) / 256)), 256, 0, 1, s, mass, n));
            rc = p->d == 128 ? run_tensor1<128, 12, 4, 1, true, true>(p, prm, s) : run_tensor1<256, 8, 4, 1, true, true>(p, prm, s);
        } else {
            // (always with a caller's workspace, which has room for two blocks per SM)
            if (p->d == 128) rc = run_tensor1<128, 8, 4, 2, true>(p, prm, s);
            else rc = two_blocks(p, B, max_blocks) ? run_tensor1<256, 4, 4, 2, true>(p, prm, s) : run_tensor1<256, 8, 4, 1, true>(p, prm, s);
        }
        if (rc != MKV_OK) return rc;
        return launch_page_mass_finish(mass, lse, lens, B, p->hkv * p->group, max_pages, p->cfg.page_size, s);
    }
    if (p->tiles > 1)                    // pages of several tiles: the default launch shapes only
        return p->d == 128 ? run_tensor1<128, 12, 4, 1, false, true>(p, prm, s) : run_tensor1<256, 8, 4, 1, false, true>(p, prm, s);
    if (p->variant == MKV_DECODE_TMEM && p->d == 256) return run_tmem<256>(p, prm, s);
    // launch shapes: warps per block, ring slots per warp, blocks per SM
    if (two_blocks(p, B, max_blocks))
        return p->d == 128 ? run_tensor1<128, 8, 4, 2>(p, prm, s) : run_tensor1<256, 4, 4, 2>(p, prm, s);
    return p->d == 128 ? run_tensor1<128, 16, 4, 1>(p, prm, s) : run_tensor1<256, 8, 4, 1>(p, prm, s);
}

}  // namespace mkv
