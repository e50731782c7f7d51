// Cut of the decode scan's work into one contiguous range per block: which pages a block scans, which blocks hold a part
// of a row, and where their partials lie.  The scan kernels run it on the device; it also compiles for the host, where a
// warp is one lane, so that every block of a grid can be walked without a GPU.
#pragma once
#include "mkv_internal.cuh"

namespace mkv {

// Work = (request, KV head, page) triples in row-major order; cum[b] = position of the first triple of
// request b.  A row of n pages takes row_cost + n positions: opening, reducing and storing a row (or a block's part of it)
// costs a block as much time as row_cost pages, so that a block with many short rows gets fewer pages.  (us a step with
// cost 0 and with row_cost: 64 requests of 1,024 to 131,072 tokens, 8 heads 524 / 480, as with 48, 503 with 16; 16 layers x
// 4 x 700..3,001 tokens, d 256 64.0 / 60 with 16, 62 with 32, 66 with 48; 16 layers x 8 x 512..16,384, one block of 16
// warps per SM 151 / 134 with 48, 139 with 32, 136 with 64.)  A block whose range lies inside a row's cost gets no page.
// Where rows are few and short that is no loss: they are split over fewer blocks, whose partials take longer to merge than
// the pages to scan.  (With the cost bounded so that every block gets pages: 4 layers x 1 x 700, d 256 13.5 -> 16.9 us;
// 8 x 400, d 256 15.3 -> 17.6, d 128 13.8 -> 17.1; 16 layers x 1 x 500, d 128 9.9 -> 12.7; 16 x 64..8,000 25.0 -> 25.8.)
//
// Two ways to cut a layer into one contiguous range per block:
//   row-aligned (few rows: B * hkv <= grid / 4): every row gets a whole number of blocks in proportion
//     to its positions (cumulative rounding), so that no block straddles two rows and pays the per-row set-up
//     and reduction twice;
//   linear (many rows): grid equal ranges that may cross row boundaries.
constexpr int kMaxAlignedRows = kMaxCtas / 4;
constexpr int kMaxBatch = 1024;         // requests per call

// and one for several layers: flat, a linear cut of all layers' triples, the layers laid end to end.
//
// Every block works this out for itself before its first page can be asked for, so the arithmetic is kept short: one
// 32-bit division per cut (quotient and remainder; block c starts at quo c + min(c, rem)), and warp 0 leaves the block's
// own range and request in shared memory.  (Time up to a block's first page with 64-bit divisions and serial searches, and
// so: 8 x 16,384 tokens, d 128 11,600 / 8,400 cycles; flat cut of 16 layers x 16 rows, d 256 18,900 / 10,100.)
struct Cut {
    long long quo;
    int rem, blocks;                    // blocks that get work (0: none)
};

struct Partition {
    Cut flat;                           // flat: all layers' triples
    Cut cut;                            // linear cut of one layer
    int aligned;                        // 1: row-aligned, 0: linear
    int start, end;                     // this block's range in the per-layer cut
    int first_layer, end_layer;         // this block's layers in the flat cut
    int first_b;                        // request of the block's first triple
    int base[kMaxAlignedRows + 1];      // row-aligned: first block of every row
};

// ---- lanes of the warp that works the cut out (on the host: one) --------------------------------
#define MKV_CUT __host__ __device__ __forceinline__
#ifdef __CUDA_ARCH__
#define MKV_CUT_WARP(on_device, on_host) on_device
constexpr int kCutLanes = 32;
#else
#define MKV_CUT_WARP(on_device, on_host) on_host
constexpr int kCutLanes = 1;
#endif
MKV_CUT float near_quotient(float a, float b) { return MKV_CUT_WARP(__fdividef(a, b), a / b); }
MKV_CUT bool any_lane(bool x) { return MKV_CUT_WARP(__any_sync(0xffffffffu, x), x); }
MKV_CUT int count_lanes(bool x) { return MKV_CUT_WARP(__popc(__ballot_sync(0xffffffffu, x)), x); }
MKV_CUT void sync_lanes() { MKV_CUT_WARP(__syncwarp(), (void)0); }
MKV_CUT int of_last_lane(int x) { return MKV_CUT_WARP(__shfl_sync(0xffffffffu, x, 31), x); }
MKV_CUT int of_lane_below(int x, int by) { return MKV_CUT_WARP(__shfl_up_sync(0xffffffffu, x, by), ((void)by, x)); }
MKV_CUT int reversed_low_5_bits(int x)
{
    return MKV_CUT_WARP((int)(__brev((unsigned)x) >> 27), (x & 1) << 4 | (x & 2) << 2 | (x & 4) | (x & 8) >> 2 | (x & 16) >> 4);
}
MKV_CUT int smaller(int a, int b) { return a < b ? a : b; }
MKV_CUT int larger(int a, int b) { return a > b ? a : b; }

// a / b for 0 <= a < 2^20: (a + 1/2) / b is at least 1 / (2 b) away from the next integer, the approximate quotient less far off
MKV_CUT int small_div(int a, int b) { return (int)near_quotient((float)a + 0.5f, (float)b); }

// What a launch shape of `warps` warps and `per_sm` blocks per SM fixes.  A row costs more pages where more warps scan them in that
// time; long pages come in few rows.
MKV_CUT constexpr int cut_row_cost(int warps, bool long_pages) { return long_pages ? 0 : 8 + 3 * warps; }
MKV_CUT constexpr int cut_min_pages(int warps, int per_sm) { return warps * per_sm; }
MKV_CUT constexpr int cut_straddle(int warps) { return 4 * warps; }

// Positions are counted in 32 bits: requests that one launch may take where a table row has room for `tiles` 16-token
// tiles, so that its positions stay below 2^31.  (A single request reaches that only with more than 32,700 KV heads.)
inline int requests_per_launch(int hkv, int tiles)
{
    constexpr long long kLargestCost = cut_row_cost(16, false);
    const long long most = 0x7FFFFFFFll / (hkv * (tiles + kLargestCost));
    return most > 1 ? (int)(most < kMaxBatch ? most : kMaxBatch) : 1;
}

// Pages (16-token tiles) of a request of len tokens
MKV_CUT int pages_of(int len) { return (len + kPage - 1) / kPage; }

// Positions of a request's rows
MKV_CUT int positions_of(int len, int hkv, int row_cost) { return len > 0 ? (pages_of(len) + row_cost) * hkv : 0; }

// Running sums over the requests, kCutLanes at a time: request b0 + lane has n positions; all lanes get the same sums.
struct RowSums {
    int positions, requests;            // positions so far, requests with pages so far
};
MKV_CUT void add_requests(RowSums& sum, int* cum, int B, int b0, int n, int lane)
{
    sum.requests += count_lanes(n > 0);
    int inc = n;                                            // over the lanes up to this one
#pragma unroll
    for (int o = 1; o < kCutLanes; o <<= 1) {
        const int v = of_lane_below(inc, o);
        if (lane >= o) inc += v;
    }
    if (b0 + lane < B) cum[b0 + lane] = sum.positions + inc - n;
    sum.positions += of_last_lane(inc);
}

// Blocks that share W positions, `pages` of them pages: all of the grid, but no more than give every block min_pages pages (a page
// per warp of an SM: below that a row's partials cost more to merge than the spreading saves).
MKV_CUT Cut make_cut(long long W, long long pages, int grid, int min_pages)
{
    Cut c;
    if (W >> 31 == 0) {
        const unsigned w = (unsigned)W, most = ((unsigned)pages + min_pages - 1) / (unsigned)min_pages;
        c.blocks = (int)(most < (unsigned)grid ? most : (unsigned)grid);
        const unsigned q = c.blocks ? w / (unsigned)c.blocks : 0u;
        c.quo = q;
        c.rem = (int)(w - q * (unsigned)c.blocks);
    } else {
        c.blocks = grid;
        c.quo = W / grid;
        c.rem = (int)(W - c.quo * grid);
    }
    return c;
}

MKV_CUT long long cut_start(const Cut& c, int block) { return c.quo * block + smaller(block, c.rem); }

// the block that holds triple x
MKV_CUT int cut_block_of(const Cut& c, long long x)
{
    const long long split = (c.quo + 1) * c.rem;          // the first `rem` blocks have one more; quo >= 1 where a triple exists
    int b = x < split ? (int)near_quotient((float)x, (float)(c.quo + 1)) : c.rem + (int)near_quotient((float)(x - split), (float)c.quo);
    b = smaller(b, c.blocks - 1);                         // near, then exact
    while (b + 1 < c.blocks && cut_start(c, b + 1) <= x) ++b;
    while (b > 0 && cut_start(c, b) > x) --b;
    return b;
}

// a row of n pages (at most 65,535) over k whole blocks
MKV_CUT Cut cut_row(int n, int k)
{
    Cut c;
    c.blocks = k;
    const int q = small_div(n, k);
    c.quo = q;
    c.rem = n - q * k;
    return c;
}

// Request that holds triple x of a layer: the number of requests that end at or before it.  All lanes of a warp.
MKV_CUT int request_of(const int* cum, int B, int x, int lane)
{
    int b = 0;
    for (int b0 = 0; b0 < B; b0 += kCutLanes) {
        const int ended = count_lanes(b0 + lane < B && cum[b0 + lane + 1] <= x);
        b += ended;
        if (ended < kCutLanes) break;
    }
    return b;
}

// Block `me` of the cut of one layer.  Called by warp 0 (all lanes) after cum[] and lens[] are complete; other warps wait at
// the next barrier.
MKV_CUT void build_partition(Partition* pt, const int* cum, const int* lens, int B, int hkv, int grid, int pages, int row_cost,
                             int min_pages, int straddle, int me, int lane)
{
    const int W = cum[B], rows = B * hkv;
    const Cut cut = make_cut(W, pages, grid, min_pages);
    grid = cut.blocks;
    int start = 0, end = 0;                             // every request of the call is empty, or more blocks than work
    // With k blocks per row the rows that get one block fewer run 1/k longer, but a block that straddles two rows
    // pays the per-row set-up, reduction and partial twice (about 8 us, a quarter of a block's pages at config-1
    // sizes).  Measured: from four blocks per row on, whole blocks per row win (16 rows: 71 -> 66 us, 32 rows: 74 -> 71).
    // The rounding to whole blocks costs about half a block's share in k of a block's pages, pages rows / (2 grid^2); from
    // `straddle` pages on that is dearer than the straddling (d 128, 8 heads, two blocks per SM: 8 x 4,096 tokens 28.9 us linear,
    // 23.6 aligned; 8 x 32,768 of which half FP8 104.7 linear, 108 aligned).
    int aligned = (rows * 4 <= grid && rows <= kMaxAlignedRows && pages >= grid &&
                   (long long)pages * rows < 2ll * straddle * grid * grid) ? 1 : 0;
    if (aligned) {
        // block boundaries at the rounded cumulative share of the rows: base[r] = round(grid * first_position(r) / W);
        // every row must end up with at least one block, otherwise the linear cut is used.  (A row's share also counts
        // row_cost, so that a row of a few pages may get more blocks than pages; those without a page do nothing, see
        // blocks_of_row.  With the linear cut for such batches, and so: 2 requests of 32 and 2,000 to 8,000 tokens, d 256,
        // 1 to 4 heads 14.2 .. 19.0 / 13.9 .. 18.5 us a step.)
        int bad = 0;
        const float scale = (float)grid / (float)W;
        for (int r = lane; r < rows; r += kCutLanes) {
            const int b = small_div(r, hkv), n = pages_of(lens[b]), len = n > 0 ? n + row_cost : 0;
            const int first = cum[b] + (r - b * hkv) * len;
            const int c0 = (int)((float)first * scale + 0.5f), c1 = r + 1 == rows ? grid : (int)((float)(first + len) * scale + 0.5f);
            pt->base[r] = c0;
            if (n > 0 && c1 <= c0) bad = 1;
            if (c0 <= me && me < c1) {                          // the one lane that holds this block's row
                const Cut row = cut_row(n, c1 - c0);
                const int j = me - c0;
                pt->start = first + (j > 0 ? row_cost + (int)cut_start(row, j) : 0);
                pt->end = first + row_cost + (int)cut_start(row, j + 1);
                pt->first_b = b;
            }
        }
        if (lane == 0) {
            pt->base[rows] = grid;
            if (me >= grid) pt->start = pt->end = 0;
        }
        if (any_lane(bad)) aligned = 0;
        sync_lanes();
    }
    if (!aligned) {
        if (me < grid) {
            start = (int)cut_start(cut, me);
            end = (int)cut_start(cut, me + 1);
        }
        const int b = request_of(cum, B, start, lane);
        if (lane == 0) {
            pt->start = start;
            pt->end = end;
            pt->first_b = b;
        }
    }
    if (lane == 0) {
        pt->aligned = aligned;
        pt->cut = cut;
    }
}

// Block `me` of the flat cut of n_layers layers: its layers, and the request of its first triple.  Warp 0, all lanes.
MKV_CUT void build_flat_partition(Partition* pt, const int* cum, int W, int B, int n_layers, int grid, int pages, int min_pages, int me, int lane)
{
    const Cut cut = make_cut((long long)W * n_layers, (long long)pages * n_layers, grid, min_pages);
    int first = 0, end = 0, b = 0;
    if (me < cut.blocks) {
        const long long s = cut_start(cut, me), e = cut_start(cut, me + 1);
        first = smaller((int)near_quotient((float)s, (float)W), n_layers - 1);
        if ((long long)first * W > s) --first;
        if ((long long)(first + 1) * W <= s) ++first;
        for (end = first + 1; (long long)end * W < e;) ++end;
        b = request_of(cum, B, (int)(s - (long long)first * W), lane);
    }
    if (lane == 0) {
        pt->flat = cut;
        pt->first_layer = first;
        pt->end_layer = end;
        pt->first_b = b;
    }
}

// Range [start, end) of block `me` of the flat cut in layer `layer`
MKV_CUT void range_in_layer(const Partition* pt, int W, int layer, int me, int& start, int& end)
{
    const long long w0 = (long long)layer * W;
    start = (int)max(cut_start(pt->flat, me) - w0, 0ll);
    end = (int)min(cut_start(pt->flat, me + 1) - w0, (long long)W);
}

// A block's part of a row
struct Segment {
    int h, n_pages;                     // KV head; pages of the row
    int row_start, row_end;             // positions of the row (the first row_cost of them are no pages)
    int end;                            // where the block goes on
    int pg0, n;                         // first page (in the order of page_at) and number of pages; n <= 0: none
};

// The segment at position pos of a block whose range ends at my_end; b, the request of pos or one before it, is brought up to date.
MKV_CUT Segment segment_at(const int* cum, const int* lens, int row_cost, int pos, int my_end, int& b)
{
    while (cum[b + 1] <= pos) ++b;
    Segment s;
    s.n_pages = pages_of(lens[b]);
    const int row_len = s.n_pages + row_cost;
    s.h = (int)near_quotient((float)(pos - cum[b]), (float)row_len);
    int off = pos - cum[b] - s.h * row_len;             // at most one row off
    if (off < 0) --s.h, off += row_len;
    if (off >= row_len) ++s.h, off -= row_len;
    s.row_start = pos - off;
    s.row_end = s.row_start + row_len;
    s.end = smaller(my_end, s.row_end);
    s.pg0 = larger(off - row_cost, 0);
    s.n = s.end - s.row_start - row_cost - s.pg0;
    return s;
}

// Blocks c0 .. c1 that hold pages of the row with index r, whose first page is at first_page and whose last before row_end
template <bool FLAT>
MKV_CUT void blocks_of_row(const Partition* pt, int W, int layer, int r, int first_page, int row_end, int& c0, int& c1)
{
    if constexpr (FLAT) {
        const long long w0 = (long long)layer * W;
        c0 = cut_block_of(pt->flat, w0 + first_page);
        c1 = cut_block_of(pt->flat, w0 + row_end - 1);
    } else if (pt->aligned) {
        c0 = pt->base[r];
        c1 = c0 + smaller(pt->base[r + 1] - c0, row_end - first_page) - 1;      // no more blocks than pages
    } else {
        c0 = cut_block_of(pt->cut, first_page);
        c1 = cut_block_of(pt->cut, row_end - 1);
    }
}

// Slot of the partial of a block's segment at pos: 2c if the segment opens the block's range (flat cut: its range in this layer)
MKV_CUT int partial_slot(int block, int pos, int my_start) { return 2 * block + (pos != my_start ? 1 : 0); }

// Slot of a row's first partial (block c0).  The row opens block c0's range of the layer where it starts at or before that
// range.  (The other blocks' ranges begin inside the row: slot 2c.)
template <bool FLAT>
MKV_CUT int first_partial_slot(const Partition* pt, int W, int layer, int c0, int row_start)
{
    long long start;
    if constexpr (FLAT) start = cut_start(pt->flat, c0) - (long long)layer * W;
    else start = pt->aligned ? row_start : cut_start(pt->cut, c0);
    return 2 * c0 + (row_start > (start > 0 ? start : 0) ? 1 : 0);
}

// Whether position x of the row [row_start, row_end) (row index r, row_cost 0) opens the run of some warp in the per-layer cut
// with n_warps warps per block.
MKV_CUT bool opens_warp_run(const Partition* pt, int r, int row_start, int row_end, int x, unsigned n_warps)
{
    int first, n;                                   // the block's share of the row
    if (pt->aligned) {
        const Cut row = cut_row(row_end - row_start, pt->base[r + 1] - pt->base[r]);
        const int j = cut_block_of(row, x - row_start);
        first = row_start + (int)cut_start(row, j);
        n = row_start + (int)cut_start(row, j + 1) - first;
    } else {
        const int c = cut_block_of(pt->cut, x);
        first = larger((int)cut_start(pt->cut, c), row_start);
        n = smaller((int)cut_start(pt->cut, c + 1), row_end) - first;
    }
    const unsigned w = ((unsigned)(x - first + 1) * n_warps - 1) / (unsigned)n;
    return (int)((unsigned)n * w / n_warps) == x - first;
}

// Pages of a row are visited in an order that gives every contiguous range of positions the row's FP8 and TQ3 pages in
// their overall proportion (spans of either format are contiguous), so that equal ranges cost equal time.  The row is cut into 32
// strips of equal length (the first n % 32 are one page longer); position x is page x / 32 of strip x % 32, the strips
// in bit-reversed order, and the pages that the longer strips have more come last.  A bijection without a division.
MKV_CUT int page_at(int x, int n)
{
    const int len = n >> 5, longer = n & 31, at = x >> 5;
    const int strip = at < len ? reversed_low_5_bits(x) : x & 31;
    return strip * len + smaller(strip, longer) + at;
}

}  // namespace mkv
