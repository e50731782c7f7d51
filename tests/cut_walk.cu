// Walks every block of the decode scan's grid through its share of the work on the host, with the scan's own arithmetic
// (decode_cut.cuh), and counts what the blocks would scan, store and merge.
#include <algorithm>
#include <cstdio>
#include <map>
#include <vector>

#include "decode_cut.cuh"

using namespace mkv;

namespace {

struct RowParts {
    int pages = 0, whole = 0, n_parts = 0, c0 = -1, first_slot = -1;
    std::vector<int> slots;                     // of the partials stored for the row, in the order of the blocks
};

template <bool FLAT>
int walk(const int* lens, int B, int hkv, int grid, int n_layers, int warps, int per_sm, int tiled, int tensor_memory,
         int* idle_blocks, int* most_pages, int* blocks, char* why, int why_size)
{
    const int cost = tensor_memory ? 0 : cut_row_cost(warps, tiled), least = tensor_memory ? 1 : cut_min_pages(warps, per_sm);
    const int straddle = tensor_memory ? 1 << 30 : cut_straddle(warps);
    std::vector<int> cum(B + 1);
    RowSums sum = {0, 0};
    for (int b = 0; b < B; ++b) add_requests(sum, cum.data(), B, b, positions_of(lens[b], hkv, cost), 0);
    const int W = cum[B] = sum.positions, pages = W - sum.requests * hkv * cost;
    std::vector<std::vector<RowParts>> part(n_layers, std::vector<RowParts>(B * hkv));
    std::vector<std::vector<std::vector<char>>> seen(n_layers, std::vector<std::vector<char>>(B * hkv));
    std::vector<std::map<int, int>> ticket_row(n_layers), slot_row(n_layers);
    *idle_blocks = *most_pages = *blocks = 0;
#define FAIL(...) do { snprintf(why, why_size, __VA_ARGS__); return 1; } while (0)
    for (int me = 0; me < grid; ++me) {
        Partition pt = {};
        int layer_first = 0, layer_end = n_layers, scanned = 0;
        if (!FLAT || tiled) build_partition(&pt, cum.data(), lens, B, hkv, grid, pages, cost, least, straddle, me, 0);
        if (FLAT) {
            build_flat_partition(&pt, cum.data(), W, B, n_layers, grid, pages, least, me, 0);
            layer_first = pt.first_layer, layer_end = pt.end_layer;
        }
        *blocks = FLAT ? pt.flat.blocks : pt.cut.blocks;
        for (int layer = layer_first; layer < layer_end; ++layer) {
            int start = pt.start, end = pt.end;
            if (FLAT) range_in_layer(&pt, W, layer, me, start, end);
            int b = FLAT && layer > layer_first ? 0 : pt.first_b;
            for (int pos = start; pos < end;) {
                const Segment s = segment_at(cum.data(), lens, cost, pos, end, b);
                if (s.end <= pos) FAIL("block %d does not move on from position %d", me, pos);
                if (s.n <= 0) {
                    pos = s.end;
                    continue;
                }
                const int r = b * hkv + s.h;
                if (b >= B || s.h < 0 || s.h >= hkv || s.pg0 < 0 || s.pg0 + s.n > pages_of(lens[b]))
                    FAIL("block %d: pages %d + %d of request %d head %d", me, s.pg0, s.n, b, s.h);
                RowParts& row = part[layer][r];
                auto& pg_seen = seen[layer][r];
                pg_seen.resize(s.n_pages);
                for (int i = s.pg0; i < s.pg0 + s.n; ++i) {
                    const int pg = tiled ? i : page_at(i, s.n_pages);
                    if (pg < 0 || pg >= s.n_pages || pg_seen[pg]++) FAIL("page %d of row %d is met twice or does not exist", pg, r);
                }
                row.pages += s.n;
                scanned += s.n;
                if (s.n == s.n_pages) {
                    row.whole++;
                } else {
                    int c0, c1;
                    blocks_of_row<FLAT>(&pt, W, layer, r, s.row_start + cost, s.row_end, c0, c1);
                    if (c0 > me || c1 < me) FAIL("row %d: blocks %d..%d do not hold block %d", r, c0, c1, me);
                    if (!row.slots.empty() && (row.c0 != c0 || row.n_parts != c1 - c0 + 1)) FAIL("row %d: blocks disagree", r);
                    row.c0 = c0;
                    row.n_parts = c1 - c0 + 1;
                    row.first_slot = first_partial_slot<FLAT>(&pt, W, layer, c0, s.row_start);
                    const int slot = partial_slot(me, pos, start);
                    row.slots.push_back(slot);
                    if (slot_row[layer].count(slot)) FAIL("slot %d holds two partials", slot);
                    slot_row[layer][slot] = r;
                    auto t = ticket_row[layer].emplace(c0, r);
                    if (t.first->second != r) FAIL("rows %d and %d share a ticket", t.first->second, r);
                }
                pos = s.end;
            }
        }
        *most_pages = std::max(*most_pages, scanned);
        if (me < *blocks && scanned == 0) ++*idle_blocks;
        if (me >= *blocks && scanned) FAIL("block %d is beyond the cut", me);
    }
    for (int layer = 0; layer < n_layers; ++layer)
        for (int r = 0; r < B * hkv; ++r) {
            const RowParts& row = part[layer][r];
            const int n = pages_of(std::max(lens[r / hkv], 0));
            if (row.pages != n) FAIL("layer %d row %d: %d of %d pages are scanned", layer, r, row.pages, n);
            if (row.whole + (row.slots.empty() ? 0 : 1) != (n > 0)) FAIL("layer %d row %d is stored twice or never", layer, r);
            if ((int)row.slots.size() != row.n_parts)
                FAIL("layer %d row %d of %d pages: %d blocks arrive where %d are waited for", layer, r, n, (int)row.slots.size(), row.n_parts);
            for (int j = 0; j < row.n_parts; ++j)
                if (row.slots[j] != (j == 0 ? row.first_slot : 2 * (row.c0 + j))) FAIL("row %d: part %d is not where it is read", r, j);
        }
    return 0;
}

}  // namespace

extern "C" int cut_walk(const int* lens, int B, int hkv, int grid, int n_layers, int flat, int warps, int per_sm, int tiled,
                        int tensor_memory, int* idle_blocks, int* most_pages, int* blocks, char* why, int why_size)
{
    return (flat ? walk<true> : walk<false>)(lens, B, hkv, grid, n_layers, warps, per_sm, tiled, tensor_memory, idle_blocks,
                                             most_pages, blocks, why, why_size);
}

// The largest number of positions of a launch when B requests of `tiles` 16-token tiles each are decoded (negative: they do not fit)
extern "C" long long cut_most_positions(int B, int hkv, int tiles)
{
    const int most = requests_per_launch(hkv, tiles);
    long long largest = 0;
    for (int b0 = 0; b0 < B; b0 += most) {
        const int n = std::min(most, B - b0);
        std::vector<int> cum(n);
        RowSums sum = {0, 0};
        long long exact = 0;
        for (int b = 0; b < n; ++b) {
            add_requests(sum, cum.data(), n, b, positions_of(tiles * kPage, hkv, cut_row_cost(16, false)), 0);
            exact += ((long long)tiles + cut_row_cost(16, false)) * hkv;
        }
        if (exact != sum.positions) return -1;
        largest = std::max(largest, exact);
    }
    return largest;
}
