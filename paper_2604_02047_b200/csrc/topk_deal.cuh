// How the items of the top-k kernel -- the chunks of all rows, in row-major order -- are dealt to its CTAs: contiguous ranges, whole rows
// where that is the better share.  Host arithmetic.
#pragma once

#include "goose.h"

namespace goose {

constexpr int kTopkChunk = 32768;                            // elements of an item, at most
constexpr int kTopkMaxChunks = GOOSE_MAX_V / kTopkChunk;     // 8

inline int topk_chunks(int V) { return (V + kTopkChunk - 1) / kTopkChunk; }   // of a row
inline int topk_items(int rows, int V) { return rows * topk_chunks(V); }

// Items that a CTA gets, at most.  A row that is spread over CTAs costs a merge behind its last part, more than an item does: where one
// item more a CTA gives every row to one CTA, that is the better share.  Top-k / harvest, us, without -> with:  4 chunks (V = 128256): 100
// rows (q = 3 -> 4) 9.8 -> 8.6 / 13.5 -> 12.1, 250 rows (7 -> 8) 16.6 -> 15.1 / 22.2 -> 20.8;  2 chunks (65536): 60 rows (1 -> 2) 6.0 ->
// 5.1, 150 rows (3 -> 4) 8.6 -> 7.9, 900 rows (13 -> 14) 23.9 -> 22.7 / 33.5 -> 31.8;  7 chunks (200000): 122 rows (6 -> 7) 15.5 -> 13.8 /
// 20.7 -> 19.1.  Two items more are even (4 chunks: 60 rows, 200 rows) or worse (30 rows 6.3 -> 7.7, 150 rows (5 -> 8) 18.2 -> 19.7), and
// so is a second item with the log-sum-exp (cycle of 32 over 8 heads, 32 rows of 65536 12.4 -> 12.8) or beside the attention of a step, where
// the CTAs that it saves would be idle (8 heads, 33 rows of 65536, 1207 keys 11.4 -> 12.2, 32 over 4 heads, 32 rows of 50000, 1507 keys
// 13.35 -> 13.9; a fourth item there: 16 heads, 64 rows of 33000, 690 keys 12.8 -> 12.1): no_second.
inline int topk_share(int items, int chunks, int ctas, bool no_second) {
    const int q = (items + ctas - 1) / ctas;
    return chunks > 1 && (q + 1) % chunks == 0 && (q > 1 || !no_second) ? q + 1 : q;
}

// CTA c's items are start(c) .. start(c + 1) - 1: `unit` items more for the first `more` CTAs than the `per` that all have
struct TopkDeal {
    int grid, per, more, unit;
    int start(int c) const { return c * per + (c < more ? c : more) * unit; }
};

// The fewest CTAs that the share allows: that loses no time.  Where the share is whole rows, rows are dealt and none is cut: items dealt one
// by one would leave a CTA with one item fewer in the middle of a row wherever they do not come out even (900 rows of 2 chunks: 123 CTAs
// with 14 and 6 with 13).  With node counts the rows that exist are known on the device alone: fewer CTAs for all rows would not get whole
// ones (the kernel works out per, more and unit for the rows that exist).
inline TopkDeal topk_deal(int rows, int chunks, int ctas, bool no_second, bool counts) {
    const int items = rows * chunks, q = counts ? (items + ctas - 1) / ctas : topk_share(items, chunks, ctas, no_second);
    const int unit = !counts && q % chunks == 0 ? chunks : 1, units = items / unit, grid = (units + q / unit - 1) / (q / unit);
    return {grid, units / grid * unit, units % grid, unit};
}

}  // namespace goose
