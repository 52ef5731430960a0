// What a draft call's row counts decide: row tiles, k-ranges, attention ranges, and
// the workspace that holds their partials.  Plain C++.
//
// A workspace for some number of sequences serves every smaller call too, so each
// size below never falls as the rows grow.  The partials of a split reduction do
// fall (k-ranges or key ranges x rows: 80 rows of 38 ranges, 96 of 19), so they are
// sized by the largest of all smaller row counts.
#pragma once

#include <algorithm>

namespace osp {

constexpr int TC_TILE_ROWS = 80;   // activation rows per tile: three accumulators fit a CTA's 256 TMEM columns
constexpr int TC_BIG_ROWS = 128;   // rows per tile of a larger GEMM ...
constexpr int TC_BIG_K = 4096;     // ... whose reduction is at least this long
constexpr int TC_MAX_ROWS = 4096;  // rows of a call on the tensor cores (beyond: the CUDA-core GEMV)
constexpr int TC_GROUP_ROWS = 512; // rows of one pass of block drafting

// A GEMM's rows as equal tiles (the MMA's N, a multiple of 16).  Up to TC_TILE_ROWS
// keep two CTAs per SM (two accumulators of 80 columns and one of the small planes
// in 256 TMEM columns, two stages of three planes in 112 KB).  More rows: with a
// reduction of TC_BIG_K or more, tiles of up to TC_BIG_ROWS and one CTA per SM
// (four accumulators of 128 columns, three stages): 120 rows at d 4096, gate and up
// 110 -> 88 us, the O and down projections 39 -> 34; with a shorter one, an even
// number of the small tiles: start and epilogue weigh more there, and two CTAs
// overlap them (96 rows, d 1024: 11.7 us a launch against 12.7).
struct TcTiles {
    int nrt, npad;     // row tiles, rows per tile
    int bps;           // CTAs per SM
    int rows() const { return nrt * npad; }   // rows of an operand plane
};
inline TcTiles tc_tiles_of(long long rows, int most, int even, int bps) {
    TcTiles t;
    t.nrt = rows <= most ? 1 : (int)((rows + most - 1) / most + even - 1) / even * even;
    t.npad = (int)(((rows + t.nrt - 1) / t.nrt + 15) / 16 * 16);
    t.bps = bps;
    return t;
}
inline TcTiles tc_tiles(long long rows, int K) {
    return rows > TC_TILE_ROWS && K >= TC_BIG_K ? tc_tiles_of(rows, TC_BIG_ROWS, 1, 1)
                                                : tc_tiles_of(rows, TC_TILE_ROWS, 2, 2);
}
// The LM head keeps two CTAs per SM at any number of rows, whose epilogues (the
// sampling partials are most of an item's time) run beside each other's MMAs:
// 96 rows, V 151936, d 1024, in two tiles of 48 132 us, in one of 96 161 (both with
// segments of 2 k-blocks).  An even number of tiles: pairs share weights through L2.
inline TcTiles tc_tiles_lm(long long rows) { return tc_tiles_of(rows, TC_TILE_ROWS, 2, 2); }
// k-ranges of block drafting's GEMMs: those of one row tile, whatever the rows
constexpr TcTiles TC_BLOCK_SPLITS{1, TC_TILE_ROWS, 2};

// k-ranges per output tile so that tiles x ranges fill the CTA slots (few
// output tiles, long K: the layer projections); 1 for wide outputs.
inline int tc_nsplit(int nout, int K, const TcTiles &t, int sms) {
    const int tiles = (nout + 127) / 128 * t.nrt, nkb = K / 64;
    // at most one item per CTA slot: one item more than the slots would take two
    // item times for barely more than one wave of work
    const int want = std::min(std::max(t.bps * sms / tiles, 1), std::max(nkb, 1));
    const int kbps = (nkb + want - 1) / want;
    return (nkb + kbps - 1) / kbps;
}

// Rows of an operand plane in a call of up to `rows` rows, whichever GEMM reads it.
inline long long tc_plane_rows(long long rows) {
    return std::max(tc_tiles(rows, 1).rows(), tc_tiles(rows, TC_BIG_K).rows());
}

// Floats of a GEMM's k-range partials in a call of up to `rows` rows; `always`: one
// range goes through them too.
inline long long tc_part_floats(int nout, int K, long long rows, int sms, bool block, bool always) {
    long long most = 0;
    auto offer = [&](long long r) {
        const int ns = tc_nsplit(nout, K, block ? TC_BLOCK_SPLITS : tc_tiles(r, K), sms);
        if (ns > 1 || always) most = std::max(most, ns * r * nout);
    };
    // within one number of tiles they grow with the rows: the last row count of each
    const int step = K >= TC_BIG_K ? TC_BIG_ROWS : 2 * TC_TILE_ROWS;
    if (!block && rows > TC_TILE_ROWS) {
        offer(TC_TILE_ROWS);
        for (long long r = step; r < rows; r += step) offer(r);
    }
    offer(rows);
    return most;
}

// Key ranges per (row, KV head) of the attention of R rows: about four blocks per SM
// over the whole grid, at most 1024 keys per block, at least 64 (one page per warp).
constexpr int ATTN_MAX_SPLITS = 128;
inline int attn_splits(int R, int Hkv, int max_ctx, int sms) {
    auto cdiv = [](long long x, long long y) { return (int)((x + y - 1) / y); };
    const int s = std::min(std::max(cdiv(4LL * sms, (long long)R * Hkv), cdiv(max_ctx, 1024)), cdiv(max_ctx, 64));
    return std::max(std::min(s, ATTN_MAX_SPLITS), 1);
}

// No call of up to R rows has more ranges x rows than this (R ceil(a / R) < a + R).
inline long long attn_ranges(long long R, int Hkv, int max_ctx, int sms) {
    const long long by_len = (max_ctx + 1023) / 1024, cap = std::min((max_ctx + 63) / 64, ATTN_MAX_SPLITS);
    return std::max(R, std::min(R * cap, std::max(R * by_len, (4LL * sms + Hkv * R - 1) / Hkv)));
}

// Whether a sequence's extend rows share one pass over their keys (attn_rows_kernel,
// 16 (row, head) queries a block) instead of streaming them once a row.  A launch of
// it takes 25 to 35 us more to start, split and merge; the row-by-row kernel takes
// about 15 us a million of (G + 2) x rows x KV heads x keys.  Measured over 1..32
// sequences of 2, 4 and 8 rows, 256..16384 keys, G 2 and 4 (582 calls): the two cross
// at 4.2 to 5 million, and with less than half a tile of queries the shared pass never
// wins.  With the line at 6 million no call is 2 % slower than row by row, and all
// together are 0.2 % off the better of the two; a line by rows x KV heads alone was
// 3.2 % off it and up to 17 % slower, at 256 to 1024 keys.  The keys are the page
// table's capacity.
inline bool attn_rows_pays(long long R, int Hq, int Hkv, int rows_per_seq, int max_ctx) {
    const int G = Hq / Hkv;
    return rows_per_seq > 1 && rows_per_seq * G >= 8 && R * Hkv * (G + 2) * max_ctx >= 6000000LL;
}

// Blocks of a tree walk's cluster, as 8 >> the index returned: the size whose waves
// take the least.  at_once: clusters of 8, 4, 2 and 1 blocks that the device holds;
// cached: their slices of two rows fit shared memory.  A walk takes a fixed time
// (barriers, exchanges: what one block takes for 95 KB of a row, 3 KB more a block of
// the cluster; greedy, without exponentials, 300 KB) and the row over the blocks, a
// third more where later passes read it again.  Walks differ in length, so waves
// overlap: x times what fits takes x + 0.4.
// us a call with clusters of 8 always / as chosen / one block a sequence in its first
// form (K 3, topk 2): float32, T 1, V 151936, 16 sequences 47 / 47 / 116, 64 134 / 82 /
// 140, 256 464 / 251 / 262; V 4096, 32 28 / 22 / 24, 128 95 / 25 / 25, 512 345 / 40 /
// 76; bf16, V 32000, 32 31 / 29 / 46, 512 375 / 120 / 146.  Of 234 such calls (V 4001
// to 200064, 1 to 512 sequences, greedy too) 6 are 4 to 10 % slower than in the first
// form, all of 96 sequences and more (float32 V 50304, bf16 V 32000 greedy).
inline int tree_cluster(int B, double row_kb, bool greedy, const bool (&cached)[4], const long long (&at_once)[4]) {
    int pick = 0;
    double best = 0;
    for (int i = 0; i < 4; ++i) {
        const int c = 8 >> i;
        const double x = (double)B / at_once[i], row = row_kb / c * (greedy || cached[i] ? 1. : 1.35);
        const double cost = (x <= 1 ? 1. : x + 0.4) * ((greedy ? 300 : 95) + 3 * c + row);
        if (i == 0 || cost < best) {
            best = cost;
            pick = i;
        }
    }
    return pick;
}

}  // namespace osp
