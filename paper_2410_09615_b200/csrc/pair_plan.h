// How the pair kernel cuts a problem, on the host: its tiles, those of T', and who makes them.  Plain C++, so that the tests can go over it.
#pragma once

namespace slim {

constexpr int kPairRows = 256, kPairTTok = 256, kPairDK = 64;     // rows of a tile; tokens (ranks) of a T' tile, its MMA's rows; columns of a stage of T'

#ifndef __CUDACC__
inline int ceil_div(int a, int b) { return (a + b - 1) / b; }
#endif

// Columns of a T' tile of the pair kernel that cuts r into `chunks`.
inline int t_width(int r, int chunks) { return r > 0 ? ceil_div(ceil_div(r, chunks), 16) * 16 : 16; }
// Chunks of r: of up to `most` columns, and as many as leave a tile up to eight of the pairs that have no other work.  (A tile's parts are added up by
// these pairs, each part of a column asked for by each of them.  us a call with as few chunks as can be and so: 4096 -> 11008, rank 416, 256
// tokens 27.3, 26.5; 8192 -> 1024, rank 112, 512 tokens 25.9, 24.7.)
inline int t_chunks(int r, int most, int token_tiles, int spare) {
    int chunks = ceil_div(r, most);
    while (spare / (token_tiles * chunks) > 8 && t_width(r, chunks + 1) >= 48) ++chunks;
    return ceil_div(r, t_width(r, chunks));      // (widths are multiples of 16: the last of the chunks counted may hold no rank)
}

// Parts of a T' tile, of up to `parts` that it may have: fewer where they are then added up in fewer rounds of loads (nine parts each) and the longest
// part grows by no more than two stages.  (us a call before and with this: 3584 -> 8192, rank 352, 600 tokens, twelve parts of up to 5 stages or
// eight of 7: 43.4, 41.1; rank 720, 300 tokens 34.6, 32.2; 8192 x 8192, rank 816, 40 tokens, ten of 13 or nine of 15: 30.0, 29.3.)
inline int t_parts(int stages, int parts) {
    int fewer = parts > 9 && parts <= 12 && ceil_div(stages, 9) <= ceil_div(stages, parts) + 2 ? 9 : parts;
    fewer = ceil_div(stages, ceil_div(stages, fewer));
    return ceil_div(fewer, 9) < ceil_div(parts, 9) ? fewer : parts;
}

// Pairs that share the work of T'.  Each tile in equal parts, one a pair, where that uses four fifths of the pairs or more
// (a pair then has one part to write, and the pairs that read the same X walk it together); else an even share each.
// Four stages (a microsecond and a half) or more for a part: below that its start and end dominate.
// Where the tiles leave pairs without one and those can make T' in about the time of the others' sparse phase, they do it
// alone (`spare` pairs, `main_stages` 128-column stages): the others start their tiles at once.
inline int t_share(int tiles, int stages, int pairs, int spare, int main_stages) {
    const int most = stages < 4 ? 1 : stages / 4;
    int parts = spare / tiles < most ? spare / tiles : most;
    if (parts >= 1 && (long long)ceil_div(stages, parts) <= main_stages) return tiles * t_parts(stages, parts);
    parts = pairs / tiles < most ? pairs / tiles : most;
    if (parts >= 1 && (parts == most || tiles * parts * 5 >= pairs * 4)) return tiles * t_parts(stages, parts);
    return (long long)tiles * most < pairs ? tiles * most : pairs;
}

// How the pair kernel cuts a problem: tokens of a tile (a multiple of 16), tiles, and the tiles of T'.
struct PairPlan { int tile_n, tiles, t_n, t_chunks, t_tiles; bool t_ranks; };
inline PairPlan plan_tiles(int b, int d_out, int r, int widest, int pairs) {
    PairPlan pl;
    pl.tile_n = ceil_div(ceil_div(b, ceil_div(b, widest)), 16) * 16;
    pl.tiles = ceil_div(d_out, kPairRows) * ceil_div(b, pl.tile_n);
    // T' tiles of narrow token tiles have up to 128 columns of tensor memory: chunks of the ranks, or, where that makes fewer tiles, the
    // tile's tokens
    const int most = pl.tile_n <= 128 ? 128 : 256;
    pl.t_ranks = pl.tile_n <= 128 && r > most && ceil_div(b, pl.tile_n) * ceil_div(r, kPairRows) < ceil_div(b, kPairTTok) * ceil_div(r, most);
    const int t_tokens = ceil_div(b, pl.t_ranks ? pl.tile_n : kPairTTok);
    pl.t_chunks = pl.t_ranks ? ceil_div(r, kPairRows) : r > 0 ? t_chunks(r, most, t_tokens, pairs - pl.tiles) : 1;
    pl.t_n = pl.t_ranks ? pl.tile_n : t_width(r, pl.t_chunks);
    pl.t_tiles = r > 0 ? t_tokens * pl.t_chunks : 0;
    return pl;
}
// The tokens cut evenly into tiles of up to 256 (so that up to 128 tokens are one narrow tile, however many tiles the rows make), or of up to 128 or 64
// where every tile then has a pair of its own: what takes the least time, in units of 10 ns.  A stage of 128 columns takes 0.40 us with 256 tokens, 0.27 with 128, 0.24 with 64; T' 7 us and 0.28 for each of its stages, on
// the pairs without a tile beside the others (of the shorter of the two a quarter counts: they share the L2), else before them.
// (4096 -> 4096, rank 416, 256 tokens in tiles of 256, 128, 64: 24.6, 22.7, 27.7 us; 5696 -> 1392, rank 288, 1024 tokens 31.1, 32.8, 49.4;
// 8192 -> 1024, rank 112, 512 tokens 32.8, 26.6, 24.7.)
inline PairPlan pair_plan(int b, int d_out, int d_in, int r, int pairs) {
    PairPlan best = {};
    long long best_cost = -1;
    for (int widest = 256; widest >= 64; widest /= 2) {
        const PairPlan pl = plan_tiles(b, d_out, r, widest, pairs);
        if (best_cost >= 0 && pl.tiles > pairs) break;
        const int stage = pl.tile_n > 128 ? 40 : pl.tile_n > 64 ? 27 : 24, t_stages = d_in / kPairDK;
        const long long main = (long long)ceil_div(pl.tiles, pairs) * ceil_div(d_in, 128) * stage;
        long long cost = main;
        if (r > 0) {
            const int spare = pairs - pl.tiles, parts = spare < pl.t_tiles ? 0 : spare / pl.t_tiles < t_stages / 4 ? spare / pl.t_tiles : t_stages < 4 ? 1 : t_stages / 4;
            if (parts > 0) {
                const long long t = 700 + (long long)ceil_div(t_stages, parts) * 28;
                cost = main > t ? main + t / 4 : t + main / 4;
            } else {
                cost = main + 700 + (long long)pl.t_tiles * t_stages * 28 / pairs;
            }
        }
        if (best_cost < 0 || cost < best_cost) { best = pl; best_cost = cost; }
    }
    return best;
}

}  // namespace slim
