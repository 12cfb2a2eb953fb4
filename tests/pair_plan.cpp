// The host's plan of the pair kernel (csrc/pair_plan.h) over a range of problems: what its tiles and those of T' have to be.
#include <cstdio>
#include <initializer_list>

#include "../paper_2410_09615_b200/csrc/handover.h"
#include "../paper_2410_09615_b200/csrc/pair_plan.h"

using namespace slim;

static int bad(const char* what, int b, int d_out, int d_in, int r, int pairs) {
    printf("%s: %d -> %d, rank %d, %d tokens, %d pairs\n", what, d_in, d_out, r, b, pairs);
    return 1;
}

int main() {
    for (int r = 16; r <= 1040; r += 16)
        for (int most : {128, 256})
            for (int token_tiles : {1, 2, 3})
                for (int spare = 0; spare <= 73; ++spare) {
                    const int chunks = t_chunks(r, most, token_tiles, spare), width = t_width(r, chunks);
                    if (width > most || width % 16 != 0 || chunks * width < r) return bad("a chunk too wide, or ranks without one", token_tiles, most, 0, r, spare);
                    if ((chunks - 1) * width >= r) return bad("a chunk without ranks", token_tiles, most, 0, r, spare);
                }
    for (int pairs : {37, 66, 74})
        for (int d_in : {64, 448, 1024, 2752, 4096, 8192})
            for (int d_out : {16, 1024, 2736, 4096, 11008, 28672})
                for (int r : {0, 16, 144, 176, 208, 272, 416, 832})
                    for (int b = 1; b <= 1100; b += b < 130 ? 1 : 57) {
                        const PairPlan pl = pair_plan(b, d_out, d_in, r, pairs);
                        const int token_tiles = ceil_div(b, pl.tile_n);
                        if (pl.tile_n % 16 != 0 || pl.tile_n < 16 || pl.tile_n > 256 || pl.tiles != token_tiles * ceil_div(d_out, kPairRows) || (token_tiles - 1) * pl.tile_n >= b)
                            return bad("tiles", b, d_out, d_in, r, pairs);
                        if (r == 0) { if (pl.t_tiles != 0) return bad("T' without adapters", b, d_out, d_in, r, pairs); continue; }
                        // columns of a T' tile: as many as its accumulator has, and no more than the partial sums have room for
                        if (pl.t_n % 16 != 0 || pl.t_n > (pl.tile_n <= 128 ? 128 : 256) || pl.t_n > t_width(r, ceil_div(r, 256))) return bad("columns of T'", b, d_out, d_in, r, pairs);
                        const int ranks_of_chunk = pl.t_ranks ? kPairTTok : pl.t_n, tokens_of_tile = pl.t_ranks ? pl.tile_n : kPairTTok;
                        if (pl.t_chunks != ceil_div(r, ranks_of_chunk) || pl.t_tiles != pl.t_chunks * ceil_div(b, tokens_of_tile)) return bad("tiles of T'", b, d_out, d_in, r, pairs);
                        const int stages = d_in / kPairDK, grid = pl.tiles < pairs ? pl.tiles : pairs;
                        const int shares = t_share(pl.t_tiles, stages, pairs, pairs - grid, ceil_div(d_in, 128));
                        if (shares < 1 || shares > pairs || shares > pl.t_tiles * stages) return bad("shares of T'", b, d_out, d_in, r, pairs);
                        // where the shares divide the tiles, tile t is made by pairs t * parts to t * parts + parts - 1
                        const int parts = shares % pl.t_tiles == 0 ? shares / pl.t_tiles : 0, units = pl.t_tiles * stages;
                        for (int t = 0; parts > 0 && t < pl.t_tiles; ++t)
                            if (share_owner(t * stages, units, shares) != t * parts || share_owner((t + 1) * stages - 1, units, shares) != (t + 1) * parts - 1)
                                return bad("owners of T'", b, d_out, d_in, r, pairs);
                    }
    printf("ok\n");
    return 0;
}
