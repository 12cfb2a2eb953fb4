// What a launch's CTAs hand to one another through the workspace: the arithmetic of its words, for the kernels and (as plain C++)
// for the CPU threads that stand in for CTAs in the tests.
//
// The first word of a workspace counts departures.  Every call of a kernel that hands words over, whatever its shape and with or
// without adapters, adds 1 << 16 to it in all: CTA 0 what is left after one from each of the others.  While a CTA of the call is
// still there the upper bits are those of the calls before, so every CTA reads the same call number whenever it looks.  A
// word carries the number of the call that wrote it in its upper half; nothing is ever cleared, and kernels and shapes may
// take turns on one workspace.
#pragma once
#include <stddef.h>
#include <stdint.h>

#ifdef __CUDACC__
#define SLIM_BOTH __host__ __device__ __forceinline__
#else
#define SLIM_BOTH inline
#endif

namespace slim {

SLIM_BOTH uint32_t call_number(unsigned long long departures) { return (uint32_t)(departures >> 16) + 1u; }
SLIM_BOTH unsigned long long departure(unsigned block, unsigned blocks) { return block == 0 ? 65536ull - (blocks - 1) : 1ull; }
SLIM_BOTH unsigned long long tagged(uint32_t call, uint32_t payload) { return ((unsigned long long)call << 32) | payload; }
SLIM_BOTH bool is_of(unsigned long long word, uint32_t call) { return (uint32_t)(word >> 32) == call; }

// The stages of T' in the pair kernel: a list, tile after tile, dealt out evenly to `pairs` pairs.
SLIM_BOTH int share_begin(int q, int units, int pairs) { return (int)((long long)q * units / pairs); }
SLIM_BOTH int share_owner(int unit, int units, int pairs) { return (int)(((long long)(unit + 1) * pairs - 1) / units); }
// A share's run inside one tile, from `unit` on.
struct Run { int tile, k0, len; };
SLIM_BOTH Run run_at(int unit, int end, int stages) {
    Run r;
    r.tile = unit / stages; r.k0 = unit - r.tile * stages;
    const int left = stages - r.k0;
    r.len = left < end - unit ? left : end - unit;
    return r;
}
// A pair's part of a tile has two words (part written; its share of the sums written), for each of its CTAs; so has a tile made
// whole (the second alone).  A pair has at most one part that starts with its tile and one that does not.
SLIM_BOTH size_t part_word(int q, bool starts, uint32_t rank) { return ((size_t)(2 * q + (starts ? 1 : 0)) * 2 + rank) * 2; }
SLIM_BOTH size_t tile_word(int pairs, int tile, uint32_t rank) { return (size_t)pairs * 8 + (size_t)tile * 2 + rank; }

}  // namespace slim
