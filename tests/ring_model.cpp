// The barriers of the pair kernel (csrc/fwd_prefill.cu) as one pair of CTAs uses them, in a model that runs its warps in many orders: the
// converters' turns are the kernel's own, from csrc/turns.h, the other warps walk as they do there.
//
// A barrier has phases; a wait by parity lets a warp pass where the phase it asks for, or one that differs from it by an even number,
// has ended.  The model knows which phase is meant.  A warp that passes before it, or all warps waiting, is an error.  Copies land in any
// order, MMAs complete in the order of their issue; who runs next is drawn, with priorities that change now and then, so that a warp
// may stay behind for as long as the others can do without it.
//
// Usage: ring_model <tile stages of 128 columns> <narrow 0 | 1> <adapter stages> <tiles> <T' runs> <T' run length> <seeds>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "../paper_2410_09615_b200/csrc/turns.h"

namespace {

using namespace slim;
constexpr int kStages = kTurnPlaces, kSlots = kTurnSlots, kGroups = kTurnGroups;

struct Barrier {
    int count = 0, pending = 0, bytes = 0, phases = 0;
    void init(int n) { count = pending = n; }
    void settle() { if (pending == 0 && bytes == 0) { ++phases; pending = count; } }
    void arrive(int n) { pending -= n; settle(); }
    bool passes(int phase) const { return (phases & 1) != (phase & 1); }
};

enum Kind { WAIT, ASK, ARRIVE, EXPECT, COPY, COMMIT };
// ASK keeps its answer (of a place or of a packed tile), and a WAIT that looks at one passes at once if it was yes.
enum Answer { NONE, PLACE, TILE, ANSWERS };
struct Op { Kind kind; int cta, bar, n; Answer answer; };

enum { FULL = 0, EMPTY = FULL + kStages, PK_FULL = EMPTY + kStages, PK_EMPTY = PK_FULL + kSlots, ACC_FULL = PK_EMPTY + kSlots, ACC_EMPTY, BARS };

struct Warp {
    std::vector<Op> ops;
    size_t at = 0;
    bool answers[ANSWERS] = {};
    void add(Kind k, int cta, int bar, int n, Answer a = NONE) { ops.push_back({k, cta, bar, n, a}); }
};

struct Shape { int n128, narrow, n2, tiles, runs, len; };

std::vector<Warp> warps_of(const Shape& s) {
    const int pk_stages = s.narrow ? 1 : 2, n1 = s.narrow ? (s.n128 + 1) / 2 : s.n128, groups_of_tile = (n1 + pk_stages - 1) / pk_stages;
    const int t_stages = s.runs * s.len, n_total = n1 + s.n2;
    std::vector<Warp> all;
    auto free_place = [&](Warp& w, int cta, int g) { if (g >= kStages) w.add(WAIT, cta, EMPTY + g % kStages, g / kStages - 1); };
    for (int cta = 0; cta < 2; ++cta) {
        for (int odd = 0; odd < 2; ++odd) {                  // token tiles and adapters
            Warp w;
            int g = 0;
            auto request = [&](int stage) { free_place(w, cta, stage); w.add(COPY, 0, FULL + stage % kStages, 1); };
            for (; g < t_stages; ++g) request(g);
            for (int t = 0; t < s.tiles; ++t) {
                for (int it = (g ^ odd) & 1; it < n1; it += 2) request(g + it);
                for (int it = n1; it < n_total; ++it) request(g + it);
                g += n_total;
            }
            all.push_back(w);
        }
        Warp packed;
        for (int i = 0; i < s.tiles * groups_of_tile; ++i) {
            if (i >= kSlots) packed.add(WAIT, cta, PK_EMPTY + i % kSlots, i / kSlots - 1);
            packed.add(EXPECT, cta, PK_FULL + i % kSlots, 1);
            packed.add(COPY, cta, PK_FULL + i % kSlots, 1);
        }
        all.push_back(packed);
        for (int warp = 0; warp < 4 * kGroups; ++warp) {     // converters
            Warp w;
            const int group = warp / 4;
            auto arrive = [&](int g, int copies) {
                if (cta == 0 && warp % 4 == 0) w.add(EXPECT, 0, FULL + g % kStages, copies);
                else w.add(ARRIVE, 0, FULL + g % kStages, 1);
            };
            for (int g = first_turn(group, 0); g < t_stages; g += kGroups) { free_place(w, cta, g); arrive(g, 4); }
            int base = t_stages;
            for (int t = 0; t < s.tiles; ++t, base += n_total) {
                Answer asked = NONE;
                const int seen = seen_from(t, n1, s.n2, pk_stages);
                for (int it = first_turn(group, base); it < n_total; it += kGroups) {
                    const int g = base + it;
                    if (it >= n1) { free_place(w, cta, g); arrive(g, 4); continue; }
                    const int gi = t * groups_of_tile + it / pk_stages, slot = gi % kSlots;
                    const bool knows = it >= seen;
                    if (!knows) free_place(w, cta, g);
                    w.add(WAIT, cta, PK_FULL + slot, gi / kSlots, asked);
                    if (knows && g >= kStages) w.add(ASK, cta, EMPTY + g % kStages, g / kStages - 1, PLACE);
                    w.add(ARRIVE, cta, PK_EMPTY + slot, it % pk_stages == 0 && it + 1 == n1 ? pk_stages : 1);
                    const int ahead = kGroups / pk_stages;
                    asked = it + kGroups < n1 && it + kGroups >= seen ? TILE : NONE;
                    if (asked) w.add(ASK, cta, PK_FULL + (gi + ahead) % kSlots, (gi + ahead) / kSlots, TILE);
                    if (knows && g >= kStages) w.add(WAIT, cta, EMPTY + g % kStages, g / kStages - 1, PLACE);
                    arrive(g, 2);
                }
            }
            all.push_back(w);
        }
        for (int warp = 0; warp < 8; ++warp) {               // epilogue
            Warp w;
            for (int i = 0; i < s.runs + s.tiles; ++i) { w.add(WAIT, cta, ACC_FULL, i); w.add(ARRIVE, 0, ACC_EMPTY, 1); }
            all.push_back(w);
        }
    }
    Warp mma;
    int g = 0, nth = 0;
    auto product = [&](int stages) {
        if (nth > 0) mma.add(WAIT, 0, ACC_EMPTY, nth - 1);
        for (int i = 0; i < stages; ++i, ++g) { mma.add(WAIT, 0, FULL + g % kStages, g / kStages); mma.add(COMMIT, 0, EMPTY + g % kStages, 1); }
        mma.add(COMMIT, 0, ACC_FULL, 1);
        ++nth;
    };
    for (int i = 0; i < s.runs; ++i) product(s.len);
    for (int t = 0; t < s.tiles; ++t) product(n_total);
    all.push_back(mma);
    return all;
}

// Returns nullptr, or what went wrong.
const char* run(const Shape& s, const std::vector<Warp>& program, unsigned seed, size_t* stuck) {
    std::mt19937 rng(seed);
    std::vector<Warp> warps = program;
    Barrier bars[2][BARS];
    for (int cta = 0; cta < 2; ++cta) {
        for (int i = 0; i < kStages; ++i) { bars[cta][FULL + i].init(8); bars[cta][EMPTY + i].init(1); }
        for (int i = 0; i < kSlots; ++i) { bars[cta][PK_FULL + i].init(1); bars[cta][PK_EMPTY + i].init(4 * (s.narrow ? 1 : 2)); }
        bars[cta][ACC_FULL].init(1); bars[cta][ACC_EMPTY].init(16);
    }
    struct Copy { int cta, bar; };
    std::vector<Copy> copies;
    std::vector<Op> mmas;
    size_t mma_at = 0;
    std::vector<unsigned> prio(warps.size() + 2);
    for (auto& p : prio) p = rng();
    auto complete = [&](int cta, int bar, int bytes) { Barrier& b = bars[cta][bar]; b.bytes -= bytes; b.settle(); };
    for (;;) {
        int best = -1;
        bool left = false;
        for (size_t i = 0; i < prio.size(); ++i) {
            bool can;
            if (i < warps.size()) {
                const Warp& w = warps[i];
                if (w.at == w.ops.size()) continue;
                left = true;
                const Op& o = w.ops[w.at];
                can = o.kind != WAIT || w.answers[o.answer] || bars[o.cta][o.bar].passes(o.n);
            } else {
                can = i == warps.size() ? !copies.empty() : mma_at < mmas.size();
            }
            if (can && (best < 0 || prio[i] > prio[best])) best = (int)i;
        }
        if (best < 0) { for (*stuck = 0; *stuck < warps.size() && warps[*stuck].at == warps[*stuck].ops.size();) ++*stuck; return left ? "all wait" : nullptr; }
        if (rng() % 64 == 0) prio[best] = rng();
        *stuck = best;
        if (best == (int)warps.size()) {
            const size_t i = rng() % copies.size();
            complete(copies[i].cta, copies[i].bar, 1);
            copies.erase(copies.begin() + i);
            continue;
        }
        if (best > (int)warps.size()) {
            const Op o = mmas[mma_at++];
            for (int cta = 0; cta < 2; ++cta) bars[cta][o.bar].arrive(1);          // on the same barrier of both CTAs
            continue;
        }
        Warp& w = warps[best];
        const Op o = w.ops[w.at++];
        Barrier& b = bars[o.cta][o.bar];
        switch (o.kind) {
        case WAIT: if (b.phases <= o.n) return "passed before the phase"; break;
        case ASK: w.answers[o.answer] = b.passes(o.n); if (b.passes(o.n) && b.phases <= o.n) return "answered before the phase"; break;
        case ARRIVE: b.arrive(o.n); break;
        case EXPECT: b.bytes += o.n; b.arrive(1); break;
        case COPY: copies.push_back({o.cta, o.bar}); break;
        case COMMIT: mmas.push_back(o); break;
        }
        if (b.pending < 0) return "an arrival too many";
    }
}

}  // namespace

int main(int argc, char** argv) {
    if (argc != 8) { fprintf(stderr, "usage: %s n128 narrow adapter_stages tiles runs run_length seeds\n", argv[0]); return 2; }
    auto arg = [&](int i) { return atoi(argv[i]); };
    const Shape s{arg(1), arg(2), arg(3), arg(4), arg(5), arg(6)};
    const std::vector<Warp> program = warps_of(s);
    for (unsigned seed = 1; seed <= (unsigned)arg(7); ++seed) {
        size_t who = 0;
        if (const char* what = run(s, program, seed, &who)) { printf("seed %u warp %zu: %s\n", seed, who, what); return 1; }
    }
    printf("ok\n");
    return 0;
}
