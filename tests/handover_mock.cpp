// The hand-over protocols of the kernels, run by CPU threads that stand in for CTAs.  The arithmetic of the words (call numbers,
// departures, shares of T' and the places of their words) is the kernels' own, from csrc/handover.h; std::atomic words stand in for
// device-scope accesses.
//
// Calls of three kinds take turns on one workspace, as kernels and shapes do:
//   0  small batch: CTAs 0 .. makers - 1 publish words of T and leave at once; the others look at the call number late, fetch every
//      word (each must be this call's), and leave.  A wait that runs out marks the call as given up, and from then on every wait
//      of the call gives up early, whichever CTA's it is;
//   1  pair kernel with adapters: a thread per CTA of a pair.  Parts of T' are written, then added up in shares of the columns by
//      the pairs that share a tile, then every CTA waits for the T' of every tile and checks it.  A CTA whose wait runs out waits no more;
//   2  pair kernel without adapters: hands nothing over, and still counts as a call.
//
// Usage: handover_mock <ctas> <makers> <words> <pairs> <t_pairs> <tiles> <stages> <calls> <withhold_call> <poll_limit>
//   In call number `withhold_call` (1-based, 0: never) maker 0, or pair 0 of the T' list, writes nothing.  One line per call: kind,
//   status word, call number, departures, wrong values, waits that ran their whole limit.
//        handover_mock shares
//   checks the shares and the places of the words over a range of sizes.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <set>
#include <thread>
#include <vector>

#include "../paper_2410_09615_b200/csrc/handover.h"

namespace {

using namespace slim;
constexpr uint32_t kTimeoutBit = 1u << 7;          // SLIM_ERR_TIMEOUT
constexpr int kColumns = 24;                       // of a tile of T'
constexpr auto relaxed = std::memory_order_relaxed;

struct Shape { int ctas, makers, words, pairs, t_pairs, tiles, stages; uint32_t poll_limit; };

struct Workspace {
    std::atomic<unsigned long long> departures{0}, gave_up{0};
    std::vector<std::atomic<unsigned long long>> words;      // T of the small batches, part and tile words: the same memory
    std::vector<long long> parts, sums;                      // [2 q + starts][rank][column], [tile][rank][column]
    explicit Workspace(const Shape& s)
        : words(std::max<size_t>(s.words, tile_word(s.t_pairs, s.tiles, 0))), parts((size_t)s.t_pairs * 4 * kColumns), sums((size_t)s.tiles * 2 * kColumns) { reset(); }
    void reset() {
        departures.store(0); gave_up.store(0);
        for (auto& w : words) w.store(0);
    }
};

struct Call {
    Workspace& ws;
    const Shape& s;
    bool withhold;
    std::atomic<uint32_t> status{0}, number{0};
    std::atomic<int> wrong{0}, expired{0};
    Call(Workspace& w, const Shape& sh, bool wh) : ws(w), s(sh), withhold(wh) {}

    void leave(unsigned block, unsigned blocks, uint32_t call) { number.store(call, relaxed); ws.departures.fetch_add(departure(block, blocks), relaxed); }

    // ---- small batches
    bool wait(const std::atomic<unsigned long long>& w, uint32_t call) {
        for (uint32_t spin = 0; !is_of(w.load(relaxed), call); ++spin) {
            if ((spin & 63u) == 63u) {
                if (is_of(ws.gave_up.load(relaxed), call)) return false;
                if (spin > s.poll_limit) { ws.gave_up.store(tagged(call, 0), relaxed); expired.fetch_add(1, relaxed); return false; }
            }
            std::this_thread::yield();
        }
        return true;
    }
    static uint32_t payload(uint32_t call, int u) { return call * 977u + (uint32_t)u; }
    void small(int cta) {
        if (cta >= s.makers) for (int i = 0; i < 50 * (cta % 3); ++i) std::this_thread::yield();
        const uint32_t call = call_number(ws.departures.load(relaxed));
        bool ok = true;
        if (cta < s.makers) {
            if (!(withhold && cta == 0))
                for (int u = cta; u < s.words; u += s.makers) ws.words[u].store(tagged(call, payload(call, u)), relaxed);
        } else {
            for (int u = 0; u < s.words; ++u) {
                ok = wait(ws.words[u], call) && ok;
                const unsigned long long w = ws.words[u].load(relaxed);
                if (!is_of(w, call) || (uint32_t)w != payload(call, u)) wrong.fetch_add(1, relaxed);
            }
        }
        if (!ok) status.fetch_or(kTimeoutBit, relaxed);
        leave(cta, s.ctas, call);
    }

    // ---- pairs
    static long long term(uint32_t call, int unit, uint32_t rank, int c) { return (long long)call * 1000003 + unit * 131 + rank * 17 + c; }
    void pair(int q, uint32_t rank) {
        const uint32_t call = call_number(ws.departures.load(relaxed));
        const int units = s.tiles * s.stages, begin = q < s.t_pairs ? share_begin(q, units, s.t_pairs) : 0, end = q < s.t_pairs ? share_begin(q + 1, units, s.t_pairs) : 0;
        bool ok = true, aborted = false;
        auto wait_word = [&](size_t at) {
            for (uint32_t spin = 0; !is_of(ws.words[at].load(std::memory_order_acquire), call); ++spin) {
                if (aborted) return false;
                if (spin > s.poll_limit) { aborted = true; expired.fetch_add(1, relaxed); return false; }
                std::this_thread::yield();
            }
            return true;
        };
        auto publish = [&](size_t at) { ws.words[at].store(tagged(call, 0), std::memory_order_release); };
        auto part = [&](int p, bool starts) { return ws.parts.data() + ((size_t)(2 * p + (starts ? 1 : 0)) * 2 + rank) * kColumns; };
        auto owner_of = [&](int unit) { return share_owner(unit, units, s.t_pairs); };
        const bool silent = withhold && q == 0;
        for (int u = begin; u < end && !silent;) {
            const Run run = run_at(u, end, s.stages);
            const bool whole = run.len == s.stages;
            long long* to = whole ? ws.sums.data() + ((size_t)run.tile * 2 + rank) * kColumns : part(q, run.k0 == 0);
            for (int c = 0; c < kColumns; ++c) {
                to[c] = 0;
                for (int i = 0; i < run.len; ++i) to[c] += term(call, u + i, rank, c);
            }
            publish(whole ? tile_word(s.t_pairs, run.tile, rank) : part_word(q, run.k0 == 0, rank));
            u += run.len;
        }
        for (int u = begin; u < end && !silent;) {
            const Run run = run_at(u, end, s.stages);
            u += run.len;
            if (run.len == s.stages) continue;
            const int q0 = owner_of(run.tile * s.stages), q1 = owner_of((run.tile + 1) * s.stages - 1);
            bool all = true;
            for (int p = q0; p <= q1; ++p) all = wait_word(part_word(p, p == q0, rank)) && all;
            ok = ok && all;
            for (int c = q - q0; c < kColumns && all; c += q1 - q0 + 1) {
                long long sum = 0;
                for (int p = q0; p <= q1; ++p) sum += part(p, p == q0)[c];
                ws.sums[((size_t)run.tile * 2 + rank) * kColumns + c] = sum;
            }
            publish(part_word(q, run.k0 == 0, rank) + 1);
        }
        for (int t = 0; t < s.tiles; ++t) {
            const int q0 = owner_of(t * s.stages), q1 = owner_of((t + 1) * s.stages - 1);
            bool all = true;
            for (int p = q0; p <= q1; ++p) all = wait_word(q0 == q1 ? tile_word(s.t_pairs, t, rank) : part_word(p, p == q0, rank) + 1) && all;
            ok = ok && all;
            for (int c = 0; c < kColumns; ++c) {
                long long want = 0;
                for (int i = 0; i < s.stages; ++i) want += term(call, t * s.stages + i, rank, c);
                if (!all || ws.sums[((size_t)t * 2 + rank) * kColumns + c] != want) { wrong.fetch_add(1, relaxed); break; }
            }
        }
        if (!ok) status.fetch_or(kTimeoutBit, relaxed);
        leave(2 * q + rank, 2 * s.pairs, call);
    }
};

int shares() {
    long long checked = 0;
    for (int pairs = 1; pairs <= 74; ++pairs)
        for (int tiles = 1; tiles <= 9; ++tiles)
            for (int stages : {1, 2, 3, 8, 27, 64, 128}) {
                const int units = tiles * stages;
                if (pairs > units) continue;
                std::set<size_t> places;
                size_t last = 0;
                for (int q = 0; q < pairs; ++q) {
                    const int b = share_begin(q, units, pairs), e = share_begin(q + 1, units, pairs);
                    for (int u = b; u < e; ++u) if (share_owner(u, units, pairs) != q) return 1;
                    int starting = 0, others = 0;
                    for (int u = b; u < e;) {
                        const Run run = run_at(u, e, stages);
                        if (run.len < 1 || run.tile * stages + run.k0 != u) return 2;
                        u += run.len;
                        for (uint32_t rank = 0; rank < 2; ++rank)
                            if (run.len == stages) places.insert(last = tile_word(pairs, run.tile, rank));
                            else for (int i = 0; i < 2; ++i) if (!places.insert(part_word(q, run.k0 == 0, rank) + i).second) return 3;
                        if (run.len < stages) ++(run.k0 == 0 ? starting : others);
                    }
                    if (starting > 1 || others > 1) return 4;
                    if (last >= (size_t)pairs * 8 + 2 * tiles) return 5;
                    ++checked;
                }
                if (share_begin(0, units, pairs) != 0 || share_begin(pairs, units, pairs) != units) return 6;
            }
    printf("shares %lld\n", checked);
    return 0;
}

}  // namespace

int main(int argc, char** argv) {
    if (argc == 2 && !strcmp(argv[1], "shares")) return shares();
    if (argc != 11) { fprintf(stderr, "usage: %s ctas makers words pairs t_pairs tiles stages calls withhold_call poll_limit\n", argv[0]); return 2; }
    auto arg = [&](int i) { return atoi(argv[i]); };
    const Shape s{arg(1), arg(2), arg(3), arg(4), arg(5), arg(6), arg(7), (uint32_t)strtoul(argv[10], nullptr, 10)};
    const int calls = arg(8), withhold = arg(9);
    if (s.makers < 1 || s.ctas <= s.makers || s.t_pairs < 1 || s.t_pairs > s.pairs || s.t_pairs > s.tiles * s.stages) return 2;
    Workspace ws(s);
    for (int k = 1; k <= calls; ++k) {
        const int kind = (k - 1) % 3;
        Call c(ws, s, k == withhold);
        std::vector<std::thread> th;
        if (kind == 0) for (int i = 0; i < s.ctas; ++i) th.emplace_back([&c, i] { c.small(i); });
        else if (kind == 1) for (int i = 0; i < 2 * s.pairs; ++i) th.emplace_back([&c, i] { c.pair(i / 2, (uint32_t)i & 1); });
        else for (int i = 0; i < 2 * s.pairs; ++i) th.emplace_back([&c, &ws, i, &s] { c.leave(i, 2 * s.pairs, call_number(ws.departures.load(relaxed))); });
        for (auto& t : th) t.join();                                            // a call ends when every CTA has left
        printf("call %d kind %d status %u number %u departures %llu wrong %d expired %d\n", k, kind, c.status.load(), c.number.load(), ws.departures.load(), c.wrong.load(), c.expired.load());
        if (c.status.load() != 0) { ws.reset(); printf("reset\n"); }            // the caller's duty after a time-out
    }
    return 0;
}
