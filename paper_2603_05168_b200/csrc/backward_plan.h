// Which output tiles of the backward GEMMs each CTA pair computes.
//
// The two parts (0: dW, 1: dX) have tiles of 256 x 256 whose lengths differ: a tile of dW runs over the tokens, one of dX
// over the features.  Longest tiles first, every further tile to the pair with the least to do; the last tiles of the
// shorter kind are cut into halves of 128 columns where that lowers the longest pair (a half costs about 0.65 of a whole:
// the loads of A are the same).  With whole waves per launch instead (fewest waves, one launch per part, the second moving
// in as pairs of the first end) 2560 -> 2560 at 4096 tokens took 95 us of GEMM where its tiles add up to 64; now 72.
#pragma once

#include <algorithm>

namespace sbn {

constexpr int kBackwardPairs = 74;               // one CTA per SM

// Entry i of a pair: index i * pairs + pair in the first `rounds` rounds, which every pair takes part in (so the pairs work
// on neighbouring tiles and share their operands in L2; a run of consecutive tiles per pair instead made a training step
// 1 % slower), then rounds * pairs + start[pair] + i - rounds.  An index is a whole tile, or a half of tile first_tile + index / 2.
struct BackwardSegment {
    int part, half, first_tile, rounds;
    int start[kBackwardPairs + 1];
#ifdef __CUDACC__
    __host__ __device__
#endif
    int count(int pair) const { return rounds + start[pair + 1] - start[pair]; }
#ifdef __CUDACC__
    __host__ __device__
#endif
    int index(int pair, int i) const { return i < rounds ? i * kBackwardPairs + pair : rounds * kBackwardPairs + start[pair] + i - rounds; }
};
struct BackwardPlan {
    int segments;
    BackwardSegment seg[3];                      // in the order of execution
};

// The pairs while they are being given work: runs of neighbouring pairs with the same load and the same item counts.  There are
// a handful (every step splits at most one run per round of leftovers), so a plan costs the host 1 to 2 us; pair by pair it was 9.
struct BackwardRun {
    int begin, end;                              // pairs
    double load;
    int n[3];                                    // items: long tiles, whole short tiles, halves of short tiles
};
struct BackwardRuns {
    int count = 1;
    BackwardRun r[kBackwardPairs];
    BackwardRuns() { r[0] = BackwardRun{0, kBackwardPairs, 0.0, {0, 0, 0}}; }
    BackwardRuns(const BackwardRuns& o) { *this = o; }
    BackwardRuns& operator=(const BackwardRuns& o) {        // the runs in use
        count = o.count;
        std::copy(o.r, o.r + o.count, r);
        return *this;
    }

    // Adds `items` items of length `cost`, counted in n[kind], to the least loaded pairs.
    void spread(int kind, int items, double cost) {
        if (items <= 0) return;
        double lo = r[0].load, total = 0.0;
        for (int i = 0; i < count; ++i) { lo = std::min(lo, r[i].load); total += r[i].load * (r[i].end - r[i].begin); }
        double hi = std::max(total / kBackwardPairs, lo) + cost * (items / kBackwardPairs + 2);
        // the highest level up to which all pairs can be filled with the items there are
        const double inv = 1.0 / cost;
        for (int it = 0; it < 10; ++it) {
            const double mid = 0.5 * (lo + hi);
            long used = 0;
            for (int i = 0; i < count; ++i)
                if (r[i].load < mid) used += static_cast<long>(static_cast<int>((mid - r[i].load) * inv)) * (r[i].end - r[i].begin);
            if (used <= items) lo = mid; else hi = mid;
        }
        int left = items;
        for (int i = 0; i < count; ++i)
            if (r[i].load < lo) {
                const int each = static_cast<int>((lo - r[i].load) * inv);
                r[i].n[kind] += each;
                r[i].load += each * cost;
                left -= each * (r[i].end - r[i].begin);
            }
        while (left > 0) {                       // one each to the least loaded: fewer than the pairs, or a few rounds of them
            const int seen = count;              // parts split off below wait for the next round
            bool served[kBackwardPairs] = {};
            for (int round_left = std::min(left, kBackwardPairs); round_left > 0;) {
                int at = -1;
                for (int i = 0; i < seen; ++i)
                    if (!served[i] && (at < 0 || r[i].load < r[at].load || (r[i].load == r[at].load && r[i].begin < r[at].begin))) at = i;
                served[at] = true;
                const int take = std::min(round_left, r[at].end - r[at].begin);
                if (take < r[at].end - r[at].begin) {
                    r[count] = r[at];
                    r[count++].begin = r[at].begin + take;
                    r[at].end = r[at].begin + take;
                }
                ++r[at].n[kind];
                r[at].load += cost;
                round_left -= take;
                left -= take;
            }
        }
    }
    double longest() const {
        double top = 0.0;
        for (int i = 0; i < count; ++i) top = std::max(top, r[i].load);
        return top;
    }
};

// tiles[part], stages[part] (64 contraction steps each).  split_hint (diagnostics): 0 no halves, 1 halves only, else as is best.
inline BackwardPlan plan_backward(const int (&tiles)[2], const int (&stages)[2], int split_hint) {
    const int lng = (tiles[1] > 0 && (tiles[0] == 0 || stages[1] >= stages[0])) ? 1 : 0;
    const int sht = tiles[1 - lng] > 0 ? 1 - lng : lng;                     // a single part is both
    // In stages (0.36 us): a tile's loads and MMAs, or its output if that takes longer, and the turnaround.  256 KB in fp32 resp.
    // 128 KB in bf16 take 15 resp. 7.5 at the 47 GB/s per pair that the memory takes; beside dW's fp32 its loads take half their
    // time again (with 15 alone the pairs that write most ended last: 54 sizes of 256 to 2048 tokens 3.5 % slower, 11008 x 4096 at 777
    // 208 us against 186).
    const double out_w = 15.0 + 0.5 * stages[0];
    auto full = [&](int part) { return std::max(stages[part] * 1.0, part == 0 ? out_w : 7.5) + 3.0; };
    auto half = [&](int part) { return std::max(stages[part] * 0.65, part == 0 ? 0.5 * out_w : 3.75) + 3.0; };
    const bool long_cut = split_hint >= 0 ? split_hint != 0 : 2 * tiles[lng] <= kBackwardPairs;   // too few to go round: all in halves
    BackwardRuns long_placed;
    if (sht != lng) long_placed.spread(0, long_cut ? 2 * tiles[lng] : tiles[lng], long_cut ? half(lng) : full(lng));
    double best_top = 1e300;
    BackwardRuns best;
    int best_h = 0, excess = 0;
    for (int option = 0; option < 4; ++option) {
        int h = 0;                                                          // tiles cut in two
        if (option == 1) h = excess;
        else if (option == 2) h = std::min(tiles[sht], excess + kBackwardPairs / 2);
        else if (option == 3) h = tiles[sht] <= kBackwardPairs ? tiles[sht] : 0;
        if (split_hint >= 0) h = split_hint ? tiles[sht] : 0;
        if (option > 0 && (h == 0 || split_hint >= 0)) continue;
        BackwardRuns runs = long_placed;
        runs.spread(1, tiles[sht] - h, full(sht));
        runs.spread(2, 2 * h, half(sht));
        const double top = runs.longest();
        if (option == 0)
            for (int i = 0; i < runs.count; ++i)
                if (runs.r[i].n[1] > 0 && runs.r[i].load > top - 0.5 * full(sht)) excess += runs.r[i].end - runs.r[i].begin;
        if (top < best_top * 0.999) {
            best_top = top;
            best_h = h;
            best = runs;
        }
    }
    BackwardPlan plan;
    plan.segments = 0;
    auto add = [&](int part, int is_half, int first_tile, int kind) {
        BackwardSegment& s = plan.seg[plan.segments];
        s.part = part; s.half = is_half; s.first_tile = first_tile;
        s.rounds = best.r[0].n[kind];
        for (int i = 1; i < best.count; ++i) s.rounds = std::min(s.rounds, best.r[i].n[kind]);
        int extra[kBackwardPairs];                                          // beyond the rounds, by pair
        for (int i = 0; i < best.count; ++i)
            for (int p = best.r[i].begin; p < best.r[i].end; ++p) extra[p] = best.r[i].n[kind] - s.rounds;
        s.start[0] = 0;
        for (int p = 0; p < kBackwardPairs; ++p) s.start[p + 1] = s.start[p] + extra[p];
        if (s.rounds > 0 || s.start[kBackwardPairs] > 0) ++plan.segments;
    };
    for (int part = 0; part < 2; ++part) {
        if (part == sht) {
            add(part, 0, 0, 1);
            add(part, 1, tiles[sht] - best_h, 2);
        } else if (part == lng) {
            add(part, long_cut ? 1 : 0, 0, 0);
        }
    }
    return plan;
}

}  // namespace sbn
