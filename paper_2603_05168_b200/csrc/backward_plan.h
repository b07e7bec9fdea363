// Which output tiles of the backward GEMMs each CTA pair computes.
//
// The two parts (0: dW, 1: dX) have tiles of 256 x 256 whose lengths differ: a tile of dW runs over the tokens, one of dX
// over the features.  Longest tiles first, every further tile to the pair with the least to do; the last tiles of the
// shorter kind are cut into halves of 128 columns where that lowers the longest pair (a half costs about 0.65 of a whole:
// the loads of A are the same).  With whole waves per launch instead (fewest waves, one launch per part, the second moving
// in as pairs of the first end) 2560 -> 2560 at 4096 tokens took 95 us of GEMM where its tiles add up to 64; now 72.
// Planning takes 10 to 20 us on the host, once per call of 25 (64 tokens) to 210 us (4096).
#pragma once

#include <algorithm>
#include <cmath>

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
    int segments, pairs;
    BackwardSegment seg[3];                      // in the order of execution
};

// Adds `count` items of length `cost` to the least loaded pairs; n[p] = how many pair p got.
inline void backward_spread(int count, double cost, double (&load)[kBackwardPairs], int (&n)[kBackwardPairs]) {
    for (int p = 0; p < kBackwardPairs; ++p) n[p] = 0;
    if (count <= 0) return;
    double lo = load[0], total = 0.0;
    for (int p = 0; p < kBackwardPairs; ++p) { lo = std::min(lo, load[p]); total += load[p]; }
    double hi = std::max(total / kBackwardPairs, lo) + cost * (count / kBackwardPairs + 2);
    // the highest level up to which all pairs can be filled with the items there are
    const double inv = 1.0 / cost;
    for (int it = 0; it < 10; ++it) {
        const double mid = 0.5 * (lo + hi);
        long used = 0;
        for (int p = 0; p < kBackwardPairs; ++p)
            if (load[p] < mid) used += static_cast<int>((mid - load[p]) * inv);
        if (used <= count) lo = mid; else hi = mid;
    }
    int left = count;
    for (int p = 0; p < kBackwardPairs; ++p)
        if (load[p] < lo) {
            n[p] = std::min(left, static_cast<int>((lo - load[p]) * inv));
            load[p] += n[p] * cost;
            left -= n[p];
        }
    while (left > 0) {                           // fewer than the pairs, or a few rounds of them
        int order[kBackwardPairs];
        for (int p = 0; p < kBackwardPairs; ++p) order[p] = p;
        const int take = std::min(left, kBackwardPairs);
        std::partial_sort(order, order + take, order + kBackwardPairs, [&](int a, int b) { return load[a] < load[b] || (load[a] == load[b] && a < b); });
        for (int i = 0; i < take; ++i) { ++n[order[i]]; load[order[i]] += cost; }
        left -= take;
    }
}

// tiles[part], stages[part] (64 contraction steps each); `first` runs first.  split_hint (diagnostics): 0 no halves, 1 halves only.
inline BackwardPlan plan_backward(const int (&tiles)[2], const int (&stages)[2], int first, int split_hint, double* longest) {
    const int lng = (tiles[1] > 0 && (tiles[0] == 0 || stages[1] >= stages[0])) ? 1 : 0;
    const int sht = tiles[1 - lng] > 0 ? 1 - lng : lng;                     // a single part is both
    // In stages (0.36 us): a tile's loads and MMAs, or its output if that takes longer (256 KB in fp32 resp. 128 KB in bf16 at
    // the 47 GB/s per pair that the memory takes), and the turnaround.
    auto full = [&](int part) { return std::max(stages[part] * 1.0, part == 0 ? 15.0 : 7.5) + 3.0; };
    auto half = [&](int part) { return std::max(stages[part] * 0.65, part == 0 ? 7.5 : 3.75) + 3.0; };
    const bool long_cut = split_hint >= 0 ? split_hint != 0 : 2 * tiles[lng] <= kBackwardPairs;   // too few to go round: all in halves
    double best = 1e300;
    int best_long[kBackwardPairs] = {}, best_short[kBackwardPairs] = {}, best_half[kBackwardPairs] = {}, best_h = 0;
    int excess = 0;
    for (int option = 0; option < 4; ++option) {
        int h = 0;                                                          // tiles cut in two
        if (option == 1) h = excess;
        else if (option == 2) h = std::min(tiles[sht], excess + kBackwardPairs / 2);
        else if (option == 3) h = tiles[sht] <= kBackwardPairs ? tiles[sht] : 0;
        if (split_hint >= 0) h = split_hint ? tiles[sht] : 0;
        if (option > 0 && (h == 0 || split_hint >= 0)) continue;
        double load[kBackwardPairs] = {};
        int nl[kBackwardPairs] = {}, ns[kBackwardPairs], nh[kBackwardPairs];
        if (sht != lng) backward_spread(long_cut ? 2 * tiles[lng] : tiles[lng], long_cut ? half(lng) : full(lng), load, nl);
        backward_spread(tiles[sht] - h, full(sht), load, ns);
        backward_spread(2 * h, half(sht), load, nh);
        const double top = *std::max_element(load, load + kBackwardPairs);
        if (option == 0)
            for (int p = 0; p < kBackwardPairs; ++p)
                if (ns[p] > 0 && load[p] > top - 0.5 * full(sht)) ++excess;
        if (top < best * 0.999) {
            best = top;
            best_h = h;
            std::copy(nl, nl + kBackwardPairs, best_long);
            std::copy(ns, ns + kBackwardPairs, best_short);
            std::copy(nh, nh + kBackwardPairs, best_half);
        }
    }
    if (longest) *longest = best;
    BackwardPlan plan;
    plan.segments = 0;
    plan.pairs = kBackwardPairs;
    auto add = [&](int part, int is_half, int first_tile, const int* n) {
        BackwardSegment& s = plan.seg[plan.segments];
        s.part = part; s.half = is_half; s.first_tile = first_tile;
        s.rounds = *std::min_element(n, n + kBackwardPairs);
        s.start[0] = 0;
        for (int p = 0; p < kBackwardPairs; ++p) s.start[p + 1] = s.start[p] + n[p] - s.rounds;
        if (s.rounds > 0 || s.start[kBackwardPairs] > 0) ++plan.segments;
    };
    for (const int part : {first, 1 - first}) {
        if (part == sht) {
            add(part, 0, 0, best_short);
            add(part, 1, tiles[sht] - best_h, best_half);
        } else if (part == lng) {
            add(part, long_cut ? 1 : 0, 0, best_long);
        }
    }
    return plan;
}

}  // namespace sbn
