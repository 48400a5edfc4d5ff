// Versions of every node for a slice set and the arena layout of one execution (host
// only; shared by the engine and a CPU test of its invariants).
//
// The arena is planned in step order: first fit, 256-byte granules, a node released after
// the step that consumes it, a gathered operand after its own step.  Batch-independent
// nodes consumed by batch steps (the stem kept for later batch groups) get a reserved
// prefix instead: batch-dependent tensors are rewritten in every group, so the two never
// share memory.  So do the results of small steps, which run out of step order (several to a
// launch, each as soon as its operands exist): see small_step.
#pragma once

#include <algorithm>
#include <array>
#include <cstddef>
#include <cstdint>
#include <unordered_map>
#include <vector>

#include "tn_internal.h"

// Sliced legs whose both values appear for every slice of the set (the set is closed
// under flipping them): those legs become layout bits, the others explicit versions.
inline uint64_t explicit_legs(const std::vector<uint64_t> &slices, int nI) {
    std::unordered_map<uint64_t, char> in;
    in.reserve(slices.size() * 2);
    for (uint64_t s : slices) in[s] = 1;
    uint64_t all = nI >= 64 ? ~0ull : ((1ull << nI) - 1);
    uint64_t fr = 0;
    for (int b = 0; b < nI; b++) {
        bool closed = true;
        for (uint64_t s : slices)
            if (!in.count(s ^ (1ull << b))) { closed = false; break; }
        if (closed) fr |= 1ull << b;
    }
    return all & ~fr;
}

struct CallLayout {
    std::vector<std::vector<uint64_t>> vals;             // per node: distinct versions
    std::vector<std::unordered_map<uint64_t, int>> index;
    std::vector<long long> nver;
    std::vector<size_t> off;
    std::vector<std::array<size_t, 2>> goff;  // per step: arena offsets of gathered operands
    std::vector<char> small;                  // per step: result kept in the reserved prefix
    size_t arena_bytes = 0;
    double flops = 0, flops_beta = 0;
};

// Steps cheap enough to share a launch: a launch costs 2 to 4 us in a replayed graph, about
// what 2^18 outputs over a short K take on the whole chip.  Their results (at most 2 MiB
// each, 48 MiB together) are never overwritten within an execution.  The memory estimates leave
// them out (they carry 64 MiB of slack), and an execution without room for them keeps its
// small steps in the arena like the others and runs them one by one.
constexpr long long kSmallOutputs = 1ll << 18, kSmallMacs = 1ll << 21, kSmallAlone = 1ll << 15;
constexpr size_t kSmallBytes = size_t(48) << 20;
inline bool small_step(const Step &s, long long nver) {
    const int out = s.nbat + s.nm + s.nn;
    return s.nk <= 6 && out <= 18 && (nver << out) <= kSmallOutputs && (nver << (out + s.nk)) <= kSmallMacs;
}

// Arena offsets of a call whose versions (L.nver) are known; small: the small steps' results
// get memory of their own in the reserved prefix.
inline void place_call(const Tree &tree, const std::vector<Step> &steps, uint64_t E, int elem, bool small, CallLayout &L) {
    const auto &nodes = tree.nodes;
    const int NN = (int)nodes.size();
    // arena: first fit, children released after their parent's step; beta-free
    // nodes consumed by beta steps stay alive (reused by later batch groups)
    auto tensor_bytes = [&](int x) {
        return (size_t)L.nver[x] * (size_t(1) << nodes[x].layout.size()) * (size_t)elem;
    };
    struct Blk { size_t off, len; };
    std::vector<Blk> freel;
    size_t top = 0;
    auto alloc = [&](size_t len) {
        len = (len + 255) & ~size_t(255);
        for (size_t i = 0; i < freel.size(); i++)
            if (freel[i].len >= len) {
                size_t o = freel[i].off;
                freel[i].off += len;
                freel[i].len -= len;
                if (!freel[i].len) freel.erase(freel.begin() + i);
                return o;
            }
        size_t o = top;
        top += len;
        return o;
    };
    auto dealloc = [&](size_t off, size_t len) {
        len = (len + 255) & ~size_t(255);
        freel.push_back({off, len});
        std::sort(freel.begin(), freel.end(), [](const Blk &a, const Blk &b) { return a.off < b.off; });
        std::vector<Blk> merged;
        for (auto &b : freel) {
            if (!merged.empty() && merged.back().off + merged.back().len == b.off) merged.back().len += b.len;
            else merged.push_back(b);
        }
        if (!merged.empty() && merged.back().off + merged.back().len == top) { top = merged.back().off; merged.pop_back(); }
        freel.swap(merged);
    };
    // Stem tensors kept for later batch groups (batch-free, consumed by a batch step)
    // get a reserved prefix: batch-dependent tensors are rewritten in every group, so
    // the two must never share memory.
    std::vector<char> keep(NN, 0);
    for (const Step &s : steps)
        for (int ch : {s.a, s.b})
            if (nodes[ch].ch[0] >= 0 && !nodes[ch].beta && nodes[s.c].beta) keep[ch] = 1;
    L.small.assign(steps.size(), 0);
    size_t small_bytes = 0;
    for (size_t i = 0; i < steps.size(); i++) {
        const Step &s = steps[i];
        if (!small || s.c == tree.root || !small_step(s, L.nver[s.c])) continue;
        const size_t b = (tensor_bytes(s.c) + 255) & ~size_t(255);
        if (small_bytes + b > kSmallBytes) continue;
        small_bytes += b;
        L.small[i] = 1;
        keep[s.c] = 1;
    }
    size_t reserved = 0;
    L.off.assign(NN, 0);
    for (const Step &s : steps)
        if (keep[s.c]) {
            L.off[s.c] = reserved;
            reserved += (tensor_bytes(s.c) + 255) & ~size_t(255);
        }
    size_t peak = 0;
    L.flops = L.flops_beta = 0;
    L.goff.assign(steps.size(), {0, 0});
    auto nver_of = [&](int x) -> long long {
        if (nodes[x].ch[0] >= 0) return L.nver[x];
        return 1LL << __builtin_popcountll(nodes[x].dep & E);  // leaf codes
    };
    for (size_t i = 0; i < steps.size(); i++) {
        const Step &s = steps[i];
        // gathered operands live for the step only
        size_t gbytes[2] = {0, 0};
        for (int o = 0; o < 2; o++)
            if (s.gat[o]) {
                gbytes[o] = (size_t)nver_of(o ? s.b : s.a) * (size_t(1) << s.g_nbits[o]) * (size_t)elem;
                L.goff[i][o] = reserved + alloc(gbytes[o]);
            }
        if (!keep[s.c]) L.off[s.c] = reserved + alloc(tensor_bytes(s.c));
        peak = std::max(peak, top);
        for (int o = 0; o < 2; o++)
            if (s.gat[o]) dealloc(L.goff[i][o] - reserved, gbytes[o]);
        for (int ch : {s.a, s.b})
            if (nodes[ch].ch[0] >= 0 && !keep[ch]) dealloc(L.off[ch] - reserved, tensor_bytes(ch));
        const double fl = s.flops_per_version * (double)L.nver[s.c];
        L.flops += fl;
        if (nodes[s.c].beta) L.flops_beta += fl;
    }
    L.arena_bytes = std::max<size_t>(reserved + peak, 256);
}

// Versions and arena of a call; small: the small steps' results are kept apart, unless that
// costs more than kSmallBytes (a first fit can do worse with fewer tensors).
inline void layout_call(const Tree &tree, const std::vector<Step> &steps, uint64_t E, int elem,
                 const std::vector<uint64_t> &slices, CallLayout &L, bool small = true) {
    const auto &nodes = tree.nodes;
    const int NN = (int)nodes.size();
    L.vals.assign(NN, {});
    L.index.assign(NN, {});
    L.nver.assign(NN, 0);
    for (int x = 0; x < NN; x++) {
        const uint64_t D = nodes[x].dep & E;
        for (uint64_t s : slices) {
            uint64_t w = s & D;
            if (L.index[x].emplace(w, (int)L.vals[x].size()).second) L.vals[x].push_back(w);
        }
        L.nver[x] = (long long)L.vals[x].size();
    }
    place_call(tree, steps, E, elem, false, L);
    if (!small) return;
    const size_t least = L.arena_bytes;
    place_call(tree, steps, E, elem, true, L);
    if (L.arena_bytes > least + kSmallBytes) place_call(tree, steps, E, elem, false, L);
}

// The launches of an execution, in order: each a group of small steps that run together
// (shared), or one step by itself.
struct LaunchItem {
    std::vector<int> steps;
    bool shared;
};

// The launch order with the small steps grouped (small: the steps that may be, a subset of
// L.small); skip_stem: without the batch-independent steps.  Every small step whose operands
// exist runs in the next shared launch, and when none is ready the next other step follows.
// The other steps keep their order and a small step never runs later than its place in it, so
// the arena's reuse (planned in step order) holds; the small steps' own results are never
// reused.
inline std::vector<LaunchItem> launch_order(const Tree &tree, const std::vector<Step> &steps, const std::vector<char> &small,
                                            const std::vector<long long> &nver, bool skip_stem) {
    std::vector<LaunchItem> out;
    std::vector<char> done(tree.nodes.size(), 1);
    std::vector<int> todo;
    for (size_t i = 0; i < steps.size(); i++)
        if (!skip_stem || tree.nodes[steps[i].c].beta) todo.push_back((int)i);
    for (int i : todo) done[steps[i].c] = 0;
    // one ready step alone shares a launch too if it is tiny (it may join a chain) or would need a
    // gather launch
    auto alone = [&](int i) {
        const Step &s = steps[i];
        return s.gat[0] || s.gat[1] || (nver[s.c] << (s.nbat + s.nm + s.nn)) <= kSmallAlone;
    };
    while (!todo.empty()) {
        std::vector<int> ready, rest;
        for (int i : todo) {
            const Step &s = steps[i];
            (small[i] && done[s.a] && done[s.b] ? ready : rest).push_back(i);
        }
        const bool shared = ready.size() > 1 || (ready.size() == 1 && alone(ready[0]));
        if (ready.empty()) {
            ready.push_back(rest[0]);
            rest.erase(rest.begin());
        }
        for (int i : ready) done[steps[i].c] = 1;
        out.push_back({ready, shared});
        todo.swap(rest);
    }
    return out;
}
