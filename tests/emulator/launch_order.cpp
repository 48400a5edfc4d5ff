// The launch order of an execution against the arena it runs in, for CPU tests: two executions in
// turn (all steps, then a later batch group that reuses the stem), every launch's writes
// ending the life of what they overlap.  Counts the operands that no longer hold their tensor
// when a launch reads them, writes over an operand of the same launch, and steps that did
// not run exactly once; -1: planning failed.  out[0] shared launches, out[1] steps that ran
// ahead of their place.  plant 1: the small results laid out like the others', 2: an order
// that runs the small steps last.
#include <cstring>

#include "tn_internal.h"
#include "planner.cpp"
#include "arena.h"

void tn_set_error(const std::string &) {}

extern "C" int launch_order_check(const void *circ, size_t len, const int32_t *openq, int32_t n_open, const tn_plan_opts *o,
                                  const uint64_t *slices, int64_t n_slices, int plant, int64_t *out) {
    tn_circuit_s c;
    if (tn_parse_circuit(circ, len, &c)) return -1;
    Merged mg;
    tn_merge(c, mg);
    std::vector<int> openv(openq, openq + n_open), closed;
    std::vector<tn_edge> I;
    Network net;
    Tree tree;
    std::vector<Step> steps;
    uint64_t E0 = 0;
    if (tn_plan_build_host(mg, *o, nullptr, 0, nullptr, 0, openv, I, net, tree, steps, closed, &E0)) return -1;
    const std::vector<uint64_t> sv(slices, slices + n_slices);
    const uint64_t E = explicit_legs(sv, (int)I.size());
    if (tn_compile(net, tree, E, steps, o->precision != TN_PREC_C64)) return -1;
    CallLayout L;
    layout_call(tree, steps, E, 8, sv, L);
    const std::vector<char> small = L.small;
    if (plant == 1) place_call(tree, steps, E, 8, false, L);
    const auto &nodes = tree.nodes;
    const int S = (int)steps.size();
    struct R { size_t lo, hi; };
    auto overlap = [](const R &a, const R &b) { return a.lo < b.hi && b.lo < a.hi; };
    auto at = [&](int x) { return R{L.off[x], L.off[x] + (size_t)L.nver[x] * (size_t(1) << nodes[x].layout.size()) * 8}; };
    auto copy_at = [&](int i, int w) {  // the gathered copy of operand w of step i
        const int x = w ? steps[i].b : steps[i].a;
        const long long nv = nodes[x].ch[0] >= 0 ? L.nver[x] : 1LL << __builtin_popcountll(nodes[x].dep & E);
        return R{L.goff[i][w], L.goff[i][w] + (size_t)nv * (size_t(1) << steps[i].g_nbits[w]) * 8};
    };
    std::vector<char> alive(nodes.size(), 0);  // the node's memory holds its tensor
    int bad = 0;
    out[0] = out[1] = 0;
    for (int skip = 0; skip < 2; skip++) {
        std::vector<LaunchItem> order = launch_order(tree, steps, small, L.nver, skip != 0);
        if (plant == 2) std::stable_partition(order.begin(), order.end(), [](const LaunchItem &t) { return !t.shared; });
        std::vector<int> runs(S, 0);
        int seen = -1;  // the last step by itself
        for (const LaunchItem &t : order) {
            out[0] += t.shared;
            std::vector<R> reads, writes;
            for (int i : t.steps) {
                const Step &s = steps[i];
                runs[i]++;
                if (t.shared || small[i]) out[1] += i > seen + 1;
                else seen = i;
                for (int w = 0; w < 2; w++) {
                    const int x = w ? s.b : s.a;
                    if (nodes[x].ch[0] >= 0) {
                        bad += !alive[x];
                        reads.push_back(at(x));
                    }
                    // shared launches read gathered operands in place, others through a copy
                    if (s.gat[w] && !t.shared) writes.push_back(copy_at(i, w));
                }
                writes.push_back(at(s.c));
            }
            for (size_t u = 0; u < writes.size(); u++) {
                for (const R &r : reads) bad += overlap(writes[u], r);
                for (size_t v = 0; v < u; v++) bad += overlap(writes[u], writes[v]);
                for (int x = 0; x < (int)nodes.size(); x++)
                    if (alive[x] && overlap(writes[u], at(x))) alive[x] = 0;
            }
            for (int i : t.steps) alive[steps[i].c] = 1;
        }
        for (int i = 0; i < S; i++) bad += runs[i] != (skip && !nodes[steps[i].c].beta ? 0 : 1);
        bad += !alive[tree.root];
    }
    return bad;
}
