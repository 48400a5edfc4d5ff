// Arena layouts with and without the small steps' results kept apart, for CPU tests: out[0] and
// out[1] arena bytes without and with them, out[2] their number.  Returns how many of the
// layouts' promises are broken (-1: planning failed): without, no step is marked; with, a small
// result shares no byte with any other tensor or gathered operand of the call.
#include <cstring>

#include "tn_internal.h"
#include "planner.cpp"
#include "arena.h"

void tn_set_error(const std::string &) {}

extern "C" int arena_small(const void *circ, size_t len, const int32_t *openq, int32_t n_open, const tn_plan_opts *o,
                           const uint64_t *slices, int64_t n_slices, int64_t *out) {
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
    CallLayout a, b;
    layout_call(tree, steps, E, 8, sv, a, false);
    layout_call(tree, steps, E, 8, sv, b);
    int bad = 0;
    for (char s : a.small) bad += s != 0;
    const auto &nodes = tree.nodes;
    struct R { size_t lo, hi; bool small; };
    std::vector<R> r;
    int n_small = 0;
    for (size_t i = 0; i < steps.size(); i++) {
        const Step &s = steps[i];
        const size_t bytes = (size_t)b.nver[s.c] * (size_t(1) << nodes[s.c].layout.size()) * 8;
        r.push_back({b.off[s.c], b.off[s.c] + bytes, b.small[i] != 0});
        n_small += b.small[i] != 0;
        for (int x = 0; x < 2; x++)
            if (s.gat[x]) {
                const int ch = x ? s.b : s.a;
                const long long nv = nodes[ch].ch[0] >= 0 ? b.nver[ch] : 1LL << __builtin_popcountll(nodes[ch].dep & E);
                r.push_back({b.goff[i][x], b.goff[i][x] + (size_t)nv * (size_t(1) << s.g_nbits[x]) * 8, false});
            }
    }
    for (size_t i = 0; i < r.size(); i++) {
        bad += r[i].hi > b.arena_bytes;
        for (size_t j = 0; j < r.size(); j++)
            bad += i != j && r[i].small && r[i].lo < r[j].hi && r[j].lo < r[i].hi;
    }
    out[0] = (int64_t)a.arena_bytes;
    out[1] = (int64_t)b.arena_bytes;
    out[2] = n_small;
    return bad;
}
