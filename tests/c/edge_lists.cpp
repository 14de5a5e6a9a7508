// Looks up an uneven timetable in the edge table (build_edges) as the round kernel does, with the
// tables of long lists, against the connections; and counts what a lookup loads: an entry, at most
// one table entry per level (a slot of 2^15 s has three) and three quads of a list.
// Arguments: seed, stops, connections of the rare edges, headway of the busy ones, days, extra day.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <random>

#include "eat_internal.h"

namespace eat {
int fail(int code, const std::string &msg) {
    std::fprintf(stderr, "%s\n", msg.c_str());
    return code;
}
void clear_error() {}
}  // namespace eat

using namespace eat;

static int loads;

static int4 quad_half(const HostNet &h, int64_t half) {
    if (half < 0 || 4 * (size_t)half + 4 > h.ex.size()) {
        std::fprintf(stderr, "outside the lists\n");
        std::exit(1);
    }
    const int32_t *w = &h.ex[4 * (size_t)half];
    return {w[0], w[1], w[2], w[3]};
}

static int32_t lookup(const HostNet &h, int64_t i, int32_t e) {
    uint32_t rel;
    int32_t start;
    const uint32_t k = std::min(edge_slot(h.e_base, h.e_shift, e, rel, start), (uint32_t)h.e_y);
    const int32_t *w = &h.ee[((size_t)k * h.etypes.size() + (size_t)i) * 4];
    int4 c = {w[0], w[1], w[2], w[3]};
    loads = 1;
    const int32_t a = edge_inline(c, rel, start);
    if (a != EAT_INF || c.w == 0) return a;
    int64_t at = 2 * ((int64_t)c.w - 1);                    // in halves of a quad
    if ((c.w & 7) == 0) {
        at -= kSubSlots;
        for (int32_t shift = h.e_shift;;) {
            shift -= kSubLog2;
            if (shift < 0) std::exit(1);
            const int32_t part = edge_part(shift, rel, start);
            c = quad_half(h, at + part);
            ++loads;
            const int32_t b = edge_inline(c, rel, start);
            if (b != EAT_INF || c.w == 0) return b;
            at = 2 * ((int64_t)std::abs(c.w) - 1);
            if (c.w > 0) break;
        }
    }
    for (;; at += 2) {
        const int4 x = quad_half(h, at), y = quad_half(h, at + 1);
        ++loads;
        for (const auto &q : {std::make_pair(x.x, x.y), std::make_pair(x.z, x.w), std::make_pair(y.x, y.y),
                              std::make_pair(y.z, y.w)})
            if (q.first >= e) return q.second;
    }
}

int main(int argc, char **argv) {
    if (argc != 7) return 2;
    std::mt19937 rng((unsigned)std::atoi(argv[1]));
    const int V = std::atoi(argv[2]), rare = std::atoi(argv[3]), headway = std::atoi(argv[4]);
    const int days = std::atoi(argv[5]), extra = std::atoi(argv[6]);
    auto draw = [&](long lo, long hi) { return (int32_t)std::uniform_int_distribution<long>(lo, hi)(rng); };
    std::vector<int32_t> u, v, dep, dur;
    auto add = [&](int32_t a, int32_t b, int32_t t, int32_t l) {
        u.push_back(a);
        v.push_back(b);
        dep.push_back(t);
        dur.push_back(l);
    };
    for (int i = 0; i < rare; ++i) add(draw(0, V - 1), draw(0, V - 1), draw(0, 86400L * days), draw(1, 90000));
    for (int s = 0; s < 3; ++s)                             // busy edges 0 -> 1 -> 2 -> 3, the last one bunched
        for (int32_t t = draw(0, 100); t < 86400 * days; t += s < 2 ? headway : draw(1, 2 * headway))
            add(s, s + 1, t, s == 1 ? draw(30, 900) : 200);
    if (extra) add(0, 1, 86400 * extra, 60);
    eat_connections c{V, (int64_t)u.size(), u.data(), v.data(), dep.data(), dur.data(), nullptr};
    HostNet h;
    if (build_host(&c, 3600, 0, h) || build_fused(h) || build_edges(h)) return 1;
    std::map<std::pair<int32_t, int32_t>, std::map<int32_t, int32_t>> edges;      // departure -> least arrival
    for (size_t i = 0; i < u.size(); ++i) {
        int32_t &a = edges[{u[i], v[i]}].emplace(dep[i], EAT_INF).first->second;
        a = std::min(a, dep[i] + dur[i]);
    }
    for (auto &e : edges) {                                 // and of any later departure
        int32_t best = EAT_INF;
        for (auto p = e.second.rbegin(); p != e.second.rend(); ++p) p->second = best = std::min(best, p->second);
    }
    int64_t checked = 0;
    int most = 0;
    for (int32_t s = 0; s < V; ++s)
        for (int32_t i = h.erow[s]; i < h.erow[s + 1]; ++i) {
            const auto &conns = edges.at({s, h.er[2 * (size_t)i] & 0xffffff});
            std::vector<int64_t> times = {INT32_MIN, -1, INT32_MAX};
            for (const auto &q : conns)
                for (int64_t t : {(int64_t)q.first - 1, (int64_t)q.first, (int64_t)q.first + 1}) times.push_back(t);
            for (int j = 0; j < 30; ++j) times.push_back(draw(0, 86400L * (std::max(days, extra) + 1)));
            for (int64_t t : times) {
                const auto q = conns.lower_bound((int32_t)t);
                const int32_t want = q == conns.end() ? EAT_INF : q->second, got = lookup(h, i, (int32_t)t);
                ++checked;
                most = std::max(most, loads);
                if (got != want) {
                    std::fprintf(stderr, "%d -> edge %d at %lld: %d, not %d\n", s, i, (long long)t, got, want);
                    return 1;
                }
            }
        }
    std::printf("%lld lookups, %d slots of %d s, %zu words of lists, %d loads at most\n", (long long)checked, h.e_y,
                1 << h.e_shift, h.ex.size(), most);
    return most <= 1 + 3 + 3 ? 0 : 1;
}
