// Checks the edge table (build_edges) against the connections it was built from: for every
// edge and every time around them, the arrival by the kernels' lookup (slot, three inline
// departures, list) equals the least dep + dur over the edge's connections with dep >= time.
// Arguments: seed, stops, connections, latest departure, longest duration, cluster width, t0.
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

static int32_t lookup(const HostNet &h, int64_t i, int32_t e) {
    uint32_t rel;
    int32_t start;
    const uint32_t k = edge_slot(h.e_base, h.e_shift, e, rel, start);
    if (k >= (uint32_t)h.e_y) return EAT_INF;
    const int32_t *w = &h.ee[((size_t)k * h.etypes.size() + (size_t)i) * 4];
    const int4 c = {w[0], w[1], w[2], w[3]};
    const int32_t a = edge_inline(c, rel, start);
    if (a != EAT_INF || c.w == 0) return a;
    for (size_t p = 8 * ((size_t)c.w - 1);; p += 8) {
        if (p + 8 > h.ex.size()) {
            std::fprintf(stderr, "list without an end\n");
            std::exit(1);
        }
        for (int j = 0; j < 8; j += 2)
            if (h.ex[p + j] >= e) return h.ex[p + j + 1];
    }
}

int main(int argc, char **argv) {
    if (argc != 8) return 2;
    std::mt19937 rng((unsigned)std::atoi(argv[1]));
    const int V = std::atoi(argv[2]), C = std::atoi(argv[3]);
    const long t_max = std::atol(argv[4]), dur_max = std::atol(argv[5]);
    const int width = std::atoi(argv[6]);
    const long t0 = std::atol(argv[7]);
    auto draw = [&](long lo, long hi) { return std::uniform_int_distribution<long>(lo, hi)(rng); };
    std::vector<int32_t> u, v, dep, dur;
    for (int i = 0; i < C; ++i) {
        u.push_back((int32_t)draw(0, V - 1));
        v.push_back((int32_t)draw(0, V - 1));
        dep.push_back((int32_t)(t0 + draw(0, t_max)));
        dur.push_back((int32_t)draw(1, dur_max));
    }
    eat_connections c{V, C, u.data(), v.data(), dep.data(), dur.data(), nullptr};
    HostNet h;
    if (build_host(&c, width, (int32_t)t0, h) || build_fused(h) || build_edges(h)) return 1;
    std::map<std::pair<int32_t, int32_t>, std::vector<std::pair<int64_t, int64_t>>> edges;
    for (int i = 0; i < C; ++i) edges[{u[i], v[i]}].push_back({dep[i], (int64_t)dep[i] + dur[i]});
    if ((int64_t)edges.size() != (int64_t)h.etypes.size() || h.erow[V] != (int32_t)edges.size()) {
        std::fprintf(stderr, "%zu edges, not %zu\n", h.etypes.size(), edges.size());
        return 1;
    }
    int64_t types = 0, checked = 0;
    for (int32_t n : h.etypes) types += n;
    if (types != h.n_types) return 1;
    for (int32_t s = 0; s < V; ++s)
        for (int32_t i = h.erow[s]; i < h.erow[s + 1]; ++i) {
            const uint32_t x = (uint32_t)h.er[2 * (size_t)i];
            const int32_t head = (int32_t)(x & 0xffffffu);
            const int32_t deg = std::min(h.erow[head + 1] - h.erow[head], kEdgeOverflow);
            if ((int32_t)(x >> 28) != deg || h.er[2 * (size_t)i + 1] != h.erow[head]) return 1;
            // the head's edge back to s, where it is one of its first 15
            int32_t back = kEdgeOverflow;
            for (int32_t j = h.erow[head]; j < h.erow[head] + deg; ++j)
                if ((h.er[2 * (size_t)j] & 0xffffff) == s) back = j - h.erow[head];
            if ((int32_t)(x >> 24 & 15) != back) return 1;
            const auto &conns = edges.at({s, head});
            std::vector<int64_t> times = {INT32_MIN, t0 - 1, t0 + t_max + 1, INT32_MAX - 1, INT32_MAX};
            for (const auto &q : conns)
                for (int64_t t : {q.first - 1, q.first, q.first + 1, q.second}) times.push_back(t);
            for (int j = 0; j < 20; ++j) times.push_back(t0 + draw(0, t_max));
            for (int64_t t : times) {
                if (t < INT32_MIN || t > INT32_MAX) continue;
                int64_t want = EAT_INF;
                for (const auto &q : conns)
                    if (q.first >= t) want = std::min(want, q.second);
                const int32_t got = lookup(h, i, (int32_t)t);
                ++checked;
                if (got != want) {
                    std::fprintf(stderr, "edge %d -> %d at %lld: %d, not %lld\n", s, head, (long long)t, got,
                                 (long long)want);
                    return 1;
                }
            }
        }
    std::printf("%lld lookups, %d slots of %d s, %zu listed pairs\n", (long long)checked, h.e_y, 1 << h.e_shift,
                h.ex.size() / 2);
    return 0;
}
