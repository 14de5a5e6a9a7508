// Internal declarations shared by libeat's translation units (not installed).
#pragma once

#include <stdint.h>
#include <stddef.h>

#include <atomic>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include <vector_types.h>

#include "eat.h"

// Functions that the kernels and the host (tests of the layouts) share.
#ifdef __CUDACC__
#define EAT_HD __host__ __device__
#else
#define EAT_HD
#endif

namespace eat {

// Device-side descriptor of one resident network (plain pointers into one blob).
//
// Device layout (derived from the logical arrays of HostNet by build_fused):
//   tr[t]         16-byte record of connection type t: {v, lambda | d << 24, row_ptr[v],
//                 last departure}: head stop, duration, types leaving v (255 = read
//                 row_ptr), the head's first type, and the type's last departure
//   ce[k*T + t]   32-byte entry of type t for cluster k_min + k, for every cluster
//                 of the network (the paper's dense CL table, cluster-major so that
//                 lookups at nearby times fall in one slab of T entries), read in
//                 one load:
//                   int4 {rel0 | rel1 << 16, sc0, sc1, next}
//                   int4 {x/2 | n << 24, rel2 | rel3 << 16, sc2, sc3}
//                 the cluster's n APs: the first four inline with first terms
//                 base + rel (base = t0 + (k_min + k) * width) and
//                 sc = (difference << 16) | terms, the others at apx[x ..] (x even);
//                 n = 255 means more: the true count heads the list in two slots;
//                 next = first departure of the next non-empty cluster (INF if none)
//   apx[]         uint2 {first term, sc} of the fifth and later APs of a cluster
//   row_ptr[V+1]  types leaving stop u are row_ptr[u] .. row_ptr[u+1]-1
// and the edge table that the round kernel reads (see EdgeDev; build_edges).
constexpr int32_t kCountOverflow = 255;
constexpr int32_t kMaxDuration = 1 << 24;
constexpr int32_t kInlineAps = 4;

// The network by edges (u, v) and time slots of 2^shift seconds.  An edge's connections of
// every duration are merged into one list ordered by departure, without those that another
// one dominates (departs no earlier, arrives no later): the earliest arrival over the edge
// for a tail reached at e is then the arrival of the first listed departure >= e, one
// relaxation for the edge instead of one per connection type (Section II-E).
//   er[i]        8-byte record of edge i = (u, v): {v | b << 24 | d << 28, erow[v]}: head stop,
//                edges leaving it (15 = read erow), which of them goes back to u (15 = none
//                of the first 15), its first edge; networks of more than 2^24 stops:
//                {v, erow[v]}, d always read from erow
//   ee[k*E + i]  16-byte entry of edge i for slot k of y + 1, slot-major (the last one, for tails
//                reached after slot y - 1, holds no departures; a round's lookups are at
//                nearby times and fall in few slabs): the listed departures inside the slot
//                and the first one after it, the first three as 16-bit numbers
//                {d0 | l0 << 16, d1 | l1 << 16, d2 | l2 << 16, x}: departure d (relative to
//                the slot's start, 0xffff = none), duration l; the others (or values that
//                do not fit 16 bits) from ex[4 * (x - 1)] on, x = 0 if there are none
//   ex[]         {departure, arrival} pairs, each list a multiple of four pairs (32 bytes, a
//                quad) ended by the first departure after the slot or by {INF, INF}.  A list of
//                more than kLongList pairs, and no other, has x a multiple of 8, and its table in
//                the 8 quads before it: 16 entries like ee's, one for each sixteenth of the slot,
//                whose x > 0 is the quad of the list to go on from and x < 0 the table at quad
//                -x - 1, of sixteenths again
//   erow[V+1]    edges leaving stop u are erow[u] .. erow[u+1]-1
// Against one 16-byte record and one 32-byte entry per (type, cluster) this reads 24 bytes
// per edge, where an edge has two (city) or three (large) types of which half have no
// departure left: a large query of a 1,024-query step looks up 65,000 edges instead of
// 194,000 types.  The table takes 2.0 GB beside the 5.1 GB of per-type entries, which the other
// modes read.
constexpr int32_t kNoDeparture = 0xffff;
constexpr int32_t kEdgeOverflow = 15;
constexpr int32_t kMaxPackedStops = 1 << 24;
constexpr int32_t kHubs = 4, kLongLists = 8;      // in EdgeDev::lanes

struct EdgeDev {
    static constexpr int32_t kUsualLanes = 2;
    const int32_t *erow;      // [V + 1]
    const int2 *er;           // [E]
    const int4 *ee;           // [(y + 1) * E], slot-major
    const int2 *ex;
    const int32_t *etypes;    // [E] connection types of each edge (work counters only)
    int32_t n_stops;
    int32_t n_edges;
    int32_t base;             // start of slot 0 (the network's first departure)
    int32_t shift;            // slots of 2^shift seconds
    int32_t y;                // slots
    int32_t big;              // more than 2^24 stops: er holds no degree
    int32_t lanes;            // log2 of the lanes per stop in a crowded round; | kHubs: some stop
                              // has kEdgeOverflow edges or more; | kLongLists: long lists are
                              // looked up through their tables
};

struct NetDev {
    const int32_t *row_ptr;   // [V + 1] types by tail stop
    const int4 *tr;           // [T] type records
    const int4 *ce;           // [2 * y * T], cluster-major
    const uint2 *apx;         // [n_apx]
    int32_t n_stops;
    int32_t n_types;
    int32_t t0;
    int32_t width;            // cluster width (seconds)
    float inv_width;          // 1 / width, for the cluster index of times < 2^22 s
    int32_t k_min;            // first cluster index stored
    int32_t y;                // clusters stored per type
};

// Slot of time e, its start, and e relative to that; e before the first slot counts as its
// start (every departure is then >= e).  A slot >= E.y: no departure at or after e.
EAT_HD inline uint32_t edge_slot(int32_t base, int32_t shift, int32_t e, uint32_t &rel, int32_t &start) {
    const int32_t t = e > base ? e : base;
    const uint32_t d = (uint32_t)t - (uint32_t)base;
    rel = d & ((1u << shift) - 1u);
    start = (int32_t)((uint32_t)t - rel);
    return d >> shift;
}

// Earliest arrival over an edge from its entry c for a tail reached at `rel` in the slot that
// starts at `start`, from the three inline departures; EAT_INF if none of them is at or after
// it (the list, if c.w is set, has the others).
EAT_HD inline int32_t edge_inline(const int4 c, uint32_t rel, int32_t start) {
    const uint32_t x = (uint32_t)c.x, y = (uint32_t)c.y, z = (uint32_t)c.z;
    const uint32_t p = rel <= (x & 0xffffu) ? x : rel <= (y & 0xffffu) ? y : z;
    const uint32_t d = p & 0xffffu;
    return rel <= d && d != (uint32_t)kNoDeparture ? (int32_t)((uint32_t)start + d + (p >> 16)) : EAT_INF;
}

// Part of a slot of 2^(shift + kSubLog2) seconds that `rel` falls into; rel and start become
// those of the part.
constexpr int32_t kSubLog2 = 4, kSubSlots = 1 << kSubLog2, kLongList = 8;

EAT_HD inline int32_t edge_part(int32_t shift, uint32_t &rel, int32_t &start) {
    const uint32_t k = rel >> shift;
    rel -= k << shift;
    start = (int32_t)((uint32_t)start + (k << shift));
    return (int32_t)k;
}

// Up to NETS networks passed by value as a kernel parameter.
template <int NETS>
struct NetTable {
    NetDev net[NETS];
};

template <int NETS>
struct EdgeTable {
    EdgeDev net[NETS];
};

// Networks of up to this many stops may leave threads of a block without work.
constexpr int32_t kFewStops = 32768;

// Host copy of the built arrays (kept for eat_net_host_view).
struct HostNet {
    int32_t n_stops = 0, n_types = 0, n_edges = 0, width = 3600, t0 = 0;
    int32_t max_clusters = 0, max_out_types = 0;
    int64_t n_conn = 0;
    int64_t n_shortcuts = 0;
    std::vector<int32_t> row_ptr;    // V + 1
    std::vector<int32_t> type_rec;   // 4 T
    std::vector<int32_t> type_cl;    // T
    std::vector<int32_t> cl;         // n_cl
    std::vector<uint32_t> ap;        // 2 n_ap
    // Device layout (see NetDev).
    int32_t k_min = 0, y = 1;
    std::vector<int32_t> tr;         // 4 T
    std::vector<int32_t> ce;         // 8 T y
    std::vector<uint32_t> apx;       // 2 n_apx
    // Edge table (see EdgeDev).
    int32_t e_base = 0, e_shift = 0, e_y = 0;
    std::vector<int32_t> erow;       // V + 1
    std::vector<int32_t> er;         // 2 E
    std::unique_ptr<int32_t[]> ee;   // 4 E (e_y + 1): written in full by the threads that fill it
    size_t ee_words = 0;
    std::vector<int32_t> ex;         // 2 per pair
    std::vector<int32_t> etypes;     // E
    int32_t e_lanes = EdgeDev::kUsualLanes;
    // Edges leaving the stops at one distance (in connections) from a source, on average over
    // the distances: the most of four sources.  What a round has work for, about.
    int32_t e_level = 0;
    // Mean duration of the kept departures, and half the mean gap between an edge's: together
    // the time that a connection takes a traveller, about.
    int32_t e_travel = 0, e_wait = 0;
};

}  // namespace eat

struct eat_net {
    eat::HostNet host;
    int32_t device = -1;
    void *blob = nullptr;            // one cudaMalloc holding every array
    int64_t blob_bytes = 0;
    eat::NetDev dev{};
    eat::EdgeDev edev{};
    int branching = 0;               // 1: two or more edges per stop that has any, 2: 2.6 or more
    // Internal workspace and staging buffers (eat_query, NULL-workspace batches).
    mutable std::mutex ws_lock;
    mutable void *ws = nullptr;
    mutable size_t ws_bytes = 0;
    mutable void *stage = nullptr;
    mutable size_t stage_bytes = 0;
    // Mapped host memory for a single query's status and counters, and its device address
    // (nullptr if it could not be had).
    int32_t *pin = nullptr, *pin_dev = nullptr;
    // Launch shape chosen by eat_autotune per batch-size class (log2 of n), packed as
    // block | vwarp << 16 | mode << 24 | horizon << 32 (0 = none) so that a query call
    // on another thread reads one whole shape.
    mutable std::atomic<uint64_t> tuned[32] = {};
};

namespace eat {

// Thread-local error message helpers (eat_api.cu).
int fail(int code, const std::string &msg);
void clear_error();

// Host preprocessing (eat_build.cpp): fills `h` from the connections.
int build_host(const eat_connections *c, int32_t width, int32_t t0, HostNet &h);

// Sub-trips (eat_build.cpp): the connections plus one artificial connection per
// sub-trip of >= 2 connections (Section II-G), as new SoA arrays.
int add_subtrips(const eat_connections *c, int32_t scheme, std::vector<int32_t> &u,
                 std::vector<int32_t> &v, std::vector<int32_t> &dep, std::vector<int32_t> &dur,
                 int64_t &n_added);

// Logical arrays from pre-encoded types / clusters / APs (eat_build.cpp).
int build_host_csr(const eat_csr_input *in, int32_t width, int32_t t0, HostNet &h);

// Device layout from the logical arrays (eat_build.cpp).
int build_fused(HostNet &h);

// Edge table from the logical arrays (eat_build.cpp).
int build_edges(HostNet &h);

// Greedy AP cover of sorted unique values (eat_build.cpp); appends (first, step, terms).
void ap_cover(const int32_t *vals, int32_t n, int32_t width_hint,
              std::vector<uint32_t> &out_ap);

// Greedy AP cover of any sorted unique values (eat_build.cpp); appends
// (first, difference, terms) as three int32 per AP.
void ap_cover_wide(const int32_t *vals, int32_t n, std::vector<int32_t> &out);

}  // namespace eat
