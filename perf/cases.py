"""What a user of this library has it do, as cases that can be timed and compared.

A case names a network (family, stops, cluster width), a call and the number of queries of
one pass.  The networks are the seeded synthetic timetables of `synth`: the 1,024-stop grid,
the 20,000-stop city, the 200,000-stop large network, the 64 ragged grids and the served mix
of a city and 16 grids, as the benchmark uses them, and other sizes drawn with the same
densities.  A network stays resident while queries on it come and go, so it is built once
per process; every seed gives other queries (source uniform over the stops that have a
departure, departure time uniform in 05:00-22:00).
"""
from __future__ import annotations

import collections
import math
import weakref

import numpy as np
import torch

import synth
from paper_1912_00966_gb300 import eat

INF = 2**31 - 1
KEEP_BYTES = 12 << 30            # device bytes of networks kept resident between cases


def listed():
    return [
        # One trip planned on a small town's network, the answer used on the GPU: latency.
        case("grid_one", "one", "grid", 1024, 1),
        # A small town's accessibility map: 256 sources at once.
        case("grid_batch", "batch", "grid", 1024, 256),
        # One interactive request on a city network, the row returned to host memory.
        case("city_one", "one_host", "city", 20000, 1),
        # A few requests gathered from users, fewer than the GPU has SMs.
        case("city_few", "batch", "city", 20000, 37),
        # The benchmark's city step: 256 queries on 10-minute clusters.
        case("city_batch", "batch", "city", 20000, 256, width=600),
        # The same step end to end from page-locked host buffers.
        case("city_host", "host", "city", 20000, 256, width=600),
        # A metropolitan region of a size between the two, an odd one, library defaults.
        case("region_batch", "batch", "region", 60013, 300),
        # One request on a country-sized network.
        case("large_one", "one", "region", 200000, 1, width=600),
        # A partly filled batch on it, library defaults.
        case("large_few", "batch", "region", 200000, 96, width=600),
        # The benchmark's default step: 1,024 queries, launch shape by the autotuner.
        case("large_batch", "batch", "region", 200000, 1024, width=600, tuned=True),
        # 64 networks of uneven size served in one launch, shape by the autotuner.
        case("ragged_batch", "multi", "grid", 50000, 4096, width=600, nets=64, tuned=True),
        # A burst of requests to the running server: a city and 16 small networks.
        case("serve_burst", "serve", "city", 20000, 256, width=600, nets=17),
    ]


def case(name, call, family, stops, queries, width=3600, nets=1, tuned=False, horizon=0):
    """family: timetable generator; stops: of the (largest) network; width: cluster width in
    seconds (3600 is the library's default); nets: networks in one call; tuned: launch shape
    chosen once by the library's autotuner, else its defaults; horizon: query option."""
    c = {"call": call, "family": family, "stops": stops, "queries": queries, "width": width,
         "nets": nets, "tuned": tuned, "horizon": horizon}
    return {"name": name, **c} if name else c


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["one", "one_host", "batch", "batch", "batch", "host", "multi"])
    width = rng.choice([600, 900, 1800, 3600])
    if call == "multi":
        return case(None, call, "grid", 50000, _log_uniform(rng, 64, 4096), width,
                    nets=rng.randint(2, 64))
    family = rng.choice(["grid", "city", "region"])
    lo, hi = {"grid": (1000, 50000), "city": (2000, 60000), "region": (20000, 200000)}[family]
    stops = _log_uniform(rng, lo, hi)
    queries = 1 if call in ("one", "one_host") else _log_uniform(rng, 2, min(1024, 80_000_000 // stops))
    horizon = rng.choice([0, 0, 3600, 7200]) if family == "region" and call in ("batch", "host") else 0
    return case(None, call, family, stops, queries, width, horizon=horizon)


# ------------------------------------------------------------------ resident networks

class Resident:
    """Networks of one case, their timetables and stops with departures, tuned shapes."""

    def __init__(self, tts, width):
        self.tts = tts
        self.nets = [eat.eat_build(t.n_stops, t.u, t.v, t.dep, t.dur, cluster_width=width)
                     for t in tts]
        self.sources = [t.sources_with_departures() for t in tts]
        self.bytes = sum(n.stats["device_bytes"] for n in self.nets)
        self.shapes = {}


_resident = collections.OrderedDict()
_servers = weakref.WeakValueDictionary()


def _timetables(c):
    n = c["stops"]
    if c["call"] == "serve":
        return [_geometric("city", n)] + [synth.small_grid(seed_offset=k) for k in range(c["nets"] - 1)]
    if c["nets"] > 1:
        return synth.ragged_grids(c["nets"])
    if c["family"] == "grid":
        return [synth.small_grid() if n == 1024 else
                synth.grid_timetable(n, math.ceil(50 * n / 1024), synth.transit.SEED_BASE + n,
                                     force_stop0=False)]
    return [_geometric(c["family"], n)]


def _geometric(family, n):
    if family == "city":
        if n == 20000:
            return synth.city()
        return synth.transit.geometric_timetable(
            n, 4, max(1, n // 50), (30, 60), (5, 20), 0.20, synth.transit.PEAK_BANDS,
            synth.transit.SEED_BASE + 1)
    if n == 200000:
        return synth.large()
    return synth.transit.geometric_timetable(
        n, 5, max(1, n // 50), (40, 80), (3, 30), 0.10,
        synth.transit.PEAK_BANDS + synth.transit.OFFPEAK_BANDS, synth.transit.SEED_BASE + 2)


def _networks(c):
    key = (c["call"] == "serve", c["family"], c["stops"], c["width"], c["nets"])
    if key not in _resident:
        _resident[key] = Resident(_timetables(c), c["width"])
        while len(_resident) > 1 and sum(r.bytes for r in _resident.values()) > KEEP_BYTES:
            _resident.popitem(last=False)
    _resident.move_to_end(key)
    return _resident[key]


def _queries(res, n, seed):
    rng = np.random.default_rng(seed)
    net = rng.permutation(np.arange(n, dtype=np.int32) % len(res.nets))   # as many on each
    src = np.empty(n, dtype=np.int32)
    for j, cand in enumerate(res.sources):
        sel = np.nonzero(net == j)[0]
        src[sel] = cand[rng.integers(0, cand.shape[0], size=sel.shape[0])]
    ts = rng.integers(synth.transit.QUERY_T_MIN, synth.transit.QUERY_T_MAX + 1, size=n)
    return net, src, ts.astype(np.int32)


def _cuda(a):
    return torch.as_tensor(a).cuda()


def _tune(c, res):
    """The options a program keeps after tuning once on a sample of its traffic."""
    n = c["queries"]
    if n not in res.shapes:
        net, src, ts = _queries(res, n, 0xA0 - 1)
        if c["call"] == "multi":
            res.shapes[n] = eat.eat_autotune_multi(res.nets, _cuda(net), _cuda(src), _cuda(ts))
        else:                    # kept inside the network: the calls then leave the shape at 0
            eat.eat_autotune(res.nets[0], _cuda(src), _cuda(ts))
            res.shapes[n] = {}
    return res.shapes[n]


def prepare(c, seed):
    res = _networks(c)
    n, call = c["queries"], c["call"]
    net, src, ts = _queries(res, n, seed)
    s = {"call": call, "res": res, "net": res.nets[0]}
    stops = np.array([t.n_stops for t in res.tts], np.int64)[net]
    opts = dict(_tune(c, res)) if c["tuned"] else {}
    if c["horizon"]:
        opts["horizon"] = c["horizon"]
    s["opts"] = opts
    if call in ("one", "one_host"):
        s["source"], s["t_s"] = int(src[0]), int(ts[0])
        if call == "one":
            s["out"] = torch.empty(int(stops[0]), dtype=torch.int32, device="cuda")
    elif call == "batch":
        s["src"], s["ts"] = _cuda(src), _cuda(ts)
        s["out"] = torch.empty((n, int(stops[0])), dtype=torch.int32, device="cuda")
        s["status"] = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        s["ws"] = torch.empty(eat.eat_workspace_bytes(s["net"], n, **opts), dtype=torch.uint8,
                              device="cuda")
    elif call == "host":
        s["src"], s["ts"] = torch.as_tensor(src).pin_memory(), torch.as_tensor(ts).pin_memory()
        s["out"] = torch.empty((n, int(stops[0])), dtype=torch.int32).pin_memory()
    elif call == "multi":
        s["idx"], s["src"], s["ts"] = _cuda(net), _cuda(src), _cuda(ts)
        offs = np.concatenate([[0], np.cumsum(stops)[:-1]]).astype(np.int64)
        s["offs"] = _cuda(offs)
        s["out"] = torch.empty(int(stops.sum()), dtype=torch.int32, device="cuda")
        s["status"] = torch.full((n,), -1, dtype=torch.int32, device="cuda")
        s["ws"] = torch.empty(eat.eat_workspace_bytes(res.nets, n, **opts), dtype=torch.uint8,
                              device="cuda")
    else:
        server = _servers.get(id(res))
        if server is None:
            server = _servers[id(res)] = eat.Server(res.nets)
        s["server"] = server
        s["requests"] = [(int(net[i]), int(src[i]), int(ts[i])) for i in range(n)]
        s["rows"] = np.empty(int(stops.sum()), dtype=np.int32)
        s["out"] = np.split(s["rows"], np.cumsum(stops)[:-1])    # one row for each request
    return s


def run(s):
    call = s["call"]
    if call == "one":
        return eat.eat_query(s["net"], s["source"], s["t_s"], s["out"])
    if call == "one_host":
        return eat.eat_query(s["net"], s["source"], s["t_s"])
    if call == "batch":
        eat.eat_query_batch(s["net"], s["src"], s["ts"], s["out"], workspace=s["ws"],
                            status=s["status"], **s["opts"])
        return {"rows": s["out"], "status": s["status"]}
    if call == "host":
        return eat.eat_query_batch(s["net"], s["src"], s["ts"], s["out"], **s["opts"])
    if call == "multi":
        eat.eat_query_batch_multi(s["res"].nets, s["idx"], s["src"], s["ts"], s["out"], s["offs"],
                                  workspace=s["ws"], status=s["status"], **s["opts"])
        return {"rows": s["out"], "status": s["status"]}
    server = s["server"]
    for tag, (net, src, ts) in enumerate(s["requests"]):
        server.submit(net, src, ts, s["out"][tag], tag)
    left = len(s["requests"])
    while left:
        for _, status, _, _ in server.poll(timeout_us=1000):
            if status != 0:
                raise RuntimeError(f"a request failed with status {status}")
            left -= 1
    return s["rows"]


def work(c):
    """Each arrival row written once, the queries read once, and of the networks one 16-byte
    record and one 4-byte departure of each connection type read once (a query may reach all
    of them, and a batch reads them together).  Types by the generators' densities: routes
    run both ways x edges per route x duration bands met."""
    n, q = c["stops"], c["queries"]
    if c["call"] == "multi":
        mean = (50000 - 1000) / math.log(50.0)
        rows, types = mean * q, mean * c["nets"] * 50 / 1024 * 19
    elif c["call"] == "serve":
        rows = q * (n + 1024 * (c["nets"] - 1)) / c["nets"]
        types = n / 50 * 88 * 1.5 + (c["nets"] - 1) * 800
    else:
        rows = q * n
        types = {"grid": n * 0.8, "city": n / 50 * 88 * 1.5, "region": n / 50 * 118 * 2.3}[c["family"]]
        types = min(types, 64.0 * q * 1000)       # a single query meets a part of them
    return {"bytes": 4 * rows + 8 * q + 20 * types, "flops": 0}


# ------------------------------------------------------------------ in 64 bits

class _Types:
    """A timetable's connections grouped by (u, v, duration), sorted by departure, as 64-bit
    torch tensors: type t leaves tail[t], its departures are the keys t << 32 | departure."""

    def __init__(self, tt):
        u, v, dep, dur = (_cuda(np.asarray(a)).long() for a in (tt.u, tt.v, tt.dep, tt.dur))
        span = int(dur.max()) + 1
        kind, of = torch.unique((u * tt.n_stops + v) * span + dur, return_inverse=True)
        self.keys = torch.unique(of << 32 | dep)
        self.dur = kind % span
        self.head = kind // span % tt.n_stops
        tail = kind // span // tt.n_stops                    # sorted: the types of a stop adjoin
        stops = torch.arange(tt.n_stops + 1, device=tail.device)
        self.row = torch.searchsorted(tail, stops)


def _arrivals(tt, src, ts):
    """Earliest arrivals by repeated relaxation of the stops that improved, in int64."""
    T, V, q = _Types(tt), tt.n_stops, len(src)
    e = torch.full((q * V,), INF, dtype=torch.int64, device="cuda")
    at = torch.arange(q, device="cuda") * V + _cuda(src).long()
    e[at] = _cuda(ts).long()
    while at.numel():
        stop = at % V
        deg = T.row[stop + 1] - T.row[stop]
        owner = torch.repeat_interleave(torch.arange(at.numel(), device="cuda"), deg)
        first = torch.cumsum(deg, 0) - deg
        t = T.row[stop][owner] + torch.arange(owner.numel(), device="cuda") - first[owner]
        want = t << 32 | e[at][owner].clamp(0, INF)
        k = torch.searchsorted(T.keys, want)
        key = T.keys[k.clamp(max=T.keys.numel() - 1)]
        ok = (k < T.keys.numel()) & (key >> 32 == t)
        owner, t, key = owner[ok], t[ok], key[ok]
        cand = (key & 0xFFFFFFFF) + T.dur[t]
        to = at[owner] // V * V + T.head[t]
        better = cand < e[to]
        to, cand = to[better], cand[better]
        e.scatter_reduce_(0, to, cand, "amin")
        at = torch.unique(to)
    return e.view(q, V)


def exact(c, seed):
    res = _networks(c)
    net, src, ts = _queries(res, c["queries"], seed)
    if c["nets"] == 1:
        rows = _arrivals(res.tts[0], src, ts)
        if c["call"] in ("one", "one_host"):
            return rows[0]
        if c["call"] == "host":
            return rows
        return {"rows": rows, "status": torch.zeros(len(src), dtype=torch.int64)}
    out = [None] * len(src)
    for j, tt in enumerate(res.tts):
        sel = np.nonzero(net == j)[0]
        if sel.size:
            for i, row in zip(sel, _arrivals(tt, src[sel], ts[sel])):
                out[i] = row
    if c["call"] == "serve":
        return torch.cat(out)
    return {"rows": torch.cat(out), "status": torch.zeros(len(src), dtype=torch.int64)}
