"""The round kernel on networks at the edges of its layout: more stops than a packed record
holds, stops of more than 255 edges, frontiers larger than the shared-memory queue, slots
with departures beyond the inline ones.  Rows equal the oracle's exactly."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]


def _timetable(n, u, v, dep, dur):
    c = [np.asarray(a, dtype=np.int32) for a in (u, v, dep, dur)]
    z = np.zeros(c[0].shape[0], np.int32)
    return synth.Timetable("edges", n, *c, z, z)


def _many_stops():
    """2^24 + 9 stops, connections between a few of them at both ends of the range."""
    rng = np.random.default_rng(1)
    ids = np.concatenate([np.arange(12), 2**24 + np.arange(-4, 9)])
    u, v = rng.choice(ids, 900), rng.choice(ids, 900)
    return _timetable(2**24 + 9, u, v, rng.integers(0, 5000, 900), rng.integers(1, 300, 900)), ids


def _star(n_spokes, n_stops):
    """A hub with an edge to every spoke, each spoke with two edges onward, some back."""
    rng = np.random.default_rng(n_spokes)
    spokes = 1 + np.arange(n_spokes)
    u = np.concatenate([np.zeros(n_spokes, int), spokes, spokes])
    v = np.concatenate([spokes, rng.integers(0, n_stops, n_spokes), rng.integers(0, n_stops, n_spokes)])
    m = u.shape[0]
    k = 3
    return _timetable(n_stops, np.tile(u, k), np.tile(v, k), rng.integers(0, 4000, k * m),
                      rng.integers(1, 500, k * m)), np.concatenate([[0], spokes[:6]])


def _dense():
    """Every second a departure of some duration on a few edges."""
    rng = np.random.default_rng(5)
    m = 20000
    u = rng.integers(0, 6, m)
    return _timetable(6, u, (u + rng.integers(1, 6, m)) % 6, rng.integers(0, 30000, m),
                      rng.integers(1, 8, m) ** 4), np.arange(6)


CASES = {"many_stops": _many_stops, "star_300": lambda: _star(300, 800),
         "star_queue_spills": lambda: _star(20000, 50000), "star_global": lambda: _star(30000, 400000),
         "dense": _dense}


@pytest.mark.parametrize("which", CASES)
def test_rows(which):
    from paper_1912_00966_gb300 import eat
    tt, ids = CASES[which]()
    sc = oracle.SortedConnections(tt)
    net = eat.eat_build(tt.n_stops, tt.u, tt.v, tt.dep, tt.dur, device=0, cluster_width=300)
    rng = np.random.default_rng(2)
    src = np.concatenate([[ids[0], ids[0]], rng.choice(ids, 2)]).astype(np.int32)
    ts = np.array([0, 1000, 2000, 29990], np.int32)
    want = np.stack([oracle.csa(sc, int(s), int(t)) for s, t in zip(src, ts)])
    out = torch.empty((4, tt.n_stops), dtype=torch.int32, device="cuda")
    for opts in ({}, {"horizon": 200}, {"block": 64, "horizon": 1500}, {"block": 256, "vwarp": 1}):
        out.fill_(-7)
        eat.eat_query_batch(net, torch.as_tensor(src).cuda(), torch.as_tensor(ts).cuda(), out, **opts)
        assert np.array_equal(out.cpu().numpy(), want), opts
    got = eat.eat_query(net, int(src[3]), int(ts[3]))
    assert np.array_equal(got, want[3])
    net.close()


@pytest.mark.parametrize("family,stops", [("grid", 1500), ("grid", 5000), ("grid", 13000), ("grid", 30000),
                                          ("city", 3000), ("city", 21000), ("city", 60000)])
def test_automatic_shapes(family, stops):
    """Every automatic launch shape (block size, threads at work, placement, horizon) by batch
    size on networks with and without a branching frontier, with and without counters."""
    import os
    from paper_1912_00966_gb300 import eat
    if family == "grid":
        tt = synth.grid_timetable(stops, max(2, stops // 25), 700 + stops, force_stop0=False)
    else:
        tt = synth.transit.geometric_timetable(stops, 4, stops // 60, (20, 40), (15, 40), 0.2,
                                               synth.transit.PEAK_BANDS, 700 + stops)
    net = eat.eat_build(tt.n_stops, tt.u, tt.v, tt.dep, tt.dur, device=0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    most = 4 * sms + 40
    q = synth.random_queries(tt, most, 71)
    src, ts = torch.as_tensor(q.source).cuda(), torch.as_tensor(q.t_s).cuda()
    want = torch.as_tensor(oracle.csa_many(oracle.SortedConnections(tt), q.source, q.t_s,
                                           os.cpu_count() or 8)[0]).cuda()
    out = torch.empty((most, stops), dtype=torch.int32, device="cuda")
    counters = torch.zeros((most, 7), dtype=torch.int64, device="cuda")
    for n in (1, 2, sms // 2, sms // 2 + 1, sms + 1, 3 * sms // 2 + 1, 2 * sms + 77, most):
        for more in ({}, {"counters": counters}, {"max_rounds": 2 * stops + 2}):
            out.fill_(-7)
            eat.eat_query_batch(net, src[:n], ts[:n], out[:n], **more)
            assert torch.equal(out[:n], want[:n]), (n, list(more))
    net.close()


@pytest.mark.parametrize("stops,degree", [(5, 3), (167, 14), (169, 15), (1001, 16), (20001, 4)])
def test_edges_back(stops, degree):
    """Edges in both directions between most pairs (of which rows in global memory leave the one
    back to the stop that queued a stop out), stops of 14 to 16 edges about, odd queue sizes."""
    from paper_1912_00966_gb300 import eat
    rng = np.random.default_rng(stops)
    a = np.tile(np.arange(stops), degree // 2 + 1)
    b = rng.integers(0, stops, a.shape[0])
    u, v = np.tile(np.concatenate([a, b]), 6), np.tile(np.concatenate([b, a]), 6)
    tt = _timetable(stops, u, v, rng.integers(0, 20000, u.shape[0]), rng.integers(1, 900, u.shape[0]))
    net = eat.eat_build(tt.n_stops, tt.u, tt.v, tt.dep, tt.dur, device=0)
    n = torch.cuda.get_device_properties(0).multi_processor_count + 9
    src, ts = rng.integers(0, stops, n).astype(np.int32), rng.integers(0, 9000, n).astype(np.int32)
    want, _ = oracle.csa_many(oracle.SortedConnections(tt), src, ts, 8)
    out = torch.empty((n, stops), dtype=torch.int32, device="cuda")
    counters = torch.zeros((n, 7), dtype=torch.int64, device="cuda")
    src, ts = torch.as_tensor(src).cuda(), torch.as_tensor(ts).cuda()
    for opts in ({"block": 512}, {"block": 1024}, {"block": 64, "vwarp": 2}, {"block": 512, "horizon": 700},
                 {"block": 1024, "horizon": 700, "counters": counters}):
        out.fill_(-7)
        eat.eat_query_batch(net, src, ts, out, placement=eat.EAT_PLACE_GLOBAL_ARR, **opts)
        assert np.array_equal(out.cpu().numpy(), want), list(opts)
    net.close()
