"""Networks unlike street networks: what their shape costs, and rows equal to the oracle's."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="no CUDA device")]

HOUR = 3600


def _service(n_stops, u, v, dur, headway, seed, first=5 * HOUR, last=23 * HOUR):
    """Edges (u, v) of `dur` seconds served every `headway` seconds from a phase of their own."""
    rng = np.random.default_rng(seed)
    u, v, dur, headway = np.broadcast_arrays(*(np.asarray(a, np.int64) for a in (u, v, dur, headway)))
    phase = (rng.random(u.shape[0]) * headway).astype(np.int64)
    trips = np.maximum(1, (last - first - phase) // headway + 1)
    e = np.repeat(np.arange(u.shape[0]), trips)
    k = np.arange(e.shape[0]) - np.repeat(np.cumsum(trips) - trips, trips)
    c = [np.asarray(a, np.int32) for a in (u[e], v[e], first + phase[e] + k * headway[e], dur[e])]
    z = np.zeros(e.shape[0], np.int32)
    return synth.Timetable("odd", n_stops, *c, z, z)


def _complete(n):
    rng = np.random.default_rng(n)
    u, v = np.divmod(np.arange(n * n), n)
    u, v = u[u != v], v[u != v]
    return _service(n, u, v, rng.integers(HOUR // 2, 6 * HOUR, u.shape[0]),
                    rng.integers(3, 6, u.shape[0]) * HOUR, n)


def _random(n, degree, headway=300):
    rng = np.random.default_rng(n)
    u = np.repeat(np.arange(n), degree)
    key = np.unique(u * n + (u + rng.integers(1, n, u.shape[0])) % n)
    return _service(n, key // n, key % n, rng.integers(60, 600, key.shape[0]), headway, n)


def _hubs(degrees, leaves, seed=1):
    """A ring of stops with `degrees` spokes each; a spoke leads back unless it is a leaf."""
    degrees = np.asarray(degrees)
    h = degrees.shape[0]
    hub = np.repeat(np.arange(h), degrees)
    spoke = h + np.arange(hub.shape[0])
    ring = np.arange(h)
    rng = np.random.default_rng(seed)
    u = np.concatenate([ring, hub] + ([] if leaves else [spoke, spoke]))
    v = np.concatenate([(ring + 1) % h, spoke] + ([] if leaves else [hub, rng.permutation(spoke)]))
    dur = rng.integers(60, 1200, u.shape[0])
    return _service(h + spoke.shape[0], u, v, dur, rng.integers(300, 2400, u.shape[0]), seed)


class _Case:
    def __init__(self, tt, n, seed=5):
        from paper_1912_00966_gb300 import eat
        self.eat, self.tt = eat, tt
        self.net = eat.eat_build(tt.n_stops, tt.u, tt.v, tt.dep, tt.dur, device=0)
        q = synth.random_queries(tt, n, seed)
        self.q = q
        self.src, self.ts = torch.as_tensor(q.source).cuda(), torch.as_tensor(q.t_s).cuda()
        self.out = torch.empty((n, tt.n_stops), dtype=torch.int32, device="cuda")

    def run(self, **opts):
        self.eat.eat_query_batch(self.net, self.src, self.ts, self.out, **opts)

    def check(self, **opts):
        self.out.fill_(-7)
        self.run(**opts)
        want, _ = oracle.csa_many(oracle.SortedConnections(self.tt), self.q.source, self.q.t_s, 8)
        assert np.array_equal(self.out.cpu().numpy(), want), opts

    def us(self, **opts):
        """Median device time of a call."""
        need = self.eat.eat_workspace_bytes(self.net, self.src.shape[0], **opts)
        ws = torch.empty(need, dtype=torch.uint8, device="cuda")
        times = []
        for _ in range(14):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda._sleep(400000)            # the GPU is busy while the host enqueues the call
            a.record()
            self.run(workspace=ws, **opts)
            b.record()
            b.synchronize()
            times.append(1e3 * a.elapsed_time(b))
        return float(np.median(times[3:]))


@pytest.mark.parametrize("make,n", [(lambda: _complete(300), 1), (lambda: _complete(300), 300),
                                    (lambda: _random(2000, 4), 1), (lambda: _random(2000, 4), 300),
                                    (lambda: _random(20000, 4), 300)])
def test_threads_fit_the_rounds(make, n):
    """The automatic shape of a small network of many or far-reaching edges is not far behind the
    explicit block sizes.  With threads chosen by the number of stops alone it took 2 to 3.4
    times the best; 1.5 leaves room for the timing."""
    c = _Case(make(), n)
    c.check()
    best = min(c.us(block=b) for b in (256, 512, 1024))
    assert c.us() < 1.5 * best
    c.net.close()


@pytest.mark.parametrize("net,horizon", [
    ("city", 14400), ("random, 10 minutes", 14400),
    ("random, 22 hours", -1), ("grid, 1 hour every three", -1), ("random, twice a day", -1),
    ("random, once a day", -1)])
def test_horizon_where_it_holds_many_connections(net, horizon):
    """An automatic horizon is for connections that are short beside it: with long or rare ones it
    moves in nearly every round."""
    if net == "city":
        tt = synth.city()
    elif net.endswith("a day"):
        tt = _random(60000, 3, (12 if "twice" in net else 24) * HOUR)
    elif net.startswith("random"):
        long = net.endswith("hours")
        t = _random(2000, 4)
        e = np.unique(t.u.astype(np.int64) * 2000 + t.v)
        dur = np.random.default_rng(3).integers(*((70000, 90000) if long else (60, 600)), e.shape[0])
        tt = _service(2000, e // 2000, e % 2000, dur, 3 * HOUR if long else 600, 4, 0, 300000 if long else 23 * HOUR)
    else:
        x, y = np.divmod(np.arange(10000), 100)
        at = np.arange(10000)
        e = [(at[m], (at + s)[m]) for m, s in ((y < 99, 1), (y > 0, -1), (x < 99, 100), (x > 0, -100))]
        u, v = (np.concatenate(a) for a in zip(*e))
        tt = _service(10000, u, v, np.random.default_rng(3).integers(2400, 4800, u.shape[0]), 3 * HOUR, 4, 0, 200000)
    c = _Case(tt, 37)
    assert c.eat.eat_launch_shape(c.net, 37)["horizon"] == horizon
    c.check()
    c.net.close()


HUBS = {
    "about a sub-warp's passes": lambda: _hubs([12, 13, 14, 15, 16, 30, 31, 32, 62, 63, 64, 126, 127, 128], False),
    "pieces of more than a warp": lambda: _hubs([2046, 2047, 2048, 5000, 9000, 15], False),
    "more pieces than room": lambda: _complete(41),
    "spilled hubs": lambda: _hubs([40] * 1200, False),
    "rows in global memory": lambda: _hubs([700] * 100, False),
    "spokes of one edge": lambda: _hubs([20] * 900, True),
}


@pytest.mark.parametrize("which", HUBS)
def test_hub_rows(which):
    """Stops of more edges than a sub-warp takes are shared by the block's warps: rows, status and
    the counted build, at block sizes and lanes of every kind."""
    tt = HUBS[which]()
    c = _Case(tt, 60)
    eat = c.eat
    want, _ = oracle.csa_many(oracle.SortedConnections(tt), c.q.source, c.q.t_s, 8)
    counters = torch.zeros((60, 7), dtype=torch.int64, device="cuda")
    for opts in ({}, {"block": 64}, {"block": 96, "vwarp": 32}, {"block": 512, "vwarp": 1}, {"block": 1024, "vwarp": 2},
                 {"block": 256, "horizon": 900}, {"block": 1024, "horizon": 900, "counters": counters},
                 {"placement": eat.EAT_PLACE_GLOBAL_ARR, "block": 512}, {"placement": eat.EAT_PLACE_GLOBAL, "block": 1024},
                 {"placement": eat.EAT_PLACE_GLOBAL_ARR, "block": 320, "horizon": 900}):
        status = torch.full((60,), -9, dtype=torch.int32, device="cuda")
        c.out.fill_(-7)
        c.run(status=status, **opts)
        assert np.array_equal(c.out.cpu().numpy(), want), list(opts.items())
        assert not status.any()
    reached = torch.as_tensor((want < 2**31 - 1).sum(axis=1)).cuda()
    assert (counters[:, 6] >= reached - 1).all() and (counters[:, 2] >= counters[:, 4]).all()
    assert np.array_equal(eat.eat_query(c.net, int(c.q.source[7]), int(c.q.t_s[7])), want[7])
    c.net.close()


def test_hubs_beside_other_networks():
    """One launch and one server over networks with hubs and without."""
    from paper_1912_00966_gb300 import eat
    tts = [_hubs([100, 40, 16, 300], False), synth.small_grid(), _hubs([20] * 200, True), _complete(30)]
    nets = [eat.eat_build(t.n_stops, t.u, t.v, t.dep, t.dur, device=0) for t in tts]
    q = synth.random_queries(tts, 400, 9)
    sizes = np.array([tts[i].n_stops for i in q.net], np.int64)
    offs = np.concatenate([[0], np.cumsum(sizes)[:-1]])
    want = np.concatenate([oracle.csa(oracle.SortedConnections(tts[i]), int(s), int(t))
                           for i, s, t in zip(q.net, q.source, q.t_s)])
    out = torch.full((int(sizes.sum()),), -7, dtype=torch.int32, device="cuda")
    dev = [torch.as_tensor(a).cuda() for a in (q.net, q.source, q.t_s)]
    for opts in ({}, {"block": 1024}, {"horizon": 1200}):
        out.fill_(-7)
        eat.eat_query_batch_multi(nets, *dev, out, torch.as_tensor(offs).cuda(), **opts)
        assert np.array_equal(out.cpu().numpy(), want), opts
    server = eat.Server(nets)
    rows = np.split(np.full(int(sizes.sum()), -7, np.int32), offs[1:])
    for k in range(400):
        server.submit(int(q.net[k]), int(q.source[k]), int(q.t_s[k]), rows[k], k)
    left = 400
    while left:
        for _, status, _, _ in server.poll(timeout_us=1000):
            assert status == 0
            left -= 1
    assert np.array_equal(np.concatenate(rows), want)
    server.close()
    for n in nets:
        n.close()


def test_hub_does_not_hold_up_its_round():
    """A ring of 40 stops, alone and with 1,000 leaves at each: with one sub-warp to a stop the leaves
    made a round some 60 times as long; the block's threads take them in one pass."""
    ring, hubs = _Case(_hubs([0] * 40, True), 1), _Case(_hubs([1000] * 40, True), 1)
    for c in (ring, hubs):
        c.q.source[0], c.q.t_s[0] = c.src[0], c.ts[0] = 0, 6 * HOUR
        c.check()
    assert hubs.us() < 10 * ring.us()
    ring.net.close()
    hubs.net.close()


def _with_extra(tt, day):
    """One more departure, `day` days on: the slots of the whole network get longer."""
    c = [np.append(a, b).astype(np.int32) for a, b in
         ((tt.u, tt.u[0]), (tt.v, tt.v[0]), (tt.dep, 86400 * day), (tt.dur, tt.dur[0]))]
    z = np.zeros(c[0].shape[0], np.int32)
    return synth.Timetable("extra", tt.n_stops, *c, z, z)


def _metro(headway):
    """A line of 60 stops served every `headway` seconds both ways, in a net of rare connections."""
    rng = np.random.default_rng(headway)
    u = np.repeat(np.arange(6000), 3)
    key = np.unique(np.concatenate([u * 6000 + (u + rng.integers(1, 6000, u.shape[0])) % 6000,
                                    np.arange(59) * 6001 + 1, np.arange(1, 60) * 6001 - 1]))
    busy = np.abs(key // 6000 - key % 6000) == 1
    busy &= (key // 6000 < 60) & (key % 6000 < 60)
    return _service(6000, key // 6000, key % 6000, rng.integers(60, 900, key.shape[0]),
                    np.where(busy, headway, 4 * HOUR), headway)


@pytest.mark.parametrize("make", [lambda: _metro(60), lambda: _metro(7),
                                  lambda: _with_extra(synth.small_grid(), 20),
                                  lambda: _with_extra(synth.small_grid(), 3000)])
def test_long_list_rows(make):
    """Long lists of departures through their tables, one to three levels deep."""
    tt = make()
    c = _Case(tt, 200)
    eat = c.eat
    want, _ = oracle.csa_many(oracle.SortedConnections(tt), c.q.source, c.q.t_s, 8)
    counters = torch.zeros((200, 7), dtype=torch.int64, device="cuda")
    for opts in ({}, {"block": 512, "horizon": 1800}, {"block": 1024, "counters": counters},
                 {"placement": eat.EAT_PLACE_GLOBAL_ARR, "block": 512},
                 {"placement": eat.EAT_PLACE_GLOBAL_ARR, "block": 1024, "horizon": 7200},
                 {"placement": eat.EAT_PLACE_GLOBAL}):
        c.out.fill_(-7)
        c.run(**opts)
        assert np.array_equal(c.out.cpu().numpy(), want), list(opts.items())
    c.net.close()


@pytest.mark.parametrize("n", [1, 300])
def test_one_far_departure_costs_little(n):
    """A city and the same city with one departure 30 days on: walked from their start, the lists that
    its longer slots bring took three times as long."""
    plain, far = _Case(synth.city(), n), _Case(_with_extra(synth.city(), 30), n)
    for c in (plain, far):
        c.run()
    assert torch.equal(plain.out, far.out)
    assert far.us() < 2 * plain.us()
    plain.net.close()
    far.net.close()


@pytest.mark.parametrize("which", ["grid", "city", "city, rows alone on an SM", "complete", "several"])
def test_workspace_holds_smaller_batches(which):
    """A program sizes one workspace for its largest batch: no smaller one needs more, whatever
    shape and horizon its size gets."""
    from paper_1912_00966_gb300 import eat
    geometric = lambda n: synth.transit.geometric_timetable(n, 4, n // 200, (30, 60), (5, 20), 0.2,
                                                            synth.transit.PEAK_BANDS, 5)
    tts = {"grid": [synth.small_grid()], "city": [geometric(10000)], "city, rows alone on an SM": [geometric(35000)],
           "complete": [_complete(200)], "several": [synth.small_grid(), geometric(9000)]}[which]
    nets = [eat.eat_build(t.n_stops, t.u, t.v, t.dep, t.dur, device=0) for t in tts]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for opts in ({}, {"block": 512}, {"max_rounds": 9}):
        need = [eat.eat_workspace_bytes(nets if len(nets) > 1 else nets[0], n, **opts) for n in range(1, 9 * sms, 3)]
        assert need[0] > 0 and need == sorted(need), opts
        need = [eat.eat_workspace_bytes(nets if len(nets) > 1 else nets[0], n, **opts) for n in range(sms - 3, 2 * sms)]
        assert need == sorted(need), opts
    for n in nets:
        n.close()


def test_horizon_around_one_query_per_sm():
    """The automatic horizon holds for batches of a little more than one query per SM as for others:
    without it they took 25 % longer than batches just below and above."""
    tt = synth.transit.geometric_timetable(10000, 4, 200, (30, 60), (5, 20), 0.2, synth.transit.PEAK_BANDS, 6)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    c = _Case(tt, sms + 8)
    for n in (2, sms - 1, sms + 2, sms + 8, sms + sms // 8, 2 * sms):
        assert c.eat.eat_launch_shape(c.net, n)["horizon"] == 14400, n
    c.check()
    c.net.close()


def test_shape_read_back_runs_alike():
    """A call with the shape that eat_launch_shape reports takes the time of the automatic call: the
    threads that a small network's rounds cannot fill leave either way (all of them: 69 -> 87 us)."""
    tt = synth.grid_timetable(1500, 75, 77, force_stop0=False)
    c = _Case(tt, 100)
    shape = c.eat.eat_launch_shape(c.net, 100)
    assert c.us(**shape) < 1.12 * c.us()
    c.check(**shape)
    c.net.close()


def test_tuned_is_not_slower_than_automatic():
    """The tuners can choose the automatic shape: 64 networks of uneven size, and one small one."""
    from paper_1912_00966_gb300 import eat
    tts = synth.ragged_grids(64)
    nets = [eat.eat_build(t.n_stops, t.u, t.v, t.dep, t.dur, device=0) for t in tts]
    q = synth.random_queries(tts, 4096, 3)
    sizes = np.array([tts[i].n_stops for i in q.net], np.int64)
    offs = torch.as_tensor(np.concatenate([[0], np.cumsum(sizes)[:-1]])).cuda()
    dev = [torch.as_tensor(a).cuda() for a in (q.net, q.source, q.t_s)]
    out = torch.empty(int(sizes.sum()), dtype=torch.int32, device="cuda")

    def us(**opts):
        times = []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda._sleep(400000)
            a.record()
            eat.eat_query_batch_multi(nets, *dev, out, offs, **opts)
            b.record()
            b.synchronize()
            times.append(1e3 * a.elapsed_time(b))
        return float(np.median(times[3:]))

    automatic, shape = us(), eat.eat_autotune_multi(nets, *dev)
    assert us(**shape) < 1.08 * automatic, shape
    for n in nets:
        n.close()
    small = _Case(synth.grid_timetable(3000, 147, 78, force_stop0=False), 1024)
    automatic = small.us()
    shape = eat.eat_autotune(small.net, small.src, small.ts)
    assert small.us() < 1.08 * automatic, shape
    small.net.close()
