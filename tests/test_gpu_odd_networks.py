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


def _random(n, degree):
    rng = np.random.default_rng(n)
    u = np.repeat(np.arange(n), degree)
    key = np.unique(u * n + (u + rng.integers(1, n, u.shape[0])) % n)
    return _service(n, key // n, key % n, rng.integers(60, 600, key.shape[0]), 300, n)


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
    ("random, 22 hours", -1), ("grid, 1 hour every three", -1)])
def test_horizon_where_it_holds_many_connections(net, horizon):
    """An automatic horizon is for connections that are short beside it: with long or rare ones it
    moves in nearly every round."""
    if net == "city":
        tt = synth.city()
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
    if horizon < 0:
        assert c.us() < 1.25 * c.us(horizon=-1)
    c.net.close()
