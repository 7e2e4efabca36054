"""The batch's paths that small batches do not take, bit for bit against each
simulation run alone: the row passes of batches of 65536 cells and more (lists of
the cells that see a potential, rows by eight per warp), more event quads than
the queue holds, and several batches whose captured runs are kept."""
import numpy as np
import pytest

import oracle
import wmc_inputs as wi
from tests._util import gpu_run, gpu_run_table, oracle_tables

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wmc():
    from paper_1806_00082_gb300 import build, wmc as w
    build.build()
    w.load()
    return w


class _Batch:
    def __init__(self, wmc, wls, Vs, hs):
        self.wmc, self.wls, self.Vs, self.hs = wmc, wls, Vs, hs
        self.ps = wmc.params_array([wmc.Params.of(w) for w in wls])
        _, self.ho = wmc.batch_layout(self.ps)
        self.ws = wmc.batch_workspace(self.ps)
        self.V = torch.from_numpy(np.concatenate(Vs)).cuda()
        self.start = torch.from_numpy(np.concatenate([h.reshape(-1) for h in hs])).cuda()
        self.a, self.b = torch.empty_like(self.start), torch.empty_like(self.start)
        wmc.batch_init(self.ps, self.ws)
        torch.cuda.synchronize()  # (the runs are on other streams)

    def run(self, t, steps, use_graph=True, **kw):
        self.a.copy_(self.start)
        self.b.fill_(7)  # (whatever the second buffer held)
        self.wmc.batch_run(self.ps, self.V, self.a, self.b, t, steps, self.ws, use_graph=use_graph, **kw)
        return self.a.cpu().numpy()

    def alone(self, s, t, steps):
        w = self.wls[s]
        return gpu_run(self.wmc, torch, self.wmc.Params.of(w), self.Vs[s], self.hs[s], t, steps)


def _sparse_state(w, rng, n):
    h = np.zeros((w.n_x, w.n_M), np.int64)
    lo = int(rng.integers(0, w.n_x // 2))
    cells = rng.integers(lo, min(w.n_x, lo + w.n_x // 3 + 1), n)
    np.add.at(h, (cells, rng.integers(0, w.n_M, n)), rng.integers(-40, 200, n))
    h[0, -1], h[-1, 0] = 90, -60  # the edges
    return h.astype(np.int32)


@pytest.mark.parametrize("ragged", [False, True])
@pytest.mark.parametrize("steps", [1, 4, 5])
def test_many_cells(wmc, steps, ragged):
    """More than 65536 cells, flat and non-flat windows, empty cells between the
    occupied ones; ragged: momentum grids that are no multiple of four (also the
    rows after them are then unaligned) and Q over all row forms."""
    rng = np.random.Generator(np.random.PCG64(steps))
    wls = wi.batch_workloads(26, seed=5, n_x_range=(2500, 3200), n0_range=(10, 20))
    wls.append(wi.batch_workloads(1, seed=6, n_x_range=(5, 5))[0].replace(sim=99))
    if ragged:
        for s, (Q, n_M) in enumerate([(30, 30), (62, 126), (64, 34), (256, 258), (130, 130), (2, 6)]):
            wls[4 * s + 1] = wls[4 * s + 1].replace(Q=Q, n_M=n_M, dt_s=1e-17, bc_potential=s & 1, child_wrap=s & 1)
    Vs = [wi.potential(w).astype(np.float32) for w in wls]
    Vs[0] = rng.uniform(-0.2, 0.2, wls[0].n_x).astype(np.float32)
    Vs[2][:] = 0.0
    hs = [_sparse_state(w, rng, 400) for w in wls]
    B = _Batch(wmc, wls, Vs, hs)
    assert sum(w.n_x for w in wls) > 65536
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        got = B.run(3, steps)
        c = wmc.batch_get_counters(B.ps, B.ws)
    pairs = absorbed = 0
    for q, w in enumerate(wls):
        ref, ca = B.alone(q, 3, steps)
        np.testing.assert_array_equal(got[B.ho[q]:B.ho[q + 1]].reshape(w.n_x, w.n_M), ref, err_msg=str(q))
        pairs += ca["pairs"]
        absorbed += ca["absorbed"]
    assert c["pairs"] == pairs > 0 and c["absorbed"] == absorbed and c["flags"] == 0


def _busy(n, seed, scale):
    """Simulations of 40 cells whose particles create a pair with probability 0.2 to 0.5 in a step."""
    rng = np.random.Generator(np.random.PCG64(seed))
    wls = [wi.BARRIER_100.replace(name=f"busy-{s}", n_x=40, Q=32, n_M=64, dt_s=8e-16, sim=s, seed=11 + s) for s in range(n)]
    Vs = [rng.uniform(-0.1, 0.1, 40).astype(np.float32) for _ in wls]
    return wls, Vs, [rng.integers(-scale, scale, size=(40, 64)).astype(np.int32) for _ in wls]


def test_more_event_quads_than_the_batch_queue(wmc):
    """2^21 queue entries of up to four ids, more than 4 x 2^21 pairs in a step:
    the pair kernel walks the ids of the whole batch again."""
    wls, Vs, hs = _busy(3, 2, 10_000)
    B = _Batch(wmc, wls, Vs, hs)
    got = B.run(5, 1, use_graph=False)
    c = wmc.batch_get_counters(B.ps, B.ws)
    pairs = 0
    for q, w in enumerate(wls):
        ref, ca = B.alone(q, 5, 1)
        np.testing.assert_array_equal(got[B.ho[q]:B.ho[q + 1]].reshape(w.n_x, w.n_M), ref)
        pairs += ca["pairs"]
    assert c["pairs"] == pairs > 4 * 2 ** 21 and c["flags"] == 0


@pytest.mark.parametrize("scale", [3, 60, 1000])
def test_events_by_ids_and_by_quads(wmc, scale):
    """The pair kernels take a thread per id of a queued quad up to a quarter of
    their threads, a thread per quad beyond (scale 1000: 4e5 quads and more): each
    simulation against the oracle, the batch against each simulation."""
    wls, Vs, hs = _busy(3, scale, scale)
    B = _Batch(wmc, wls, Vs, hs)
    got = B.run(5, 2, use_graph=False)
    c = wmc.batch_get_counters(B.ps, B.ws)
    pairs = 0
    for q, w in enumerate(wls):
        ref, ca = B.alone(q, 5, 2)
        np.testing.assert_array_equal(got[B.ho[q]:B.ho[q + 1]].reshape(w.n_x, w.n_M), ref)
        pairs += ca["pairs"]
        full, half = oracle_tables(w, Vs[q])
        want, st = oracle.simulate(oracle.params(w), hs[q], 5, 2, table=full)
        out, co = gpu_run_table(wmc, torch, wmc.Params.of(w), half, hs[q], 5, 2)
        np.testing.assert_array_equal(out, want)
        assert co["pairs"] == st[oracle.ST_PAIRS] and co["flags"] == 0
    assert c["pairs"] == pairs > 0 and c["flags"] == 0


def test_more_event_quads_than_the_queue_of_one_simulation(wmc):
    """The same for one simulation, against the oracle."""
    wls, Vs, hs = _busy(1, 3, 30_000)
    wl, V, h0 = wls[0], Vs[0], hs[0]
    full, half = oracle_tables(wl, V)
    ref, st = oracle.simulate(oracle.params(wl), h0, 1, 1, table=full)
    got, c = gpu_run_table(wmc, torch, wmc.Params.of(wl), half, h0, 1, 1)
    assert st[oracle.ST_PAIRS] > 4 * 2 ** 21
    np.testing.assert_array_equal(got, ref)
    assert c["pairs"] == st[oracle.ST_PAIRS] and c["flags"] == 0


def test_captured_runs_of_several_batches(wmc):
    """Batches in turn, more of them than the captured runs that are kept, each
    with its own buffers, potentials and parameters: the bits of direct launches."""
    Bs = []
    for k in range(6):
        wls = wi.batch_workloads(3, seed=30 + k // 2, n_x_range=(60, 90), n0_range=(5_000, 9_000))
        if k % 2:  # the same but for one seed
            wls[1] = wls[1].replace(seed=77)
        Vs = [wi.potential(w).astype(np.float32) + np.float32(0.01 * k) * (np.arange(w.n_x) > 40) for w in wls]
        Bs.append(_Batch(wmc, wls, [v.astype(np.float32) for v in Vs], [wi.initial_histogram(w) for w in wls]))
    direct = [B.run(1, 4, use_graph=False) for B in Bs]
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        for order in ([0, 1, 2, 3], [3, 0, 2, 1], [0, 1, 2, 3, 4, 5], [5, 0, 4, 1, 3, 2], [0, 5, 0, 5]):
            for k in order:
                np.testing.assert_array_equal(Bs[k].run(1, 4), direct[k], err_msg=str((order, k)))
