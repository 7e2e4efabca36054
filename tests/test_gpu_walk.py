"""The particle step's walk over the survivors and the snapshot of the explicit
particles, bit for bit against the oracle, at the edges of the walk's cases:
windows of 128 ids in one bucket, in a few, in many; column blocks of 32 that
are empty, partial or beyond the first 32 blocks; cells of one particle; ranges
that start inside a cell; more quads with events than the queue holds."""
import numpy as np
import pytest

import oracle
import wmc_inputs as wi
from tests._util import gpu_run_table, oracle_tables

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wmc():
    from paper_1806_00082_gb300 import build, wmc as w
    build.build()
    w.load()
    return w


def _workload(n_x, Q, n_M):
    wl = wi.BARRIER_100.replace(name=f"walk-{n_x}-{Q}-{n_M}", n_x=n_x, Q=Q, n_M=n_M, child_wrap=int(n_M == 34))
    rng = np.random.Generator(np.random.PCG64(n_M))
    V = 0.2 * min(1.0, Q / n_M)  # gamma grows with the periods on the grid
    return wl, rng.uniform(-V, V, n_x).astype(np.float32)


def _state(kind, wl, rng):
    n_x, n_M = wl.n_x, wl.n_M
    h = np.zeros((n_x, n_M), np.int64)
    sign = rng.choice([-1, 1], size=(n_x, n_M))
    if kind == "ones":  # every bucket one particle, some cells empty
        h[:] = sign
        h[::3] = 0
    elif kind == "sizes":  # bucket sizes around a quad, a lane's limit, a window
        sizes = np.array([0, 0, 1, 2, 3, 4, 5, 7, 8, 9, 31, 127, 128, 129, 255, 256, 260, 1000])
        h[:] = sign * rng.choice(sizes, size=(n_x, n_M), p=np.r_[0.3, 0.3, np.full(16, 0.4 / 16)])
    elif kind == "far":  # a few particles in columns far apart
        for i in range(0, n_x, 2):
            k = rng.choice(n_M, size=min(n_M, 5), replace=False)
            h[i, k] = rng.integers(1, 4, size=k.size)
        h[n_x // 2, n_M - 1] = -70_000
    return h.astype(np.int32)


@pytest.mark.parametrize("kind", ["ones", "sizes", "far"])
@pytest.mark.parametrize("n_x,Q,n_M", [(7, 2, 2), (40, 32, 30), (40, 32, 34), (33, 64, 128), (24, 64, 1026), (9, 64, 2052)])
def test_walk_bit_exact(wmc, kind, n_x, Q, n_M):
    wl, V = _workload(n_x, Q, n_M)
    h0 = _state(kind, wl, np.random.Generator(np.random.PCG64(7 * n_x + n_M)))
    full, half = oracle_tables(wl, V)
    ref, st = oracle.simulate(oracle.params(wl), h0, 3, 2, table=full)
    got, c = gpu_run_table(wmc, torch, wmc.Params.of(wl), half, h0, 3, 2)
    np.testing.assert_array_equal(got, ref)
    assert c["pairs"] == st[oracle.ST_PAIRS] and c["flags"] == 0


def test_more_event_quads_than_the_queue(wmc):
    """2^21 queue entries, more quads with events in a step."""
    wl, V = _workload(40, 32, 64)
    rng = np.random.Generator(np.random.PCG64(1))
    h0 = rng.integers(-32000, 32000, size=(40, 64)).astype(np.int32)
    wl = wl.replace(dt_s=4e-16)
    full, half = oracle_tables(wl, V)
    ref, st = oracle.simulate(oracle.params(wl), h0, 1, 1, table=full)
    got, c = gpu_run_table(wmc, torch, wmc.Params.of(wl), half, h0, 1, 1)
    assert st[oracle.ST_PAIRS] > 2 * 2 ** 21
    np.testing.assert_array_equal(got, ref)
    assert c["pairs"] == st[oracle.ST_PAIRS] and c["flags"] == 0


@pytest.mark.parametrize("id_base", [0, 1, 3, 130])
@pytest.mark.parametrize("n_x,n_M", [(7, 2), (40, 34), (9, 2052)])
def test_snapshot_places_and_words(wmc, id_base, n_x, n_M):
    """Every particle at place id - id_base, its offset word from its id."""
    wl, _ = _workload(n_x, 64 if n_M > 64 else 32, n_M)
    h0 = _state("sizes", wl, np.random.Generator(np.random.PCG64(n_x + id_base)))
    p = wmc.Params.of(wl)
    ws = wmc.workspace(p)
    wmc.init(p, ws)
    wmc.set_id_base(p, ws, id_base)
    hd = torch.from_numpy(h0).cuda()
    wmc.annihilate(p, hd, ws)
    P = int(np.abs(h0).sum())
    cell, f, M, s = (x.cpu().numpy() for x in wmc.materialize(p, hd, 5, ws, P))
    n = np.abs(h0).reshape(-1)
    at = np.repeat(np.arange(n.size), n)
    np.testing.assert_array_equal(cell, at // n_M)
    np.testing.assert_array_equal(M, at % n_M - n_M // 2)
    np.testing.assert_array_equal(s, np.sign(h0.reshape(-1))[at])
    ids = np.unique(np.concatenate([np.arange(min(P, 40)), np.arange(max(0, P - 40), P), np.arange(0, P, max(1, P // 50))]))
    for i in ids:
        gid = int(i) + id_base
        w = int(oracle.philox((gid // 4, 5, 2, wl.sim), (wl.seed & 0xffffffff, wl.seed >> 32))[gid % 4])
        assert f[i] == np.float32((w >> 8) * 2.0 ** -24)


@pytest.mark.parametrize("sizes", [(15, 16, 17, 18), (17, 19, 20, 21, 24), (12, 30, 33, 40, 43), (0, 0, 31, 48, 60, 63, 64),
                                   (0, 16, 17, 90, 110, 127), (1, 2, 0, 0, 45, 80)])
@pytest.mark.parametrize("n_x,Q,n_M", [(7, 2, 2), (33, 32, 30), (33, 32, 34), (33, 64, 64), (12, 64, 1026)])
def test_windows_of_mid_sized_buckets(wmc, sizes, n_x, Q, n_M):
    """Windows that hold one, two and more buckets of more than 16 ids, beside small
    and empty ones, in columns that are few or all of a block: counted under masks, by
    a lane each or by several lanes each; drift only and with pairs."""
    wl, V = _workload(n_x, Q, n_M)
    rng = np.random.Generator(np.random.PCG64(sum(sizes) + n_M))
    h0 = (rng.choice(sizes, size=(n_x, n_M)) * rng.choice([-1, 1], size=(n_x, n_M))).astype(np.int32)
    for v in (V, np.zeros_like(V)):
        full, half = oracle_tables(wl, v)
        ref, st = oracle.simulate(oracle.params(wl), h0, 3, 2, table=full)
        got, c = gpu_run_table(wmc, torch, wmc.Params.of(wl), half, h0, 3, 2)
        np.testing.assert_array_equal(got, ref)
        assert c["pairs"] == st[oracle.ST_PAIRS] and c["flags"] == 0


@pytest.mark.parametrize("one_in", [1, 3, 8, 30])
@pytest.mark.parametrize("n_x,Q,n_M", [(5, 64, 386), (5, 64, 1026), (4, 64, 4096)])
def test_sparse_rows(wmc, n_x, Q, n_M, one_in):
    """Windows whose ids lie in more and in fewer than a dozen column blocks of a few
    ids each, over the edges of 32 blocks, with a large bucket between them; the
    step with and without pairs, and the snapshot."""
    wl, V = _workload(n_x, Q, n_M)
    if n_M > 2052:
        wl = wl.replace(dt_s=wl.dt_s / 2)  # (a particle moves one cell at most)
    rng = np.random.Generator(np.random.PCG64(one_in + n_M))
    h0 = np.where(rng.random((n_x, n_M)) < 1 / one_in, rng.choice([-3, -1, -1, 1, 1, 2], size=(n_x, n_M)), 0).astype(np.int32)
    h0[1, n_M // 2 + 5], h0[2, -1] = 333, -40
    p = wmc.Params.of(wl)
    for v in (V, np.zeros_like(V)):
        full, half = oracle_tables(wl, v)
        ref, st = oracle.simulate(oracle.params(wl), h0, 3, 2, table=full)
        got, c = gpu_run_table(wmc, torch, p, half, h0, 3, 2)
        np.testing.assert_array_equal(got, ref)
        assert c["pairs"] == st[oracle.ST_PAIRS] and c["flags"] == 0
    ws = wmc.workspace(p)
    wmc.init(p, ws)
    hd = torch.from_numpy(h0).cuda()
    wmc.annihilate(p, hd, ws)
    n = np.abs(h0).reshape(-1).astype(np.int64)
    at = np.repeat(np.arange(n.size), n)
    cell, f, M, s = (x.cpu().numpy() for x in wmc.materialize(p, hd, 5, ws, int(n.sum())))
    np.testing.assert_array_equal(cell, at // n_M)
    np.testing.assert_array_equal(M, at % n_M - n_M // 2)
    np.testing.assert_array_equal(s, np.sign(h0.reshape(-1))[at])
    for i in range(0, at.size, max(1, at.size // 300)):
        w = int(oracle.philox((i // 4, 5, 2, wl.sim), (wl.seed & 0xffffffff, wl.seed >> 32))[i % 4])
        assert f[i] == np.float32((w >> 8) * 2.0 ** -24)
