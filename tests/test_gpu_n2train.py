"""The trained N = 2 network on the GPU (wmc_n2_train / wmc_n2_eval) against
the FP64 oracle (oracle/n2train.py): the model's rows at the analytic weights
and at perturbed weights, SGD trajectories of several learning rates in one
launch fed the oracle's targets (trained weights and per-epoch losses), zero
loss where N = 2 is exact, determinism."""
import numpy as np
import pytest

import oracle
import wmc_inputs as wi
from oracle import n2train as nt
from tests._util import normwise

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N_X, Q = 64, 16


@pytest.fixture(scope="module")
def wmc():
    from paper_1806_00082_gb300 import build, wmc as w
    build.build()
    w.load()
    return w


def _wl(n_x=N_X, q=Q, bc=0):
    return wi.N2_TRAIN.replace(n_x=n_x, Q=q, n_M=q, bc_potential=bc)


def _targets(w, Vs):
    p = oracle.params(w)
    return np.stack([oracle.kernel_rows(p, V, np.arange(w.n_x))[:, w.Q // 2:] for V in Vs]).astype(np.float32)


@pytest.mark.parametrize("bc", [0, 1])
def test_eval_at_analytic_weights_is_the_n2_network(wmc, bc):
    w = _wl(n_x=256, q=64, bc=bc)
    V = np.random.default_rng(1).uniform(-0.2, 0.3, w.n_x).astype(np.float32)
    p = wmc.Params.of(w)
    prm = torch.from_numpy(nt.initial_params(w.Q).astype(np.float32)).cuda()
    got = wmc.n2_eval(p, prm, torch.from_numpy(V).cuda()).cpu().numpy()
    ref = oracle.kernel_rows_n2(oracle.params(w), V, np.arange(w.n_x))[:, w.Q // 2:]
    assert normwise(got, ref) <= 1e-6


def test_eval_at_perturbed_weights_matches_oracle_model(wmc):
    w = _wl(n_x=256, q=64)
    rng = np.random.default_rng(2)
    Vs = wi.gaussian_bumps(3, n_x=w.n_x)
    prm = nt.initial_params(w.Q) + rng.normal(0.0, 0.05, w.Q + 4)
    got = wmc.n2_eval(wmc.Params.of(w), torch.from_numpy(prm.astype(np.float32)).cuda(),
                      torch.from_numpy(Vs).cuda()).cpu().numpy()
    ref = np.concatenate([nt.model(prm.astype(np.float32).astype(np.float64), V, w.Q) for V in Vs]) / nt.target_scale(w.Q)
    assert normwise(got, ref) <= 2e-6


def test_sgd_trajectories_match_oracle(wmc):
    w = _wl()
    n_ex, epochs = 8, 10
    lrs = np.array([3e-2, 1e-2, 3e-3], np.float32)
    Vs = wi.gaussian_bumps(n_ex, n_x=w.n_x, seed=4)
    T = _targets(w, Vs)
    order = wi.sgd_order(epochs, n_ex)
    p0 = nt.initial_params(w.Q)
    prm = torch.from_numpy(np.tile(p0.astype(np.float32), (lrs.size, 1))).cuda()
    loss = torch.zeros((lrs.size, epochs), device="cuda")
    wmc.n2_train(wmc.Params.of(w), torch.from_numpy(Vs).cuda(), torch.from_numpy(T).cuda(),
                 torch.from_numpy(order).cuda(), torch.from_numpy(lrs).cuda(), prm, loss)
    got, got_loss = prm.cpu().numpy().astype(np.float64), loss.cpu().numpy()
    Ts = T.astype(np.float64) * nt.target_scale(w.Q)
    for r, lr in enumerate(lrs):
        pf, hist = nt.train(p0, Vs, Ts, order, float(lr), w.Q)
        delta_ref = pf - p0
        assert np.linalg.norm(got[r] - pf) <= 1e-2 * np.linalg.norm(delta_ref), (r, lr)
        assert np.all(np.abs(got_loss[r] - hist) <= 1e-4 * hist), (r, got_loss[r], hist)
        assert hist[-1] < hist[0]


def test_zero_loss_where_n2_is_exact_and_determinism(wmc):
    w = _wl()
    V = np.zeros(w.n_x, np.float32)
    V[20:44] = np.repeat(np.random.default_rng(3).uniform(0.05, 0.3, 12), 2).astype(np.float32)
    Vs = np.stack([V, V])
    T = _targets(w, Vs)
    order = np.array([[0, 1]], np.int32)
    p0 = nt.initial_params(w.Q).astype(np.float32)
    prm = torch.from_numpy(np.tile(p0, (2, 1))).cuda()
    loss = torch.zeros((2, 1), device="cuda")
    wmc.n2_train(wmc.Params.of(w), torch.from_numpy(Vs).cuda(), torch.from_numpy(T).cuda(),
                 torch.from_numpy(order).cuda(), torch.tensor([1e-2, 1e-2], device="cuda"), prm, loss)
    scale2 = float(((T.astype(np.float64) * nt.target_scale(w.Q)) ** 2).mean())
    assert float(loss[0, 0]) <= 1e-10 * scale2
    out = prm.cpu().numpy()
    assert np.array_equal(out[0], out[1])
    assert np.abs(out[0] - p0).max() <= 1e-5


@pytest.mark.parametrize("n_x,q,runs", [(2, 6, 1), (34, 10, 3), (66, 14, 30), (96, 30, 152)])
def test_sgd_with_the_rows_split_over_ctas(wmc, n_x, q, runs):
    """Row pairs that fill no group of four and do not divide over the CTAs of a
    run (8, 4 and 1 of them), windows whose half is odd."""
    w = _wl(n_x=n_x, q=q)
    n_ex, epochs = 4, 3
    lrs = np.linspace(3e-3, 3e-2, runs).astype(np.float32)
    Vs = np.random.default_rng(n_x).uniform(-0.2, 0.3, (n_ex, n_x)).astype(np.float32)
    T = _targets(w, Vs)
    order = wi.sgd_order(epochs, n_ex)
    p0 = nt.initial_params(w.Q)
    prm = torch.from_numpy(np.tile(p0.astype(np.float32), (runs, 1))).cuda()
    loss = torch.zeros((runs, epochs), device="cuda")
    wmc.n2_train(wmc.Params.of(w), torch.from_numpy(Vs).cuda(), torch.from_numpy(T).cuda(),
                 torch.from_numpy(order).cuda(), torch.from_numpy(lrs).cuda(), prm, loss)
    got, got_loss = prm.cpu().numpy().astype(np.float64), loss.cpu().numpy()
    Ts = T.astype(np.float64) * nt.target_scale(w.Q)
    for r in sorted({0, runs // 2, runs - 1}):
        pf, hist = nt.train(p0, Vs, Ts, order, float(lrs[r]), w.Q)
        assert np.linalg.norm(got[r] - pf) <= 1e-2 * np.linalg.norm(pf - p0) + 1e-6
        assert np.all(np.abs(got_loss[r] - hist) <= 1e-4 * hist + 1e-12)


@pytest.mark.parametrize("n_x,q,companions", [(256, 64, 2), (256, 64, 29), (256, 64, 59), (256, 64, 151), (66, 14, 151),
                                              (98, 30, 39), (70, 190, 151), (4, 222, 151)])
def test_a_run_does_not_depend_on_the_other_runs(wmc, n_x, q, companions):
    """One learning rate alone (its rows over up to eight CTAs) and among others
    (over fewer, down to one): the same weights and losses, bit for bit."""
    w = _wl(n_x=n_x, q=q)
    n_ex, epochs = 3, 2
    rng = np.random.default_rng(n_x + companions)
    Vs = torch.from_numpy(rng.uniform(-0.2, 0.3, (n_ex, n_x)).astype(np.float32)).cuda()
    p = wmc.Params.of(w)
    ws = wmc.workspace(p)
    wmc.init(p, ws)
    T = wmc.kernel_eval_rows(p, Vs, ws)
    order = torch.from_numpy(wi.sgd_order(epochs, n_ex)).cuda()
    lrs = torch.from_numpy(rng.uniform(1e-3, 1e-2, 1 + companions).astype(np.float32)).cuda()
    start = torch.from_numpy((nt.initial_params(w.Q) + rng.normal(0.0, 0.02, w.Q + 4)).astype(np.float32)).cuda()

    def train(rates):
        prm, loss = start.repeat(rates.numel(), 1), torch.zeros((rates.numel(), epochs), device="cuda")
        wmc.n2_train(p, Vs, T, order, rates, prm, loss)
        return prm, loss

    prm, loss = train(lrs)
    assert torch.isfinite(prm).all() and torch.isfinite(loss).all()
    for r in {0, companions // 2, companions}:
        alone_p, alone_l = train(lrs[r:r + 1].contiguous())
        assert torch.equal(alone_p[0], prm[r]) and torch.equal(alone_l[0], loss[r])
