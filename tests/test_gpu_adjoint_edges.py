"""The adjoint's sums and the smooth potential at their edges: window lengths and
domains that fill no chunk of rows, barriers whose edges lie just inside and far
outside the reach of FP32 exponentials, and a gradient that is not finite."""
import numpy as np
import pytest

import wmc_inputs as wi
from oracle import adjoint as oa  # noqa: F401  (the oracle package is importable here)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def wmc():
    from paper_1806_00082_gb300 import build, wmc as w
    build.build()
    w.load()
    return w


def _params(wmc, n_x, Q):
    return wmc.Params.of(wi.TANH_BARRIERS_4096.replace(n_x=n_x, Q=Q, n_M=Q))


@pytest.mark.parametrize("n_x,Q", [(1, 4), (31, 64), (255, 62), (257, 130), (300, 256), (513, 90)])
def test_vbar_sums(wmc, n_x, Q):
    """Vbar against the FP64 sum over the FP32 Abar the call leaves: compensated
    FP32 sums of at most 2 h terms, so within 2^-22 of the magnitudes."""
    h, n_pot = Q // 2, 3
    p = _params(wmc, n_x, Q)
    ws = wmc.workspace(p)
    wmc.init(p, ws)
    g = torch.Generator(device="cuda").manual_seed(n_x)
    VWh = torch.randn((n_pot * n_x, h), device="cuda", generator=g)
    gV = torch.randn((n_pot * n_x, h), device="cuda", generator=g)
    abar = torch.empty_like(VWh)
    Vbar = torch.empty((n_pot, n_x), dtype=torch.float32, device="cuda")
    import ctypes
    wmc._check("wmc_kernel_vjp", wmc.load().wmc_kernel_vjp(ctypes.byref(p), wmc._ptr(VWh), wmc._ptr(gV), None, n_pot,
                                                           wmc._ptr(abar), wmc._ptr(Vbar), wmc._ptr(ws), wmc._stream()))
    A = abar.double().cpu().numpy().reshape(n_pot, n_x, h)
    ref, mag = np.zeros((n_pot, n_x)), np.zeros((n_pot, n_x))
    for m in range(1, h):
        if m >= n_x:
            break
        ref[:, m:] += A[:, :n_x - m, m - 1]
        ref[:, :n_x - m] -= A[:, m:, m - 1]
        mag[:, m:] += np.abs(A[:, :n_x - m, m - 1])
        mag[:, :n_x - m] += np.abs(A[:, m:, m - 1])
    assert np.all(np.abs(Vbar.cpu().numpy() - ref) <= 2.0 ** -22 * mag + 1e-30)


@pytest.mark.parametrize("n_x,nb,ns", [(64, 2, 3), (700, 3, 0), (4096, 16, 16), (1000, 0, 300)])
def test_smooth_potential_and_its_adjoint(wmc, n_x, nb, ns):
    """V and its adjoint against FP64 tanh: a few units of FP32 rounding per window
    on the value and on its sums."""
    p = _params(wmc, n_x, 64)
    rng = np.random.Generator(np.random.PCG64(n_x))
    L, eps = n_x * 0.25, 0.5
    th = np.concatenate([rng.uniform(0.05, 0.3, (2, nb)), rng.uniform(1, 5, (2, nb)), rng.uniform(0, L, (2, nb)),
                         rng.uniform(-0.02, 0.02, (2, ns))], 1).astype(np.float32)
    T = torch.from_numpy(th).cuda()
    V = wmc.potential_tanh(p, T, nb, ns, eps).cpu().numpy()
    t = torch.from_numpy(th.astype(np.float64)).requires_grad_(True)
    x = (torch.arange(n_x, dtype=torch.float64) + 0.5) * 0.25
    ref = torch.zeros(2, n_x, dtype=torch.float64)
    for k in range(nb):
        h, w, c = t[:, k:k + 1], t[:, nb + k:nb + k + 1], t[:, 2 * nb + k:2 * nb + k + 1]
        ref = ref + 0.5 * h * (torch.tanh((x - c + w / 2) / eps) - torch.tanh((x - c - w / 2) / eps))
    for s in range(ns):
        o = t[:, 3 * nb + s:3 * nb + s + 1]
        ref = ref + 0.5 * o * (torch.tanh((x - L * s / ns) / eps) - torch.tanh((x - L * (s + 1) / ns) / eps))
    # an edge position is rounded at |x| <= 1024 nm: 2^-14 nm over eps in the argument of a window
    assert np.abs(V - ref.detach().numpy()).max() <= 0.3 * (nb + ns) * 2.0 ** -13
    gb = torch.randn((2, n_x), generator=torch.Generator().manual_seed(1))
    got = wmc.potential_tanh_vjp(p, T, nb, ns, eps, gb.cuda()).cpu().double()
    grad, = torch.autograd.grad(ref, t, gb.double())
    assert float((got - grad).abs().max()) <= 2e-3 * float(grad.abs().max())


def test_a_gradient_that_is_not_finite_shows_in_every_parameter(wmc):
    p = _params(wmc, 4096, 64)
    T = torch.from_numpy(wi.tanh_parameters(1)).cuda()
    gb = torch.zeros((1, 4096), device="cuda")
    gb[0, 7] = float("inf")
    got = wmc.potential_tanh_vjp(p, T, 16, 16, 0.5, gb)
    assert not torch.isfinite(got).any()


def _fma32(a, b, c):
    """a b + c of FP32 arrays, rounded once: the product is exact in FP64, the
    FP64 sum is rounded to odd (by its TwoSum error), which rounds on correctly."""
    p, c = a.astype(np.float64) * b.astype(np.float64), c.astype(np.float64)
    s = p + c
    t = s - p
    err = (p - (s - t)) + (c - t)
    even = (s.view(np.int64) & 1) == 0
    s = np.where((err != 0) & even, np.nextafter(s, np.where(err > 0, np.inf, -np.inf)), s)
    return s.astype(np.float32)


@pytest.mark.parametrize("n_x,nb,ns", [(300, 2, 0), (700, 3, 5), (1000, 0, 300), (4096, 16, 16)])
def test_potential_sums_each_window_by_one_rounding(wmc, n_x, nb, ns):
    """V bit for bit: the windows' values (each by itself, with height one) times
    their heights, added in turn with one rounding each, whether a window lies
    within the reach of the exponentials or is passed over."""
    p = _params(wmc, n_x, 64)
    rng = np.random.Generator(np.random.PCG64(n_x + ns))
    L, eps = n_x * 0.25, 0.5
    heights = np.r_[rng.uniform(0.05, 0.3, nb), rng.uniform(-0.02, 0.02, ns)].astype(np.float32)
    centres, widths = rng.uniform(0, L, nb), rng.uniform(1, 5, nb)
    if nb:  # edges 52.9 and 53.1 eps from the centre of cell 0, where windows begin to be passed over
        widths[0], centres[0] = 0.2 * eps, 0.125 + 53.0 * eps
    place = np.r_[widths, centres].astype(np.float32)

    def potential(hs):  # hs [n, nb + ns]
        th = np.concatenate([hs[:, :nb], np.tile(place, (len(hs), 1)), hs[:, nb:]], 1).astype(np.float32)
        return wmc.potential_tanh(p, torch.from_numpy(th).cuda(), nb, ns, eps).cpu().numpy()

    w = potential(np.eye(nb + ns))
    assert (w == 0).any() and ((w != 0) & (w < 1)).any()
    ref = np.zeros(n_x, np.float32)
    for k in range(nb + ns):
        ref = _fma32(np.full(n_x, heights[k]), w[k], ref)
    np.testing.assert_array_equal(potential(heights[None])[0], ref)
    for k in {0, nb + ns - 1}:
        bad = heights.copy()
        bad[k] = np.inf
        assert not np.isfinite(potential(bad[None])).any()


@pytest.mark.parametrize("n_x", [64, 106, 107, 4096])
@pytest.mark.parametrize("ns", [1, 255, 256, 257, 513])
def test_segments_beyond_one_round_of_edges(wmc, n_x, ns):
    """The edges are staged 256 segments at a time: each segment by itself at its
    place, and all of them added in turn with one rounding each, on domains that
    every window reaches (53 eps and less) and on wider ones."""
    p = _params(wmc, n_x, 64)
    rng = np.random.Generator(np.random.PCG64(n_x + ns))
    eps, L = 0.5, n_x * 0.25
    heights = rng.uniform(-0.02, 0.02, ns).astype(np.float32)
    w = wmc.potential_tanh(p, torch.from_numpy(np.eye(ns, dtype=np.float32)).cuda(), 0, ns, eps).cpu().numpy()
    x = (np.arange(n_x) + 0.5) * 0.25
    s = np.arange(ns)[:, None]
    exact = 0.5 * (np.tanh((x - L * s / ns) / eps) - np.tanh((x - L * (s + 1) / ns) / eps))
    # an edge position is rounded at |x| <= 1024 nm: 2^-14 nm over eps in the argument of a window
    assert np.abs(w - exact).max() <= 2.0 ** -13
    ref = np.zeros(n_x, np.float32)
    for k in range(ns):
        ref = _fma32(np.full(n_x, heights[k]), w[k], ref)
    got = wmc.potential_tanh(p, torch.from_numpy(heights[None]).cuda(), 0, ns, eps).cpu().numpy()[0]
    np.testing.assert_array_equal(got, ref)
