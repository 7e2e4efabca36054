"""The hi/lo split contraction (3xTF32, FP16 split) at the edges of its tiles and
of the window staging, against the FP64 oracle: row counts about a 128-row tile,
windows that fill no column tile or K block, cell lists too scattered or out of
order for one window, and rows over several potentials.  1e-6 normwise is the
accuracy the split forms are stated for."""
import numpy as np
import pytest

import oracle
import wmc_inputs as wi
from tests._util import normwise

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-6


@pytest.fixture(scope="module")
def wmc():
    from paper_1806_00082_gb300 import build, wmc as w
    build.build()
    w.load()
    return w


def _cells(kind, n, n_x, rng):
    if kind == "run":
        return np.arange(n) + (n_x - n) // 2
    if kind == "scattered":  # every tile spans more cells than one window holds
        return np.sort(rng.choice(n_x, size=n, replace=False))
    return rng.permutation(n_x)[:n]


@pytest.mark.parametrize("form", ["tf32x3", "fp16_split"])
@pytest.mark.parametrize("kind,n", [("run", 1), ("run", 129), ("run", 300), ("scattered", 127), ("scattered", 260),
                                    ("shuffled", 128)])
@pytest.mark.parametrize("Q", [4, 66, 258, 602, 1024])
def test_split_rows(wmc, form, kind, n, Q):
    wl = wi.DOUBLE_BARRIER_16384.replace(n_x=6001, Q=Q, n_M=Q, barriers=(wi.Barrier(0.25, 4e-9, 300e-9),))
    V = wi.potential(wl)
    cells = _cells(kind, n, wl.n_x, np.random.Generator(np.random.PCG64(n + Q))).astype(np.int32)
    p = wmc.Params.of(wl)
    ws = wmc.workspace(p)
    wmc.init(p, ws)
    got = wmc.kernel_eval(p, torch.from_numpy(V).cuda(), torch.from_numpy(cells).cuda(), ws,
                          prec=wmc.PRECISIONS[form]).cpu().numpy()
    pick = np.unique(np.r_[0, 1, n // 2, n - 2, n - 1, np.arange(0, n, 37)]).clip(0, n - 1)
    ref = oracle.kernel_rows(oracle.params(wl.replace(n_M=Q)), V, cells[pick])[:, Q // 2:]
    assert normwise(got[pick], ref) <= TOL
    assert wmc.get_counters(p, ws)["flags"] == 0


def _operands(V, cells, Q, net):
    """FP32 window terms [n, h] and matrix [h, h] of the N = 1 or N = 2 network, V = 0 outside."""
    h = Q // 2
    Vp = np.pad(V, h + 1).astype(np.float32)
    u = np.arange(h)[None, :]
    i = cells[:, None].astype(np.int64)
    at = lambda l: Vp[l + h + 1]
    r = np.arange(h)
    if net == 1:
        A = at(i + u + 1) - at(i - u - 1)
        A[:, h - 1] = 0
        S = np.sin(2 * np.pi * (((r[:, None] + 1) * r[None, :]) % Q) / Q)
    else:
        A = np.where((i + u) % 2 == 0, at(i + u) + at(i + u + 1), -(at(i - u - 1) + at(i - u)))
        S = np.cos(np.pi * r / Q) * np.sin(np.pi * (((2 * r[:, None] + 1) * r[None, :]) % (2 * Q)) / Q)
    return A.astype(np.float32), S.astype(np.float32)


@pytest.mark.parametrize("form", ["bf16", "fp16"])
@pytest.mark.parametrize("kind,n", [("run", 1), ("run", 300), ("scattered", 260), ("shuffled", 128)])
@pytest.mark.parametrize("Q", [4, 258, 602, 1024])
def test_one_pass_forms_and_n2(wmc, form, kind, n, Q):
    """BF16 and FP16 rows of both networks against the FP64 product of the rounded
    operands: what is left is the FP32 accumulation, one truncation of the running
    sum per MMA of 16 terms and of each product's alignment, at most
    (K / 16 + 2) 2^-22 of the sum of the terms' magnitudes."""
    wl = wi.DOUBLE_BARRIER_16384.replace(n_x=6001, Q=Q, n_M=Q, barriers=(wi.Barrier(0.25, 4e-9, 300e-9),))
    V = wi.potential(wl)
    cells = _cells(kind, n, wl.n_x, np.random.Generator(np.random.PCG64(n + Q))).astype(np.int32)
    p = wmc.Params.of(wl)
    ws = wmc.workspace(p)
    wmc.init(p, ws)
    Vd, cd = torch.from_numpy(V).cuda(), torch.from_numpy(cells).cuda()
    c = 2.0 / (6.582119569e-16 * Q)
    for net, f in ((1, wmc.kernel_eval), (2, wmc.kernel_eval_n2)):
        got = f(p, Vd, cd, ws, prec=wmc.PRECISIONS[form]).cpu().numpy().astype(np.float64)
        A, S = (torch.from_numpy(x).to(torch.bfloat16 if form == "bf16" else torch.float16).double().numpy()
                for x in _operands(V, cells, Q, net))
        bound = c * ((Q // 32 + 2) * 2.0 ** -22 * (np.abs(A) @ np.abs(S))) + 1e-6 * np.abs(A @ S) * c + 1e-30
        assert np.all(np.abs(got + c * (A @ S)) <= bound)
    assert wmc.get_counters(p, ws)["flags"] == 0


@pytest.mark.parametrize("n_pot,n_x", [(3, 50), (5, 333), (2, 128)])
def test_split_rows_over_several_potentials(wmc, n_pot, n_x):
    """Rows r over potential r / n_x: tiles that straddle two potentials or more."""
    Q = 130
    wl = wi.TANH_BARRIERS_4096.replace(n_x=n_x, Q=Q, n_M=Q)
    V = np.random.Generator(np.random.PCG64(n_x)).uniform(-0.2, 0.2, (n_pot, n_x)).astype(np.float32)
    p = wmc.Params.of(wl)
    ws = wmc.workspace(p)
    wmc.init(p, ws)
    got = wmc.kernel_eval_rows(p, torch.from_numpy(V).cuda(), ws, wmc.TF32X3).cpu().numpy().reshape(n_pot, n_x, -1)
    for b in range(n_pot):
        ref = oracle.kernel_rows(oracle.params(wl), V[b], np.arange(n_x))[:, Q // 2:]
        assert normwise(got[b], ref) <= TOL


@pytest.mark.parametrize("form,net", [("tf32x3", 1), ("fp16_split", 1), ("fp16_split", 2)])
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("Q", [2, 4, 34, 66, 258, 1024, 3580, 3582, 4096])
def test_rows_without_a_window_are_the_windows_rows(wmc, form, net, bc, Q):
    """Cells in any order, whose 128-row tiles fit no window, and rows over several
    potentials: the bits of consecutive cells (Q = 3580 is the widest window beside
    which the rows' stages have room of their own), at the domain's edges too and
    with values that are not finite."""
    n_x = 1300
    wl = wi.DOUBLE_BARRIER_16384.replace(n_x=n_x, Q=Q, n_M=Q, bc_potential=bc)
    p = wmc.Params.of(wl)
    ws = wmc.workspace(p)
    wmc.init(p, ws)
    rng = np.random.Generator(np.random.PCG64(Q + bc))
    f, prec = wmc.kernel_eval if net == 1 else wmc.kernel_eval_n2, wmc.PRECISIONS[form]
    for bad in (False, True):
        V = rng.uniform(-0.2, 0.3, n_x).astype(np.float32)
        if bad:
            V[700], V[3] = np.inf, np.nan
        Vd = torch.from_numpy(V).cuda()
        run = f(p, Vd, torch.arange(n_x, dtype=torch.int32, device="cuda"), ws, prec)
        for n in (2, 129, n_x):
            cells = np.r_[0, n_x - 1, rng.permutation(np.arange(1, n_x - 1))][:n]
            got = f(p, Vd, torch.from_numpy(cells.astype(np.int32)).cuda(), ws, prec)
            np.testing.assert_array_equal(got.cpu().numpy(), run[torch.from_numpy(cells).cuda()].cpu().numpy())
    assert wmc.get_counters(p, ws)["flags"] == 0


@pytest.mark.parametrize("form", ["tf32x3", "fp16_split"])
@pytest.mark.parametrize("Q,n_pot,n_x", [(66, 300, 1), (258, 7, 37), (1024, 3, 333), (130, 2, 129)])
def test_implicit_rows_are_the_rows_of_each_potential(wmc, form, Q, n_pot, n_x):
    wl = wi.TANH_BARRIERS_4096.replace(n_x=n_x, Q=Q, n_M=Q)
    p = wmc.Params.of(wl)
    ws = wmc.workspace(p)
    wmc.init(p, ws)
    V = torch.from_numpy(np.random.Generator(np.random.PCG64(Q)).uniform(-0.2, 0.2, (n_pot, n_x)).astype(np.float32)).cuda()
    prec = wmc.PRECISIONS[form]
    got = wmc.kernel_eval_rows(p, V, ws, prec).view(n_pot, n_x, -1)
    occ = torch.arange(n_x, dtype=torch.int32, device="cuda")
    for b in range(n_pot):
        assert torch.equal(got[b], wmc.kernel_eval(p, V[b].contiguous(), occ, ws, prec))


@pytest.mark.parametrize("n_x,Q", [(7168, 1276), (7169, 1276), (7169, 1280), (7400, 2048)])
def test_permuted_cells_of_a_domain_beyond_the_cache(wmc, n_x, Q):
    """Both sides of the line from which lists of many cells have their terms fetched
    by coalesced loads: any order gives the bits of consecutive cells."""
    wl = wi.DOUBLE_BARRIER_16384.replace(n_x=n_x, Q=Q, n_M=Q)
    p = wmc.Params.of(wl)
    ws = wmc.workspace(p)
    wmc.init(p, ws)
    rng = np.random.Generator(np.random.PCG64(n_x + Q))
    V = torch.from_numpy(rng.uniform(-0.2, 0.3, n_x).astype(np.float32)).cuda()
    run = wmc.kernel_eval(p, V, torch.arange(n_x, dtype=torch.int32, device="cuda"), ws, wmc.TF32X3)
    for n in (n_x // 2, n_x - 1, n_x):
        cells = rng.permutation(n_x)[:n]
        for c in (cells, np.sort(cells)):
            got = wmc.kernel_eval(p, V, torch.from_numpy(c.astype(np.int32)).cuda(), ws, wmc.TF32X3)
            assert torch.equal(got, run[torch.from_numpy(c).cuda()])
    assert wmc.get_counters(p, ws)["flags"] == 0
