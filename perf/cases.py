"""What a user of this package has it do, as cases that can be timed: whole simulations and batches of them, snapshots
of the explicit particles, kernel rows in every precision form, the differentiation form forward and backward, and the
training of the N = 2 network.  All of it goes through the public entry points (wmc, sim, adjoint, n2train).

A case is a dict of plain values; prepare() makes its inputs on the GPU from a seed alone, run() is one pass, work()
what such a pass cannot do without, exact() the same outputs in 64 bits by plain torch (for computed numbers;
histograms and snapshots are whole numbers drawn from a counter-based generator)."""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1806_00082_gb300 import adjoint, n2train, sim, wmc

M_E = 9.1093837015e-31       # electron mass [kg]
HBAR_JS = 1.054571817e-34    # [J s]
HBAR_EVS = 6.582119569e-16   # [eV s]
EV_J = 1.602176634e-19       # [J / eV]

FORMS = ("fp32", "bf16", "fp16", "fp16_split")


def listed():
    return [
        # One simulation advanced by wmc_run's step graphs.  The smallest (a quick look at one barrier: 1e5 particles,
        # 100 cells): every step is a handful of short launches.
        {"name": "sim 100 cells", "kind": "sim", "n_x": 100, "dx_nm": 1.0, "Q": 32, "n_M": 64, "dt_fs": 0.1,
         "n0": 100_000, "x0": 0.25, "sigma_nm": 5.0, "energy": 0.1, "barriers": 1, "height": 0.2, "width_nm": 6.0,
         "noise": 0.0, "warm": 60, "steps": 100, "form": "fp32"},
        # An ordinary one, the packet still on its way to the barrier (no pairs are created): drift and annihilation.
        {"name": "sim 2000 cells", "kind": "sim", "n_x": 2000, "dx_nm": 0.5, "Q": 128, "n_M": 256, "dt_fs": 0.05,
         "n0": 10_000_000, "x0": 0.25, "sigma_nm": 20.0, "energy": 0.15, "barriers": 1, "height": 0.3,
         "width_nm": 10.0, "noise": 0.0, "warm": 20, "steps": 20, "form": "fp32"},
        # The largest: double barrier with disorder, 1e8 particles, every cell creates pairs.
        {"name": "sim 16384 cells", "kind": "sim", "n_x": 16384, "dx_nm": 0.1, "Q": 1024, "n_M": 1024,
         "dt_fs": 0.05, "n0": 100_000_000, "x0": 0.25, "sigma_nm": 50.0, "energy": 0.1, "barriers": 2,
         "height": 0.25, "width_nm": 2.0, "noise": 5e-3, "warm": 60, "steps": 4, "form": "fp32"},
        # A sweep over barriers and energies: many uneven simulations stepped together.
        {"name": "batch of 512", "kind": "batch", "n_sims": 512, "n_x_lo": 200, "n_x_hi": 4000, "n0_lo": 10_000,
         "n0_hi": 1_000_000, "shapes": 2, "steps": 4},
        # Output of a run: the explicit particles (cell, offset, momentum, sign) and the density.
        {"name": "snapshot 2000 cells", "kind": "snapshot", "n_x": 2000, "dx_nm": 0.5, "Q": 128, "n_M": 256,
         "dt_fs": 0.05, "n0": 10_000_000, "x0": 0.4, "sigma_nm": 20.0, "energy": 0.15, "t": 400},
        # Kernel rows on request.  The smallest call: every cell of a small domain, where the launch counts.
        {"name": "rows fp32 100 cells", "kind": "rows", "n_x": 100, "dx_nm": 1.0, "Q": 32, "net": 1, "form": "fp32",
         "cells": "all", "n_occ": 100},
        # The kernel table of a whole domain at full accuracy ...
        {"name": "rows fp32 16384 cells", "kind": "rows", "n_x": 16384, "dx_nm": 0.1, "Q": 1024, "net": 1,
         "form": "fp32", "cells": "all", "n_occ": 16384},
        # ... and in the fast form.
        {"name": "rows bf16 16384 cells", "kind": "rows", "n_x": 16384, "dx_nm": 0.1, "Q": 1024, "net": 1,
         "form": "bf16", "cells": "all", "n_occ": 16384},
        # Scattered occupied cells and a window that fits no tile, in the split form.
        {"name": "rows split 5001 cells", "kind": "rows", "n_x": 9001, "dx_nm": 0.1, "Q": 602, "net": 1,
         "form": "fp16_split", "cells": "ragged", "n_occ": 5001},
        # The N = 2 network's rows on a run of cells around a barrier.
        {"name": "rows n2 fp16 3600 cells", "kind": "rows", "n_x": 16384, "dx_nm": 0.1, "Q": 1024, "net": 2,
         "form": "fp16", "cells": "run", "n_occ": 3600},
        # Fitting potentials: kernel rows and gamma of 64 parametrised potentials, and the gradient of the parameters.
        {"name": "adjoint 64 potentials", "kind": "adjoint", "n_pot": 64, "n_x": 4096, "dx_nm": 0.25, "Q": 256,
         "n_M": 512, "nb": 16, "ns": 16},
        # Training the N = 2 network at the three learning rates that the paper tried.
        {"name": "train 3 rates", "kind": "train", "n_ex": 100, "n_x": 256, "dx_nm": 0.5, "Q": 64, "epochs": 3,
         "runs": 3},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(n):
    return max(2, n - (n & 1))


def _draw_domain(rng):
    Q = _even(_log(rng, 32, 1024))
    n_M = Q * rng.choice((1, 2)) if Q <= 512 else Q
    n_x = _log(rng, 100, 16384)
    dx = rng.choice((0.1, 0.25, 0.5, 1.0))
    # a particle moves at most one cell a step: |D| < 1 at the largest momentum
    most = M_E * Q * (dx * 1e-9) ** 2 / (HBAR_JS * math.pi * (n_M / 2)) * 1e15
    return {"n_x": n_x, "dx_nm": dx, "Q": Q, "n_M": n_M, "dt_fs": round(min(0.05, 0.9 * most), 4)}


def _draw_packet(rng, c, n0):
    L = c["n_x"] * c["dx_nm"]
    c.update(n0=n0, x0=round(rng.uniform(0.2, 0.6), 3), sigma_nm=round(L * rng.uniform(0.03, 0.08), 3),
             energy=round(rng.uniform(0.05, 0.3), 3), barriers=rng.choice((1, 1, 2)),
             height=round(rng.uniform(0.05, 0.4), 3), width_nm=round(L * rng.uniform(0.01, 0.05), 3),
             noise=rng.choice((0.0, 5e-3)))
    return c


def draw(rng):
    kind = rng.choice(("sim", "sim", "sim", "batch", "snapshot", "rows", "rows", "rows", "adjoint", "train"))
    if kind == "sim":
        n0 = _log(rng, 50_000, 50_000_000)
        c = _draw_packet(rng, {"kind": kind, **_draw_domain(rng)}, n0)
        steps = max(2, min(60, 120_000_000 // n0))
        c.update(warm=20, steps=steps, form=rng.choice(("fp32", "fp32", "bf16", "fp16_split")))
        return c
    if kind == "batch":
        n = _log(rng, 8, 400)
        return {"kind": kind, "n_sims": n, "n_x_lo": rng.randint(100, 400), "n_x_hi": rng.randint(500, 4000),
                "n0_lo": 5_000, "n0_hi": _log(rng, 10_000, 1_000_000), "shapes": rng.randrange(1 << 16), "steps": rng.choice((2, 3, 4))}
    if kind == "snapshot":
        c = _draw_domain(rng)
        return {"kind": kind, **c, "n0": _log(rng, 50_000, 10_000_000), "x0": round(rng.uniform(0.2, 0.6), 3),
                "sigma_nm": round(c["n_x"] * c["dx_nm"] * rng.uniform(0.03, 0.08), 3),
                "energy": round(rng.uniform(0.05, 0.3), 3), "t": rng.randint(1, 2000)}
    if kind == "rows":
        net = rng.choice((1, 1, 2))
        Q, n_x = _even(_log(rng, 32, 4096 if net == 1 else 1024)), _log(rng, 100, 16384)
        while n_x * Q * Q > 16384 * 1024 * 1024:
            n_x = max(100, n_x // 2)
        cells = rng.choice(("all", "run", "ragged"))
        n_occ = n_x if cells == "all" else rng.randint(max(1, n_x // 8), n_x)
        return {"kind": kind, "n_x": n_x, "dx_nm": rng.choice((0.1, 0.25, 0.5)), "Q": Q, "net": net,
                "form": rng.choice(FORMS), "cells": cells, "n_occ": n_occ}
    if kind == "adjoint":
        Q = _even(_log(rng, 32, 256))
        return {"kind": kind, "n_pot": _log(rng, 1, 48), "n_x": _log(rng, 300, 4096), "dx_nm": 0.25, "Q": Q,
                "n_M": Q * rng.choice((1, 2)), "nb": rng.randint(2, 16), "ns": rng.randint(2, 16)}
    return {"kind": kind, "n_ex": rng.randint(10, 100), "n_x": _even(rng.randint(96, 256)), "dx_nm": 0.5,
            "Q": _even(rng.randint(32, 64)), "epochs": rng.randint(1, 3), "runs": rng.choice((1, 3, 8, 64))}


# ---------------------------------------------------------------- inputs
def _rng(seed, salt):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 16 + salt)


def _params(c, seed, index=0):
    return wmc.Params(dx_m=c["dx_nm"] * 1e-9, mass_kg=M_E, dt_s=c.get("dt_fs", 0.01) * 1e-15, seed=int(seed) + 1,
                      n_x=c["n_x"], Q=c["Q"], n_M=c.get("n_M", c["Q"]), bc_potential=0, child_wrap=0, sim=index)


def _barriers(c, seed):
    """Potential [n_x] (FP32, eV): one or two rectangular barriers about the middle, and disorder."""
    x = (torch.arange(c["n_x"], device="cuda", dtype=torch.float64) + 0.5) * c["dx_nm"]
    L, w = c["n_x"] * c["dx_nm"], c["width_nm"]
    V = torch.zeros_like(x)
    for centre in ([L / 2] if c["barriers"] == 1 else [L / 2 - 1.75 * w, L / 2 + 1.75 * w]):
        V += c["height"] * ((x >= centre - w / 2) & (x < centre + w / 2))
    if c["noise"]:
        V += c["noise"] * (2 * torch.rand(c["n_x"], device="cuda", dtype=torch.float64, generator=_rng(seed, 1)) - 1)
    return V.float()


def _packet_weights(n_x, dx_nm, Q, n_M, x0_nm, sigma_nm, energy):
    """The Gaussian initial Wigner function's distributions over the cells and over the momenta."""
    x = (torch.arange(n_x, device="cuda", dtype=torch.float64) + 0.5) * dx_nm
    px = torch.exp(-((x - x0_nm) / sigma_nm) ** 2)
    dk = math.pi / (Q * dx_nm * 1e-9)
    k0 = math.sqrt(2 * M_E * energy * EV_J) / HBAR_JS
    M = torch.arange(n_M, device="cuda", dtype=torch.float64) - n_M // 2
    pM = torch.exp(-((M * dk - k0) * sigma_nm * 1e-9) ** 2)
    if float(pM.sum()) < 1e-30:  # the momentum falls between or outside the grid's: the nearest one
        pM = torch.zeros_like(pM)
        pM[min(n_M - 1, max(0, int(round(k0 / dk)) + n_M // 2))] = 1.0
    return px / px.sum(), pM / pM.sum()


def _packet(n_x, dx_nm, Q, n_M, x0_nm, sigma_nm, energy, n0, gen):
    """Signed counts [n_x, n_M] (int32) of about n0 positive particles of the initial packet."""
    px, pM = _packet_weights(n_x, dx_nm, Q, n_M, x0_nm, sigma_nm, energy)
    return torch.poisson((n0 * px[:, None] * pM[None, :]).float(), generator=gen).to(torch.int32)


def _snapshot_state(c, seed):
    """Signed counts of exactly n0 particles: the packet, and one in fifty scattered by pair creation, both signs."""
    g = _rng(seed, 8)
    n, far = c["n0"], c["n0"] // 50
    px, pM = _packet_weights(c["n_x"], c["dx_nm"], c["Q"], c["n_M"], c["x0"] * c["n_x"] * c["dx_nm"], c["sigma_nm"],
                             c["energy"])
    cell = torch.multinomial(px.float(), n - far, replacement=True, generator=g)
    k = torch.multinomial(pM.float(), n - far, replacement=True, generator=g)
    at = torch.cat([cell * c["n_M"] + k, torch.randint(c["n_x"] * c["n_M"], (far,), device="cuda", generator=g)])
    h = torch.bincount(at, minlength=c["n_x"] * c["n_M"])
    minus = torch.rand(h.shape, device="cuda", generator=g) < torch.where(h > 4, 0.05, 0.5)
    return torch.where(minus, -h, h).to(torch.int32).reshape(c["n_x"], c["n_M"])


def _simulation(c, seed):
    p = _params(c, seed)
    h0 = _packet(c["n_x"], c["dx_nm"], c["Q"], c["n_M"], c["x0"] * c["n_x"] * c["dx_nm"], c["sigma_nm"], c["energy"],
                 c["n0"], _rng(seed, 2))
    s = sim.Simulation(p, _barriers(c, seed).cpu().numpy(), h0.cpu().numpy(), prec=wmc.PRECISIONS[c.get("form", "fp32")])
    s.run(c["warm"])  # into the run: annihilated pairs and their leftovers are part of the state
    return s


def _bumps(c, seed):
    """Potentials [n_ex, n_x] (FP32, eV) of single Gaussian bumps."""
    g = _rng(seed, 3)
    L = c["n_x"] * c["dx_nm"]
    x = (torch.arange(c["n_x"], device="cuda", dtype=torch.float64) + 0.5) * c["dx_nm"]
    u = torch.rand((3, c["n_ex"], 1), device="cuda", dtype=torch.float64, generator=g)
    return ((0.05 + 0.25 * u[0]) * torch.exp(-((x - L * (0.25 + 0.5 * u[1])) / (1 + 4 * u[2])) ** 2)).float()


def _theta(c, seed):
    """Parameters [n_pot, 3 nb + ns] (FP32) of the tanh-edged potential: heights, widths, centres, offsets."""
    g = _rng(seed, 4)
    nb, ns, n = c["nb"], c["ns"], c["n_pot"]
    L = c["n_x"] * c["dx_nm"]
    u = torch.rand((n, 3 * nb + ns), device="cuda", dtype=torch.float64, generator=g)
    mid = (torch.arange(nb, device="cuda", dtype=torch.float64) + 0.5) * (L / nb)
    return torch.cat([0.05 + 0.25 * u[:, :nb], 1 + 4 * u[:, nb:2 * nb],
                      mid + (L / nb) * (u[:, 2 * nb:3 * nb] - 0.5) / 2, 0.04 * u[:, 3 * nb:] - 0.02], 1).float()


def _rows_inputs(c, seed):
    L = c["n_x"] * c["dx_nm"]
    V = _barriers({**c, "barriers": 2, "height": 0.25, "width_nm": L / 100, "noise": 5e-3}, seed)
    if c["cells"] == "ragged":
        occ = torch.randperm(c["n_x"], device="cuda", generator=_rng(seed, 5))[:c["n_occ"]].sort().values
    else:
        occ = torch.arange(c["n_occ"], device="cuda") + (c["n_x"] - c["n_occ"]) // 2
    return V, occ.to(torch.int32)


def _batch(c, seed):
    rng = np.random.Generator(np.random.PCG64(c["shapes"]))
    gen = _rng(seed, 6)
    ps, Vs, hs = [], [], []
    for s in range(c["n_sims"]):
        n_x, n_M = int(rng.integers(c["n_x_lo"], c["n_x_hi"] + 1)), int(rng.choice([128, 256]))
        height, width, energy = rng.uniform(0.05, 0.5), rng.uniform(2, 20), rng.uniform(0.05, 0.3)
        n0 = int(rng.integers(c["n0_lo"], c["n0_hi"] + 1))
        one = {"n_x": n_x, "dx_nm": 0.5, "Q": n_M // 2, "n_M": n_M, "dt_fs": 0.05, "barriers": 1, "height": height,
               "width_nm": width, "noise": 0.0}
        L = n_x * 0.5
        ps.append(_params(one, seed + s, s))
        Vs.append(_barriers(one, seed))
        hs.append(_packet(n_x, 0.5, n_M // 2, n_M, L / 4, L / 20, energy, n0, gen).reshape(-1))
    return wmc.params_array(ps), torch.cat(Vs), torch.cat(hs)


def prepare(case, seed):
    c, kind = case, case["kind"]
    state = {"case": c}
    if kind == "sim":
        # graphs need a stream of the simulation's own; a pass goes on from a checkpoint
        state["stream"] = torch.cuda.Stream()
        state["stream"].wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(state["stream"]):
            s = _simulation(c, seed)
            state.update(sim=s, checkpoint=s.hist.clone(), t=s.t)
    elif kind == "batch":
        state["stream"] = torch.cuda.Stream()
        state["stream"].wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(state["stream"]):
            ps, V, a = _batch(c, seed)
            ws = wmc.batch_workspace(ps)
            wmc.batch_init(ps, ws)
            state.update(ps=ps, V=V, a=a, b=torch.empty_like(a), ws=ws, t=1)
    elif kind == "snapshot":
        p = _params(c, seed)
        ws = wmc.workspace(p)
        wmc.init(p, ws)
        state.update(p=p, ws=ws, hist=_snapshot_state(c, seed))
    elif kind == "rows":
        p = _params(c, seed)
        V, occ = _rows_inputs(c, seed)
        ws = wmc.workspace(p)
        wmc.init(p, ws)
        state.update(p=p, V=V, occ=occ, ws=ws, eval=wmc.kernel_eval if c["net"] == 1 else wmc.kernel_eval_n2)
    elif kind == "adjoint":
        p = _params(c, seed)
        ws = wmc.workspace(p)
        wmc.init(p, ws)
        g = _rng(seed, 7)
        rows = c["n_pot"] * c["n_x"]
        # the loss's gradients, as a fit's would be: of the rows (1/s) and of gamma
        gV = torch.randn((rows, c["Q"] // 2), device="cuda", generator=g)
        gg = torch.randn(rows, device="cuda", generator=g)
        state.update(p=p, ws=ws, theta=_theta(c, seed).requires_grad_(True), gV=gV, gg=gg)
    else:
        p = _params(c, seed)
        ws = wmc.workspace(p)
        wmc.init(p, ws)
        g = torch.Generator().manual_seed(int(seed))
        order = torch.stack([torch.randperm(c["n_ex"], generator=g) for _ in range(c["epochs"])]).to(torch.int32).cuda()
        state.update(p=p, ws=ws, V=_bumps(c, seed), order=order, lrs=_rates(c["runs"]).cuda())
    return state


def _rates(runs):
    """The paper's three learning rates first, then a sweep between them."""
    if runs <= 3:
        return torch.tensor([1e-4, 1e-3, 1e-5][:runs], dtype=torch.float32)
    return torch.logspace(-5, -3, runs, dtype=torch.float32)


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "sim":
        s = state["sim"]
        with torch.cuda.stream(state["stream"]):
            s.hist.copy_(state["checkpoint"])
            s.t = state["t"]
            s.run(c["steps"])
            return {"hist": s.hist, "rho": s.density()}
    if kind == "batch":
        with torch.cuda.stream(state["stream"]):
            wmc.batch_run(state["ps"], state["V"], state["a"], state["b"], state["t"], c["steps"], state["ws"])
        state["t"] += c["steps"]
        return {"hist": state["a"]}
    if kind == "snapshot":
        p, hist, ws = state["p"], state["hist"], state["ws"]
        wmc.annihilate(p, hist, ws)
        cell, f, M, sign = wmc.materialize(p, hist, c["t"], ws, c["n0"])
        return {"cell": cell, "f": f, "M": M, "sign": sign, "rho": wmc.density(p, hist)}
    if kind == "rows":
        return {"rows": state["eval"](state["p"], state["V"], state["occ"], state["ws"], wmc.PRECISIONS[c["form"]])}
    if kind == "adjoint":
        theta = state["theta"]
        rows, gamma = adjoint.kernel_of_potential(theta, state["p"], c["nb"], c["ns"], 0.5, state["ws"])
        grad, = torch.autograd.grad((rows, gamma), theta, (state["gV"], state["gg"]))
        return {"rows": rows.detach(), "gamma": gamma.detach(), "grad": grad}
    params, loss = n2train.train(state["p"], state["V"], state["order"], state["lrs"], state["ws"])
    return {"params": params, "loss": loss}


def work(case):
    """Bytes: inputs once, outputs once.  Flops: the contraction's, over the distinct columns; for particles, the
    operations of their counter-based draws (a quarter of a ten-round generator call of 40 operations each for the
    offset and for the creation word) and two comparisons."""
    c, kind = case, case["kind"]
    h = c.get("Q", 2) // 2
    if kind == "sim":
        return {"bytes": 8 * c["n_x"] * c["n_M"] + 4 * c["n_x"], "flops": 22.0 * c["n0"] * c["steps"]}
    if kind == "batch":
        cells, n0 = c["n_sims"] * (c["n_x_lo"] + c["n_x_hi"]) / 2, c["n_sims"] * (c["n0_lo"] + c["n0_hi"]) / 2
        return {"bytes": 8 * cells * 192 + 4 * cells, "flops": 22.0 * n0 * c["steps"]}
    if kind == "snapshot":
        return {"bytes": 4 * c["n_x"] * c["n_M"] + 11 * c["n0"] + 8 * c["n_x"], "flops": 11.0 * c["n0"]}
    if kind == "rows":
        return {"bytes": 4 * c["n_occ"] * h + 4 * c["n_occ"] + 4 * c["n_x"], "flops": 2.0 * max(1, h - 1) ** 2 * c["n_occ"]}
    if kind == "adjoint":
        rows = c["n_pot"] * c["n_x"]
        # forward: rows and gamma out; backward: the rows and their gradients in
        return {"bytes": rows * (3 * 4 * h + 8) + 8 * c["n_pot"] * (3 * c["nb"] + c["ns"]), "flops": 4.0 * rows * (h - 1) * h}
    steps = c["epochs"] * c["n_ex"] * c["runs"]
    return {"bytes": 4 * c["n_ex"] * c["n_x"] * (h + 1), "flops": 6.0 * c["n_x"] * h * (h - 1) * steps}


# ---------------------------------------------------------------- the same in 64 bits
def _exact_rows(V, cells, Q):
    """Rows [len(cells), Q / 2] of the N = 1 network for one FP64 potential V (zero outside the domain)."""
    h = Q // 2
    dev = V.device
    Vp = torch.nn.functional.pad(V, (h, h))
    m = torch.arange(1, max(2, h), device=dev)
    A = Vp[cells[:, None] + h + m] - Vp[cells[:, None] + h - m]
    r = torch.arange(h, device=dev)
    S = torch.sin(2 * math.pi / Q * ((m[:, None] * r[None, :]) % Q).double())
    return (-2.0 / (HBAR_EVS * Q)) * (A @ S)


def _exact_rows_n2(V, cells, Q):
    """Rows of the N = 2 network: absolute cell pairs (2 q, 2 q + 1) inside the window, each with its mean potential."""
    h = Q // 2
    dev = V.device
    Vp = torch.nn.functional.pad(V, (h + 2, h + 2))
    d = torch.arange(-h, h, device=dev)
    first = ((cells[:, None] + d) % 2) == 0
    P = (Vp[cells[:, None] + d + h + 2] + Vp[cells[:, None] + d + h + 3]) * first
    r = torch.arange(h, device=dev)
    S = torch.sin(math.pi / Q * (((2 * d[:, None] + 1) * r[None, :]) % (2 * Q)).double())
    return (-2.0 / (HBAR_EVS * Q)) * torch.cos(math.pi * r.double() / Q) * (P @ S)


def _exact_potential(theta, c, eps):
    nb, ns, n_x = c["nb"], c["ns"], c["n_x"]
    dx = float(np.float32(c["dx_nm"]))
    L = n_x * dx
    x = ((torch.arange(n_x, device=theta.device, dtype=torch.float64) + 0.5) * dx)[None, :]
    V = 0.0
    for b in range(nb):
        hb, wb, cb = theta[:, b:b + 1], theta[:, nb + b:nb + b + 1], theta[:, 2 * nb + b:2 * nb + b + 1]
        V = V + 0.5 * hb * (torch.tanh((x - cb + wb / 2) / eps) - torch.tanh((x - cb - wb / 2) / eps))
    for s in range(ns):
        V = V + 0.5 * theta[:, 3 * nb + s:3 * nb + s + 1] * (torch.tanh((x - L * s / ns) / eps)
                                                             - torch.tanh((x - L * (s + 1) / ns) / eps))
    return V


def _exact_adjoint(c, seed):
    Q, n_M, n_pot, n_x = c["Q"], c["n_M"], c["n_pot"], c["n_x"]
    h = Q // 2
    g = _rng(seed, 7)
    gV = torch.randn((n_pot * n_x, h), device="cuda", generator=g).double().reshape(n_pot, n_x, h)
    gg = torch.randn(n_pot * n_x, device="cuda", generator=g).double().reshape(n_pot, n_x)
    theta = _theta(c, seed).double().requires_grad_(True)
    V = _exact_potential(theta, c, 0.5)
    r = torch.arange(h, device="cuda")
    M = torch.arange(n_M, device="cuda") - n_M // 2
    count = torch.zeros(Q, device="cuda", dtype=torch.float64).index_add_(0, M % Q, torch.ones(n_M, device="cuda", dtype=torch.float64))
    pos, neg = count[:h].clone(), count[(Q - r) % Q].clone()
    pos[0] = neg[0] = 0
    rows_out, gamma_out, Vbar = [], [], []
    for b in range(n_pot):
        Vb = V[b].detach().requires_grad_(True)
        rows = _exact_rows(Vb, torch.arange(n_x, device="cuda"), Q)
        gamma = rows.clamp(min=0) @ pos + (-rows).clamp(min=0) @ neg
        Vbar.append(torch.autograd.grad((rows, gamma), Vb, (gV[b], gg[b]))[0])
        rows_out.append(rows.detach())
        gamma_out.append(gamma.detach())
    grad, = torch.autograd.grad(V, theta, torch.stack(Vbar))
    return {"rows": torch.cat(rows_out), "gamma": torch.cat(gamma_out), "grad": grad}


def _exact_train(c, seed):
    Q, n_x, h, runs = c["Q"], c["n_x"], c["Q"] // 2, c["runs"]
    V = _bumps(c, seed).double()
    g = torch.Generator().manual_seed(int(seed))
    order = [torch.randperm(c["n_ex"], generator=g).tolist() for _ in range(c["epochs"])]
    lr = _rates(runs).cuda().double()
    i = torch.arange(n_x, device="cuda")
    j = torch.arange(1, h, device="cuda").double()
    d = torch.arange(-h, h, device="cuda")
    first = (((i[:, None] + d) % 2) == 0).double()
    target = torch.stack([_exact_rows(v, i, Q) for v in V])[:, :, 1:] * (HBAR_EVS * Q / 2)
    Vp = torch.nn.functional.pad(V, (h, h + 1))
    Va, Vb = Vp[:, i[:, None] + d + h], Vp[:, i[:, None] + d + h + 1]
    phi = 2 * math.pi / Q * j
    cj = torch.cos(phi / 2)
    W = -torch.ones((runs, Q), device="cuda", dtype=torch.float64)
    w4 = torch.tensor([1.0, 1.0, 0.5, 0.5], device="cuda", dtype=torch.float64).repeat(runs, 1)
    n_out = n_x * (h - 1)
    df = d.double()
    losses = []
    for epoch in order:
        total = 0.0
        for e in epoch:
            a = w4[:, 2:3] * df + w4[:, 3:4] * (df + 1)                       # [R, Q]
            S, C = torch.sin(a[:, :, None] * phi), torch.cos(a[:, :, None] * phi) * phi  # [R, Q, h-1]
            A1, A2 = Va[e] * first, Vb[e] * first                               # [n_x, Q]
            P = w4[:, 0, None, None] * A1 + w4[:, 1, None, None] * A2         # [R, n_x, Q]
            res = cj * torch.bmm(P * W[:, None, :], S) - target[e]
            total = total + res.square().mean((1, 2))
            dy = res * cj * (2.0 / n_out)
            G, H = torch.bmm(dy, S.transpose(1, 2)), torch.bmm(dy, C.transpose(1, 2))  # [R, n_x, Q]
            gW = (P * G).sum(1)
            WG, WPH = W[:, None, :] * G, W[:, None, :] * P * H
            g4 = torch.stack([(WG * A1).sum((1, 2)), (WG * A2).sum((1, 2)), (WPH * df).sum((1, 2)),
                              (WPH * (df + 1)).sum((1, 2))], 1)
            W, w4 = W - lr[:, None] * gW, w4 - lr[:, None] * g4
        losses.append(total / c["n_ex"])
    return {"params": torch.cat([W, w4], 1), "loss": torch.stack(losses, 1)}


def exact(case, seed):
    if case["kind"] == "rows":
        V, occ = _rows_inputs(case, seed)
        f = _exact_rows if case["net"] == 1 else _exact_rows_n2
        parts = [f(V.double(), o.long(), case["Q"]) for o in occ.split(4096)]
        return {"rows": torch.cat(parts)}
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    if case["kind"] == "train":
        return _exact_train(case, seed)
    return None
