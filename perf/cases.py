"""The work this package is measured on: its public entry points at the sizes its configurations, tests and benchmark
use, from single calls on a few hundred nodes to the 608,256-node density current and the 308,097-node warm bubble.

Kinds of case (case["kind"]):
  run      a Navier-Stokes run of `steps` RK4 steps from a given state (Problem.run)
  rhs      one right-hand side with its ghost solve (Problem.rhs), the call of a user's own time stepper
  advect   a scalar-advection run in the deformational or the vortex flow (Problem.run)
  ensemble `steps` steps of a batch of uneven density currents (Ensemble.run)
  setup    stencils and weights of scattered nodes (build_stencils, build_weights)
  learned  a corrected coarse run (Mlp.run)
  train    Adam iterations on the correction's network from given parameters (Mlp.train)

Every run starts from a copy of the same state, so a pass can be repeated.  Ghost records are solved for by the
library and differ in meaning between its run modes: the prognostic records are the result.
"""
import dataclasses
import functools
import math

import numpy as np
import torch

from paper_1509_02615_gb300 import configs, learned, rbffd
from paper_1509_02615_gb300 import inputs as inp


def listed():
    return [
        # Sec. 6.1 on 64 x 64 nodes: the smallest problem of the package, bound by latency; 1000 steps are one period
        {"name": "advect_64_fp64", "kind": "advect", "flow": "deformational", "layout": "cart", "m": 64,
         "precision": 64, "steps": 100},
        # the paper's vortex flow (two velocity parts) on its hexagonal nodes at h = 0.005
        {"name": "vortex_200_fp32", "kind": "advect", "flow": "vortex", "layout": "hex", "m": 201, "precision": 32,
         "steps": 20},
        # one tendency of the rising bubble in its walled box, Cartesian, for a caller's own time stepper
        {"name": "rhs_box_125m_fp64", "kind": "rhs", "problem": "box", "layout": "cart", "h": 125.0, "n": 37, "l": 4,
         "precision": 64, "storage": "per-node"},
        # coarse density current (the learned correction's grid): a stage is a few microseconds
        {"name": "current_400m_fp32", "kind": "run", "problem": "current", "layout": "hex", "h": 400.0, "n": 37,
         "l": 4, "precision": 32, "storage": "per-node", "steps": 50},
        # Sec. 6.3 at 100 m, the middle of the paper's table, in both precisions
        {"name": "current_100m_fp32", "kind": "run", "problem": "current", "layout": "hex", "h": 100.0, "n": 37,
         "l": 4, "precision": 32, "storage": "per-node", "steps": 40},
        {"name": "current_100m_fp64", "kind": "run", "problem": "current", "layout": "hex", "h": 100.0, "n": 37,
         "l": 4, "precision": 64, "storage": "per-node", "steps": 20},
        # Sec. 6.3 at 25 m, the paper's finest: operators far larger than L2
        {"name": "current_25m_fp32", "kind": "run", "problem": "current", "layout": "hex", "h": 25.0, "n": 37, "l": 4,
         "precision": 32, "storage": "per-node", "steps": 8},
        # the warm bubble at 25 m on scattered nodes, r^9 + degree 5, n = 56, FP64: the benchmark's headline
        {"name": "bubble_25m_fp64", "kind": "run", "problem": "bubble", "layout": "scattered", "h": 25.0, "n": 56,
         "l": 5, "precision": 64, "storage": "per-node", "steps": 8},
        # a batch of density currents of uneven spacing, layout and stencil
        {"name": "ensemble_12_fp32", "kind": "ensemble", "members": 12, "draw": 7, "precision": 32,
         "storage": "per-node", "steps": 8},
        # stencils and all six operators of the warm bubble's nodes at 50 m
        {"name": "setup_50m", "kind": "setup", "h": 50.0, "n": 56, "p": 9, "l": 5, "hv_k": 3},
        # corrected coarse run, the network evaluated once per step
        {"name": "learned_400m", "kind": "learned", "h": 400.0, "steps": 50},
        # the network's training loop at its default batch
        {"name": "train_400m", "kind": "train", "h": 400.0, "batch": 4096, "iters": 8},
    ]


_MOST = 8 * 308097 * 56 * 5.0   # slot updates (an FP64 one counts as 5) of the largest listed run


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def _steps(rng, nodes, n, precision, most):
    fit = int(0.5 * _MOST / (nodes * n * (5.0 if precision == 64 else 1.0)))
    return max(1, min(int(_log(rng, 2, most)), fit))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "rhs", "advect", "ensemble", "setup", "learned", "train"])
    precision = rng.choice([32, 64])
    if kind in ("run", "rhs"):
        problem = rng.choice(["current", "box", "bubble"])
        storage = "lattice" if rng.random() < 0.2 else "per-node"
        if problem == "current":
            layout, n_l = rng.choice(["hex", "cart", "scattered"]), rng.choice([(31, 3), (37, 4), (45, 4), (56, 5)])
            h = _log(rng, 50.0 if layout == "scattered" else 26.0, 800.0)
            area = 51200.0 * 6400.0
        elif problem == "box":
            layout, n_l, h = rng.choice(["hex", "cart", "scattered"]), (37, 4), _log(rng, 40.0, 500.0)
            area = 1e8
        else:
            layout, n_l, h, area = "scattered", (56, 5), _log(rng, 40.0, 1000.0), 2e8
        if layout == "scattered":
            storage = "per-node"
        c = {"kind": kind, "problem": problem, "layout": layout, "h": round(h, 2), "n": n_l[0], "l": n_l[1],
             "precision": precision, "storage": storage}
        if kind == "run":
            c["steps"] = _steps(rng, area / h ** 2 * 1.2, n_l[0], precision, 60)
        return c
    if kind == "advect":
        flow, m = rng.choice(["deformational", "vortex"]), int(_log(rng, 24, 240))
        return {"kind": kind, "flow": flow, "layout": rng.choice(["hex", "cart"]) if flow == "vortex" else "cart",
                "m": m, "precision": precision, "steps": _steps(rng, m * m * 1.2, 37, precision, 120)}
    if kind == "ensemble":
        return {"kind": kind, "members": rng.randint(3, 10), "draw": rng.randint(8, 1000), "precision": precision,
                "storage": rng.choice(["per-node", "per-node", "lattice"]), "steps": rng.randint(2, 6)}
    if kind == "setup":
        n, p, l, k = rng.choice([(31, 7, 3, 3), (37, 7, 4, 3), (37, 9, 4, 4), (45, 7, 4, 3), (56, 9, 5, 3), (75, 7, 5, 3)])
        return {"kind": kind, "h": round(_log(rng, 60.0, 1000.0), 2), "n": n, "p": p, "l": l, "hv_k": k}
    h = rng.choice([400.0, 500.0, 800.0, round(rng.uniform(300.0, 800.0), 1)])
    if kind == "learned":
        return {"kind": kind, "h": h, "steps": rng.randint(5, 60)}
    return {"kind": kind, "h": h, "batch": rng.choice([1000, 2048, 4096, rng.randint(200, 4096)]), "iters": rng.randint(2, 10)}


# ---- inputs ---------------------------------------------------------------------------------------------------------

_FLOW = {"u": 8.0, "w": 4.0, "theta": 1.5, "pi": 1.5e-4}   # amplitudes of a developed density current's fields


def _flow(nodes, seed):
    """A developed flow [4, n_all] as a run is in after some minutes: smooth in all four fields (twelve modes of 1 to
    12 km), w = 0 on the bottom and top, u = 0 on side walls, over the case's cold or warm bubble."""
    rng = np.random.default_rng(seed)
    x0, x1, z0, z1 = nodes.domain
    x, z = (nodes.x - x0) / (x1 - x0), (nodes.z - z0) / (z1 - z0)
    across = np.ones_like(x) if nodes.period_x > 0 else np.sin(np.pi * x)
    nx, nz = max(2, int((x1 - x0) / 2000.0)), max(1, int((z1 - z0) / 2000.0))
    U = np.zeros((4, nodes.n_all))
    for f, amp in enumerate(_FLOW.values()):
        for _ in range(12):
            kx, kz = int(rng.integers(1, nx + 1)), int(rng.integers(1, nz + 1))
            v = np.cos(2 * np.pi * kx * x + rng.uniform(0, 2 * np.pi))
            v = v * (np.sin(np.pi * kz * z) if f == 1 else np.cos(np.pi * kz * z + rng.uniform(0, 0.5)))
            U[f] += amp / 4.0 * rng.uniform(0.3, 1.0) * v * (across if f == 0 else 1.0)
    U[1, :nodes.n_prog][(nodes.kind == inp.KIND_BOTTOM) | (nodes.kind == inp.KIND_TOP)] = 0.0
    U[0, :nodes.n_prog][(nodes.kind == inp.KIND_LEFT) | (nodes.kind == inp.KIND_RIGHT)] = 0.0
    return U


@functools.lru_cache(maxsize=6)
def _nodes(problem, layout, h):
    if problem == "box":
        return inp.rising_bubble_nodes(h, layout)
    if problem == "bubble":
        return inp.poisson_disk_nodes(0.0, 20000.0, 0.0, 10000.0, h, seed=1)
    if layout == "scattered":
        return inp.poisson_disk_nodes(-25600.0, 25600.0, 0.0, 6400.0, h, seed=1, periodic_x=True)
    return inp.density_current_nodes(h, layout)


def _method(case):
    """Keyword arguments of rbffd.ns_problem: the configurations' constants."""
    if case["problem"] == "bubble":
        return dict(configs.BUBBLE_METHOD)
    gamma_c = inp.ENSEMBLE_GAMMA_C.get((case["layout"], case["n"], case["l"]), 2.0 ** -6)
    return dict(n=case["n"], p=7, l=case["l"], hv_k=3, hv_p=7, mu=75.0 if case["problem"] == "current" else 10.0,
                gamma_c=gamma_c)


def _state(case, seed):
    """Nodes and initial state [4, n_all] of a Navier-Stokes case."""
    nodes = _nodes(case["problem"], case["layout"], case["h"])
    U = _flow(nodes, seed)
    if case["problem"] == "current":
        U += inp.perturbed_density_current(nodes, seed)
    elif case["problem"] == "box":
        U += inp.cone_bubble_state(nodes)
    else:
        U += inp.warm_bubble_state(nodes, amp=2.0 + 0.001 * (seed % 97))
    return nodes, U


def _advection(case, seed):
    if case["flow"] == "vortex":
        wl = configs.vortex(1.0 / (case["m"] - 1), case["layout"], "paper")
    else:
        wl = configs.advection(case["m"])
        wl.dt = 5.0 * 64 / 1000.0 / case["m"]
    rng = np.random.default_rng(seed)   # the bell, displaced, over a smooth background
    P = wl.nodes.n_prog
    x, z = wl.nodes.x[:P], wl.nodes.z[:P]
    U = inp.cosine_bell(x, z, 0.3 + 0.1 * rng.uniform(), 0.4 + 0.2 * rng.uniform(), 0.2)
    for _ in range(4):
        U = U + 0.1 * np.cos(np.pi * rng.integers(1, 5) * x) * np.cos(np.pi * rng.integers(1, 5) * z) * rng.uniform()
    return wl, U[None, :]


@functools.lru_cache(maxsize=4)
def _members(count, which):
    return inp.ensemble_members(count, seed=which, t_end=900.0)


def _ensemble(case, seed):
    return [dataclasses.replace(m, U0=m.U0 + _flow(m.nodes, 1000 * seed + r))
            for r, m in enumerate(_members(case["members"], case["draw"]))]


def _points(case, seed):
    """The warm bubble's scattered nodes with every interior node moved by up to a tenth of the spacing."""
    nodes = _nodes("bubble", "scattered", case["h"])
    move = 0.1 * case["h"] * np.random.default_rng(seed).uniform(-1.0, 1.0, (2, nodes.n_all))
    move[:, nodes.n_prog:] = 0.0
    move[:, :nodes.n_prog][:, nodes.kind != inp.KIND_INTERIOR] = 0.0
    return nodes, nodes.x + move[0], nodes.z + move[1]


_TRAIN = {"runs": 4, "snaps": 8, "lr": 2e-3}
_ALPHA = (0.25, 0.25, 0.375, 0.25)


def _network(seed):
    """Parameters of a network a while into its training: every bias and output weight non-zero."""
    P = learned.init_params(4 * 36 + 4, seed=seed % 100003)
    rng = np.random.default_rng(seed)
    return P + (0.05 * rng.standard_normal(P.shape)).astype(np.float32)


def _dataset(case, seed):
    """Coarse nodes, snapshots [runs, snaps, n_all, 4] (ghost records filled) and targets [.., snaps - 1, n_prog, 4]."""
    nodes = _nodes("current", "hex", case["h"])
    R, K = _TRAIN["runs"], _TRAIN["snaps"]
    S = np.stack([np.stack([_flow(nodes, 100 * seed + K * r + k).T for k in range(K)]) for r in range(R)])
    T = np.stack([np.stack([1e-3 * _flow(nodes, 100 * seed + 50 + K * r + k).T[:nodes.n_prog] for k in range(K - 1)])
                  for r in range(R)])
    return nodes, np.ascontiguousarray(S, np.float32), np.ascontiguousarray(T, np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("run", "rhs"):
        nodes, U = _state(case, seed)
        pb = rbffd.ns_problem(nodes, precision=case["precision"], storage=case["storage"], **_method(case))
        U0 = rbffd.state_tensor(U, case["precision"])
        return {"case": case, "pb": pb, "U0": U0, "U": U0.clone(), "dt": nodes.h / 400.0}
    if kind == "advect":
        wl, U = _advection(case, seed)
        pb = rbffd.advection_problem(wl.nodes, precision=case["precision"], **wl.params)
        U0 = rbffd.state_tensor(U, case["precision"])
        return {"case": case, "pb": pb, "U0": U0, "U": U0.clone(), "dt": wl.dt}
    if kind == "ensemble":
        pb = rbffd.ensemble_problem(_ensemble(case, seed), precision=case["precision"], storage=case["storage"])
        U0 = pb.state()
        keep = np.concatenate([np.arange(m.nodes.n_prog) + r for m, r in zip(pb.members, pb.rec0)])
        return {"case": case, "pb": pb, "U0": U0, "U": U0.clone(), "keep": torch.as_tensor(keep, device="cuda")}
    if kind == "setup":
        nodes, x, z = _points(case, seed)
        return {"case": case, "n_prog": nodes.n_prog, "x": torch.as_tensor(x, device="cuda"),
                "z": torch.as_tensor(z, device="cuda")}
    if kind == "learned":
        nodes = _nodes("current", "hex", case["h"])
        pb = rbffd.ns_problem(nodes, precision=32)
        mlp = rbffd.Mlp(pb)
        mlp.set_params(_network(seed))
        mlp.set_scales(_scales(nodes.h))
        mlp.tune_run()
        U0 = rbffd.state_tensor(_flow(nodes, seed) + inp.perturbed_density_current(nodes, seed), 32)
        return {"case": case, "pb": pb, "mlp": mlp, "U0": U0, "U": U0.clone(), "dt": nodes.h / 400.0}
    nodes, S, T = _dataset(case, seed)
    pb = rbffd.ns_problem(nodes, precision=32)
    mlp = rbffd.Mlp(pb)
    S, T = torch.as_tensor(S, device="cuda"), torch.as_tensor(T, device="cuda")
    mlp.fit_scales(S, T, _TRAIN["runs"], _TRAIN["snaps"])
    return {"case": case, "pb": pb, "mlp": mlp, "S": S, "T": T, "P0": _network(seed), "seed": seed}


def _scales(h):
    """Feature, output and own-value scales of the developed flow at spacing h."""
    a = np.array(list(_FLOW.values()))
    return np.concatenate([a * min(1.0, h / 2000.0), 1e-3 * a, a]).astype(np.float32)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "rhs":
        return s["pb"].rhs(0.0, s["U"])
    if kind in ("run", "advect"):
        s["U"].copy_(s["U0"])
        s["pb"].run(0.0, s["dt"], case["steps"], s["U"])
        return s["U"][:s["pb"].n_prog]
    if kind == "ensemble":
        s["U"].copy_(s["U0"])
        s["pb"].run(case["steps"], s["U"])
        return s["U"][s["keep"]]
    if kind == "setup":
        idx = rbffd.build_stencils(s["x"], s["z"], s["n_prog"], case["n"])
        return idx, rbffd.build_weights(s["x"], s["z"], idx, case["p"], case["l"], _OPS, case["hv_k"])
    if kind == "learned":
        s["U"].copy_(s["U0"])
        skipped = s["mlp"].run(0.0, s["dt"], case["steps"], s["U"], alpha=_ALPHA)
        return s["U"][:s["pb"].n_prog], skipped
    s["mlp"].set_params(s["P0"])
    loss = s["mlp"].train(s["S"], s["T"], _TRAIN["runs"], _TRAIN["snaps"], case["iters"], batch=case["batch"],
                          lr=_TRAIN["lr"], seed=s["seed"])
    return s["mlp"].params(), loss


_OPS = ("dx", "dz", "lap", "dxx", "dzz", "hv")


def _count(case):
    """Prognostic nodes of a single-problem case, from its geometry."""
    kind = case["kind"]
    if kind == "advect":
        return case["m"] ** 2 * (1.155 if case["layout"] == "hex" else 1.0)
    if kind == "setup" or case.get("problem") == "bubble":
        return 20000.0 * 10000.0 / case["h"] ** 2 * 0.963
    if kind in ("run", "rhs"):
        area = 1e8 if case["problem"] == "box" else 51200.0 * 6400.0
        return area / case["h"] ** 2 * (1.155 if case["layout"] == "hex" else 1.0)
    return 51200.0 * 6400.0 / case["h"] ** 2 * 1.155


def work(case):
    """Bytes: operators and indices, or node positions, read once; the state, or parameters and samples, read and
    written once.  Flops: the stencil sums of every stage, the elimination of every system, the network's products."""
    kind = case["kind"]
    ts = case.get("precision", 32) // 8
    if kind in ("run", "rhs"):
        N, n, stages = _count(case), case["n"], 4 * case.get("steps", 0.25)
        return {"bytes": N * (n * (4 * ts + 4) + 8 * ts), "flops": stages * N * (24 * n + 56)}
    if kind == "advect":
        N, parts = _count(case), 2 if case["flow"] == "vortex" else 1
        return {"bytes": N * (37 * ((parts + 1) * ts + 4) + 2 * ts), "flops": 4 * case["steps"] * N * 37 * 2 * (parts + 1)}
    if kind == "ensemble":
        b = f = 0.0
        for m in _members(case["members"], case["draw"]):
            b += m.nodes.n_prog * (m.n * (4 * ts + 4) + 8 * ts)
            f += 4 * case["steps"] * m.nodes.n_prog * (24.0 * m.n + 56)
        return {"bytes": b, "flops": f}
    if kind == "setup":
        N, n = _count(case), case["n"]
        S = n + (case["l"] + 1) * (case["l"] + 2) // 2
        return {"bytes": N * (16 + n * (4 + 8 * len(_OPS))), "flops": N * (2 / 3 * S ** 3 + 2 * len(_OPS) * S ** 2)}
    macs = 148 * 64 + 64 * 64 + 64 * 4
    if kind == "learned":
        N = _count(case)
        return {"bytes": N * (37 * 20 + 32) + 4 * macs,
                "flops": case["steps"] * N * (4 * (24 * 37 + 56) + 2 * macs)}
    return {"bytes": 8 * macs + case["iters"] * case["batch"] * (37 + 1) * 16,
            "flops": case["iters"] * case["batch"] * 2.0 * (3 * macs - 148 * 64)}


# ---- the same in 64 bits, in plain torch ------------------------------------------------------------------------------

def _dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda").to(dtype)


def _offset(d, period):
    if period > 0.0:
        d = torch.where(d > 0.5 * period, d - period, torch.where(d < -0.5 * period, d + period, d))
    return d


def _nearest(x, z, count, n, h, period):
    """The n nearest of all nodes for each of the first `count`, by (squared distance, index): candidates from 3 x 3
    cells at least as wide as the widest stencil."""
    R = 2.6 * h * math.sqrt(n / math.pi)
    x0, z0 = x.min(), z.min()
    W = period if period > 0 else float(x.max() - x0)
    nx = max(1, int(W / R))
    nz = max(1, int(float(z.max() - z0) / R))
    assert period <= 0 or nx >= 3
    cx = ((x - x0) / (W / nx)).long().clamp(0, nx - 1)
    cz = ((z - z0) / (float(z.max() - z0) / nz)).long().clamp(0, nz - 1)
    cell = cz * nx + cx
    order = torch.argsort(cell, stable=True)
    size = torch.bincount(cell, minlength=nx * nz)
    cap = int(size.max())
    start = torch.cumsum(size, 0) - size
    slot = torch.arange(x.numel(), device="cuda") - start[cell[order]]
    table = torch.full((nx * nz + 1, cap), x.numel(), dtype=torch.long, device="cuda")
    table[cell[order], slot] = order
    out = torch.empty((count, n), dtype=torch.long, device="cuda")
    xp, zp = torch.cat([x, x.new_tensor([math.inf])]), torch.cat([z, z.new_tensor([math.inf])])
    for a in range(0, count, 16384):
        i = torch.arange(a, min(count, a + 16384), device="cuda")
        near = []
        for dz in (-1, 0, 1):
            for dx in (-1, 0, 1):
                ax, az = cx[i] + dx, cz[i] + dz
                ok = (az >= 0) & (az < nz)
                if period > 0:
                    ax = ax % nx
                else:
                    ok &= (ax >= 0) & (ax < nx)
                near.append(torch.where(ok, az * nx + ax, nx * nz))
        c, _ = torch.sort(table[torch.stack(near, 1)].reshape(i.numel(), -1), dim=1)
        ex, ez = _offset(xp[c] - x[i, None], period), zp[c] - z[i, None]
        d, at = torch.sort(ex * ex + ez * ez, dim=1, stable=True)
        assert float(d[:, n - 1].max()) < min(W / nx, float(z.max() - z0) / nz) ** 2 or nx * nz == 1
        out[i] = torch.gather(c, 1, at[:, :n])
    return out


_ORDER = {"dx": 1, "dz": 1, "lap": 2, "dxx": 2, "dzz": 2}


def _weights(x, z, idx, p, l, ops, k, period):
    """RBF-FD weights [len(ops), N, n] of r^p with polynomials to degree l, in coordinates scaled to each stencil."""
    mono = [(d - b, b) for d in range(l + 1) for b in range(d + 1)]
    N, n = idx.shape
    out = torch.empty((len(ops), N, n), dtype=torch.float64, device="cuda")
    for a in range(0, N, 8192):
        q = idx[a:a + 8192]
        ex, ez = _offset(x[q] - x[q[:, :1]], period), z[q] - z[q[:, :1]]
        r = torch.hypot(ex, ez)
        s = r.max(dim=1, keepdim=True).values
        ex, ez, r = ex / s, ez / s, r / s
        A = torch.zeros((q.shape[0], n + len(mono), n + len(mono)), dtype=torch.float64, device="cuda")
        A[:, :n, :n] = torch.hypot(ex[:, :, None] - ex[:, None, :], ez[:, :, None] - ez[:, None, :]) ** p
        b = torch.zeros((q.shape[0], n + len(mono), len(ops)), dtype=torch.float64, device="cuda")
        for c, (i, j) in enumerate(mono):
            A[:, :n, n + c] = A[:, n + c, :n] = ex ** i * ez ** j
        for o, op in enumerate(ops):
            if op in ("dx", "dz"):
                b[:, :n, o] = -p * r ** (p - 2) * (ex if op == "dx" else ez)
            elif op == "lap":
                b[:, :n, o] = p * p * r ** (p - 2)
            elif op in ("dxx", "dzz"):
                e = ex if op == "dxx" else ez
                b[:, :n, o] = p * r ** (p - 2) + p * (p - 2) * torch.where(r > 0, r, 1.0) ** (p - 4) * e * e
            else:
                b[:, :n, o] = math.prod((p - 2 * t) ** 2 for t in range(k)) * torch.where(r > 0, r, 0.0) ** (p - 2 * k)
            if op == "hv":
                b[:, 0, o] = 0.0
            for c, (i, j) in enumerate(mono):
                v = {"dx": {(1, 0): 1.0}, "dz": {(0, 1): 1.0}, "lap": {(2, 0): 2.0, (0, 2): 2.0}, "dxx": {(2, 0): 2.0},
                     "dzz": {(0, 2): 2.0}}.get(op, {}).get((i, j), 0.0)
                if op == "hv" and i % 2 == 0 and j % 2 == 0 and i + j == 2 * k:
                    v = float(math.comb(k, i // 2) * math.factorial(i) * math.factorial(j))
                b[:, n + c, o] = v
        w = torch.linalg.solve(A, b)[:, :n]
        for o, op in enumerate(ops):
            out[o, a:a + 8192] = w[:, :, o] / s ** _ORDER.get(op, 2 * k)
    return out


def _rk4(rhs, t, dt, y):
    a = rhs(t, y)
    b = rhs(t + 0.5 * dt, y + 0.5 * dt * a)
    c = rhs(t + 0.5 * dt, y + 0.5 * dt * b)
    d = rhs(t + dt, y + dt * c)
    return y + dt / 6.0 * (a + 2.0 * b + 2.0 * c + d)


class _Flow:
    """The Navier-Stokes right-hand side of a node set."""

    def __init__(self, nodes, n, p, l, hv_k, hv_p, mu, gamma_c):
        assert hv_p == p
        x, z = _dev(nodes.x), _dev(nodes.z)
        self.P, self.mu = nodes.n_prog, mu
        self.idx = _nearest(x, z, self.P, n, nodes.h, nodes.period_x)
        W = dict(zip(_OPS, _weights(x, z, self.idx, p, l, _OPS, hv_k, nodes.period_x)))
        self.dx, self.dz = W["dx"], W["dz"]
        self.hv = (-1.0) ** (hv_k + 1) * gamma_c * nodes.h ** (2 * hv_k - 1) * W["hv"]
        self.diss = mu * W["lap"] + self.hv
        self.pibar, self.dpibar = 1.0 - inp.G * z[:self.P] / (inp.CP * inp.THETA_BAR), -inp.G / (inp.CP * inp.THETA_BAR)
        kind = _dev(nodes.kind, torch.long)
        self.free = torch.ones((self.P, 4), dtype=torch.float64, device="cuda")
        self.free[:, 1][(kind == 1) | (kind == 2)] = 0.0
        self.free[:, 0][(kind == 3) | (kind == 4)] = 0.0
        own = _dev(nodes.ghost_owner, torch.long)
        self.own, self.tb = own, (kind[own] <= 2)
        self.solve = []
        for f in range(4):
            tb, lr = (("dz", "dxx"), ("dzz", "dx"), ("dz", "dx"), ("dz", "dx"))[f]
            w = torch.where(self.tb[:, None], W[tb][own], W[lr][own])
            ghost = self.idx[own] >= self.P
            G = torch.zeros((own.numel(), own.numel()), dtype=torch.float64, device="cuda")
            rows = torch.arange(own.numel(), device="cuda")[:, None].expand_as(w)
            G[rows[ghost], self.idx[own][ghost] - self.P] = w[ghost]
            same = self.solve[2] if f == 3 else self.solve[0] if f == 2 and bool(self.tb.all()) else None
            self.solve.append((torch.where(ghost, 0.0, w), same[1] if same else torch.linalg.lu_factor(G)))

    def fill(self, y):
        """All records [n_all, 4]: the prognostic ones of y and the ghosts that the boundary conditions give."""
        g = torch.empty((self.own.numel(), 4), dtype=torch.float64, device="cuda")
        at = torch.where(self.idx[self.own] >= self.P, 0, self.idx[self.own])
        for f, (w, lu) in enumerate(self.solve):
            r = -(w * y[:, f][at]).sum(1)
            if f == 3:
                th = y[self.own, 2]
                r = r + torch.where(self.tb, inp.G * th / (inp.CP * inp.THETA_BAR * (inp.THETA_BAR + th)), 0.0)
            g[:, f] = torch.linalg.lu_solve(*lu, r[:, None])[:, 0]
        return torch.cat([y[:self.P], g])

    def rhs(self, t, y):
        V = self.fill(y)
        S = [V[:, f][self.idx] for f in range(4)]
        u, w, th, pi = y[:, 0], y[:, 1], y[:, 2], y[:, 3]
        dx, dz = [(self.dx * s).sum(1) for s in S], [(self.dz * s).sum(1) for s in S]
        d = [((self.hv if f == 3 else self.diss) * s).sum(1) for f, s in enumerate(S)]
        cp = inp.CP * (inp.THETA_BAR + th)
        return self.free * torch.stack([
            -u * dx[0] - w * dz[0] - cp * dx[3] + d[0],
            -u * dx[1] - w * dz[1] - cp * dz[3] + inp.G / inp.THETA_BAR * th + d[1],
            -u * dx[2] - w * dz[2] + d[2],
            -u * dx[3] - w * (self.dpibar + dz[3]) - inp.RD / inp.CV * (self.pibar + pi) * (dx[0] + dz[1]) + d[3]], 1)

    def run(self, y, dt, steps, after=None):
        for _ in range(steps):
            add = after(self.fill(y)) if after else 0.0
            y = _rk4(self.rhs, 0.0, dt, y) + add
        return y


def _start(U, P, precision):
    """The state as the library is given it, in 64 bits."""
    return _dev(U.T[:P].astype(np.float32 if precision == 32 else np.float64))


class _Net:
    """The correction's network: weights as BF16 values, a width of 64."""

    def __init__(self, P):
        self.W1, self.b1, self.W2, self.b2, self.W3, self.b3 = (
            t.reshape(s) for t, s in zip(torch.split(P, [148 * 64, 64, 4096, 64, 256, 4]),
                                         [(148, 64), (64,), (64, 64), (64,), (64, 4), (4,)]))

    def __call__(self, X):
        def f(X):
            return torch.tanh(torch.tanh(X @ self.W1 + self.b1) @ self.W2 + self.b2) @ self.W3 + self.b3
        return f(X) - f(X.new_zeros((1, 148)))


def _round(P):
    """Parameters as the products see them: weights rounded to BF16, biases as they are."""
    at = torch.ones_like(P, dtype=torch.bool)
    for b, n in ((148 * 64, 64), (148 * 64 + 64 + 4096, 64), (148 * 64 + 128 + 4096 + 256, 4)):
        at[b:b + n] = False
    return torch.where(at, P.float().bfloat16().double(), P)


def _features(V, idx, i, scales):
    """[rows, 148]: scaled differences to the 36 neighbours, field by field, then the node's own scaled values."""
    own = V[i]
    D = (V[idx[i][:, 1:]] - own[:, None]) / scales[:4]
    return torch.cat([D.permute(0, 2, 1).reshape(own.shape[0], -1), own / scales[8:]], 1)


def _mix(v):
    """One round of the 64-bit counter hash that draws the samples."""
    v = v + np.uint64(0x9E3779B97F4A7C15)
    v = (v ^ (v >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    v = (v ^ (v >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return v ^ (v >> np.uint64(31))


def _train(case, seed):
    nodes, S, T = _dataset(case, seed)
    R, K, N = _TRAIN["runs"], _TRAIN["snaps"], nodes.n_prog
    idx = _nearest(_dev(nodes.x), _dev(nodes.z), N, 37, nodes.h, nodes.period_x)
    S, T = _dev(S), _dev(T)
    A = S[:, :-1].reshape(-1, nodes.n_all, 4)
    B = T.reshape(-1, N, 4)
    diff = torch.stack([((V[idx[:, 1:]] - V[:N, None]) ** 2).mean(dim=(0, 1)) for V in A]).mean(0)
    scales = torch.cat([diff, (B ** 2).mean(dim=(0, 1)), (A[:, :N] ** 2).mean(dim=(0, 1))]).sqrt().float().double()
    P = _dev(_network(seed))
    m, v, losses = torch.zeros_like(P), torch.zeros_like(P), []
    s = np.arange(case["batch"], dtype=np.uint64)
    with np.errstate(over="ignore"):
        for it in range(case["iters"]):
            key = _mix(np.uint64(seed) ^ _mix(np.uint64(it) * np.uint64(0x100000001) + s))
            k = _dev((key % np.uint64(R * (K - 1))).astype(np.int64), torch.long)
            i = _dev(((key >> np.uint64(32)) % np.uint64(N)).astype(np.int64), torch.long)
            V = A.reshape(-1, 4)
            own = V[k * nodes.n_all + i]
            D = (V[k[:, None] * nodes.n_all + idx[i][:, 1:]] - own[:, None]) / scales[:4]
            X = torch.cat([D.permute(0, 2, 1).reshape(own.shape[0], -1), own / scales[8:]], 1)
            q = _round(P).requires_grad_()
            loss = ((_Net(q)(X) - B[k, i] / scales[4:8]) ** 2).mean()
            g, = torch.autograd.grad(loss, q)
            losses.append(float(loss.detach()))
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            lr = _TRAIN["lr"] * 0.5 * (1.0 + math.cos(math.pi * it / case["iters"]))
            P = P - lr * (m / (1 - 0.9 ** (it + 1))) / ((v / (1 - 0.999 ** (it + 1))).sqrt() + 1e-8)
    return P.cpu().numpy(), np.array(losses)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("run", "rhs"):
        nodes, U = _state(case, seed)
        flow, y = _Flow(nodes, **_method(case)), _start(U, nodes.n_prog, case["precision"])
        return flow.rhs(0.0, y) if kind == "rhs" else flow.run(y, nodes.h / 400.0, case["steps"])
    if kind == "advect":
        wl, U = _advection(case, seed)
        q, prm, x, z = wl.nodes, wl.params, _dev(wl.nodes.x), _dev(wl.nodes.z)
        idx = _nearest(x, z, q.n_prog, prm["n"], q.h, 0.0)
        dx, dz = _weights(x, z, idx, prm["p"], prm["l"], ("dx", "dz"), 0, 0.0)
        hv, = _weights(x, z, idx, prm["hv_p"], prm["l"], ("hv",), prm["hv_k"], 0.0)
        hv = (-1.0) ** (prm["hv_k"] + 1) * prm["gamma_c"] * q.h ** (2 * prm["hv_k"] - 1) * hv
        if case["flow"] == "vortex":
            parts, coef = inp.vortex_flow_parts(q.x, q.z, prm["T"])
        else:
            parts, coef = [inp.deformational_velocity(q.x, q.z)], [(0.0, 1.0, 1.0)]
        A = [-(dx * _dev(u)[idx] + dz * _dev(v)[idx]) for u, v in parts]
        col = _dev(q.src, torch.long)[idx]

        def rhs(t, y):
            c = [a + b * math.cos(m * math.pi * t / prm["T"]) for a, b, m in coef]
            return ((sum(ck * Ak for ck, Ak in zip(c, A)) + hv) * y[:, 0][col]).sum(1, keepdim=True)

        y = _start(U, q.n_prog, case["precision"])
        for step in range(case["steps"]):
            y = _rk4(rhs, step * wl.dt, wl.dt, y)
        return y
    if kind == "ensemble":
        out = []
        for m in _ensemble(case, seed):
            flow = _Flow(m.nodes, m.n, 7, m.l, 3, 7, 75.0, m.gamma_c)
            out.append(flow.run(_start(m.U0, m.nodes.n_prog, case["precision"]), m.dt, min(case["steps"], m.n_steps)))
        return torch.cat(out)
    if kind == "setup":
        nodes, x, z = _points(case, seed)
        x, z = _dev(x), _dev(z)
        idx = _nearest(x, z, nodes.n_prog, case["n"], nodes.h, 0.0)
        return idx.int(), _weights(x, z, idx, case["p"], case["l"], _OPS, case["hv_k"], 0.0)
    if kind == "learned":
        nodes = _nodes("current", "hex", case["h"])
        flow = _Flow(nodes, 37, 7, 4, 3, 7, 75.0, 2.0 ** -6)
        net, sc = _Net(_round(_dev(_network(seed)))), _dev(_scales(nodes.h))
        dt, every = nodes.h / 400.0, torch.arange(nodes.n_prog, device="cuda")

        def correction(V):
            y = net(_features(V, flow.idx, every, sc)).clamp(-4.0, 4.0)
            return dt * _dev(np.array(_ALPHA)) * y * sc[4:8] * flow.free

        y = _start(_flow(nodes, seed) + inp.perturbed_density_current(nodes, seed), nodes.n_prog, 32)
        return flow.run(y, dt, case["steps"], correction), None
    return _train(case, seed)
