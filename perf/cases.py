"""Performance cases of the CPM library: what its users run, at the sizes they run it.

Single lattices (``cpm.Sim``), ensembles of lattices (``cpm.Batch``) and the
emulator network (``emulator.Ensemble``), each through its public entry
points.  The models, schedules and parameters are those of the workload
generators in ``cpm_workloads``; the large 3D tissue is laid out here at its
grown size, so that a state need not be grown from seeds first.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges,
``prepare(case, seed)`` makes a state, ``run(state)`` is one pass,
``work(case)`` the bytes and operations a pass cannot do without, and
``exact(case, seed)`` the floating-point outputs in 64 bits.
"""
from __future__ import annotations

import numpy as np
import torch

import cpm_workloads as cw
from paper_2312_09317_gb300 import cpm, emulator


def listed():
    return [
        # The 2D point-cell model, 200 x 200 with 100 cells: lattice and per-cell volumes every
        # 10 MCS.  The smallest calls: 16 rounds of 2,500 attempts per MCS.
        {"name": "points_2d_200", "kind": "lattice", "model": "points", "n": 200, "cells": 100, "a": 4, "P": 1, "mcs": 10},
        # The same model on the schedule that matches the serial chain (areas of 40 x 40, one
        # round per colour visit): 1,600 rounds of 25 attempts per MCS.
        {"name": "points_2d_200_a40", "kind": "lattice", "model": "points", "n": 200, "cells": 100, "a": 40, "P": 400, "mcs": 1},
        # A migrating 2D tissue: chemotaxis along a circular field and persistence (whose update
        # observes the lattice every MCS), centroids tracked.
        {"name": "motile_2d_256", "kind": "lattice", "model": "motile", "n": 256, "cells": 160, "a": 8, "P": 4, "mcs": 10},
        # The 3D model without Act, 256^3 with about 17,600 cells: one MCS, lattice and tallies read.
        {"name": "cubes_3d_256", "kind": "lattice", "model": "cubes", "n": 256, "a": 4, "P": 8, "mcs": 1},
        # The 3D Act tissue with fibres on a mid-size lattice, on the schedule that matches the
        # serial chain: 4,096 rounds of 4,096 attempts.
        {"name": "tissue_3d_256", "kind": "lattice", "model": "tissue", "n": 256, "a": 16, "P": 64, "mcs": 1},
        # The tissue-scale lattice: 1024^3 sites, about 0.9 M motile cells, 4,096 rounds of 262,144 attempts.
        {"name": "tissue_3d_1024", "kind": "lattice", "model": "tissue", "n": 1024, "a": 16, "P": 64, "mcs": 1},
        # Training data of the emulator: 1,024 runs of 64 x 64 sites with 16 cells, parameters from
        # a Latin hypercube; the 10 MCS between two observations, and the observation.
        {"name": "emulator_runs_1024", "kind": "runs", "members": 1024, "side": 64, "cells": 16, "mcs": 10},
        # A parameter sweep over lattices of uneven sizes (2D 64^2..512^2, 3D 64^3..128^3, 10..2,000
        # cells): one MCS of every member, and an observation of all of them.
        {"name": "ensemble_64", "kind": "ensemble", "members": 64, "recipe": 1, "mcs": 1},
        # The sixteen statistics of 512 runs from 81 observations each.
        {"name": "summarize_512", "kind": "summarize", "members": 512, "cells": 16, "snapshots": 81, "every": 10},
        # Emulator queries: a block of sweep points, and a sweep of a million.
        {"name": "predict_4001", "kind": "predict", "rows": 4001, "width": 256, "max_rows": 8192},
        {"name": "predict_1m", "kind": "predict", "rows": 1 << 20, "width": 256, "max_rows": 65536},
        # 32 Adam steps of 1,024 rows on the ensemble of five networks, and the new weights.
        {"name": "train_32x1024", "kind": "train", "steps": 32, "batch_rows": 1024, "width": 256},
    ]


def draw(rng):
    """One more case: every size spread over its range, odd ones among them."""

    def log(lo, hi):
        return lo * (hi / lo) ** rng.random()

    kind = rng.choice(["points", "motile", "cubes", "tissue", "runs", "ensemble", "summarize", "predict", "predict", "train"])
    if kind in ("points", "motile"):
        a = rng.choice([4, 4, 8, 20, 40])
        n = a * max(3, round(log(64, 512) / a))
        s = (a // 2) ** 2
        return {"kind": "lattice", "model": kind, "n": n, "cells": max(4, int(n * n / log(200, 800))), "a": a,
                "P": rng.choice([p for p in (1, 4, 25, 100, 400) if s % p == 0]), "mcs": rng.randint(1, 20)}
    if kind == "cubes":
        a = rng.choice([4, 8])
        return {"kind": "lattice", "model": kind, "n": a * round(log(48, 384) / a), "a": a, "P": rng.choice([1, 2, 4, 8]),
                "mcs": rng.randint(1, 3)}
    if kind == "tissue":
        a = rng.choice([4, 8, 16, 16])
        return {"kind": "lattice", "model": kind, "n": 16 * round(log(64, 640) / 16), "a": a,
                "P": {4: 8, 8: 16, 16: 64}[a], "mcs": 1}
    if kind == "runs":
        return {"kind": "runs", "members": int(log(20, 2048)), "side": rng.choice([32, 48, 64, 64, 80, 96]),
                "cells": rng.randint(6, 30), "mcs": rng.randint(1, 12)}
    if kind == "ensemble":
        return {"kind": "ensemble", "members": int(log(6, 96)), "recipe": rng.randint(2, 10000), "mcs": rng.randint(1, 2)}
    if kind == "summarize":
        return {"kind": "summarize", "members": int(log(20, 2048)), "cells": rng.choice([9, 16, 25, 36]),
                "snapshots": rng.randint(22, 101), "every": 10}
    if kind == "predict":
        return {"kind": "predict", "rows": int(log(100, 1 << 20)), "width": rng.choice([64, 128, 256, 256]),
                "max_rows": rng.choice([8192, 65536])}
    return {"kind": "train", "steps": rng.randint(4, 32), "batch_rows": int(log(200, 2048)),
            "width": rng.choice([64, 128, 256, 256])}


# --------------------------------------------------------------------------
# states
# --------------------------------------------------------------------------

MEMBERS, N_IN, N_HIDDEN, N_OUT = 5, 7, 4, 16
ADAM = {"lr": 5e-4, "beta1": 0.9, "beta2": 0.999, "eps": 1e-8}


def tissue(n, a, P, seed):
    """The fibre tissue of ``cpm_workloads.fibre_tissue_3d`` laid out at its grown size on the
    GPU: every site of a ball of about V_t sites around a jittered centre belongs to that
    centre's cell (the nearest one), Act values on the cells' borders; the fibre network of a
    256^3 tissue (a smaller one for a smaller lattice), repeated."""
    dev = torch.device("cuda")
    base = cw.fibre_tissue_3d(seed=seed % 1000 + 1, n=48, a=a if 48 % a == 0 else 16, c=2, P=1)  # the model's parameters
    m = min(256, n)
    fib = torch.from_numpy(cw.fibre_mask((m, m, m), np.random.default_rng(seed), cell_spacing=min(48.0, m / 4),
                                         device="cuda")).to(dev)
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    g = max(3, round(n / 10))                       # cells per axis
    step = n / g
    ctr = (torch.rand((g, g, g, 3), generator=gen, device=dev) - 0.5) * 4.0
    grid = torch.arange(g, device=dev)
    for d in range(3):
        ctr[..., d] += (grid.view([-1 if k == d else 1 for k in range(3)]) + 0.5) * step
    at = torch.remainder(ctr.floor().long(), m)
    alive = ~fib[at[..., 0], at[..., 1], at[..., 2]]
    n_cells = int(0.84 * g ** 3)                    # about 85% of the centres lie outside the fibres
    rank = torch.randperm(g ** 3, generator=gen, device=dev).view(g, g, g)
    rank = torch.where(alive, rank, g ** 3 + rank).flatten().argsort().argsort().view(g, g, g)
    alive &= rank < n_cells
    ids = torch.where(alive, rank + 1, torch.zeros_like(rank)).to(torch.int32)
    lat = np.empty((n, n, n), dtype=np.int32)
    act = np.empty((n, n, n), dtype=np.uint8)
    ax = torch.arange(n, device=dev, dtype=torch.float32) + 0.5
    cell = (ax / step).floor().long().clamp(max=g - 1)
    zc = max(1, min(n, (1 << 26) // (n * n)))
    for z0 in range(0, n, zc):
        z = slice(z0, min(n, z0 + zc))
        shape = (z.stop - z.start, n, n)
        best = torch.full(shape, 6.4 ** 2, device=dev)
        own = torch.zeros(shape, dtype=torch.int32, device=dev)
        for k in range(27):
            o = [k // 9 - 1, (k // 3) % 3 - 1, k % 3 - 1]
            i = [torch.remainder(c + d, g) for c, d in zip((cell[z], cell, cell), o)]
            idx = (i[0][:, None, None], i[1][None, :, None], i[2][None, None, :])
            d2 = torch.zeros(shape, device=dev)
            for d in range(3):
                x = (ax[z], ax, ax)[d].view([-1 if q == d else 1 for q in range(3)]) - ctr[..., d][idx]
                d2 += (x - n * torch.round(x / n)) ** 2
            near = (d2 < best) & alive[idx]
            best = torch.where(near, d2, best)
            own = torch.where(near, ids[idx], own)
        zi = torch.remainder(torch.arange(z.start, z.stop, device=dev), m)
        xi = torch.remainder(torch.arange(n, device=dev), m)
        own[fib[zi][:, xi][:, :, xi]] = -1
        border = (own > 0) & (best > 4.0 ** 2)
        draw_ = torch.randint(0, 60, shape, generator=gen, device=dev, dtype=torch.uint8)
        value = torch.where(border & (draw_ <= 30), draw_, torch.zeros_like(draw_))
        lat[z] = own.cpu().numpy()
        act[z] = value.cpu().numpy()
    return base.replace(name="tissue_%d" % n, nx=n, ny=n, nz=n, a=a, c=2, P=P, seed=int(seed) + 1, lattice=lat, act=act,
                        cell_type=np.concatenate([[0], np.ones(n_cells)]).astype(np.uint8))


def lattice_state(case, seed):
    n, a, P = case["n"], case["a"], case["P"]
    burn = 50
    if case["model"] in ("points", "motile"):
        w = cw.point_cells_2d(seed=seed + 1, n=n, n_cells=case["cells"], a=a, c=2, P=P)
        if case["model"] == "motile":
            w = cw.with_motility(w, chem=cw.circular_field(n, n, 1, 2), lambda_chem=15, lambda_pers=10, mu=0.5, dt=2)
        burn = 50 if P < 100 else 10
    elif case["model"] == "cubes":
        w = cw.cube_cells_3d(seed=seed + 1, n=n, a=a, c=2, P=P)
        burn = 20
    else:
        w = tissue(n, a, P, seed)
        burn = 6  # the balls settle at V_t; their Act values become the model's own
    sim = cpm.Sim(w)
    sim.w = w.replace(lattice=w.lattice[:1], act=None, chem_field=None)  # the host copies are not needed any more
    if case["model"] == "motile":
        sim.track_centroids(True)
    sim.step(burn)
    return {"sim": sim, "mcs": case["mcs"], "track": case["model"] == "motile",
            "out": torch.empty((w.nz, w.ny, w.nx), dtype=torch.int32, device="cuda")}


def batch_state(ws, burn, case):
    batches = []
    for dim in sorted({w.dim for w in ws}):
        b = cpm.Batch([w for w in ws if w.dim == dim])
        b.step(burn)
        rows = int(b.observation_rows()[-1])
        batches.append((b, torch.empty((rows, cpm.OBS_FIELDS), dtype=torch.int64, device="cuda"),
                        torch.empty((len(b), 2), dtype=torch.int64, device="cuda")))
    return {"batches": batches, "mcs": case["mcs"]}


def history(case, seed):
    """Observations of drifting, slowly turning cells, stacked: [S, rows, 12] and [S, members, 2]."""
    rng = np.random.default_rng([seed, 7])
    n, c, S, side = case["members"], case["cells"], case["snapshots"], cw.EMULATOR_SIDE
    cells = np.zeros((S, n, c + 1, cpm.OBS_FIELDS), dtype=np.int64)
    angle = rng.uniform(0, 2 * np.pi, (1, n, c)) + np.cumsum(rng.normal(0, 0.5, (S, n, c)), axis=0)
    speed = rng.uniform(0.2, 3.0, (1, n, 1))
    px = rng.uniform(0, side, (1, n, c)) + np.cumsum(speed * np.cos(angle) + rng.normal(0, 0.3, (S, n, c)), axis=0)
    py = rng.uniform(0, side, (1, n, c)) + np.cumsum(speed * np.sin(angle) + rng.normal(0, 0.3, (S, n, c)), axis=0)
    V = np.maximum(60, np.round(rng.normal(128, 6, (S, n, c))))
    ax, ay = np.floor(px), np.floor(py) - 6
    ox, oy = px - ax, py - ay
    cxx, cyy, cxy = rng.uniform(8, 20, (S, n, c)), rng.uniform(8, 20, (S, n, c)), rng.uniform(-4, 4, (S, n, c))
    row = cells[:, :, 1:]
    row[..., 0] = (np.mod(ay, side) * side + np.mod(ax, side)).astype(np.int64)
    row[..., 1] = V
    row[..., 2], row[..., 3] = np.round(V * ox), np.round(V * oy)
    row[..., 5] = np.round(rng.normal(170, 10, (S, n, c)))
    row[..., 6], row[..., 7] = np.round(V * (ox * ox + cxx)), np.round(V * (oy * oy + cyy))
    row[..., 9] = np.round(V * (ox * oy + cxy))
    cells[:, :, 0, 0] = -1
    member = np.empty((S, n, 2), dtype=np.int64)
    member[..., 0] = np.round(row[..., 5].sum(axis=2) * rng.uniform(0.2, 0.9, (S, n)))
    member[..., 1] = np.cumsum(rng.integers(200, 2000, (S, n)), axis=0)
    return cells.reshape(S, n * (c + 1), cpm.OBS_FIELDS), member


def network(case, seed, max_rows):
    sizes = [N_IN] + [case["width"]] * N_HIDDEN + [N_OUT]
    init = cw.mlp_init(seed + 1, MEMBERS, sizes)
    net = emulator.Ensemble(init, MEMBERS, N_IN, case["width"], N_HIDDEN, N_OUT, max_rows)
    return net, init, sizes


def transform(seed):
    """Shift, scale, log mask and validation RMSE of the outputs, as a fit sets them."""
    rng = np.random.default_rng([seed, 3])
    mask = np.array([s in emulator.LOG_STATS for s in emulator.STATS], dtype=np.uint8)
    return rng.normal(0, 1, N_OUT), rng.uniform(0.05, 0.5, N_OUT), mask, rng.uniform(0.3, 0.6, N_OUT)


def data(case, seed):
    """Training rows: inputs in [0, 1], smooth standardised targets with noise."""
    rng = np.random.default_rng([seed, 5])
    n = case["steps"] * case["batch_rows"]
    X = rng.random((n, N_IN), dtype=np.float32)
    Y = np.sin(X @ rng.normal(0, 2, (N_IN, N_OUT)) + rng.uniform(0, 6, N_OUT)) * 1.4 + rng.normal(0, 0.2, (n, N_OUT))
    return X, Y.astype(np.float32), rng.permutation(n).astype(np.int32)


def queries(case, seed):
    return np.random.default_rng([seed, 4]).random((case["rows"], N_IN), dtype=np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        return {"kind": kind, **lattice_state(case, seed)}
    if kind == "runs":
        X = cw.sweep_points(case["members"], seed + 1)
        ws = [cw.emulator_run(x, seed * 5003 + k, side=case["side"], n_cells=case["cells"]) for k, x in enumerate(X)]
        return {"kind": "batch", **batch_state(ws, 60, case)}
    if kind == "ensemble":
        # the recipe fixes sizes and parameters; the seed the Philox keys and where the cells start
        rng = np.random.default_rng(seed)
        ws = [w.replace(seed=seed * 5003 + k, lattice=np.roll(w.lattice, rng.integers(0, w.nx, w.dim), axis=(1, 2) if w.dim == 2 else (0, 1, 2)))
              for k, w in enumerate(cw.ensemble(case["members"], seed=case["recipe"]))]
        return {"kind": "batch", **batch_state(ws, 20, case)}
    if kind == "summarize":
        X = cw.sweep_points(case["members"], seed + 1)
        batch = cpm.Batch([cw.emulator_run(x, seed * 5003 + k, n_cells=case["cells"]) for k, x in enumerate(X)])
        cells, member = history(case, seed)
        return {"kind": kind, "batch": batch, "every": case["every"], "cells": torch.from_numpy(cells).cuda(),
                "member": torch.from_numpy(member).cuda(),
                "out": torch.empty((case["members"], N_OUT), dtype=torch.float64, device="cuda")}
    if kind == "predict":
        net, _, _ = network(case, seed, case["max_rows"])
        net.set_output_transform(*transform(seed), factor=3.0)
        return {"kind": kind, "net": net, "X": torch.from_numpy(queries(case, seed)).cuda()}
    net, _, _ = network(case, seed, max(case["batch_rows"], 8))
    X, Y, order = (torch.from_numpy(v).cuda() for v in data(case, seed))
    return {"kind": kind, "net": net, "X": X, "Y": Y, "order": order, "batch_rows": case["batch_rows"]}


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------

def run(state):
    kind = state["kind"]
    if kind == "lattice":
        sim = state["sim"]
        sim.step(state["mcs"])
        V, A = sim.read_tallies()
        got = {"lattice": sim.read_lattice(state["out"]), "V": V, "A": A}
        if state["track"]:
            got["sums"] = sim.read_centroid_sums()
        return got
    if kind == "batch":
        for b, cells, member in state["batches"]:
            b.step(state["mcs"])
            b.observe(cells, member)
        return [(cells, member) for _, cells, member in state["batches"]]
    if kind == "summarize":
        state["batch"].summarize(state["cells"], state["member"], state["every"], state["out"])
        return state["out"]
    if kind == "predict":
        return state["net"].predict(state["X"])
    trace = state["net"].train(state["X"], state["Y"], state["order"], state["batch_rows"], trace=True, **ADAM)
    return state["net"].get_params(), trace


# --------------------------------------------------------------------------
# work and exact values
# --------------------------------------------------------------------------

def parameters(width):
    return width * N_IN + width + (N_HIDDEN - 1) * (width * width + width) + N_OUT * width + N_OUT


def work(case):
    """Lattices: the int32 word of a site read and written once per MCS, and the read-out;
    observations and histories: read or written once; networks: two operations per weight and row
    (six with the backward pass), inputs read and outputs written once."""
    kind = case["kind"]
    if kind == "lattice":
        sites = case["n"] ** (2 if case["model"] in ("points", "motile") else 3)
        return {"bytes": sites * (8 * case["mcs"] + 8), "flops": 0}
    if kind == "runs":
        sites = case["members"] * case["side"] ** 2
        return {"bytes": sites * (8 * case["mcs"] + 4) + case["members"] * (case["cells"] + 1) * 96, "flops": 0}
    if kind == "ensemble":
        # the generator's mean over 2D members of 64^2..512^2 and 3D ones of 64^3..128^3 sites
        return {"bytes": case["members"] * 400_000 * (8 * case["mcs"] + 4), "flops": 0}
    if kind == "summarize":
        return {"bytes": case["snapshots"] * case["members"] * (case["cells"] + 1) * 96, "flops": 0}
    P = parameters(case["width"])
    if kind == "predict":
        return {"bytes": case["rows"] * (4 * N_IN + 8 * N_OUT + 1) + 2 * MEMBERS * P, "flops": 2 * MEMBERS * P * case["rows"]}
    rows = case["steps"] * case["batch_rows"]
    return {"bytes": rows * 4 * (N_IN + N_OUT + 1) + case["steps"] * MEMBERS * P * 28, "flops": 6 * MEMBERS * P * rows}


def layers(params, sizes):
    """[members, P] -> per layer (W [members, out, in], b [members, 1, out]) in 64 bits."""
    got, o = [], 0
    for i, n in zip(sizes[:-1], sizes[1:]):
        got.append((params[:, o:o + i * n].reshape(-1, n, i), params[:, o + i * n:o + i * n + n].reshape(-1, 1, n)))
        o += i * n + n
    return got


def network_output(params, sizes, X):
    H = X[None].expand(params.shape[0], -1, -1)
    net = layers(params, sizes)
    for k, (W, b) in enumerate(net):
        H = torch.baddbmm(b, H, W.transpose(1, 2))
        if k + 1 < len(net):
            H = torch.nn.functional.gelu(H)
    return H


def exact(case, seed):
    kind = case["kind"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if kind in ("predict", "train"):
        sizes = [N_IN] + [case["width"]] * N_HIDDEN + [N_OUT]
        params = torch.from_numpy(cw_init(seed + 1, sizes)).double().to(dev)
    if kind == "predict":
        shift, scale, mask, _ = (torch.from_numpy(np.asarray(v, dtype=np.float64)).to(dev) for v in transform(seed))
        means, stds = [], []
        for x in torch.from_numpy(queries(case, seed)).to(dev).split(1 << 16):
            out = network_output(params, sizes, x.double())
            y = out.mean(dim=0) * scale + shift
            means.append(torch.where(mask[None] != 0, y.exp(), y))
            stds.append(out.std(dim=0, unbiased=False))
        return torch.cat(means), torch.cat(stds), None
    if kind == "train":
        X, Y, order = (torch.from_numpy(v).to(dev) for v in data(case, seed))
        params.requires_grad_(True)
        m, v = torch.zeros_like(params), torch.zeros_like(params)
        trace = []
        for s in range(case["steps"]):
            rows = order[s * case["batch_rows"]:(s + 1) * case["batch_rows"]].long()
            loss = (network_output(params, sizes, X[rows].double()) - Y[rows].double()).square().mean(dim=(1, 2))
            (grad,) = torch.autograd.grad(loss.sum(), params)
            trace.append(loss.detach())
            with torch.no_grad():
                m = ADAM["beta1"] * m + (1 - ADAM["beta1"]) * grad
                v = ADAM["beta2"] * v + (1 - ADAM["beta2"]) * grad * grad
                mh, vh = m / (1 - ADAM["beta1"] ** (s + 1)), v / (1 - ADAM["beta2"] ** (s + 1))
                params -= ADAM["lr"] * mh / (vh.sqrt() + ADAM["eps"])
        return params.detach().cpu().numpy(), torch.stack(trace)
    if kind == "summarize":
        return torch.from_numpy(statistics_of(case, seed))
    return None  # lattices, tallies and observations are whole numbers


def cw_init(seed, sizes):
    """The initial weights, He-normal per member, as the input generator draws them."""
    out = []
    for e in range(MEMBERS):
        rng = np.random.default_rng([seed, e])
        parts = []
        for i, o in zip(sizes[:-1], sizes[1:]):
            parts += [rng.normal(0.0, (2.0 / i) ** 0.5, (o, i)).ravel(), np.zeros(o)]
        out.append(np.concatenate(parts))
    return np.asarray(out, dtype=np.float32)


def statistics_of(case, seed):
    """The sixteen statistics of the histories, every cell present throughout."""
    n, c, S, every, side = case["members"], case["cells"], case["snapshots"], case["every"], 64
    cells, member = history(case, seed)
    row = cells.reshape(S, n, c + 1, -1)[:, :, 1:].astype(np.float64)
    V, A = row[..., 1], row[..., 5]
    v_t = max(10, int(0.5 * side * side / c))
    a_t = int(round(1.2 * 12.5 * v_t ** 0.5))
    mx, my = row[..., 2] / V, row[..., 3] / V
    x, y = np.mod(row[..., 0], side) + mx, np.floor(row[..., 0] / side) + my
    step = np.diff(np.stack([x, y], axis=-1), axis=0)
    step -= side * np.rint(step / side)
    track = np.concatenate([np.zeros((1, n, c, 2)), np.cumsum(step, axis=0)])
    out = np.full((n, 16), np.nan)
    out[:, 0], out[:, 2] = V.mean(axis=(0, 2)) / v_t, A.mean(axis=(0, 2)) / a_t
    out[:, 1] = np.sqrt(V.var(axis=2).mean(axis=0)) / v_t
    out[:, 3] = np.sqrt(A.var(axis=2).mean(axis=0)) / a_t
    for j, lag in enumerate((10, 50, 200)):
        k = lag // every
        if k < S:
            out[:, 4 + j] = np.square(track[k:] - track[:-k]).sum(axis=-1).mean(axis=(0, 2))
    length = np.sqrt(np.square(step).sum(axis=-1))
    out[:, 7], out[:, 8] = (length / every).mean(axis=(0, 2)), (length / every).std(axis=(0, 2))
    k = 50 // every
    far = track[k:] - track[:-k]
    reach = np.sqrt(np.square(far).sum(axis=-1))
    out[:, 11] = (reach / 50.0 < 0.05).mean(axis=(0, 2))
    unit = np.divide(far, reach[..., None], out=np.zeros_like(far), where=reach[..., None] > 0)
    both = (reach[:-k] > 0) & (reach[k:] > 0)
    out[:, 9] = (unit[:-k] * unit[k:]).sum(axis=(0, 2, 3)) / both.sum(axis=(0, 2))
    unit = np.divide(step, length[..., None], out=np.zeros_like(step), where=length[..., None] > 0)
    pers, open_ = np.full(n, 0.5 * every), np.ones(n, dtype=bool)
    for lag in range(1, min(S - 1, 21)):
        ck = (unit[:-lag] * unit[lag:]).sum(axis=(0, 2, 3)) / ((length[:-lag] > 0) & (length[lag:] > 0)).sum(axis=(0, 2))
        open_ &= ck > 0
        pers += np.where(open_, ck * every, 0.0)
    out[:, 10] = pers
    out[:, 12] = (member[-1, :, 1] - member[0, :, 1]) / ((S - 1.0) * every * side * side)
    cm = member[..., 0]
    cc = (A.sum(axis=2) - cm) / 2.0
    out[:, 13] = (cc / (cc + cm)).mean(axis=0)
    out[:, 14] = (np.sqrt(np.square(track[-1]).sum(axis=-1)) / length.sum(axis=0)).mean(axis=1)
    xx, yy = row[..., 6] / V - mx * mx, row[..., 7] / V - my * my
    xy = row[..., 9] / V - mx * my
    t, det = xx + yy, xx * yy - xy * xy
    d = np.sqrt(np.maximum(t * t / 4 - det, 0))
    out[:, 15] = np.sqrt((t / 2 + d) / (t / 2 - d)).mean(axis=(0, 2))
    return out
