"""The work that a program has this library do, as measurable cases.

Kinds of case, each through the entry point that a program calls:

  lap      rlt2_lap_batched on device tiles
  ascent   one dual ascent: Context, iterate, then its duals, reduced costs and
           checkpoint copied to device buffers
  nodes    rlt2_bound_nodes on a batch of branch-and-bound nodes
  bnb      rlt2_bnb_solve to the proven optimum
  predict  Mlp.predict, row duals for Z-LAP tiles from the trained network
  grad     Mlp.grad, loss and gradients of one training batch

The reference values of `exact` are plain torch in FP64: a batched shortest
augmenting path solver, the canonical duals by Bellman-Ford, and the ascent
written on index tensors.
"""
import itertools
import math
import os

import numpy as np
import torch

from paper_1710_03732_gb300 import rlt2

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # the smallest call: a few hundred small LAPs, all launch and latency
        {"name": "lap small", "kind": "lap", "m": 7, "batch": 400, "mode": 1, "warm": False},
        # a program with its own large batch of LAPs, started from duals it kept
        {"name": "lap large", "kind": "lap", "m": 29, "batch": 150000, "mode": 1, "warm": True},
        # small grid problem with the default parameters (cold LAPs), its 50 iterations
        {"name": "ascent n8", "kind": "ascent", "n": 8, "grid": 2, "iters": 50, "mode": 1, "warm": 0, "scheme": "S1"},
        # grid problem of a branch-and-bound root, its 200 iterations
        {"name": "ascent n12", "kind": "ascent", "n": 12, "grid": 3, "iters": 200, "mode": 1, "warm": 1, "scheme": "S1"},
        # odd size, defaults (cold LAPs), dense: what a first call of the library does
        {"name": "ascent n17 cold", "kind": "ascent", "n": 17, "grid": 0, "iters": 40, "mode": 1, "warm": 0,
         "scheme": "S1"},
        # the headline problem: n = 20 dense, warm-started LAPs
        {"name": "ascent n20", "kind": "ascent", "n": 20, "grid": 0, "iters": 40, "mode": 1, "warm": 1, "scheme": "S1"},
        # the largest problem: n = 30 grid, the z array is 4.75 GB
        {"name": "ascent n30", "kind": "ascent", "n": 30, "grid": 5, "iters": 10, "mode": 1, "warm": 1, "scheme": "S1"},
        # the paper's F variant with two Z phases, on the Hungarian's own FP64 duals
        {"name": "ascent n16 F2 raw", "kind": "ascent", "n": 16, "grid": 4, "iters": 30, "mode": 0, "warm": 1,
         "scheme": "F2"},
        # 64 open nodes of an n = 22 search at depths 4 to 8, bounded together
        {"name": "nodes n22", "kind": "nodes", "n": 22, "grid": 2, "nodes": 64, "iters": 20},
        # a small problem solved to optimality, children bounded in batches
        {"name": "bnb n11", "kind": "bnb", "n": 11},
        # learned starts for every Z-LAP of an n = 20 problem
        {"name": "predict n20", "kind": "predict", "m": 18, "tiles": 144400},
        # a training batch of the learned start
        {"name": "grad", "kind": "grad", "rows": 65536, "hidden": 256},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lap", "lap", "ascent", "ascent", "ascent", "ascent", "nodes", "bnb", "predict", "grad"])
    if kind == "lap":
        m = rng.randint(3, 32)
        most = min(400000, 150000 * 29 * 29 // (m * m))
        return {"kind": kind, "m": m, "batch": _log_int(rng, 100, most), "mode": rng.choice([1, 1, 1, 0, 2]),
                "warm": rng.random() < 0.5}
    if kind == "ascent":
        n = rng.randint(6, 29)
        scheme = rng.choice(["S1", "S1", "S1", "S1", "S2", "F1", "F2", "half"])
        grid = rng.choice([g for g in (0, 2, 3, 4, 5) if g == 0 or (n % g == 0 and n > 2 * g)])
        # as many iterations as keep the pass below the largest one
        iters = _log_int(rng, 5, max(6, min(150, int(4 * (30 / n) ** 6))))
        return {"kind": kind, "n": n, "grid": grid, "iters": iters, "mode": rng.choice([1, 1, 1, 1, 0, 2]),
                "warm": rng.choice([0, 1]), "scheme": scheme}
    if kind == "nodes":
        n = rng.randint(12, 22)
        return {"kind": kind, "n": n, "grid": 0, "nodes": _log_int(rng, 3, 60), "iters": rng.randint(5, 20)}
    if kind == "bnb":
        return {"kind": kind, "n": rng.randint(7, 11)}
    if kind == "predict":
        m = rng.randint(4, 30)
        return {"kind": kind, "m": m, "tiles": _log_int(rng, 100, 144400 * 18 // m)}
    return {"kind": kind, "rows": _log_int(rng, 300, 250000), "hidden": rng.choice([256, 256, 256, 64, 128])}


# ------------------------------------------------------------------- inputs --
def _qap(case, seed):
    """F, D, B of a QAP: dense symmetric integers 0..99, or flows 0..9 at density
    one half on a Manhattan grid of case["grid"] rows; odd dense sizes get fixed
    costs and an asymmetric F."""
    n, rows = case["n"], case["grid"]
    rng = np.random.default_rng([seed, n, rows])

    def sym(hi, density):
        a = np.triu(rng.integers(0, hi + 1, (n, n)) * (rng.random((n, n)) < density), 1).astype(np.float64)
        return a + a.T

    if rows:
        cols = n // rows
        r, c = np.divmod(np.arange(n), cols)
        dist = np.abs(r[:, None] - r[None, :]) + np.abs(c[:, None] - c[None, :])
        return sym(9, 0.5), dist.astype(np.float64), np.zeros((n, n))
    F, D, B = sym(99, 1.0), sym(99, 1.0), np.zeros((n, n))
    if n % 2:
        F = F + np.triu(rng.integers(0, 20, (n, n)), 1)
        B = rng.integers(0, 2000, (n, n)).astype(np.float64)
    return F, D, B


def _partials(case, seed):
    """Nodes of depth 4..8 (less for small n): random facilities at random locations."""
    n, nodes = case["n"], case["nodes"]
    rng = np.random.default_rng([seed, n, nodes, 7])
    out = -np.ones((nodes, n), dtype=np.int32)
    for row in out:
        depth = int(rng.integers(min(4, n - 7), min(8, n - 4) + 1))
        row[rng.permutation(n)[:depth]] = rng.permutation(n)[:depth]
    return out


def _tiles(batch, m, seed):
    """Tiles as the Z stage meets them: row and column potentials of either sign
    plus slacks of which many are near zero; and row duals near the optimal ones."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 1000003 + m)
    u = 200 * torch.randn(batch, m, generator=g, device=DEV, dtype=F64)
    v = 200 * torch.randn(batch, m, generator=g, device=DEV, dtype=F64)
    slack = -60 * torch.log1p(-torch.rand(batch, m, m, generator=g, device=DEV, dtype=F64))
    tiles = u[:, :, None] + v[:, None, :] + slack
    near = u - u[:, :1] + 5 * torch.randn(batch, m, generator=g, device=DEV, dtype=F64)
    return tiles, near


def _params(case):
    scheme, kw = case["scheme"], dict(dual_mode=case["mode"], warm=case["warm"], feas_tol=0.0)
    if scheme == "half":
        return rlt2.half_z_params(**kw)
    return rlt2.params(variant=int(scheme[0] == "F"), two_phase=int(scheme[1] == "2"), **kw)


def _empty(*shape):
    return torch.empty(shape, device=DEV, dtype=F64)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "lap":
        b, m = case["batch"], case["m"]
        s["cost"], near = _tiles(b, m, seed)
        s["u0"] = near if case["warm"] else None
        s["out"] = dict(value=_empty(b), u=_empty(b, m), v=_empty(b, m),
                        row_to_col=torch.empty(b, m, device=DEV, dtype=torch.int32))
    elif kind == "ascent":
        s["F"], s["D"], s["B"] = _qap(case, seed)
        s["prm"] = _params(case)
        n = case["n"]
        m, T = n - 2, (n * (n - 1)) ** 2
        yd = n * n * (n - 1)
        s["duals"] = dict(alpha=_empty(n), beta=_empty(n), gamma=_empty(yd), delta=_empty(yd), xi=_empty(T * m),
                          psi=_empty(T * m))
        s["red"] = dict(pi_x=_empty(n * n), pi_y=_empty(T))
        s["state"] = dict(Dhat=_empty(T * m * m), Chat=_empty(T))
    elif kind == "nodes":
        s["F"], s["D"], s["B"] = _qap(case, seed)
        s["partials"] = _partials(case, seed)
        s["prm"] = rlt2.params(warm=1, feas_tol=0.0)
    elif kind == "bnb":
        s["F"], s["D"], s["B"] = _qap({"n": case["n"], "grid": 0}, seed)
        s["prm"], s["opts"] = rlt2.params(warm=1), rlt2.bnb_options(iters_root=100, iters_node=60)
    elif kind == "predict":
        s["net"] = rlt2.Mlp(hidden=256)
        s["net"].load(os.path.join(os.path.dirname(rlt2.__file__), "weights", "warmstart_h256.npz"))
        s["tiles"], s["prev"] = _tiles(case["tiles"], case["m"], seed)
        s["u0"] = _empty(case["tiles"], case["m"])
    else:
        s["net"] = rlt2.Mlp(hidden=case["hidden"])
        s["net"].set_weights(*_weights(case, seed))
        s["net"].add_samples(*_samples(case, seed))
    return s


def _weights(case, seed):
    """A network in training: He-scaled weights, small biases."""
    H, rng = case["hidden"], np.random.default_rng([seed, case["hidden"], 3])
    return (rng.normal(0, math.sqrt(2 / 34), (34, H)).astype(np.float32), rng.normal(0, 0.1, H).astype(np.float32),
            rng.normal(0, math.sqrt(2 / H), (H, H)).astype(np.float32), rng.normal(0, 0.1, H).astype(np.float32),
            rng.normal(0, math.sqrt(1 / H), H).astype(np.float32), 0.1)


def _samples(case, seed):
    """(tiles, target duals, previous duals) of at least case["rows"] rows of size 18."""
    tiles, near = _tiles(-(-case["rows"] // 18), 18, seed)
    return tiles, near + 200 + 40 * torch.cos(near), near


# ---------------------------------------------------------------------- run --
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "lap":
        rlt2.rlt2_lap_batched(state["cost"], u0=state["u0"], dual_mode=case["mode"], **state["out"])
        return state["out"]
    if kind == "ascent":
        with rlt2.Context(state["F"], state["D"], state["B"], prm=state["prm"]) as ctx:
            bounds, done = ctx.iterate(case["iters"])
            rlt2.rlt2_duals(ctx.ctx, on_device=1, **state["duals"])
            rlt2.rlt2_reduced_costs(ctx.ctx, on_device=1, **state["red"])
            rlt2.rlt2_export_state(ctx.ctx, on_device=1, **state["state"])
        return {"bounds": bounds, "done": done, **state["duals"], **state["red"], **state["state"]}
    if kind == "nodes":
        best, hist, its, _ = rlt2.rlt2_bound_nodes(state["F"], state["D"], state["partials"], case["iters"],
                                                   B=state["B"], prm=state["prm"])
        return {"best": best, "bounds": hist, "done": its}
    if kind == "bnb":
        best, perm, root, stats = rlt2.rlt2_bnb_solve(state["F"], state["D"], state["B"], prm=state["prm"],
                                                      opts=state["opts"])
        return {"best": best, "perm": perm, "root": root, "proven": stats["proven"]}
    if kind == "predict":
        state["net"].predict(state["tiles"], state["u0"], prev_u=state["prev"])
        return state["u0"]
    loss, gW1, gb1, gW2, gb2, gw3, gb3 = state["net"].grad(case["rows"])
    return {"loss": loss, "gW1": gW1, "gb1": gb1, "gW2": gW2, "gb2": gb2, "gw3": gw3, "gb3": gb3}


# --------------------------------------------------------------------- work --
def _lap_flops(m):
    """Additions of one LAP that no method here avoids: the column reduction, the
    optimum, and the canonical duals' relaxations (three each) and outputs."""
    return m * m + m + 3 * (m - 1) * (m - 2) / 2 + 3 * m


def _ascent_work(n, iters, scheme):
    m, T = n - 2, (n * (n - 1)) ** 2
    E = T * m * m
    solves = 2 if scheme.endswith("2") else 1
    share = 0.5 if scheme == "half" else 1.0
    flops = iters * (share * solves * T * _lap_flops(m) + n * n * _lap_flops(n - 1) + _lap_flops(n)
                     + share * E * 29 / 6 * solves + 6 * T)
    # the z array is read and written once per iteration where it does not fit on the chip
    z = 16 * E * share * solves * iters if 8 * E > 129e6 else 0
    out = 8 * (E + 2 * T * m + 2 * T)
    return z + out + 24 * n * n, flops


def work(case):
    kind = case["kind"]
    if kind == "lap":
        b, m = case["batch"], case["m"]
        return {"bytes": b * (8 * m * m + 8 + 20 * m + (8 * m if case["warm"] else 0)), "flops": b * _lap_flops(m)}
    if kind == "ascent":
        by, fl = _ascent_work(case["n"], case["iters"], case["scheme"])
        return {"bytes": by, "flops": fl}
    if kind == "nodes":
        by, fl = _ascent_work(case["n"] - 6, case["iters"], "S1")
        return {"bytes": by * case["nodes"], "flops": fl * case["nodes"]}
    if kind == "bnb":  # at least the root's ascent
        by, fl = _ascent_work(case["n"], 100, "S1")
        return {"bytes": by, "flops": fl}
    if kind == "predict":
        rows = case["tiles"] * case["m"]
        return {"bytes": rows * (8 * case["m"] + 16), "flops": rows * 2 * (34 * 256 + 256 * 256 + 256)}
    H, rows = case["hidden"], case["rows"]
    return {"bytes": rows * (34 * 2 + 4) + 4 * (36 * H + H * H), "flops": rows * 6 * (34 * H + H * H + H)}


# -------------------------------------------------------- values in 64 bits --
def _lap64(c):
    """Optima, assignments and canonical duals (the largest optimal row duals with
    u_0 = 0) of a batch of LAPs c[b, m, m]."""
    b, m = c.shape[0], c.shape[1]
    at = torch.arange(b, device=c.device)
    inf = torch.tensor(math.inf, device=c.device, dtype=F64)
    u, v = torch.zeros(b, m, device=c.device, dtype=F64), c.min(1).values
    r2c = torch.full((b, m), -1, device=c.device)
    c2r = torch.full((b, m), -1, device=c.device)
    for i in range(m):  # one shortest augmenting path per row
        seen = torch.zeros(b, m, device=c.device, dtype=torch.bool)
        d = c[:, i] - u[:, i, None] - v
        pred = torch.full((b, m), i, device=c.device)
        sink, dist = torch.full((b,), -1, device=c.device), torch.zeros(b, device=c.device, dtype=F64)
        for _ in range(i + 1):
            open_ = sink < 0
            low, col = torch.where(seen, inf, d).min(1)
            row = c2r[at, col]
            hit = open_ & (row < 0)
            sink, dist = torch.where(hit, col, sink), torch.where(hit, low, dist)
            go = open_ & (row >= 0)
            seen[at, col] |= go
            row = row.clamp(min=0)
            new = low[:, None] + c[at, row] - u[at, row][:, None] - v
            better = go[:, None] & ~seen & (new < d)
            d, pred = torch.where(better, new, d), torch.where(better, row[:, None], pred)
            if not bool((sink < 0).any()):
                break
        gain = torch.where(seen, d - dist[:, None], torch.zeros_like(d))  # <= 0 on the scanned columns
        v = v + gain
        rows = torch.where(seen, c2r, torch.full_like(c2r, m))
        u = torch.cat([u, u[:, :1]], 1).scatter_add_(1, rows, -gain)[:, :m]
        u[:, i] += dist
        col, live = sink, torch.ones(b, device=c.device, dtype=torch.bool)
        while bool(live.any()):
            row = pred[at, col]
            before = r2c[at, row]
            c2r[at[live], col[live]] = row[live]
            r2c[at[live], row[live]] = col[live]
            live = live & (row != i)
            col = torch.where(live, before, col)
    own = c.gather(2, r2c[:, :, None])[:, :, 0]
    arcs = c.gather(2, r2c[:, None, :].expand(b, m, m)) - own[:, None, :]  # u_r <= u_s + arcs[r, s]
    can = arcs[:, :, 0].clone()
    for _ in range(m):
        new = torch.minimum(can, (arcs + can[:, None, :]).min(2).values)
        if torch.equal(new, can):
            break
        can = new
    can = can - can[:, :1]
    return own.sum(1), r2c, can, (own - can).gather(1, c2r)


def _members(n):
    """Flat positions in D^ of the six members of every class {(i,p),(j,q),(k,r)}."""
    m = n - 2
    fac = torch.tensor(list(itertools.combinations(range(n), 3)), device=DEV)
    loc = torch.tensor(list(itertools.permutations(range(n), 3)), device=DEV)
    out = []
    for o in itertools.permutations(range(3)):
        i, j, k = (fac[:, x][:, None] for x in o)
        p, q, r = (loc[:, x][None, :] for x in o)
        tile = ((i * n + p) * (n - 1) + j - (j > i).long()) * (n - 1) + q - (q > p).long()
        kk = k - (k > i).long() - (k > j).long()
        rr = r - (r > p).long() - (r > q).long()
        out.append(((tile * m + kk) * m + rr).reshape(-1))
    return torch.stack(out)


def _ascent64(F, D, B, const, iters):
    """S1 dual ascent with the default parameters and canonical duals."""
    n = F.shape[0]
    m, T = n - 2, (n * (n - 1)) ** 2
    other = torch.tensor([[j for j in range(n) if j != i] for i in range(n)], device=DEV)
    back = torch.tensor([[j - (j > i) for j in range(n)] for i in range(n)], device=DEV)
    i, p = torch.arange(n, device=DEV)[:, None, None, None], torch.arange(n, device=DEV)[None, :, None, None]
    j, q = other[:, None, :, None], other[None, :, None, :]
    C = (F[i, j] * D[p, q]).reshape(T)
    mirror = (((j * n + q) * (n - 1) + back[j, i]) * (n - 1) + back[q, p]).reshape(T)
    b = B + F.diagonal()[:, None] * D.diagonal()[None, :]
    Z = torch.zeros(T, m, m, device=DEV, dtype=F64)
    members = _members(n)
    bounds, o = [], None
    for _ in range(iters):
        if o:
            term = 0.5 / m * o["pi_y"] + o["pi_x"].reshape(n * n, 1).expand(-1, (n - 1) ** 2).reshape(T) / ((n - 1) * m)
            C = C - 0.5 * o["pi_y"] + 0.5 * o["pi_y"][mirror]
            pool = (Z - o["xi"][:, :, None] - o["psi"][:, None, :] + term[:, None, None]).reshape(-1)[members]
            flat = Z.reshape(-1)
            flat[members] = flat[members] - pool + 0.2 * (pool.sum(0) - pool)
        theta, _, xi, psi = _lap64(Z)
        Y = (C + theta).reshape(n * n, n - 1, n - 1)
        delta, _, gu, gv = _lap64(Y)
        X = (b + delta.reshape(n, n))[None]
        val, _, al, be = _lap64(X)
        bounds.append(float(val[0]) + const)
        o = {"xi": xi, "psi": psi, "pi_y": (Y - gu[:, :, None] - gv[:, None, :]).reshape(T), "gamma": gu.reshape(-1),
             "delta": gv.reshape(-1), "alpha": al[0], "beta": be[0],
             "pi_x": (X - al[:, :, None] - be[:, None, :]).reshape(-1)}
    return {"bounds": np.array(bounds), **{k: o[k].reshape(-1) for k in ("alpha", "beta", "gamma", "delta", "xi", "psi",
                                                                      "pi_x", "pi_y")},
            "Dhat": Z.reshape(-1), "Chat": C}


def _residual(F, D, B, part):
    """The QAP left by a partial assignment, and the constant of its fixed part."""
    fix = np.flatnonzero(part >= 0)
    at = part[fix]
    fac = np.flatnonzero(part < 0)
    loc = np.setdiff1d(np.arange(len(part)), at)
    b = B[np.ix_(fac, loc)] + F[np.ix_(fac, fix)] @ D[np.ix_(loc, at)].T + F[np.ix_(fix, fac)].T @ D[np.ix_(at, loc)]
    const = B[fix, at].sum() + (F[np.ix_(fix, fix)] * D[np.ix_(at, at)]).sum()
    return F[np.ix_(fac, fac)], D[np.ix_(loc, loc)], b, float(const)


def _features64(tiles, prev):
    """Network inputs per row: sorted column-reduced scaled costs (32), the row's
    previous dual, m/32; and the tile scales."""
    nt, m = prev.shape
    red = tiles - tiles.min(1).values[:, None, :]
    scale = red.amax((1, 2))
    x = torch.zeros(nt, m, 34, device=DEV, dtype=F64)
    x[:, :, :m] = (red / scale[:, None, None]).sort(2).values
    x[:, :, 32] = prev / scale[:, None]
    x[:, :, 33] = m / 32
    return x.reshape(nt * m, 34), scale


def _on_gpu(*arrays):
    return [torch.as_tensor(np.ascontiguousarray(a), device=DEV, dtype=F64) for a in arrays]


def exact(case, seed):
    kind = case["kind"]
    if kind == "lap":
        if case["mode"] == 0 and case["m"] > 1:  # the Hungarian's own duals are one choice of many
            value, r2c, _, _ = _lap64(_tiles(case["batch"], case["m"], seed)[0])
            return {"value": value, "u": None, "v": None, "row_to_col": r2c.int()}
        value, r2c, u, v = _lap64(_tiles(case["batch"], case["m"], seed)[0])
        return {"value": value, "u": u, "v": v, "row_to_col": r2c.int()}
    if kind == "ascent":
        if case["scheme"] != "S1" or case["mode"] == 0:  # other rules, or duals that are one choice of many
            return None
        return {**_ascent64(*_on_gpu(*_qap(case, seed)), 0.0, case["iters"]), "done": case["iters"]}
    if kind == "nodes":
        if case["nodes"] * case["iters"] > 250:
            return None
        hist = []
        for part in _partials(case, seed):
            Fr, Dr, b, const = _residual(*_qap(case, seed), part)
            hist.append(_ascent64(*_on_gpu(Fr, Dr, b), const, case["iters"])["bounds"])
        hist = np.array(hist)
        return {"best": hist.max(1), "bounds": hist, "done": None}
    if kind == "bnb":
        n = case["n"]
        if n > 9:
            return None
        F, D, B = _qap({"n": n, "grid": 0}, seed)
        perms = np.array(list(itertools.permutations(range(n))))
        cost = sum(F[i, j] * D[perms[:, i], perms[:, j]] for i in range(n) for j in range(n))
        cost = cost + sum(B[i, perms[:, i]] for i in range(n))
        return {"best": float(cost.min()), "perm": None, "root": None, "proven": None}
    if kind == "predict":
        tiles, prev = _tiles(case["tiles"], case["m"], seed)
        path = os.path.join(os.path.dirname(rlt2.__file__), "weights", "warmstart_h256.npz")
        with np.load(path) as w:
            W1, b1, W2, b2, w3, b3 = _on_gpu(*(w[k] for k in ("W1", "b1", "W2", "b2", "w3", "b3")))
        x, scale = _features64(tiles, prev)
        out = ((x @ W1 + b1).relu() @ W2 + b2).relu() @ w3 + b3
        return prev + out.reshape(prev.shape) * scale[:, None]
    tiles, target, prev = _samples(case, seed)
    W1, b1, W2, b2, w3, b3 = _on_gpu(*_weights(case, seed))
    x, scale = _features64(tiles, prev)
    rows = case["rows"]
    x, t = x[:rows], ((target - prev) / scale[:, None]).reshape(-1)[:rows]
    h1 = (x @ W1 + b1).relu()
    h2 = (h1 @ W2 + b2).relu()
    e = (h2 @ w3 + b3 - t) / rows
    d2 = e[:, None] * w3 * (h2 > 0)
    d1 = (d2 @ W2.T) * (h1 > 0)
    return {"loss": float((e * e).sum() * rows / 2), "gW1": x.T @ d1, "gb1": d1.sum(0), "gW2": h1.T @ d2,
            "gb2": d2.sum(0), "gw3": h2.T @ e, "gb3": float(e.sum())}
