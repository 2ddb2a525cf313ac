"""The work that users of this package have it do, as cases that can be timed and checked.

A case is one call pattern of the public API ("op") on one problem ("data" and sizes):

    solve     a new problem: create a context, solve within an iteration budget, read the state
    iterate   a kept context is restarted from the start of Alg. 2 and run for some iterations
    train     one step of a loss: lamp_ot_loss forward and backward on new points
    gradient  a kept context is put to a saved state: the envelope gradient of both point sets
    map       a kept context applies its transport map to value columns (colour transfer)
    evaluate  a kept context at some iterate: objective with dual bound and gap, and Round

The problems are drawn on the GPU from the seed alone, with the distributions of the package's
synthetic workloads; ``exact`` computes the same outputs in float64 with plain torch.
"""
from __future__ import annotations

import math

import torch

import paper_2511_11359_gb300 as L

DEV = "cuda"
# float64 checks of more entry evaluations than this take too long
EXACT_ENTRIES = 4.0e10
# no drawn case evaluates more entries than the largest listed one (2^36 entries, twice)
DRAW_ENTRIES = 5.0e10
ROW_BLOCK_ENTRIES = 1 << 26


def case(name, op, data, n, m, d=0, *, cost="sqeuclid", prec="fp32", eta=0.0, scale=1.0, iters=10, k=0):
    return {"name": name, "op": op, "data": data, "n": n, "m": m, "d": d, "cost": cost, "prec": prec, "eta": eta,
            "scale": scale, "iters": iters, "k": k}


def listed():
    return [
        # a small problem solved from nothing, context and all: launches and latency are everything
        case("plain_2d_solve", "solve", "uniform", 256, 256, 2, scale=-1.0, iters=200),
        # one minibatch of 64-dimensional features in a training loop: create, solve, loss, backward
        case("minibatch_bf16_train", "train", "gauss", 1024, 1024, 64, prec="bf16_tc", eta=0.05, scale=1.0 / 64, iters=50),
        # a pair of 64 x 64 images, cost stored (67 MB), entropic
        case("image_grid_iterate", "iterate", "grid", 4096, 4096, eta=1e-3, iters=50),
        # a stored rectangular cost of odd extents: its rows are not a multiple of 16 bytes apart
        case("stored_odd_iterate", "iterate", "matrix", 3001, 2777, iters=50),
        # a stored cost far larger than the caches (1.07 GB): streamed from memory twice an iteration
        case("stored_16384_iterate", "iterate", "matrix", 16384, 16384, iters=5),
        # the differentiable loss between 3-d point clouds, forward and backward
        case("diffloss_train", "train", "sphere", 8192, 8192, 3, eta=1e-2, iters=100),
        # the same with 64-dimensional features in the default precision
        case("features_fp32_train", "train", "gauss", 8192, 8192, 64, eta=0.05, scale=1.0 / 64, iters=20),
        # high-dimensional clouds on tensor cores: the largest ordinary problem
        case("highdim_bf16_iterate", "iterate", "gauss", 1 << 15, 1 << 15, 64, prec="bf16_tc", iters=10),
        # the gradient of that problem with respect to both point sets
        case("highdim_bf16_gradient", "gradient", "gauss", 1 << 15, 1 << 15, 64, prec="bf16_tc", iters=10),
        # the transport map of one image's colours applied to another's palette
        case("colour_map", "map", "uniform", 65536, 16384, 3, iters=10, k=3),
        # a ground metric compared on its certificates: odd sizes, l1, objective, dual, gap, Round
        case("metric_l1_evaluate", "evaluate", "uniform", 5003, 3001, 8, cost="l1", iters=10),
        # the largest problem: 2^18 points a side, cost never stored
        case("largescale_iterate", "iterate", "uniform", 1 << 18, 1 << 18, 3, iters=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ones' ranges: any size between, odd ones among them."""
    while True:
        c = _draw(rng)
        if float(c["n"]) * c["m"] * c["iters"] * max(1, c["d"] / 8.0) <= DRAW_ENTRIES:
            return c


def _draw(rng):
    kind = rng.choice(["solve", "train_low", "train_high", "stored", "points", "highdim", "gradient", "map", "evaluate"])
    side = lambda lo, hi: (_log_int(rng, lo, hi), _log_int(rng, lo, hi))  # noqa: E731
    if kind == "solve":
        n, m = side(100, 2000)
        c = case("", "solve", "uniform", n, m, rng.randint(1, 4), scale=-1.0, iters=rng.randint(60, 200))
    elif kind == "train_low":
        n, m = side(500, 9000)
        c = case("", "train", "sphere", n, m, rng.randint(2, 8), eta=1e-2, iters=rng.randint(30, 100))
    elif kind == "train_high":
        n, m = side(500, 8192)
        d = rng.randint(9, 64)
        c = case("", "train", "gauss", n, m, d, prec=rng.choice(["fp32", "bf16_tc"]), eta=0.05, scale=1.0 / d,
                 iters=rng.randint(10, 40))
    elif kind == "stored":
        n, m = side(1000, 16384)
        if rng.random() < 0.5:
            m = m // 4 * 4
        c = case("", "iterate", "matrix", n, m, eta=rng.choice([0.0, 1e-3]), iters=rng.randint(5, 40))
    elif kind == "points":
        n, m = side(2000, 100000)
        c = case("", "iterate", "uniform", n, m, rng.randint(1, 8), cost=rng.choice(["sqeuclid", "sqeuclid", "l1", "linf"]),
                 iters=rng.randint(3, 30))
    elif kind == "highdim":
        n, m = side(2000, 40000)
        c = case("", "iterate", "gauss", n, m, rng.randint(9, 64), cost=rng.choice(["sqeuclid", "sqeuclid", "cosine"]),
                 prec=rng.choice(["bf16_tc", "bf16_tc", "fp32"]), iters=rng.randint(3, 20))
    elif kind == "gradient":
        n, m = side(2000, 32768)
        low = rng.random() < 0.4
        c = case("", "gradient", "sphere" if low else "gauss", n, m, rng.randint(1, 8) if low else rng.randint(16, 64),
                 prec="fp32" if low else "bf16_tc", iters=rng.randint(3, 10))
    elif kind == "map":
        n, m = side(2000, 65536)
        stored = n * m < 1 << 27 and rng.random() < 0.4
        c = case("", "map", "matrix" if stored else "uniform", n, m, 0 if stored else 3, iters=rng.randint(3, 10),
                 k=rng.randint(1, 4))
    else:
        n, m = side(1000, 10000)
        cost = rng.choice(["sqeuclid", "l1", "linf"])
        c = case("", "evaluate", "uniform", n, m, rng.randint(2, 8), cost=cost, eta=rng.choice([0.0, 1e-2]),
                 iters=rng.randint(3, 20))
    del c["name"]
    return c


# ------------------------------------------------------------------------------------------
# inputs


def _rows(g, n, lo=0.1):
    v = lo + (1.0 - lo) * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    return v / v.sum()


def _mixture(g, side):
    """Eight isotropic Gaussians with random weights on a side x side unit grid, a floor of 1e-6."""
    t = torch.arange(side, device=DEV, dtype=torch.float64) / max(side - 1, 1)
    gx, gy = torch.meshgrid(t, t, indexing="ij")
    p = torch.stack([gx.reshape(-1), gy.reshape(-1)], 1)
    mu = torch.rand(8, 2, generator=g, device=DEV, dtype=torch.float64)
    sig = 0.03 + 0.17 * torch.rand(8, generator=g, device=DEV, dtype=torch.float64)
    wt = torch.rand(8, generator=g, device=DEV, dtype=torch.float64)
    d2 = ((p[:, None, :] - mu[None]) ** 2).sum(2)
    dens = (wt / (2 * math.pi * sig ** 2) * torch.exp(-0.5 * d2 / sig ** 2)).sum(1)
    v = dens / dens.sum() + 1e-6
    return v / v.sum()


def inputs(case, seed):
    """The problem's arrays: marginals, points or a stored cost, value columns."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    n, m, d = case["n"], case["m"], case["d"]
    a = {}
    if case["data"] == "grid":
        side = math.isqrt(n)
        a["r"], a["c"] = _mixture(g, side), _mixture(g, side)
        q = torch.arange(side, device=DEV)
        i, j = (v.reshape(-1) for v in torch.meshgrid(q, q, indexing="ij"))
        d2 = (i[:, None] - i[None]) ** 2 + (j[:, None] - j[None]) ** 2
        a["C"] = (d2.double() / float(2 * (side - 1) ** 2)).float()
        return a
    normal = lambda *s: torch.randn(*s, generator=g, device=DEV)  # noqa: E731
    if case["data"] == "matrix":
        a["C"] = torch.rand(n, m, generator=g, device=DEV)
    elif case["data"] == "uniform":
        a["x"] = torch.rand(n, d, generator=g, device=DEV)
        a["y"] = torch.rand(m, d, generator=g, device=DEV)
    elif case["data"] == "gauss":
        a["x"], a["y"] = normal(n, d), normal(m, d) + 0.5
    else:
        y = normal(m, d)
        a["x"], a["y"] = normal(n, d), y / y.norm(dim=1, keepdim=True) + 0.05 * normal(m, d)
    if case["data"] in ("gauss", "sphere"):
        a["r"] = torch.full((n,), 1.0 / n, dtype=torch.float64, device=DEV)
        a["c"] = torch.full((m,), 1.0 / m, dtype=torch.float64, device=DEV)
    else:
        a["r"], a["c"] = _rows(g, n), _rows(g, m)
    if case["k"]:
        a["V"] = torch.rand(m, case["k"], generator=g, device=DEV)
    return a


def context(case, a, **params):
    if "C" in a:
        return L.Lamp(a["r"], a["c"], C=a["C"], eta=case["eta"], **params)
    return L.Lamp(a["r"], a["c"], x=a["x"], y=a["y"], cost=case["cost"], cost_scale=case["scale"], eta=case["eta"],
                  prec=case["prec"], **params)


def prepare(case, seed):
    a = inputs(case, seed)
    state = {"case": case, "a": a}
    if case["op"] == "train":
        a["x"].requires_grad_(True)
        a["y"].requires_grad_(True)
    elif case["op"] != "solve":
        s = state["s"] = context(case, a)
        if case["op"] == "iterate":
            zero = s.get_state()  # the start of Alg. 2
            state["start"] = {"nu": zero["nu"], "theta": zero["theta"], "kappa": 0.0, "t": 0}
        else:
            s.iterate(case["iters"])
            state["saved"] = s.get_state()
    return state


# ------------------------------------------------------------------------------------------
# one pass


def run(state):
    case, a = state["case"], state["a"]
    op, T = case["op"], case["iters"]
    if op == "solve":
        with context(case, a, max_iter=T) as s:
            info = s.solve()
            st = s.get_state()
        return {"iters": info["iters"], "infeas": info["infeas"], "cost": info["cost"], "K": info["K"],
                "kappa": info["kappa"], "nu": st["nu"], "theta": st["theta"], "logZ": st["logZ"]}
    if op == "train":
        loss = L.lamp_ot_loss(a["x"], a["y"], eta=case["eta"], cost_scale=case["scale"], prec=case["prec"], max_iter=T)
        dx, dy = torch.autograd.grad(loss, (a["x"], a["y"]))
        return {"loss": loss.detach(), "dx": dx, "dy": dy}
    s = state["s"]
    if op == "iterate":
        s.set_state(**state["start"])
        s.iterate(T)
        st = s.get_state()
        return {"nu": st["nu"], "theta": st["theta"], "kappa": st["kappa"], "t": st["t"], "row_shifts": st["row_shifts"]}
    if op == "gradient":
        st = state["saved"]
        s.set_state(st["nu"], st["theta"], st["kappa"], st["t"], st["row_shifts"])
        dx, dy = s.grad()
        return {"dx": dx, "dy": dy}
    if op == "map":
        return {"out": s.apply_map(a["V"], side=0)}
    ob = s.objective()
    rd = s.round(want_vectors=True)
    return {"objective": ob, "round": rd}


def work(case):
    n, m, d, T, op = case["n"], case["m"], case["d"], case["iters"], case["op"]
    stored = case["data"] in ("grid", "matrix")
    E = float(n) * m
    # per entry: the cost, and per stream of an iteration its exponent, exponential, row sum
    # and column sum
    cost = 0 if stored else (2 * d + 2 if case["cost"] in ("sqeuclid", "cosine") and d > 8 else 3 * d)
    iteration = E * (cost + 2 * 6)
    evaluation = E * (cost + 8)
    vectors = 8.0 * (2 * n + 4 * m) + (0 if stored else 4.0 * d * (n + m))
    C = 4.0 * E if stored else 0.0  # a stored cost is read at least once an iteration
    if op in ("solve", "iterate"):
        return {"bytes": T * C + vectors, "flops": T * iteration}
    if op == "train":
        return {"bytes": vectors + 4.0 * d * (n + m), "flops": T * iteration + evaluation + E * 4 * d}
    if op == "gradient":
        return {"bytes": vectors + 4.0 * d * (n + m), "flops": evaluation + E * 4 * d}
    if op == "map":
        return {"bytes": C + vectors + 4.0 * case["k"] * (n + m), "flops": evaluation + E * 2 * case["k"]}
    return {"bytes": vectors + 8.0 * (n + 2 * m), "flops": 2 * evaluation + 2 * E * (cost + 2)}


# ------------------------------------------------------------------------------------------
# float64 values of the outputs


class Plain:
    """Alg. 2 and the quantities read from its iterates in float64, blocks of rows at a time."""

    def __init__(self, case, a):
        self.n, self.m, self.eta = case["n"], case["m"], case["eta"]
        self.r = a["r"] if "r" in a else None
        self.c = a["c"]
        self.C = a.get("C")
        self.cost, self.s, self.d = case["cost"], 1.0, case["d"]
        if self.C is None:
            x, y = a["x"].detach().double(), a["y"].detach().double()
            if self.cost == "cosine":
                x = (x / (math.sqrt(2.0) * x.norm(dim=1, keepdim=True))).float().double()
                y = (y / (math.sqrt(2.0) * y.norm(dim=1, keepdim=True))).float().double()
            if case["prec"] == "bf16_tc":
                x, y = x.float().bfloat16().double(), y.float().bfloat16().double()
            self.x, self.y = x, y
        step = max(1, ROW_BLOCK_ENTRIES // self.m)
        self.blocks = [(i, min(i + step, self.n)) for i in range(0, self.n, step)]
        self.K = max(float(self.block(b).max()) for b in self.blocks)
        if self.C is None:
            self.s = 1.0 / self.K if case["scale"] < 0 else case["scale"]
            self.K *= self.s
        self.tau = 1.0 / (2.0 * self.K)
        self.nu = torch.zeros(self.m, dtype=torch.float64, device=DEV)
        self.theta = torch.zeros_like(self.nu)
        self.kappa, self.t = 0.0, 0

    def block(self, b):
        i, j = b
        if self.C is not None:
            return self.C[i:j].double()
        x = self.x[i:j]
        if self.cost in ("sqeuclid", "cosine") and self.d > 8:
            z = (x * x).sum(1)[:, None] + (self.y * self.y).sum(1)[None] - 2.0 * (x @ self.y.T)
        else:
            z = torch.zeros(j - i, self.m, dtype=torch.float64, device=DEV)
            for q in range(self.d):
                df = x[:, q, None] - self.y[None, :, q]
                z = torch.maximum(z, df.abs()) if self.cost == "linf" else z + (df.abs() if self.cost == "l1" else df * df)
        return z * self.s

    def coupling(self, C, b, phi, kappa):
        """(X, log Z) of rows b[0] .. b[1] for the potentials phi at 1 / eta = kappa."""
        v = -kappa * (C + 2.0 * self.K * phi[None])
        lz = torch.logsumexp(v, 1)
        return self.r[b[0]:b[1], None] * torch.exp(v - lz[:, None]), lz

    def iterate(self, T):
        alpha, clip = 0.01 / self.m, math.tanh(0.55)
        for _ in range(T):
            kn = self.tau + self.kappa * (1.0 - self.tau * self.eta)
            w = self.tau / kn
            bar = self.nu + w * (self.theta - self.nu)
            A, B = torch.zeros_like(self.nu), torch.zeros_like(self.nu)
            for b in self.blocks:
                C = self.block(b)
                A += self.coupling(C, b, self.nu, self.kappa)[0].sum(0)
                B += self.coupling(C, b, bar, kn)[0].sum(0)
            g = 2.0 * self.tau * self.K / (self.c + alpha)
            at = torch.atanh(self.theta)
            self.nu = self.nu + w * (torch.tanh(g * (A - self.c) + at) - self.nu)
            self.theta = torch.tanh(g * (B - self.c) + at).clamp(-clip, clip)
            self.kappa, self.t = kn, self.t + 1

    def evaluate(self):
        """col(X), log Z, <C, X> and H(X) of the current iterate."""
        col = torch.zeros_like(self.nu)
        lz, cost, H = [], 0.0, 0.0
        for b in self.blocks:
            C = self.block(b)
            X, z = self.coupling(C, b, self.nu, self.kappa)
            col += X.sum(0)
            lz.append(z)
            cost += float((C * X).sum())
            logp = -self.kappa * (C + 2.0 * self.K * self.nu[None]) - z[:, None]
            H -= float((X * (logp + self.r[b[0]:b[1]].log()[:, None])).sum())
        return col, torch.cat(lz), cost, H

    def dual(self, phi):
        v = 0.0
        for b in self.blocks:
            u = self.block(b) + 2.0 * self.K * phi[None]
            row = u.min(1).values if self.eta == 0.0 else -self.eta * torch.logsumexp(-u / self.eta, 1)
            v += float((self.r[b[0]:b[1]] * row).sum())
        v -= 2.0 * self.K * float((self.c * phi).sum())
        if self.eta > 0.0:
            v += self.eta * float((self.r * self.r.log()).sum())
        return v


def exact(case, seed):
    op, T = case["op"], case["iters"]
    if float(case["n"]) * case["m"] * (T + 2) > EXACT_ENTRIES:
        return None
    a = inputs(case, seed)
    p = Plain(case, a)
    p.iterate(T)
    if op == "iterate":
        return {"nu": p.nu, "theta": p.theta, "kappa": p.kappa, "t": p.t, "row_shifts": None}
    if op == "solve":
        col, lz, cost, _ = p.evaluate()
        return {"iters": p.t, "infeas": float((col - p.c).abs().sum()), "cost": cost, "K": p.K, "kappa": p.kappa,
                "nu": p.nu, "theta": p.theta, "logZ": lz}
    if op == "map":
        out = []
        for b in p.blocks:
            X, _ = p.coupling(p.block(b), b, p.nu, p.kappa)
            out.append((X @ a["V"].double()) / p.r[b[0]:b[1], None])
        return {"out": torch.cat(out)}
    if op in ("train", "gradient"):
        dx, dy = torch.empty_like(p.x), torch.zeros_like(p.y)
        col = torch.zeros_like(p.nu)
        for b in p.blocks:
            X, _ = p.coupling(p.block(b), b, p.nu, p.kappa)
            dx[b[0]:b[1]] = 2.0 * p.s * (p.r[b[0]:b[1], None] * p.x[b[0]:b[1]] - X @ p.y)
            dy -= 2.0 * p.s * (X.T @ p.x[b[0]:b[1]])
            col += X.sum(0)
        dy += 2.0 * p.s * col[:, None] * p.y
        if op == "gradient":
            return {"dx": dx, "dy": dy}
        _, _, cost, H = p.evaluate()
        return {"loss": cost - p.eta * H, "dx": dx, "dy": dy}
    col, _, cost, H = p.evaluate()
    res = float((col - p.c).abs().sum())
    P = cost + 2.0 * p.K * res - p.eta * H
    D = max(p.dual(p.theta), p.dual(p.nu))
    ob = {"cost": cost, "col_res": res, "row_res": 0.0, "entropy": H, "P_eta": P, "dual": D, "K": p.K,
          "certificate": 4.0 * p.K * res + 2.0 * p.K * math.log(p.m) / p.t if p.eta == 0.0 else math.nan,
          "L": cost - p.eta * H, "gap": P - D}
    y = torch.clamp(p.c / col, max=1.0)
    dc = torch.clamp(p.c - col, min=0.0)
    dr, scaled, cross = torch.empty_like(p.r), 0.0, 0.0
    for b in p.blocks:
        C = p.block(b)
        X, _ = p.coupling(C, b, p.nu, p.kappa)
        dr[b[0]:b[1]] = (X * (1.0 - y)[None]).sum(1)
        scaled += float((C * X * y[None]).sum())
        cross += float((dr[b[0]:b[1]] * (C @ dc)).sum())
    return {"objective": ob, "round": {"cost": scaled + cross / float(dr.sum()), "dr_l1": float(dr.sum()),
                                       "dc_l1": float(dc.sum()), "cost_scaled": scaled, "y": y, "dr": dr, "dc": dc}}
