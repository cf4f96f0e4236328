"""The framework's work as its users have it done, as timed cases on one GPU.

Every case goes through the public Python entry points. Five kinds:

  estimate  the Monte Carlo estimate at given nodes over one mesh step
            (sdd_set_w, sdd_interface_mc): plain, Brownian-bridge or exponential
            time-stepping, without or with a control variate
  step      whole mesh steps (sdd_set_w, sdd_step) and the mesh they end at
  batch     the estimate of many independent problems in one call
            (sdd_batch_interface_mc)
  solve     the implicit subdomain solve with given interface values
            (sdd_subdomain_solve)
  train     loss and gradient of the control variate's two networks over a batch
            of path samples (sdd_mlp_grad)

exact() restates each kind in 64 bits with plain torch and numpy: the same
random streams (Philox4x32-10, counter = path, node, draw, mesh step), the same
Euler-Maruyama paths, exit tests, scores, interface fill and implicit step.
"""
import math
import random

import numpy as np
import torch

import paper_1402_0266_gb300 as sdd

CV_MODES = {"off": sdd.SDD_CV_OFF, "fields": sdd.SDD_CV_FIELDS, "model": sdd.SDD_CV_MODEL}


def _estimate(name, n, ny, sub, density, dt, K, nodes, paths, spread=1.0, mode=0, cv="off"):
    return {"name": name, "kind": "estimate", "n": n, "ny": ny, "sub": sub, "density": density, "dt": dt, "K": K,
            "nodes": nodes, "paths": paths, "spread": spread, "exit_mode": mode, "cv": cv}


def _step(name, n, sub, density, dt, K, paths, steps, spacing=-1):
    return {"name": name, "kind": "step", "n": n, "sub": sub, "density": density, "dt": dt, "K": K, "paths": paths,
            "steps": steps, "spacing": spacing}


def listed():
    return [
        # the smallest estimate of the test suite and the bench: the heat problem's line of 33 nodes, where latency counts
        _estimate("heat65", 65, 65, 2, "const", 1e-3, 50, 33, 1000),
        # few paths per node with the learned control variate, its table rebuilt from the current w at every estimate
        _estimate("cv65_model", 65, 65, 2, "const", 1e-3, 50, 31, 2000, cv="model"),
        # the paper's own experiment: short mesh steps on a small grid, key points filled by PCHIP
        _step("ring41_step", 41, 2, "paper_ring", 5e-5, 20, 10000, 10, spacing=8),
        # the moving front: pipelined mesh steps, the ordinary size
        _step("front257_step", 257, 2, "front", 1e-4, 100, 10000, 4),
        # the Brownian-bridge exit test on the same problem with coarser sub-steps
        _estimate("front257_bridge", 257, 257, 2, "front", 4e-4, 25, 509, 10000, mode=1),
        # exponential time-stepping around a Gaussian bump
        _estimate("bump129_exp", 129, 129, 2, "bump", 5e-4, 20, 253, 8000, mode=2),
        # a rectangular grid of odd sizes, drift everywhere, an odd number of sub-steps, path counts that differ by node
        _estimate("rect_ragged", 194, 131, 3, "smooth", 2e-4, 45, 601, 5000, spread=4.0),
        # many independent problems at once: 65^2 to 513^2 bumps with their own node sets and path counts
        {"name": "batch16", "kind": "batch", "count": 16, "dt": 1e-4, "K": 100, "nodes": 180, "paths": 6000,
         "spread": 4.0},
        # a fine grid with the previous fields' gradient as control variate: few paths per node are enough
        _estimate("ring1025_fields", 1025, 1025, 4, "ring", 2e-5, 50, 6129, 2000, cv="fields"),
        # the largest: one mesh step of the 2049^2 ring, 28,609 interface nodes, 8 x 8 subdomains
        _step("ring2049_step", 2049, 8, "ring", 1e-5, 100, 20000, 1),
        # the implicit subdomain solve alone, for interface values from elsewhere
        {"name": "solve513", "kind": "solve", "n": 513, "ny": 513, "sub": 2, "density": "ring", "Dt": 2e-3},
        # one gradient of the control variate's networks
        {"name": "mlp_grad", "kind": "train", "rows": 65536},
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def draw(rng):
    kind = rng.choice(["estimate", "estimate", "estimate", "step", "step", "batch", "solve", "train"])
    density = rng.choice(["front", "ring", "bump", "smooth", "paper_ring"])
    if kind == "estimate":
        n, ny = round(_log(rng, 41, 1025)), round(_log(rng, 41, 1025))
        K = round(_log(rng, 10, 120))
        mode = rng.choice([0, 0, 0, 1, 2])
        cv = "off" if mode == 2 else rng.choice(["off", "off", "fields"])
        nodes, paths = round(_log(rng, 30, 4000)), round(_log(rng, 1000, 20000))
        paths = max(1000, min(paths, int(2e9 / (K * nodes))))
        c = _estimate("", n, ny, rng.choice([2, 3, 4]), density, _log(rng, 1e-3, 1e-2) / K, K, nodes, paths,
                      rng.choice([1.0, 1.0, 4.0]), mode, cv)
    elif kind == "step":
        sub = rng.choice([2, 2, 3, 4])
        # subdomains of one size or of several
        n = sub * round(_log(rng, 20, 384) / sub) + 1 if rng.random() < 0.6 else round(_log(rng, 41, 385))
        K = round(_log(rng, 10, 100))
        paths = max(1000, min(round(_log(rng, 1000, 20000)), int(1e9 / (K * 2 * (sub - 1) * n))))
        c = _step("", n, sub, density, _log(rng, 1e-3, 1e-2) / K, K, paths, rng.randint(1, 6),
                  rng.choice([-1, -1, 8]))
    elif kind == "batch":
        K = round(_log(rng, 20, 100))
        c = {"kind": "batch", "count": rng.randint(3, 24), "dt": _log(rng, 2e-3, 1e-2) / K, "K": K,
             "nodes": round(_log(rng, 33, 300)), "paths": round(_log(rng, 1000, 8000)), "spread": 4.0}
    elif kind == "solve":
        m, sub = rng.choice([15, 19, 31, 63, 64, 100, 127, 200, 255]), rng.choice([1, 2, 3, 4])
        n = sub * (m + 1) + 1
        c = {"kind": "solve", "n": n, "ny": n + rng.choice([0, 0, -1]), "sub": sub, "density": density,
             "Dt": _log(rng, 5e-4, 5e-3)}
    else:
        c = {"kind": "train", "rows": 64 * round(_log(rng, 16, 4096))}
    c.pop("name", None)
    return c


# ------------------------------------------------------------------ inputs

def _grid(n, ny):
    x = torch.arange(n, dtype=torch.float64, device="cuda") / (n - 1)
    y = torch.arange(ny, dtype=torch.float64, device="cuda") / (ny - 1)
    return x[None, :].expand(ny, n), y[:, None].expand(ny, n)


def _density(kind, n, ny, t, rng):
    """Mesh density w on the grid (float32): the workloads' formulas at time t, their places and widths by the seed."""
    X, Y = _grid(n, ny)
    if kind == "const":
        w = torch.ones_like(X)
    elif kind == "front":
        w = 1.0 + 10.0 * torch.exp(-((X - 0.3 - 0.4 * t) ** 2) / 0.05 ** 2)
    elif kind == "ring":
        r = torch.sqrt((X - 0.5) ** 2 + (Y - 0.5) ** 2)
        w = 1.0 + 50.0 * torch.exp(-((r - 0.25 - 0.1 * math.sin(2 * math.pi * t)) ** 2) / 0.02 ** 2)
    elif kind == "paper_ring":
        q = (X - 0.5 - 0.25 * math.cos(2 * math.pi * t)) ** 2 + (Y - 0.5 - 0.25 * math.sin(2 * math.pi * t)) ** 2
        w = 1.0 / (1.0 + 10.0 * torch.exp(-50.0 * torch.abs(q - 0.01)))
    elif kind == "bump":
        cx, cy, width, alpha = rng.uniform(0.2, 0.8), rng.uniform(0.2, 0.8), rng.uniform(0.05, 0.15), rng.uniform(1, 50)
        w = 1.0 + alpha * torch.exp(-((X - cx) ** 2 + (Y - cy) ** 2) / width ** 2)
    else:  # smooth: a few low Fourier modes
        w = torch.ones_like(X)
        for _ in range(3):
            kx, ky, a = rng.randint(1, 3), rng.randint(1, 3), rng.uniform(-0.13, 0.13)
            px, py = rng.uniform(0, 6.28), rng.uniform(0, 6.28)
            w = w + a * torch.cos(math.pi * kx * X + px) * torch.cos(math.pi * ky * Y + py)
    return w.to(torch.float32).contiguous()


def _fields(n, ny, rng, noise):
    """A deformed mesh: the uniform one, a smooth displacement, and the noise that interface estimates leave."""
    X, Y = _grid(n, ny)
    a, b = rng.uniform(-0.03, 0.03), rng.uniform(-0.03, 0.03)
    xi = X + a * torch.sin(2 * math.pi * X) * torch.cos(math.pi * Y)
    eta = Y + b * torch.sin(2 * math.pi * Y) * torch.cos(math.pi * X)
    if noise:
        g = torch.Generator(device="cuda").manual_seed(rng.randrange(1 << 30))
        xi = xi + noise * torch.randn(xi.shape, generator=g, device="cuda", dtype=torch.float64)
        eta = eta + noise * torch.randn(eta.shape, generator=g, device="cuda", dtype=torch.float64)
    return xi.contiguous(), eta.contiguous()


def _lines(n, parts):
    return [int(math.floor(k * (n - 1) / parts + 0.5)) for k in range(1, parts)]


def _interface(n, ny, sub):
    """Grid indices of the interface nodes: vertical lines bottom to top, then horizontal ones without the crossings."""
    vi, hj = _lines(n, sub), _lines(ny, sub)
    return [(i, j) for i in vi for j in range(1, ny - 1)] + [(i, j) for j in hj for i in range(1, n - 1) if i not in vi]


def _node_set(n, ny, sub, count, paths, spread, rng):
    """`count` nodes taken evenly from the interface (all of them if there are fewer), and their path counts."""
    every = _interface(n, ny, sub)
    pick = np.unique(np.linspace(0, len(every) - 1, min(count, len(every))).round().astype(np.int64))
    x = np.array([every[k][0] / (n - 1) for k in pick])
    y = np.array([every[k][1] / (ny - 1) for k in pick])
    # between paths / spread (1000 at least) and paths
    lo = max(min(1000, paths), paths / spread)
    np_ = np.array([round(math.exp(rng.uniform(math.log(lo), math.log(paths)))) for _ in pick], dtype=np.int64)
    return x, y, np_


def _batch_sizes(c):
    """Grid size and node count of each problem of a batch: the case's own, whatever the seed."""
    rng = random.Random(c["count"] * 1000003 + c["nodes"])
    return [(rng.choice([65, 129, 257, 513]), round(_log(rng, c["nodes"] / 5, c["nodes"]))) for _ in range(c["count"])]


def _network(rng):
    """A parameter block with Glorot-uniform weights and small biases, and a standardisation."""
    g = torch.Generator(device="cuda").manual_seed(rng.randrange(1 << 30))
    theta = torch.zeros(2, sdd.MLP_STRIDE, device="cuda")
    o = 0
    for size, fan in ((320, 69), (64, 0), (4096, 128), (64, 0), (64, 65), (1, 0)):
        u = 2 * torch.rand(2, size, generator=g, device="cuda") - 1
        theta[:, o:o + size] = u * (math.sqrt(6 / fan) if fan else 0.1)
        o += size
    norm = torch.tensor([0.5, 0.5, 0.51, 1.0, 0.0, 3.46, 3.46, 3.4, 0.0, 0.0], device="cuda")
    return theta.reshape(-1).contiguous(), norm


def prepare(case, seed):
    rng = random.Random(seed)
    c, kind = case, case["kind"]
    s = {"case": c, "seed": rng.randrange(1 << 40)}
    if kind == "estimate":
        t = rng.uniform(0.0, 1.0)
        s["w"] = _density(c["density"], c["n"], c["ny"], t, rng)
        if c["density"] == "const":
            # the heat problem: separable modes, zero boundary data, the line x = 1/2
            X, Y = _grid(c["n"], c["ny"])
            a = rng.uniform(0.5, 1.5)
            s["xi"] = (a * torch.sin(math.pi * X) * torch.sin(math.pi * Y)).contiguous()
            s["eta"] = (a * torch.sin(math.pi * X) * torch.sin(2 * math.pi * Y)).contiguous()
            s["faces"] = torch.zeros(sdd.faces_len(c["n"], c["ny"]), dtype=torch.float64, device="cuda")
            y = np.arange(c["nodes"]) / (c["nodes"] - 1) if c["cv"] == "off" else (np.arange(c["nodes"]) + 1) / (c["nodes"] + 1)
            s["nodes"] = np.full(c["nodes"], 0.5), y, np.full(c["nodes"], c["paths"], dtype=np.int64)
        else:
            s["xi"], s["eta"] = _fields(c["n"], c["ny"], rng, 1e-6 if c["cv"] == "fields" else 0.0)
            s["nodes"] = _node_set(c["n"], c["ny"], c["sub"], c["nodes"], c["paths"], c["spread"], rng)
        ctx = sdd.sdd_init(c["n"], c["ny"], c["sub"], c["sub"], w=s["w"], xi0=s["xi"], eta0=s["eta"])
        if "faces" in s:
            sdd.sdd_set_boundary(ctx, s["faces"])
        if c["cv"] == "model":
            s["theta"], s["norm"] = _network(rng)
            sdd.sdd_cv_set_model(ctx, s["theta"], s["norm"], c["K"])
        sdd.sdd_cv_enable(ctx, CV_MODES[c["cv"]])
        s["ctx"] = ctx
    elif kind == "step":
        t = rng.uniform(0.0, 0.7)
        again = rng.randrange(1 << 30)
        s["w"] = [_density(c["density"], c["n"], c["n"], t + k * c["dt"] * c["K"], random.Random(again))
                  for k in range(c["steps"])]
        s["ctx"] = sdd.sdd_init(c["n"], c["n"], c["sub"], c["sub"], w=s["w"][0])
        if c["spacing"] >= 0:
            sdd.sdd_set_keypoints(s["ctx"], True, c["spacing"])
    elif kind == "batch":
        s["parts"], s["ctxs"] = [], []
        for n, count in _batch_sizes(c):
            w = _density("bump", n, n, 0.0, rng)
            xi, eta = _fields(n, n, rng, 0.0)
            nodes = _node_set(n, n, 2, count, c["paths"], c["spread"], rng)
            s["parts"].append((w, xi, eta, nodes))
            s["ctxs"].append(sdd.sdd_init(n, n, 2, 2, w=w, xi0=xi, eta0=eta))
        s["batch"] = sdd.sdd_batch_create(s["ctxs"])
    elif kind == "solve":
        s["w"] = _density(c["density"], c["n"], c["ny"], rng.uniform(0.0, 1.0), rng)
        s["xi"], s["eta"] = _fields(c["n"], c["ny"], rng, 0.0)
        s["ctx"] = sdd.sdd_init(c["n"], c["ny"], c["sub"], c["sub"], w=s["w"], xi0=s["xi"], eta0=s["eta"])
        ij = np.array(_interface(c["n"], c["ny"], c["sub"]), dtype=np.int64).reshape(-1, 2)
        at = torch.from_numpy(ij[:, 1] * c["n"] + ij[:, 0]).cuda()
        g = torch.Generator(device="cuda").manual_seed(rng.randrange(1 << 30))
        # Monte Carlo values: the fields there and an error of their size
        s["iface"] = [(f.reshape(-1)[at] + 2e-4 * torch.randn(at.numel(), generator=g, device="cuda", dtype=torch.float64))
                      .contiguous() for f in (s["xi"], s["eta"])]
    else:
        s["theta"], s["norm"] = _network(rng)
        g = torch.Generator(device="cuda").manual_seed(rng.randrange(1 << 30))
        m = c["rows"]
        s["norm"] = torch.tensor([0.5, 0.5, 0.51, 1.5, 4.0, 3.46, 3.46, 3.4, 0.7, 0.2], device="cuda")
        f = torch.rand(m, 5, generator=g, device="cuda")
        f[:, 3] = 1 + 3 * f[:, 3] ** 4
        f[:, 4] = 16 * f[:, 4] ** 2
        s["feats"] = f.contiguous()
        # single-path scores: the smooth solution and the path's own noise
        s["targets"] = (f[:, :2] + 0.1 * torch.randn(m, 2, generator=g, device="cuda")).contiguous()
        s["ctx"] = sdd.sdd_init(65, 65, 2, 2)
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "estimate":
        sdd.sdd_set_w(s["ctx"], s["w"])
        x, y, n_paths = s["nodes"]
        return sdd.sdd_interface_mc(s["ctx"], x, y, n_paths, dt=c["dt"], Dt=c["dt"] * c["K"], seed=s["seed"],
                                    exit_mode=c["exit_mode"])
    if kind == "step":
        for w in s["w"]:
            sdd.sdd_set_w(s["ctx"], w)
            sdd.sdd_step(s["ctx"], dt=c["dt"], Dt=c["dt"] * c["K"], seed=s["seed"], paths_per_node=c["paths"])
        out = dict(sdd.sdd_last_interface_stats(s["ctx"]))
        out["xi"], out["eta"] = sdd.sdd_get_fields(s["ctx"])
        return out
    if kind == "batch":
        for ctx, (w, _, _, _) in zip(s["ctxs"], s["parts"]):
            sdd.sdd_set_w(ctx, w)
        got = sdd.sdd_batch_interface_mc(s["batch"], [p[3] for p in s["parts"]], dt=c["dt"], Dt=c["dt"] * c["K"],
                                         seed=s["seed"])
        return {k: torch.cat([g[k] for g in got]) for k in got[0]}
    if kind == "solve":
        sdd.sdd_set_w(s["ctx"], s["w"])
        xi, eta, _ = sdd.sdd_subdomain_solve(s["ctx"], c["Dt"], s["iface"][0], s["iface"][1], want_iters=False)
        return {"xi": xi, "eta": eta}
    grad, loss = sdd.sdd_mlp_grad(s["ctx"], s["theta"], s["norm"], s["feats"], s["targets"])
    return {"grad": grad, "loss": loss}


def work(case):
    """Bytes of inputs and outputs, and operations: a path's sub-step takes 58 (half a Philox block 20, a normal pair
    12, cell 12, drift 6, update 4, exit test 4); paths that leave early are counted in full."""
    c, kind = case, case["kind"]
    if kind == "estimate":
        grid = c["n"] * c["ny"]
        mean = c["paths"] if c["spread"] == 1.0 else c["paths"] * (1 - 1 / c["spread"]) / math.log(c["spread"])
        return {"bytes": grid * (4 + 16) + c["nodes"] * (24 + 48), "flops": 58.0 * c["nodes"] * mean * c["K"]}
    if kind == "step":
        grid, nodes = c["n"] * c["n"], len(_interface(c["n"], c["n"], c["sub"]))
        # the solve: a few tens of operations per unknown at the least
        return {"bytes": c["steps"] * (grid * (4 + 16 + 16) + nodes * 48),
                "flops": c["steps"] * (58.0 * nodes * c["paths"] * c["K"] + 100.0 * grid)}
    if kind == "batch":
        sizes = _batch_sizes(c)
        nodes = sum(k for _, k in sizes)
        mean = c["paths"] * (1 - 1 / c["spread"]) / math.log(c["spread"])
        return {"bytes": sum(n * n for n, _ in sizes) * 20 + nodes * 72, "flops": 58.0 * nodes * mean * c["K"]}
    if kind == "solve":
        return {"bytes": c["n"] * c["ny"] * (4 + 16 + 16), "flops": 100.0 * c["n"] * c["ny"]}
    return {"bytes": c["rows"] * 28 + 4 * 4 * sdd.MLP_STRIDE, "flops": c["rows"] * 2 * 6.0 * 4480}


# ------------------------------------------------------------------ 64-bit restatement

M32 = 0xFFFFFFFF


def _mulhilo(a, m):
    p1 = (a >> 16) * m
    t = (a & 0xFFFF) * m + ((p1 & 0xFFFF) << 16)
    return (p1 >> 16) + (t >> 32), t & M32


def _philox(c0, c1, c2, c3, seed):
    """Ten rounds on int64 tensors (or numbers) holding 32-bit words."""
    k0, k1 = seed & M32, seed >> 32
    for _ in range(10):
        h0, l0 = _mulhilo(c0, 0xD2511F53)
        h1, l1 = _mulhilo(c2, 0xCD9E8D57)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


def _unit(word):
    return (word & 0x7FFFFF).double() * 2.0 ** -23


def _normals(a, b, sigma):
    r = sigma * torch.sqrt(-2.0 * torch.log1p(-_unit(a)))
    ang = 2 * math.pi * _unit(b)
    return r * torch.cos(ang), r * torch.sin(ang)


def _fd(f):
    """Second-order differences of node values, one-sided on the edges."""
    ny, nx = f.shape
    gx, gy = torch.empty_like(f), torch.empty_like(f)
    gx[:, 1:-1] = (f[:, 2:] - f[:, :-2]) / 2
    gx[:, 0] = (-3 * f[:, 0] + 4 * f[:, 1] - f[:, 2]) / 2
    gx[:, -1] = (3 * f[:, -1] - 4 * f[:, -2] + f[:, -3]) / 2
    gy[1:-1] = (f[2:] - f[:-2]) / 2
    gy[0] = (-3 * f[0] + 4 * f[1] - f[2]) / 2
    gy[-1] = (3 * f[-1] - 4 * f[-2] + f[-3]) / 2
    return gx * (nx - 1), gy * (ny - 1)


def _faces(w):
    """The 1D Winslow solution along each face: cumulative trapezoids of w."""
    def line(v):
        s = torch.cat([torch.zeros(1, dtype=torch.float64, device=v.device), torch.cumsum(0.5 * (v[1:] + v[:-1]), 0)])
        return s / s[-1]
    ny, nx = w.shape
    z = lambda n, v: torch.full((n,), v, dtype=torch.float64, device=w.device)  # noqa: E731
    return torch.cat([z(ny, 0.0), z(ny, 1.0), line(w[0]), line(w[-1]), line(w[:, 0]), line(w[:, -1]), z(nx, 0.0), z(nx, 1.0)])


class _Walk:
    """The estimate of one problem: node means, standard errors, exits and sub-steps."""

    def __init__(self, w, xi, eta, faces, model=None, model_cells=False):
        self.w = w.double()
        self.ny, self.nx = w.shape
        bx, by = _fd(self.w)
        self.b = torch.stack([-bx / self.w, -by / self.w], -1).reshape(-1, 2)
        self.f = torch.stack([xi, eta], -1).reshape(-1, 2)
        self.faces = _faces(self.w) if faces is None else faces
        self.model, self.model_cells = model, model_cells

    def cell(self, x, y):
        gx, gy = x * (self.nx - 1), y * (self.ny - 1)
        i = gx.floor().clamp(0, self.nx - 2)
        j = gy.floor().clamp(0, self.ny - 2)
        return i.long(), j.long(), gx - i, gy - j

    def at(self, table, i, j, s, t):
        k = j * self.nx + i
        s, t = s[:, None], t[:, None]
        return ((1 - s) * table[k] + s * table[k + 1]) * (1 - t) + ((1 - s) * table[k + self.nx] + s * table[k + self.nx + 1]) * t

    def face(self, field, face, s):
        n = torch.where(face < 2, self.ny, self.nx)
        off = field * 2 * (self.nx + self.ny) + torch.where(face < 2, face * self.ny, 2 * self.ny + (face - 2) * self.nx)
        g = s * (n - 1)
        k = torch.minimum(g.floor().clamp(min=0).long(), n - 2)
        a = self.faces[off + k]
        return a + (g - k) * (self.faces[off + k + 1] - a)

    def chunk(self, x0, y0, node, path, K, dt, seed, step, mode):
        """Scores, exit flags and sub-steps of paths from (x0, y0); node, path: their Philox words."""
        n, T = x0.numel(), K * dt
        x, y = x0.clone(), y0.clone()
        alive = torch.ones(n, dtype=torch.bool, device=x.device)
        score = torch.zeros(n, 2, dtype=torch.float64, device=x.device)
        acc = torch.zeros_like(score)
        steps = torch.zeros(n, dtype=torch.int64, device=x.device)
        left = torch.zeros_like(alive)
        tm = torch.zeros_like(x)
        pair = None
        zero = torch.zeros_like(path)
        limit = 4 * K + 16 if mode == 2 else K
        for j in range(limit):
            last = None
            if mode == 0:
                if j % 2 == 0:
                    pair = _philox(path, node, zero + j // 2, zero + step, seed)
                zx, zy = _normals(pair[2 * (j % 2)], pair[2 * (j % 2) + 1], math.sqrt(2 * dt))
                tau = dt
            else:
                p = _philox(path, node, zero + j, zero + step, seed)
                tau = dt
                if mode == 2:
                    tau = -dt * torch.log1p(-_unit(p[3]))
                    last = (tm + tau >= T) | (j + 1 >= limit)
                    tau = torch.where(last, T - tm, tau)
                zx, zy = _normals(p[0], p[1], 1.0)
                sigma = torch.sqrt(2 * tau) if mode == 2 else math.sqrt(2 * dt)
                zx, zy = zx * sigma, zy * sigma
                ub = _unit(p[2]) + 2.0 ** -23
            i_, j_, s_, t_ = self.cell(x, y)
            if self.model is not None:
                if self.model_cells:
                    G = self.model[j_ * (self.nx - 1) + i_]
                else:
                    G = self.at(self.model[j * self.model.shape[0] // K], i_, j_, s_, t_)
                g = torch.stack([G[:, 0] * zx + G[:, 1] * zy, G[:, 2] * zx + G[:, 3] * zy], -1)
                acc += torch.where(alive[:, None], g, 0.0)
            b = self.at(self.b, i_, j_, s_, t_)
            xn, yn = x + b[:, 0] * tau + zx, y + b[:, 1] * tau + zy
            steps += alive
            # the plain test: the first face of the smallest crossing fraction
            out = (xn <= 0) | (xn >= 1) | (yn <= 0) | (yn >= 1)
            inf = torch.full_like(x, 2.0)
            cut = torch.stack([torch.where(xn <= 0, x / (x - xn), inf), torch.where(xn >= 1, (1 - x) / (xn - x), inf),
                               torch.where(yn <= 0, y / (y - yn), inf), torch.where(yn >= 1, (1 - y) / (yn - y), inf)])
            frac, face = cut.min(0)
            tang = torch.where(face < 2, y + frac * (yn - y), x + frac * (xn - x)).clamp(0, 1)
            if mode:
                # the Brownian bridge between two inside points
                q = torch.stack([x * xn, (1 - x) * (1 - xn), y * yn, (1 - y) * (1 - yn)])
                p4 = torch.exp(-q / tau)
                hit = ~out & (ub < 1 - torch.prod(1 - p4, 0))
                fb = p4.argmax(0)
                face = torch.where(hit, fb, face)
                tang = torch.where(hit, torch.where(fb < 2, 0.5 * (y + yn), 0.5 * (x + xn)).clamp(0, 1), tang)
                out = out | hit
            new = out & alive
            if bool(new.any()):
                k = new.nonzero()[:, 0]
                score[k, 0], score[k, 1] = self.face(0, face[k], tang[k]), self.face(1, face[k], tang[k])
            left |= new
            alive &= ~out
            x, y = torch.where(alive, xn, x), torch.where(alive, yn, y)
            if last is not None:
                tm = torch.where(alive, tm + tau, tm)
                done = alive & last
                if bool(done.any()):
                    k = done.nonzero()[:, 0]
                    score[k] = self.at(self.f, *self.cell(x[k], y[k]))
                alive &= ~last
                if not bool(alive.any()):
                    break
        if mode != 2:
            score = torch.where(alive[:, None], self.at(self.f, *self.cell(x, y)), score)
        return score - acc, left, steps

    def estimate(self, xs, ys, n_paths, K, dt, seed, step=0, mode=0, word0=0):
        dev = self.w.device
        count = len(xs)
        out = {k: torch.zeros(count, dtype=torch.float64, device=dev) for k in ("mean_xi", "mean_eta", "se_xi", "se_eta")}
        out |= {k: torch.zeros(count, dtype=torch.int64, device=dev) for k in ("n_exit", "path_steps")}
        inside = [k for k in range(count) if 0 < xs[k] < 1 and 0 < ys[k] < 1]
        for k in sorted(set(range(count)) - set(inside)):
            f = 0 if xs[k] <= 0 else 1 if xs[k] >= 1 else 2 if ys[k] <= 0 else 3
            t = torch.tensor([ys[k] if f < 2 else xs[k]], dtype=torch.float64, device=dev)
            for q, name in enumerate(("mean_xi", "mean_eta")):
                out[name][k] = self.face(q, torch.tensor([f], device=dev), t)[0]
            out["n_exit"][k] = int(n_paths[k])
        at = 0
        while at < len(inside):
            end, total = at, 0
            while end < len(inside) and (end == at or total + n_paths[inside[end]] <= 3_000_000):
                total += int(n_paths[inside[end]])
                end += 1
            ids = torch.tensor(inside[at:end], device=dev)
            cnt = torch.tensor([int(n_paths[k]) for k in inside[at:end]], device=dev)
            which = torch.repeat_interleave(torch.arange(end - at, device=dev), cnt)
            first = torch.cumsum(cnt, 0) - cnt
            path = torch.arange(total, device=dev) - first[which]
            X = torch.from_numpy(np.asarray(xs, dtype=np.float64)).to(dev)[ids][which]
            Y = torch.from_numpy(np.asarray(ys, dtype=np.float64)).to(dev)[ids][which]
            score, left, steps = self.chunk(X, Y, word0 + ids[which], path, K, dt, seed, step, mode)
            for q, f in enumerate(("xi", "eta")):
                add = lambda v: torch.zeros(end - at, dtype=v.dtype, device=dev).index_add_(0, which, v)  # noqa: E731
                mean = add(score[:, q]) / cnt
                var = add((score[:, q] - mean[which]) ** 2) / (cnt - 1).clamp(min=1)
                out["mean_" + f][ids], out["se_" + f][ids] = mean, torch.sqrt(var / cnt)
            out["n_exit"][ids], out["path_steps"][ids] = add(left.long()), add(steps)
            at = end
        return out


def _solve(w, prev, new, sub, Dt):
    """Implicit Euler of w div((1/w) grad f) on every subdomain: conjugate gradients with the diagonal, to rounding."""
    ny, nx = w.shape
    free = torch.ones(ny, nx, dtype=torch.bool, device=w.device)
    for i in [0, nx - 1] + _lines(nx, sub):
        free[:, i] = False
    for j in [0, ny - 1] + _lines(ny, sub):
        free[j] = False
    cx = 2.0 / (w[:, 1:] + w[:, :-1]) * (nx - 1) ** 2
    cy = 2.0 / (w[1:] + w[:-1]) * (ny - 1) ** 2
    m = 1.0 / (w * Dt)
    d = m.clone()
    d[:, 1:] += cx
    d[:, :-1] += cx
    d[1:] += cy
    d[:-1] += cy

    def apply(u):
        r = d * u
        r[:, :, 1:] -= cx * u[:, :, :-1]
        r[:, :, :-1] -= cx * u[:, :, 1:]
        r[:, 1:] -= cy * u[:, :-1]
        r[:, :-1] -= cy * u[:, 1:]
        return torch.where(free, r, 0.0)

    u = torch.stack([torch.where(free, p, b) for p, b in zip(prev, new)])
    rhs = torch.where(free, m * torch.stack(list(prev)), 0.0)
    dot = lambda a, b: (a * b).sum((1, 2), keepdim=True)  # noqa: E731
    for _ in range(2):  # the second pass takes out what rounding left in the first's recurrence
        r = rhs - apply(u)
        z = r / d
        p, rz = z.clone(), dot(r, z)
        stop = 1e-30 * dot(m * u, m * u)
        for k in range(6000):
            q = apply(p)
            a = rz / dot(p, q).clamp(min=1e-300)
            u = u + a * p
            r = r - a * q
            z = r / d
            new_rz = dot(r, z)
            p = z + new_rz / rz.clamp(min=1e-300) * p
            rz = new_rz
            if k % 50 == 49 and bool((dot(r, r) <= stop).all()):
                break
    return u[0], u[1]


def _key_mask(w, lines, nodes, sub, spacing):
    """Key positions: extrema (of at least a hundredth of the largest) of the first and second differences of 1 / w
    along the interface lines, every position divisible by the spacing, and the crossings."""
    rho = 1.0 / w
    index = {p: k for k, p in enumerate(nodes)}
    mask = np.zeros(len(nodes), dtype=bool)
    vi, hj = set(_lines(w.shape[1], sub)), set(_lines(w.shape[0], sub))
    for pts in lines:
        r = np.array([rho[j, i] for i, j in pts])
        for p in (r[2:] - r[:-2], (r[2:] - r[1:-1]) - (r[1:-1] - r[:-2])):
            big = np.abs(p).max()
            for k in range(1, len(p) - 1):
                top = (p[k] > p[k - 1] and p[k] >= p[k + 1]) or (p[k] < p[k - 1] and p[k] <= p[k + 1])
                if big > 0 and abs(p[k]) * 100 >= big and top:
                    mask[index[pts[k + 1]]] = True
        for t in range(1, len(pts) - 1):
            if (spacing > 0 and t % spacing == 0) or (pts[t][0] in vi and pts[t][1] in hj):
                mask[index[pts[t]]] = True
    return mask


def _pchip(x, y, at):
    """Monotone cubic Hermite interpolation (Fritsch-Butland derivatives, three-point ends)."""
    h, d = np.diff(x), np.diff(y) / np.diff(x)
    if len(x) == 2:
        return y[0] + d[0] * (at - x[0])
    m = np.zeros(len(x))
    for k in range(1, len(x) - 1):
        if d[k - 1] * d[k] > 0:
            a, b = 2 * h[k] + h[k - 1], h[k] + 2 * h[k - 1]
            m[k] = (a + b) / (a / d[k - 1] + b / d[k])
    for e, (h0, h1, d0, d1) in ((0, (h[0], h[1], d[0], d[1])), (-1, (h[-1], h[-2], d[-1], d[-2]))):
        v = ((2 * h0 + h1) * d0 - h0 * d1) / (h0 + h1)
        m[e] = 0.0 if v * d0 <= 0 else 3 * d0 if d0 * d1 < 0 and abs(v) > 3 * abs(d0) else v
    k = np.clip(np.searchsorted(x, at, side="right") - 1, 0, len(h) - 1)
    t = (at - x[k]) / h[k]
    return ((1 + 2 * t) * (1 - t) ** 2 * y[k] + t * (1 - t) ** 2 * h[k] * m[k]
            + t * t * (3 - 2 * t) * y[k + 1] + t * t * (t - 1) * h[k] * m[k + 1])


def _step_exact(s):
    c = s["case"]
    n, sub, K, dt = c["n"], c["sub"], c["K"], c["dt"]
    X, Y = _grid(n, n)
    xi, eta = X.clone(), Y.clone()
    nodes = _interface(n, n, sub)
    xs, ys = np.array([i / (n - 1) for i, _ in nodes]), np.array([j / (n - 1) for _, j in nodes])
    at = torch.tensor([j * n + i for i, j in nodes], device="cuda")
    lines = [[(i, t) for t in range(n)] for i in _lines(n, sub)] + [[(t, j) for t in range(n)] for j in _lines(n, sub)]
    index = {p: k for k, p in enumerate(nodes)}
    for k, w32 in enumerate(s["w"]):
        w = w32.double()
        walk = _Walk(w, xi, eta, None)
        n_paths = np.full(len(nodes), c["paths"])
        if c["spacing"] < 0:
            out = walk.estimate(xs, ys, n_paths, K, dt, s["seed"], step=k)
        else:
            key = _key_mask(w.cpu().numpy(), lines, nodes, sub, c["spacing"])
            out = {q: torch.zeros(len(nodes), dtype=torch.float64, device="cuda") for q in ("mean_xi", "mean_eta", "se_xi", "se_eta")}
            out |= {q: torch.zeros(len(nodes), dtype=torch.int64, device="cuda") for q in ("n_exit", "path_steps")}
            # the node words stay the nodes' own: every key node is estimated under its index
            for a in np.nonzero(key)[0]:
                one = walk.estimate(xs[a:a + 1], ys[a:a + 1], n_paths[a:a + 1], K, dt, s["seed"], step=k, word0=int(a))
                for q in out:
                    out[q][a] = one[q][0]
            F = walk.faces.cpu().numpy()
            for f, name in enumerate(("mean_xi", "mean_eta")):
                v = out[name].cpu().numpy()
                base = f * 4 * n
                for pts in lines:
                    vertical = pts[0][0] == pts[1][0]
                    fixed = pts[0][0] if vertical else pts[0][1]
                    ends = (F[base + 2 * n + fixed], F[base + 3 * n + fixed]) if vertical else (F[base + fixed], F[base + n + fixed])
                    ks = [index[p] for p in pts[1:-1]]
                    ts = [t for t in range(1, n - 1) if key[ks[t - 1]]]
                    got = _pchip(np.array([0.0] + ts + [n - 1.0]), np.array([ends[0]] + [v[ks[t - 1]] for t in ts] + [ends[1]]),
                                 np.arange(1.0, n - 1))
                    for t in range(1, n - 1):
                        if not key[ks[t - 1]]:
                            v[ks[t - 1]] = got[t - 1]
                out[name] = torch.from_numpy(v).cuda()
        new = []
        for f, name in enumerate(("mean_xi", "mean_eta")):
            g = torch.zeros(n, n, dtype=torch.float64, device="cuda")
            F = walk.faces[f * 4 * n:(f + 1) * 4 * n].reshape(4, n)
            g.reshape(-1)[at] = out[name]
            g[:, 0], g[:, -1], g[0], g[-1] = F[0], F[1], F[2], F[3]
            if f == 0:
                g[:, 0], g[:, -1] = F[0], F[1]
            new.append(g)
        xi, eta = _solve(w, (xi, eta), new, sub, K * dt)
    return out | {"xi": xi, "eta": eta}


def _model_table(s):
    """Spatial gradients of the two networks at the nodes, one slice per sub-step."""
    c = s["case"]
    w = s["w"].double()
    ny, nx = w.shape
    wx, wy = _fd(w)
    r = torch.sqrt(wx * wx + wy * wy) / w
    rx, ry = _fd(r)
    X, Y = _grid(nx, ny)
    one, zero = torch.ones_like(X), torch.zeros_like(X)
    mu, sc = s["norm"].double()[:5], s["norm"].double()[5:]
    K, tables = c["K"], []
    for q in range(K):
        F = torch.stack([X, Y, one * ((K - q) / K), w, r], -1).reshape(-1, 5)
        Z = (F - mu) * sc
        dx = torch.stack([one, zero, zero, wx, rx], -1).reshape(-1, 5) * sc
        dy = torch.stack([zero, one, zero, wy, ry], -1).reshape(-1, 5) * sc
        cols = []
        for W1, b1, W2, b2, w3, _ in _unpack(s["theta"]):
            h1 = torch.tanh(Z @ W1.T + b1)
            k2 = 1 - torch.tanh(h1 @ W2.T + b2) ** 2
            for d in (dx, dy):
                cols.append((k2 * (((1 - h1 * h1) * (d @ W1.T)) @ W2.T)) @ w3)
        tables.append(torch.stack(cols, -1))
    return torch.stack(tables)


def _unpack(theta):
    for f in range(2):
        t, o, got = theta.double()[f * sdd.MLP_STRIDE:], 0, []
        for shape in ((64, 5), (64,), (64, 64), (64,), (64,), (1,)):
            size = math.prod(shape)
            got.append(t[o:o + size].reshape(shape))
            o += size
        yield got


def _cells_model(xi, eta):
    """The fields' differences smoothed by the binomial filter of the grid's order, one value per cell."""
    m = max(xi.shape) - 1
    order = max(1, min(2 * (m * m // 16384) - 1, 33))
    g = torch.stack([*_fd(xi), *_fd(eta)], -1)
    for axis in (1, 0):
        L = g.shape[axis]
        at, out = torch.arange(L - 1, device=g.device), 0
        for k in range(order + 1):
            out = out + math.comb(order, k) / 2.0 ** order * g.index_select(axis, (at - (order - 1) // 2 + k).clamp(0, L - 1))
        g = out
    return g.reshape(-1, 4)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "step" and c["n"] > 600:
        return None  # 5e10 path steps: minutes in 64 bits
    s = prepare(case, seed)
    if kind == "estimate":
        model = _cells_model(s["xi"], s["eta"]) if c["cv"] == "fields" else _model_table(s) if c["cv"] == "model" else None
        walk = _Walk(s["w"], s["xi"], s["eta"], s.get("faces"), model, c["cv"] == "fields")
        return walk.estimate(*s["nodes"], c["K"], c["dt"], s["seed"], mode=c["exit_mode"])
    if kind == "step":
        return _step_exact(s)
    if kind == "batch":
        got, word = [], 0
        for w, xi, eta, nodes in s["parts"]:
            got.append(_Walk(w, xi, eta, None).estimate(*nodes, c["K"], c["dt"], s["seed"], word0=word))
            word += len(nodes[0])
        return {k: torch.cat([g[k] for g in got]) for k in got[0]}
    if kind == "solve":
        w, n = s["w"].double(), c["n"]
        F = _faces(w)
        ij = _interface(n, c["ny"], c["sub"])
        new = []
        for f in range(2):
            base, ny = f * 2 * (n + c["ny"]), c["ny"]
            g = torch.zeros(ny, n, dtype=torch.float64, device="cuda")
            if ij:
                g.reshape(-1)[torch.tensor([j * n + i for i, j in ij], device="cuda")] = s["iface"][f]
            g[0], g[-1] = F[base + 2 * ny:base + 2 * ny + n], F[base + 2 * ny + n:base + 2 * ny + 2 * n]
            g[:, 0], g[:, -1] = F[base:base + ny], F[base + ny:base + 2 * ny]
            new.append(g)
        xi, eta = _solve(w, (s["xi"], s["eta"]), new, c["sub"], c["Dt"])
        return {"xi": xi, "eta": eta}
    grads, losses = [], []
    Z = (s["feats"].double() - s["norm"].double()[:5]) * s["norm"].double()[5:]
    for f, (W1, b1, W2, b2, w3, b3) in enumerate(_unpack(s["theta"])):
        h1 = torch.tanh(Z @ W1.T + b1)
        h2 = torch.tanh(h1 @ W2.T + b2)
        e = h2 @ w3 + b3 - s["targets"][:, f].double()
        d = 2 * e / e.numel()
        g2 = d[:, None] * w3 * (1 - h2 * h2)
        g1 = (g2 @ W2) * (1 - h1 * h1)
        flat = torch.cat([(g1.T @ Z).reshape(-1), g1.sum(0), (g2.T @ h1).reshape(-1), g2.sum(0), h2.T @ d, d.sum()[None]])
        grads.append(torch.cat([flat, torch.zeros(sdd.MLP_STRIDE - flat.numel(), dtype=torch.float64, device="cuda")]))
        losses.append((e * e).mean())
    return {"grad": torch.cat(grads), "loss": torch.stack(losses)}
