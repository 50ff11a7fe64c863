"""Workloads of the library as a user's program runs them, for timing.

Five kinds, each through the public entry points (the binding's Solver,
Batch and Solver3, and the C ABI's device-pointer forms where the binding
only copies to the host):

* ``lattice``: advance the resident state of one D2Q9 lattice by a chunk of
  steps and write its fields (rho, u, mu) to device tensors, as a simulation
  loop does between two looks at its state;
* ``relax``: one relax-to-equilibrium request from its initial density, with
  a check every ``check`` steps and a step budget, and its fields;
* ``batch``: a round of the batched persistent kernel over many uneven
  cases, then the fields of eight of them to the host, as the serving loop
  delivers the requests that finished;
* ``d3q19``: the three-dimensional lattice, advanced like ``lattice``;
* ``sequence``: several initial states relaxed one after another from and to
  page-locked host memory.

Initial densities are tanh droplets or slabs (Sec. IV of Guo, arXiv
2012.11075) whose places, sizes and noise follow the seed.  The relaxation
times are ones at which the scheme stays stable for long runs, so that a
state can be advanced as often as a measurement wants.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2012_11075_gb300 import wblbe

SCHEMES = {"well_balanced": wblbe.WELL_BALANCED, "standard": wblbe.STANDARD}
PRECISIONS = {"fp64": wblbe.FP64, "fp32": wblbe.FP32_SHIFTED}
FETCHED = 8                      # finished requests a serving round delivers


def listed():
    wb, std = "well_balanced", "standard"
    return [
        # the flat-interface run: the smallest lattice, thousands of steps in
        # a row, where latency per step is everything
        dict(name="flat_4x256_fp64", kind="lattice", shape="slab", nx=4, ny=256, scheme=wb,
             precision="fp64", ratio=10.0, width=4.0, tau=1.0, noise=0.01, steps=256),
        # the paper's 100 x 100 droplet with the scheme it is compared against
        dict(name="droplet_100_fp64_std", kind="lattice", shape="droplets", nx=100, ny=100,
             count=1, scheme=std, precision="fp64", ratio=5.0, width=4.0, tau=0.85, noise=0.0,
             steps=200),
        # the stationary droplet of the verification runs (100000 steps in use)
        dict(name="droplet_256_fp64", kind="lattice", shape="droplets", nx=256, ny=256, count=1,
             scheme=wb, precision="fp64", ratio=10.0, width=4.0, tau=1.0, noise=0.0, steps=200),
        # large domain, FP64: the arithmetic-bound end
        dict(name="large_4096_fp64", kind="lattice", shape="droplets", nx=4096, ny=4096, count=64,
             scheme=wb, precision="fp64", ratio=10.0, width=5.0, tau=0.9, noise=0.0, steps=8),
        # large domain, FP32-shifted: the throughput headline
        dict(name="large_4096_fp32", kind="lattice", shape="droplets", nx=4096, ny=4096, count=64,
             scheme=wb, precision="fp32", ratio=10.0, width=5.0, tau=0.9, noise=0.0, steps=100),
        # odd sides: rows that no vector load divides
        dict(name="ragged_1023x771_fp32", kind="lattice", shape="droplets", nx=1023, ny=771,
             count=6, scheme=wb, precision="fp32", ratio=10.0, width=4.0, tau=1.0, noise=0.0,
             steps=100),
        # the comparison scheme at a medium size
        dict(name="medium_1024_fp32_std", kind="lattice", shape="droplets", nx=1024, ny=1024,
             count=8, scheme=std, precision="fp32", ratio=5.0, width=4.0, tau=1.0, noise=0.0,
             steps=100),
        # one serving-size request on its own: init, checks, budget, fields
        dict(name="relax_320x192_fp32", kind="relax", shape="droplets", nx=320, ny=192, count=1,
             scheme=wb, precision="fp32", ratio=10.0, width=4.0, tau=1.0, noise=0.0, tol=1e-9,
             budget=1000, check=250),
        # many uneven cases at once
        dict(name="batch_128_fp32", kind="batch", cases=128, side_min=64, side_max=512,
             precision="fp32", tile_x=128, rows=128, per_launch=64, launches=8),
        # three dimensions, both precisions
        dict(name="d3q19_256_fp32", kind="d3q19", nx=256, ny=256, nz=256, scheme=wb,
             precision="fp32", ratio=10.0, width=4.0, tau=1.0, steps=16),
        dict(name="d3q19_128_fp64", kind="d3q19", nx=128, ny=128, nz=128, scheme=wb,
             precision="fp64", ratio=10.0, width=4.0, tau=1.0, steps=8),
        # host to host: density in, density and statistics out
        dict(name="sequence_2048_fp32", kind="sequence", shape="droplets", nx=2048, ny=2048,
             count=16, scheme=wb, precision="fp32", ratio=10.0, width=5.0, tau=0.9, noise=0.0,
             states=3, steps=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lattice", "lattice", "lattice", "relax", "batch", "d3q19", "sequence"])
    precision = rng.choice(["fp64", "fp32"])
    scheme = rng.choice(["well_balanced", "well_balanced", "standard"])
    wb = scheme == "well_balanced"
    common = dict(scheme=scheme, precision=precision,
                  ratio=round(rng.uniform(5.0, 20.0), 2) if wb else round(rng.uniform(2.0, 5.0), 2),
                  width=float(rng.choice([4, 5])), tau=round(rng.uniform(0.9, 1.2), 3))
    rate = 2.5e9 if precision == "fp64" else 3.0e10          # updates per second, roughly
    if kind == "lattice":
        nx, ny = _log_int(rng, 4, 2048), _log_int(rng, 32, 2048)
        shape = "slab" if nx < 48 or ny < 48 or rng.random() < 0.3 else "droplets"
        c = dict(kind=kind, shape=shape, nx=nx, ny=ny, **common,
                 noise=0.01 if shape == "slab" else 0.0)
        if shape == "droplets":
            c["count"] = rng.randint(1, max(1, min(16, nx * ny // 40000)))
        c["steps"] = max(4, min(rng.randint(60, 260), int(0.02 * rate / (nx * ny))))
        return c
    if kind == "relax":
        nx, ny = _log_int(rng, 48, 1024), _log_int(rng, 48, 1024)
        budget = max(50, min(1000, int(0.02 * rate / (nx * ny))))
        return dict(kind=kind, shape="droplets", nx=nx, ny=ny, count=1, **common, noise=0.0,
                    tol=1e-9 if precision == "fp32" else 1e-13, budget=budget,
                    check=max(10, budget // rng.randint(2, 5)))
    if kind == "batch":
        return dict(kind=kind, cases=rng.randint(16, 128), side_min=64,
                    side_max=rng.randint(160, 400), precision="fp32",
                    tile_x=rng.choice([64, 128]), rows=rng.choice([32, 64, 128]),
                    per_launch=rng.choice([32, 64]), launches=rng.randint(2, 8))
    if kind == "d3q19":
        nx, ny, nz = (_log_int(rng, 24, 200) for _ in range(3))
        rate3 = 1.5e9 if precision == "fp64" else 1.0e10
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, **common,
                    steps=max(2, min(50, int(0.01 * rate3 / (nx * ny * nz)))))
    nx, ny = _log_int(rng, 100, 1500), _log_int(rng, 100, 1500)
    return dict(kind=kind, shape="droplets", nx=nx, ny=ny, count=1, **common, noise=0.0,
                states=rng.randint(2, 4),
                steps=max(4, min(100, int(0.01 * rate / (nx * ny)))))


# ---- inputs -----------------------------------------------------------------

KAPPA = 0.01


def _physics(case):
    rho_l, rho_g = 1.0, 1.0 / case["ratio"]
    beta = 8.0 * KAPPA / (case["width"] * (rho_l - rho_g)) ** 2
    return rho_l, rho_g, beta


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _profile(r, radius, rho_l, rho_g, width):
    return 0.5 * (rho_l + rho_g) - 0.5 * (rho_l - rho_g) * torch.tanh(2.0 * (r - radius) / width)


def _sphere(shape, centre, radius, rho_l, rho_g, width):
    """Liquid sphere (or disc) in vapour on a periodic lattice, any dimension;
    shape and centre in array order."""
    r2 = None
    for d, (n, c) in enumerate(zip(shape, centre)):
        x = (torch.arange(n, dtype=torch.float64, device=_device()) - c).abs()
        x = torch.minimum(x, n - x).square()
        x = x.reshape([-1 if k == d else 1 for k in range(len(shape))])
        r2 = x if r2 is None else r2 + x
    return _profile(r2.sqrt(), radius, rho_l, rho_g, width)


def _density(case, seed):
    """Initial density [ny][nx] on the device."""
    rho_l, rho_g, _ = _physics(case)
    nx, ny, width = case["nx"], case["ny"], case["width"]
    rng = np.random.default_rng([seed, nx, ny])
    if case["shape"] == "slab":
        y = torch.arange(ny, dtype=torch.float64, device=_device())
        centre, half = ny * rng.uniform(0.4, 0.6), ny * rng.uniform(0.2, 0.3)
        d = (y - centre).abs()
        row = _profile(torch.minimum(d, ny - d), half, rho_l, rho_g, width)
        rho = row[:, None].expand(ny, nx).clone()
    else:
        # one droplet in each of some cells of a grid, so that none overlap
        n = case["count"]
        cols = max(1, min(n, int(round(math.sqrt(n * nx / ny)))))
        rows = -(-n // cols)
        cx, cy = nx / cols, ny / rows
        rho = torch.full((ny, nx), rho_g, dtype=torch.float64, device=_device())
        for k in range(n):
            radius = min(64.0, min(cx, cy) * rng.uniform(0.2, 0.3))
            at = ((k // cols + rng.uniform(0.45, 0.55)) * cy,
                  (k % cols + rng.uniform(0.45, 0.55)) * cx)
            # the profile is vapour outside a few widths: only a window of it
            reach = int(radius + 10 * width) + 2
            y0, x0 = int(at[0]) - reach, int(at[1]) - reach
            if 2 * reach < min(nx, ny) and n > 1:
                side = 2 * reach
                ys = torch.arange(y0, y0 + side, device=_device()) % ny
                xs = torch.arange(x0, x0 + side, device=_device()) % nx
                # a lattice of its own, larger than the window: no wrap inside it
                w = _sphere((4 * side, 4 * side), (at[0] - y0, at[1] - x0), radius, rho_l,
                            rho_g, width)[:side, :side]
                rho[ys[:, None], xs[None, :]] = torch.maximum(rho[ys[:, None], xs[None, :]], w)
            else:
                rho = torch.maximum(rho, _sphere((ny, nx), at, radius, rho_l, rho_g, width))
    if case["noise"]:
        r = torch.from_numpy(rng.uniform(-1.0, 1.0, (ny, nx))).to(rho.device)
        rho = rho * (1.0 + case["noise"] * r)
    return rho.contiguous()


def _density3(case, seed):
    rho_l, rho_g, _ = _physics(case)
    shape = (case["nz"], case["ny"], case["nx"])
    rng = np.random.default_rng([seed, *shape])
    centre = [n * rng.uniform(0.45, 0.55) for n in shape]
    return _sphere(shape, centre, min(shape) * rng.uniform(0.2, 0.3), rho_l, rho_g, case["width"])


def _batch_specs(case, seed):
    """The uneven mix: sides log-uniform, flat slab or droplet, density ratio
    2-50, kappa 0.005-0.02, W in {3, 4, 5}; tau in the stable range."""
    # sizes follow the case, so that every seed has the same amount of work
    sizes = np.random.default_rng(case["cases"] * 1000 + case["side_max"])
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(case["cases"]):
        nx, ny = (int(round(math.exp(sizes.uniform(math.log(case["side_min"]),
                                                   math.log(case["side_max"])))))
                  for _ in range(2))
        out.append(dict(nx=nx, ny=ny, shape="slab" if rng.random() < 0.5 else "droplets", count=1,
                        ratio=float(rng.uniform(2.0, 50.0)), width=float(rng.choice([3, 4, 5])),
                        tau=float(rng.uniform(0.9, 1.2)), kappa=float(rng.uniform(0.005, 0.02)),
                        noise=0.001, seed=int(rng.integers(1 << 30))))
    for s in out:
        s["beta"] = 8.0 * s["kappa"] / (s["width"] * (1.0 - 1.0 / s["ratio"])) ** 2
    return out


def _params(case):
    rho_l, rho_g, beta = _physics(case)
    return wblbe.Params(case["nx"], case["ny"], case["tau"], KAPPA, beta, rho_l, rho_g,
                        scheme=SCHEMES[case["scheme"]], precision=PRECISIONS[case["precision"]])


# ---- the passes -------------------------------------------------------------


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        specs = _batch_specs(case, seed)
        cases = [(wblbe.Params(s["nx"], s["ny"], s["tau"], s["kappa"], s["beta"], 1.0,
                               1.0 / s["ratio"], precision=PRECISIONS[case["precision"]]),
                  _density(s, s["seed"]).cpu().numpy()) for s in specs]
        b = wblbe.Batch(precision=PRECISIONS[case["precision"]], max_cases=len(cases),
                        max_case_nodes=max(p.nx * p.ny for p, _ in cases),
                        arena_bytes=sum(_case_bytes(p) for p, _ in cases) + (1 << 20),
                        tile_x=case["tile_x"], rows_per_tile=case["rows"],
                        steps_per_launch=case["per_launch"])
        ids = [b.admit(p, rho, 0.0, 10 ** 12) for p, rho in cases]
        return dict(case=case, batch=b, ids=ids)
    if kind == "d3q19":
        rho_l, rho_g, beta = _physics(case)
        s = wblbe.Solver3(wblbe.Params3(case["nx"], case["ny"], case["nz"], case["tau"], KAPPA,
                                        beta, rho_l, rho_g, scheme=SCHEMES[case["scheme"]],
                                        precision=PRECISIONS[case["precision"]]))
        s.init_rho(_density3(case, seed))
        out = {"rho": torch.empty(s.shape, dtype=torch.float64, device="cuda"),
               "u": torch.empty((3,) + s.shape, dtype=torch.float64, device="cuda"),
               "mu": torch.empty(s.shape, dtype=torch.float64, device="cuda")}
        return dict(case=case, solver=s, out=out)
    s = wblbe.Solver(_params(case))
    if kind == "sequence":
        rho_in = [_density(case, seed + 1000 * k).cpu().pin_memory()
                  for k in range(case["states"])]
        rho_out = [torch.empty(s.shape, dtype=torch.float64).pin_memory() for _ in rho_in]
        return dict(case=case, solver=s, rho_in=rho_in, rho_out=rho_out)
    rho = _density(case, seed)
    out = {"rho": torch.empty(s.shape, dtype=torch.float64, device="cuda"),
           "u": torch.empty((2,) + s.shape, dtype=torch.float64, device="cuda"),
           "mu": torch.empty(s.shape, dtype=torch.float64, device="cuda")}
    if kind == "lattice":
        s.init_rho(rho)
    return dict(case=case, solver=s, rho=rho, out=out)


def _case_bytes(p):
    cp = p.c()
    return int(wblbe.load_library().wblbe_batch_case_bytes(ctypes.byref(cp)))


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "batch":
        b = state["batch"]
        b.advance(case["launches"])
        return [b.fetch(i)[0] for i in state["ids"][:FETCHED]]
    s = state["solver"]
    if kind == "sequence":
        s.run_sequence(state["rho_in"], case["steps"], state["rho_out"])
        return state["rho_out"]
    out = state["out"]
    if kind == "d3q19":
        s.step(case["steps"])
        stats = wblbe.CStats()
        s._check(s.lib.wblbe3_moments(s.h, out["rho"].data_ptr(), out["u"].data_ptr(),
                                      out["mu"].data_ptr(), 1, ctypes.byref(stats)))
        return out
    if kind == "relax":
        s.init_rho(state["rho"])
        s.run_until_equilibrium(case["tol"], case["budget"], case["check"])
    else:
        s.step(case["steps"])
    s.moments_into(out["rho"], out["u"][0], out["u"][1], out["mu"])
    return out


def work(case):
    """The resident state read once and written once, host and field data
    once; FP64 and FP32 operations of the update (each operation counts one,
    a multiply-add two), for every step."""
    kind = case["kind"]
    size = 8 if case["precision"] == "fp64" else 4
    if kind == "batch":
        specs = _batch_specs(case, 0)
        nodes = [s["nx"] * s["ny"] for s in specs]
        return {"bytes": 2 * 9 * size * sum(nodes) + 2 * 4 * 8 * sum(nodes[:FETCHED]),
                "flops": 160 * sum(nodes) * case["per_launch"] * case["launches"]}
    if kind == "d3q19":
        nodes = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": (2 * 19 * size + 5 * 8) * nodes, "flops": 320 * nodes * case["steps"]}
    nodes = case["nx"] * case["ny"]
    if kind == "sequence":
        return {"bytes": case["states"] * 4 * 8 * nodes,
                "flops": 160 * nodes * case["steps"] * case["states"]}
    if kind == "relax":
        return {"bytes": (8 + 4 * 8) * nodes, "flops": 160 * nodes * case["budget"]}
    return {"bytes": (2 * 9 * size + 4 * 8) * nodes, "flops": 160 * nodes * case["steps"]}


# ---- the same in plain torch, in 64 bits ------------------------------------


def _velocities(dim):
    """Velocities in array order ((y, x) or (z, y, x)) and weights of D2Q9
    and D3Q19."""
    axes = range(-1, 2)
    if dim == 2:
        c = [(y, x) for y in axes for x in axes]
        w = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}
    else:
        c = [(z, y, x) for z in axes for y in axes for x in axes if abs(x) + abs(y) + abs(z) < 3]
        w = {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
    return c, [w[sum(abs(a) for a in v)] for v in c]


class _Reference:
    """f_i(x, t) after streaming, before the collision (Eq. D2Q9)."""

    def __init__(self, rho, tau, kappa, beta, rho_l, rho_g, well_balanced):
        self.c, self.w = _velocities(rho.dim())
        self.dims = tuple(range(rho.dim()))
        self.p = (tau, kappa, beta, rho_l, rho_g, well_balanced)
        self.f = [self._feq(c, w, rho, [torch.zeros_like(rho)] * rho.dim())
                  for c, w in zip(self.c, self.w)]

    def _at(self, phi, c):                       # phi(x + c)
        return torch.roll(phi, tuple(-a for a in c), self.dims) if any(c) else phi

    def _dot(self, c, v):
        s = None
        for a, b in zip(c, v):
            if a:
                b = b if a > 0 else -b
                s = b if s is None else s + b
        return s

    def _feq(self, c, w, rho, u):
        uu = sum(a * a for a in u)
        s = -1.5 * uu
        if any(c):
            cu = self._dot(c, u)
            s = s + 3.0 * cu + 4.5 * cu * cu
        if self.p[5]:                            # Eq. mFeq with rho0 = 0
            return w * rho * s if any(c) else rho + w * rho * s
        return w * rho * (1.0 + s)               # Eq. feq

    def _grad(self, phi):
        g = [torch.zeros_like(phi) for _ in self.dims]
        for c, w in zip(self.c, self.w):
            if any(c):
                v = (3.0 * w) * self._at(phi, c)
                for k, a in enumerate(c):
                    if a:
                        g[k] += a * v
        return g

    def macro(self):
        tau, kappa, beta, rho_l, rho_g, wb = self.p
        rho = sum(self.f)
        lap = torch.zeros_like(rho)
        for c, w in zip(self.c, self.w):
            if any(c):
                lap += (6.0 * w) * (self._at(rho, c) - rho)
        mu = 2.0 * beta * (rho - rho_l) * (rho - rho_g) * (2.0 * rho - rho_l - rho_g) - kappa * lap
        gm, gr = self._grad(mu), self._grad(rho)
        F = [-rho * m for m in gm] if wb else [r / 3.0 - rho * m for r, m in zip(gr, gm)]
        j = [torch.zeros_like(rho) for _ in self.dims]
        for c, f in zip(self.c, self.f):
            for k, a in enumerate(c):
                if a:
                    j[k] += a * f
        u = [(a + 0.5 * b) / rho for a, b in zip(j, F)]
        return rho, u, mu, F, gr

    def step(self):
        tau, wb, dim = self.p[0], self.p[5], len(self.dims)
        rho, u, _, F, gr = self.macro()
        G = [a + b / 3.0 for a, b in zip(F, gr)] if wb else F
        uG = sum(a * b for a, b in zip(u, G))
        ur = sum(a * b for a, b in zip(u, gr)) if wb else None
        for i, (c, w) in enumerate(zip(self.c, self.w)):
            s = -3.0 * uG
            if any(c):
                s = s + 3.0 * self._dot(c, F) + 9.0 * self._dot(c, u) * self._dot(c, G)
            if wb:
                s = s + 0.5 * (3.0 * sum(abs(a) for a in c) - dim) * ur
            out = self.f[i] - (self.f[i] - self._feq(c, w, rho, u)) / tau
            out += (1.0 - 0.5 / tau) * w * s
            self.f[i] = torch.roll(out, c, self.dims) if any(c) else out

    def run(self, n):
        for _ in range(n):
            self.step()
        return self


def exact(case, seed):
    kind, wb = case["kind"], case.get("scheme", "well_balanced") == "well_balanced"
    if kind == "batch":
        out = []
        for s in _batch_specs(case, seed)[:FETCHED]:
            r = _Reference(_density(s, s["seed"]), s["tau"], s["kappa"], s["beta"], 1.0,
                           1.0 / s["ratio"], True).run(case["per_launch"] * case["launches"])
            rho, u, mu = r.macro()[:3]
            out.append({"rho": rho, "ux": u[1], "uy": u[0], "mu": mu})
        return out
    rho_l, rho_g, beta = _physics(case)

    def after(rho, n):
        r = _Reference(rho, case["tau"], KAPPA, beta, rho_l, rho_g, wb).run(n)
        rho, u, mu = r.macro()[:3]
        return {"rho": rho, "u": torch.stack(u[::-1]), "mu": mu}

    if kind == "d3q19":
        return after(_density3(case, seed), case["steps"])
    if kind == "sequence":
        return [after(_density(case, seed + 1000 * k), case["steps"])["rho"]
                for k in range(case["states"])]
    return after(_density(case, seed), case["budget"] if kind == "relax" else case["steps"])
