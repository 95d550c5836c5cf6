"""The particle-in-tree work that is timed: time steps, re-binning and re-refinement through the public calls of
``paper_1508_02435_gb300.pic`` at the sizes of the repository's own workloads, configurations and tests.

Every case is one pass of a program's main loop: a few time steps (or one re-bin) queued on the GPU, then the native
particle state, the vertex charges and the field read into device arrays.  Inputs are drawn on the GPU from the seed.
"""
import functools
import math

import numpy as np
import torch

from paper_1508_02435_gb300 import pic
from paper_1508_02435_gb300.workloads import tree_flags_from_predicate, uniform_tree_flags

DT = 0.1        # omega_p dt of the plasma workloads
OMEGA = 0.8     # damping of the built-in Jacobi solve
Q3 = 774840978  # 2 * 3^18: quantisation of positions


def _plasma(name, d, depth, n, scheme, precision, mode, steps, sweeps=100, quiet=0, graph=False, vth=0.05):
    """A Langmuir wave on the uniform tree of `depth`: quiet = particles per cell and axis of a regular lattice start,
    0 = n random positions.  mode "step": deposit, built-in solve, push and re-bin; "fixed": the field stays."""
    return {"name": name, "kind": "plasma", "d": d, "depth": depth, "n": n, "scheme": scheme, "precision": precision,
            "mode": mode, "steps": steps, "sweeps": sweeps, "quiet": quiet, "graph": graph, "vth": vth}


def listed():
    return [
        # the smallest configuration: 27 x 27 cells, 16 particles per cell, whole steps; launches and latency count
        _plasma("langmuir2d_27_fp64", 2, 3, 11664, "pit", "fp64", "step", 1, quiet=4),
        # a small 3D plasma (27^3 cells, 8 per cell) stepped as a captured graph, ten whole steps between read-outs
        _plasma("langmuir3d_27_fp32_graph", 3, 3, 157464, "pit", "fp32", "step", 10, quiet=2, graph=True),
        # the validation plasma: 243 x 243 cells of one Debye length, 100 random particles per cell, field held
        _plasma("thermal2d_243_fp32", 2, 5, 5904900, "pit", "fp32", "fixed", 5, vth=1 / 243),
        # a whole step in 3D at ordinary size: 81^3 cells, 8 per cell, 100 Jacobi sweeps
        _plasma("langmuir3d_81_fp32", 3, 4, 4251528, "pit", "fp32", "step", 1, quiet=2),
        # the same in FP64 (the generic kernels)
        _plasma("langmuir3d_81_fp64", 3, 4, 4251528, "pit", "fp64", "step", 1, quiet=2),
        # the headline: 243^3 cells, 8 per cell, five fixed-field steps between read-outs
        _plasma("langmuir3d_243_fp32", 3, 5, 114791256, "pit", "fp32", "fixed", 5, quiet=2),
        # the headline plasma with its field solve: the largest pass
        _plasma("langmuir3d_243_fp32_solve", 3, 5, 114791256, "pit", "fp32", "step", 1, quiet=2),
        # adaptive 2D (Gaussian bump, 1e6 particles, levels 4-6, 64 per cell), PIDT: restart from a saved state and
        # take five whole steps
        {"name": "bump2d_1e6_fp64_pidt", "kind": "bump", "d": 2, "n": 1000000, "dmin": 4, "dmax": 6, "ppc": 64,
         "scheme": "pidt", "precision": "fp64", "steps": 5, "sweeps": 100},
        # adaptive 3D two-stream (levels 4-6, 32 per cell), PIDT: five fixed-field steps between read-outs
        {"name": "twostream3d_2e8_fp32_pidt", "kind": "beams", "d": 3, "n": 200000000, "dmin": 4, "dmax": 6, "ppc": 32,
         "scheme": "pidt", "precision": "fp32", "steps": 5, "sweeps": 20},
        # 256 uneven 2D plasmas in one handle (1e3 to 1e6 particles each), ten captured fixed-field steps
        {"name": "batch256_2d_fp32", "kind": "batch", "d": 2, "n_inst": 256, "n_min": 1000, "n_max": 1000000,
         "scheme": "pit", "precision": "fp32", "steps": 10, "sweeps": 100},
        # the particle-handling experiment: 1e7 free particles in a reflecting box, re-refined before every step
        {"name": "handling2d_1e7_fp32", "kind": "handling", "d": 2, "n": 10000000, "dmin": 1, "dmax": 8, "ppc": 1000,
         "scheme": "pit", "precision": "fp32", "dt": 1e-3, "steps": 5},
        # particles that another code moved (unordered native state) handed over, re-binned and deposited
        {"name": "rebin3d_5e6_fp32", "kind": "rebin", "d": 3, "depth": 4, "n": 5000011, "scheme": "pit",
         "precision": "fp32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plasma", "plasma", "plasma", "bump", "beams", "batch", "handling", "rebin"])
    scheme, precision = rng.choice(["pit", "pit", "pidt"]), rng.choice(["fp32", "fp32", "fp64"])
    d = rng.choice([2, 3])
    if kind == "plasma":
        depth = rng.randint(2, 7 if d == 2 else 5)
        cells = 3 ** (d * depth)
        n = _log(rng, max(1000, cells // 2), min(30_000_000, cells * 200)) | 1
        c = _plasma("", d, depth, n, scheme, precision, rng.choice(["step", "fixed"]), rng.randint(1, 5),
                    sweeps=rng.choice([20, 50, 100]), graph=rng.random() < 0.25, vth=rng.choice([0.02, 0.05, 0.1]))
        del c["name"]
        return c
    if kind == "bump":
        dmin = rng.randint(2, 4) if d == 2 else rng.randint(2, 3)
        return {"kind": kind, "d": d, "n": _log(rng, 20_000, 4_000_000) | 1, "dmin": dmin, "dmax": dmin + 2,
                "ppc": rng.choice([16, 32, 64]), "scheme": scheme, "precision": precision, "steps": rng.randint(1, 5),
                "sweeps": rng.choice([20, 50, 100])}
    if kind == "beams":
        dmin = rng.randint(3, 5) if d == 2 else rng.randint(2, 3)
        return {"kind": kind, "d": d, "n": _log(rng, 100_000, 30_000_000) | 1, "dmin": dmin, "dmax": dmin + 2,
                "ppc": rng.choice([16, 32, 64]), "scheme": scheme, "precision": precision, "steps": rng.randint(1, 5),
                "sweeps": 20}
    if kind == "batch":
        return {"kind": kind, "d": 2, "n_inst": rng.randint(2, 64), "n_min": 100, "n_max": _log(rng, 10_000, 500_000),
                "scheme": scheme, "precision": precision, "steps": rng.randint(2, 10), "sweeps": rng.choice([20, 100])}
    if kind == "handling":
        return {"kind": kind, "d": d, "n": _log(rng, 30_000, 10_000_000) | 1, "dmin": 1, "dmax": 8 if d == 2 else 5,
                "ppc": rng.choice([100, 1000]), "scheme": scheme, "precision": precision,
                "dt": rng.choice([1e-4, 1e-3, 1e-2]), "steps": rng.randint(1, 5)}
    return {"kind": "rebin", "d": d, "depth": rng.randint(2, 6 if d == 2 else 4), "n": _log(rng, 5_000, 20_000_000) | 1,
            "scheme": scheme, "precision": precision}


# ---- inputs --------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _randn(g, *shape):
    # drawn in single precision: the values are random either way and half the preparation time is saved
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32).double()


def _perturb(u, amp=0.01, k=1):
    """Inverse CDF of the density 1 + amp cos(2 pi k x)."""
    w = 2 * math.pi * k
    x = u.clone()
    for _ in range(8):
        x -= (x + amp / w * torch.sin(w * x) - u) / (1 + amp * torch.cos(w * x))
    return torch.remainder(x, 1.0)


def _plasma_particles(c, seed):
    g, d, n = _gen(seed), c["d"], c["n"]
    if c["quiet"]:
        m = 3 ** c["depth"] * c["quiet"]
        line = (torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) / m
        axes = [line] * (d - 1) + [_perturb(line)]
        x = torch.stack([a.reshape(-1) for a in torch.meshgrid(*axes, indexing="ij")][::-1])
    else:
        x = _rand(g, d, n)
        x[0] = _perturb(x[0])
    return x.contiguous(), _randn(g, d, n) * c["vth"]


def _batch_particles(c, seed):
    """Per instance: particles and depth (log-uniform counts, depths 3 to 5, v_th 0.02 to 0.1, mode 1, 2 or 4: one
    mix of sizes for all seeds)."""
    host, g, out = np.random.default_rng(2), _gen(seed), []
    for _ in range(c["n_inst"]):
        n = int(round(math.exp(host.uniform(math.log(c["n_min"]), math.log(c["n_max"])))))
        depth, vth, k = int(host.integers(3, 6)), float(host.uniform(0.02, 0.1)), int(host.choice([1, 2, 4]))
        u = (torch.arange(n, device="cuda", dtype=torch.float64) + _rand(g, n)) / n
        out.append((torch.stack([_perturb(u, k=k), _rand(g, n)]), _randn(g, 2, n) * vth, depth))
    return out


def _bump_particles(c, seed):
    """Uniform background and a Gaussian bump of ten times its density (sigma 0.1), Maxwellian velocities with a 5% Cauchy tail
    clipped to 20 finest cells per step."""
    g, d, n, sigma, vth = _gen(seed), c["d"], c["n"], 0.1, 0.02
    nb = n - int(round(n / (1 + 9 * (2 * math.pi * sigma * sigma) ** (d / 2))))
    x = _rand(g, d, n)
    x[:, :nb] = torch.remainder(0.5 + sigma * _randn(g, d, nb), 1.0)
    x = torch.where(x >= 1.0, 0.0, x)[:, torch.randperm(n, generator=g, device="cuda")].contiguous()
    v = _randn(g, d, n) * vth
    nt = n // 20
    tail = torch.tan(math.pi * (_rand(g, nt) - 0.5)).abs().mul(vth).clamp(max=20 * 3.0 ** -c["dmax"] / DT)
    way = _randn(g, d, nt)
    v[:, :nt] = way / way.norm(dim=0) * tail
    return x, v


def _beam_particles(c, seed):
    """Thermal background and two beams of a tenth each along x at eight level-(dmin + 1) cells per step."""
    g, d, n = _gen(seed), c["d"], c["n"]
    x, v, nb = _rand(g, d, n), _randn(g, d, n) * 0.05, c["n"] // 10
    u = 8 * 3.0 ** -(c["dmin"] + 1) / DT
    v[:, :2 * nb] *= 0.2
    v[0, :nb] += u
    v[0, nb:2 * nb] -= u
    return x, v


def _handling_particles(c, seed):
    """Free particles: uniform positions, speeds uniform in [0, 1], directions uniform."""
    g, d, n = _gen(seed), c["d"], c["n"]
    x, way = _rand(g, d, n), _randn(g, d, n)
    return x, way / way.norm(dim=0).clamp(min=1e-9) * _rand(g, n)


@functools.lru_cache(maxsize=4)
def _tree(kind, d, n, dmin, dmax, ppc):
    """Flags of the tree that the particles-per-cell criterion leaves for such particles: a cell is refined where a
    draw of its count, from its expectation, is over ppc (one draw for all seeds: every seed has the same vertices)."""
    rng = np.random.default_rng(1)

    def refine(level, coords):
        if level < dmin:
            return np.ones(len(coords), bool)
        density = 1.0
        if kind == "bump":
            r2 = (((coords + 0.5) / 3 ** level - 0.5) ** 2).sum(1)
            density = (1 + 9 * np.exp(-r2 / 0.02)) / (1 + 9 * (0.02 * math.pi) ** (d / 2))
        return rng.poisson(density * n / 3.0 ** (d * level), len(coords)) > ppc

    return tree_flags_from_predicate(d, dmax, refine)


def _kw(c, q, sweeps=0):
    return dict(scheme=pic.PIT if c["scheme"] == "pit" else pic.PIDT,
                precision=pic.FP64 if c["precision"] == "fp64" else pic.FP32_SPLIT,
                q=q, qm=-1.0, ion=1.0, sweeps=sweeps, omega=OMEGA, track_ids=False)


def _buffers(h, c, n, field=True):
    """Device arrays that a program reads the results of a pass into."""
    ft = torch.float64 if c["precision"] == "fp64" else torch.float32
    e = lambda *s, t=ft: torch.empty(*s, device="cuda", dtype=t)  # noqa: E731
    out = {"leaf": e(n, t=torch.int32), "pos": e(c["d"], n), "vel": e(c["d"], n)}
    if field:
        if not c.get("graph") and c["kind"] != "batch":  # captured steps go on from the charges that they hold
            out["Q"] = e(h.n_vertices, t=torch.float64)
        out["E"] = e(c["d"], h.n_vertices, t=torch.float64)
    return out


def prepare(case, seed):
    c = dict(case)
    kind, d = c["kind"], c["d"]
    st = {"case": c, "stream": torch.cuda.Stream() if c.get("graph") or kind == "batch" else None}
    if kind == "plasma":
        x, v = _plasma_particles(c, seed)
        torch.cuda.synchronize()
        h = pic.Pic(d, uniform_tree_flags(d, c["depth"]), x, v, stream=st["stream"], **_kw(c, -1.0 / c["n"], c["sweeps"]))
        h.init_leapfrog(DT)
        if c["graph"]:
            (h.graph_capture_step if c["mode"] == "step" else h.graph_capture)(DT)
        st["out"] = _buffers(h, c, c["n"])
    elif kind == "batch":
        parts = _batch_particles(c, seed)
        torch.cuda.synchronize()
        h = pic.Pic.batch(2, [uniform_tree_flags(2, p[2]) for p in parts], [p[0] for p in parts], [p[1] for p in parts],
                          [-1.0 / p[0].shape[1] for p in parts], stream=st["stream"], **_kw(c, -1.0, c["sweeps"]))
        h.init_leapfrog(DT)
        h.graph_capture(DT)
        st["out"] = _buffers(h, c, h.n)
    elif kind in ("bump", "beams"):
        x, v = (_bump_particles if kind == "bump" else _beam_particles)(c, seed)
        flags = _tree(kind, d, c["n"], c["dmin"], c["dmax"], c["ppc"])
        h = pic.Pic(d, flags, x, v, **_kw(c, -1.0 / c["n"], c["sweeps"]))
        h.init_leapfrog(DT)
        st["out"] = _buffers(h, c, c["n"])
        if kind == "bump":
            st["saved"] = _buffers(h, c, c["n"], field=False)
            h.get_state(*st["saved"].values())
    elif kind == "handling":
        x, v = _handling_particles(c, seed)
        h = pic.Pic(d, uniform_tree_flags(d, c["dmin"]), x, v, **dict(_kw(c, 0.0), qm=0.0, ion=0.0))
        st["out"] = _buffers(h, c, c["n"], field=False)
    else:  # rebin: the state that comes in, in no order
        h, st["state"] = _rebin_handle(c, seed)
        st["out"] = _buffers(h, c, c["n"])
        del st["out"]["E"]
    st["h"] = h
    return st


def _rebin_state(c, seed):
    """Leaf (depth-first index), position and velocity in the handle's native form, in random order."""
    g, d, n, depth = _gen(seed), c["d"], c["n"], c["depth"]
    v = _randn(g, d, n) * 0.05
    if c["precision"] == "fp64":
        x = _rand(g, d, n)
        return _dfs((x * Q3).long() // (Q3 // 3 ** depth), depth).int(), x, v
    cell = torch.randint(0, 3 ** depth, (d, n), generator=g, device="cuda")
    o = torch.rand(d, n, generator=g, device="cuda", dtype=torch.float32)
    return _dfs(cell, depth).int(), o, v.float()


def _rebin_handle(c, seed):
    g, d, n = _gen(seed + 1), c["d"], c["n"]
    state = _rebin_state(c, seed)
    return pic.Pic(d, uniform_tree_flags(d, c["depth"]), _rand(g, d, n), _rand(g, d, n), **_kw(c, -1.0 / n)), state


# ---- one pass ------------------------------------------------------------------

def run(st):
    c, h, out = st["case"], st["h"], st["out"]
    kind = c["kind"]
    if st["stream"] is not None:
        st["stream"].wait_stream(torch.cuda.current_stream())
    if kind == "rebin":
        h.set_state(*st["state"])
    elif kind == "handling":
        for _ in range(c["steps"]):
            h.adapt(c["ppc"], c["dmin"], c["dmax"])
            h.step_particles(c["dt"], reflect=True)
    elif kind == "batch" or c.get("graph"):
        h.graph_launch(c["steps"])
    else:
        if kind == "bump":
            h.set_state(*st["saved"].values())
        step = h.step_fixed_field if kind == "beams" or c.get("mode") == "fixed" else h.step
        for _ in range(c["steps"]):
            step(DT)
    h.get_state(out["leaf"], out["pos"], out["vel"])
    if "Q" in out:
        h.deposit(out["Q"])
    if "E" in out:
        h.field(out["E"])
    if st["stream"] is not None:
        torch.cuda.current_stream().wait_stream(st["stream"])
    return out


# ---- what a pass cannot do without ---------------------------------------------

def work(case):
    c, d = case, case["d"]
    w = 8 if c["precision"] == "fp64" else 4
    if c["kind"] == "batch":  # the log-uniform mean count; 81^2 cells at the median
        n = c["n_inst"] * (c["n_max"] - c["n_min"]) / math.log(c["n_max"] / c["n_min"])
        nv = c["n_inst"] * (27 ** 2 + 81 ** 2 + 243 ** 2) / 3
    else:
        n, nv = c["n"], 3 ** (d * c.get("depth", c.get("dmin", 0)))
    state = 2 * d * w + 4                      # position, velocity, leaf
    per = 30 * (1 << d)                        # shape functions, deposit and gather per particle
    steps = c.get("steps", 1)
    if c["kind"] in ("handling", "rebin"):     # state in and out once per step
        return {"bytes": steps * 2.0 * n * state, "flops": steps * 10.0 * d * n}
    solve = c["sweeps"] if c["kind"] == "bump" or c.get("mode") == "step" else 0
    grid = nv * w * (1 + d + (2 if solve else 0))   # charges, field, potential in and out
    return {"bytes": steps * (2.0 * n * state + grid), "flops": steps * (float(per) * n + solve * 2.0 * 3 ** d * nv)}


# ---- the same in 64 bits, plainly ----------------------------------------------

def _dfs(cell, depth):
    """Depth-first leaf index of cells (d, n) of the uniform tree: base-3 digits interleaved, x fastest."""
    d, key, mul = cell.shape[0], torch.zeros_like(cell[0]), 1
    rest = cell.clone()
    for _ in range(depth):
        dg = rest[0] % 3 + 3 * (rest[1] % 3) + (9 * (rest[2] % 3) if d == 3 else 0)
        key += dg * mul
        mul *= 3 ** d
        rest //= 3
    return key


class _Plain:
    """Particles and grid of one uniform plasma in FP64: grid arrays indexed [z][y][x]."""

    def __init__(self, d, depth, x, v, q, scheme, sweeps):
        self.d, self.depth, self.M, self.q, self.scheme, self.sweeps = d, depth, 3 ** depth, q, scheme, sweeps
        self.x, self.v = x - torch.floor(x), v.clone()
        self.V = torch.zeros((self.M,) * d, dtype=torch.float64, device=x.device)
        self.key, self.leaf = self.keys(self.x)
        self.order(torch.argsort(self.key, stable=True))

    def order(self, p):
        self.x, self.v, self.key, self.leaf = self.x[:, p], self.v[:, p], self.key[p], self.leaf[p]

    def keys(self, x):
        s = Q3 // self.M
        quant = torch.floor(x * float(Q3)).long().clamp(0, Q3 - 1)
        cell = quant // s
        leaf = _dfs(cell, self.depth)
        if self.scheme == "pit":
            return leaf, leaf
        up = (2 * (quant % s) >= s).long()
        vert, a = torch.zeros_like(leaf), torch.zeros_like(leaf)
        for k in range(self.d):
            vert += ((cell[k] + up[k]) % self.M) * self.M ** k
            a += up[k] << k
        nc = 1 << self.d
        return vert * nc + (nc - 1 - a), leaf

    def corners(self):
        """(vertex, weight) per corner: cells from the leaf that holds the particle."""
        cell, rest = torch.zeros_like(self.x, dtype=torch.int64), self.leaf.clone()
        for i in range(self.depth):
            for k in range(self.d):
                cell[k] += (rest % 3 ** self.d) // 3 ** k % 3 * 3 ** i
            rest = rest // 3 ** self.d
        t = (self.x * self.M - cell).clamp(0.0, 1.0)
        for e in range(1 << self.d):
            vert, w = torch.zeros_like(self.leaf), torch.ones_like(t[0])
            for k in range(self.d):
                b = e >> k & 1
                vert += ((cell[k] + b) % self.M) * self.M ** k
                w = w * (t[k] if b else 1 - t[k])
            yield vert, w

    def deposit(self):
        S = torch.zeros(self.M ** self.d, dtype=torch.float64, device=self.x.device)
        for vert, w in self.corners():
            S.index_add_(0, vert, w)
        self.Q = self.q * S + 1.0 / self.M ** self.d
        return self.Q

    def solve(self):
        d, M = self.d, self.M
        h = 1.0 / M
        b = self.Q.view((M,) * d) - self.Q.sum() / M ** d
        # per leaf and corner pair that differ in k axes; a vertex pair shares 2^(d - k) leaves
        K = (4 / 6, -1 / 6, -2 / 6) if d == 2 else (4 / 12, 0.0, -1 / 12, -1 / 12)
        K = [K[k] * h ** (d - 2) * 2 ** (d - k) for k in range(d + 1)]
        rim = lambda a, ax: torch.roll(a, 1, ax) + torch.roll(a, -1, ax)  # noqa: E731
        for _ in range(self.sweeps):
            s = [self.V]                      # s[k]: sum over the neighbours that differ in k axes
            for ax in range(d):
                r = [rim(a, ax) for a in s]
                s = [s[0]] + [s[k] + r[k - 1] for k in range(1, len(s))] + [r[-1]]
            AV = sum(K[k] * s[k] for k in range(d + 1))
            self.V = self.V + OMEGA * (b - AV) / K[0]
        self.E = torch.stack([-(torch.roll(self.V, -1, d - 1 - a) - torch.roll(self.V, 1, d - 1 - a)).reshape(-1) / (2 * h)
                              for a in range(d)])

    def gather(self):
        E = torch.zeros_like(self.x)
        for vert, w in self.corners():
            for k in range(self.d):
                E[k] += w * self.E[k][vert]
        return E

    def start(self):
        self.deposit()
        self.solve()
        self.v = self.v + 0.5 * DT * self.gather()

    def step(self, fixed):
        if not fixed:
            self.deposit()
            self.solve()
        self.v = self.v - DT * self.gather()
        x = self.x + self.v * DT
        x = x - torch.floor(x)
        self.x = torch.where(x >= 1.0, 0.0, x)
        old = self.key
        self.key, self.leaf = self.keys(self.x)
        self.order(torch.argsort(2 * self.key + (self.key != old), stable=True))


def _answer(parts, split, charges):
    """Outputs of one or several plasmas.  The split state's storage order follows its single-precision cells: no
    64-bit value for it."""
    cat = lambda f, dim: torch.cat([f(p) for p in parts], dim)  # noqa: E731
    out = {"leaf": None, "pos": None if split else cat(lambda p: p.x, 1), "vel": None if split else cat(lambda p: p.v, 1),
           "E": cat(lambda p: p.E, 1)}
    if charges:
        out["Q"] = cat(lambda p: p.deposit(), 0)
    return out


def exact(case, seed):
    c, kind, split = case, case["kind"], case["precision"] == "fp32"
    if kind == "plasma":
        x, v = _plasma_particles(c, seed)
        parts = [_Plain(c["d"], c["depth"], x, v, -1.0 / c["n"], c["scheme"], c["sweeps"])]
    elif kind == "batch":
        parts = [_Plain(2, depth, x, v, -1.0 / x.shape[1], c["scheme"], c["sweeps"])
                 for x, v, depth in _batch_particles(c, seed)]
    elif kind == "rebin":
        return _rebin_exact(c, seed)
    elif kind == "handling":
        return None if split or c["scheme"] == "pidt" else _handling_exact(c, seed)
    else:
        return None  # adaptive grids: hanging vertices have no plain closed form
    # a captured graph was preceded by one ordinary step
    graph = kind == "batch" or c["graph"]
    steps = c["steps"] + int(graph)
    for p in parts:
        p.start()
        for _ in range(steps):
            p.step(kind == "batch" or c["mode"] == "fixed")
    return _answer(parts, split, not graph)


def _rebin_exact(c, seed):
    leaf, pos, vel = _rebin_state(c, seed)
    d, depth, n, M = c["d"], c["depth"], c["n"], 3 ** c["depth"]
    if c["precision"] == "fp64":
        x = pos
    else:
        cell, rest = torch.zeros(d, n, dtype=torch.float64, device="cuda"), leaf.long()
        for i in range(depth):
            for k in range(d):
                cell[k] += rest % 3 ** d // 3 ** k % 3 * 3 ** i
            rest = rest // 3 ** d
        x = (cell + pos.double()) / M
    p = _Plain.__new__(_Plain)
    p.d, p.depth, p.M, p.q, p.scheme = d, depth, M, -1.0 / n, c["scheme"]
    p.x, p.v, p.leaf = x, vel.double(), leaf.long()
    if c["precision"] == "fp64":
        p.key, p.leaf = p.keys(x)
    else:  # the cell and the offset say it, not their sum
        p.key = p.leaf
        if c["scheme"] == "pidt":
            nc = 1 << d
            up = (pos >= 0.5).long()
            vert = sum((cell[k].long() + up[k]) % M * M ** k for k in range(d))
            p.key = vert * nc + (nc - 1 - sum(up[k] << k for k in range(d)))
    o = torch.argsort(p.key, stable=True)
    p.order(o)
    return {"leaf": None, "pos": pos.double()[:, o], "vel": p.v, "Q": p.deposit()}


def _handling_exact(c, seed):
    """FP64, PIT: positions and velocities in the order of the re-refined trees' leaves."""
    x, v = _handling_particles(c, seed)
    d, top = c["d"], c["dmax"]
    nch = 3 ** d

    def fine(x):
        return _dfs(torch.floor(x * float(Q3)).long().clamp(0, Q3 - 1) // (Q3 // 3 ** top), top)

    def levels(key):
        """Which level's cell is the leaf, per finest cell."""
        lev = torch.full_like(torch.arange(nch ** top, device="cuda"), top)
        cells = torch.bincount(key, minlength=nch ** top)
        counts = {top: cells}
        for m in range(top - 1, c["dmin"] - 1, -1):
            counts[m] = counts[m + 1].view(-1, nch).sum(1)
        for m in range(top - 1, c["dmin"] - 1, -1):
            lev = torch.where((counts[m] <= c["ppc"]).repeat_interleave(nch ** (top - m)), m, lev)
        return lev

    def leaf_key(key, lev):
        width = nch ** (top - lev[key])
        return key // width

    def order(key, lev, moved=None):
        k = leaf_key(key, lev) * nch ** (top - lev[key])
        return torch.argsort(k if moved is None else 2 * k + moved, stable=True)

    base = torch.full((nch ** top,), c["dmin"], device="cuda", dtype=torch.int64)
    o = order(fine(x), base)
    x, v = x[:, o], v[:, o]
    lev = base
    for _ in range(c["steps"]):
        key = fine(x)
        new = levels(key)
        if not torch.equal(new, lev):
            lev = new
            o = order(key, lev)
            x, v, key = x[:, o], v[:, o], key[o]
        y = x + v * c["dt"]
        y = y - 2.0 * torch.floor(y * 0.5)
        flip = y >= 1.0
        x = torch.where(flip, (2.0 - y).clamp(max=1.0 - 2.0 ** -53), y)
        v = torch.where(flip, -v, v)
        after = fine(x)
        same = leaf_key(key, lev) * nch ** (top - lev[key]) == leaf_key(after, lev) * nch ** (top - lev[after])
        o = order(after, lev, (~(same & (lev[key] == lev[after]))).long())
        x, v = x[:, o], v[:, o]
    return {"leaf": None, "pos": x, "vel": v}
