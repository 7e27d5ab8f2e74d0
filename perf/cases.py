"""What a user of the library has it do, as measurable cases: charge deposits,
space-charge steps call by call, and whole tracked turns of one bunch, of a
sliced bunch and of a batch of bunches, through the public calls of
paper_2010_11540_gb300.sc.

A case is a dict of plain values:

  kind       "deposit"  sc.deposit of a bunch -> the charge grid
             "cell"     the step-wise calls over one lattice cell (deposit, solve,
                        kick_push per space-charge location) -> the bunch
             "turn"     sc.track_turns, one turn of the ring -> the bunch
             "batch"    sc.batch_track_turns, one turn of many bunches -> all bunches
             "moments"  sc.moments_noalloc -> the 14 beam moments
  n          macroparticles (batch: of the largest bunch)
  grid       nodes per axis
  precision  the solve's arithmetic (sc.PRECISION)
  lattice    "c1" (24 FODO cells, 48 locations) or "c2" (72 cells with
             sextupoles, 216 locations), the rings of synth.CONFIGS
  slices     longitudinal slices (1: none)
  and the options rf, tunes, lon, bezier, ordered, bunches.

Bunch, ring and beam follow synth.CONFIGS' recipes (Gaussian transversally, cut
at 4 sigma; grids over +-5 sigma), drawn on the GPU from the seed.  The
tensor-core solves' tiling is fixed (sc.set_solver_tiling), because the tiling
found by timing may differ from one process to the next and with it the order
of the float32 sums: a program that wants the same bits from run to run fixes it
too.
"""
import math

import numpy as np
import torch

from paper_2010_11540_gb300 import sc, synth

KEYS = ("x", "px", "y", "py", "sigma", "psigma")
SIG_Z = 15.0       # m, rms length of a sliced bunch, cut at 4 sigma
N_PPB = 1.0e13     # protons per sliced bunch
N_LAMBDA = 1e11 / 20.0


def _case(kind, n, grid, precision="fp64", lattice="c2", slices=1, **opts):
    c = dict(kind=kind, n=n, grid=grid, precision=precision, lattice=lattice, slices=slices, rf=False, tunes=False,
             lon=False, bezier=False, ordered=False, bunches=1)
    c.update(opts)
    return c


def listed():
    return [
        # the smallest call: the charge of a 2e4-particle bunch (a launch and its latency)
        dict(_case("deposit", 20000, 64, lattice="c1"), name="deposit-20k-64"),
        # the charge of a production-size bunch
        dict(_case("deposit", 1000000, 128), name="deposit-1M-128"),
        # the charge of a long bunch in 32 longitudinal slices
        dict(_case("deposit", 10000000, 128, slices=32), name="deposit-10M-32x128"),
        # a program that drives the loop itself, small bunch, float64: latency of each call
        dict(_case("cell", 20000, 64, lattice="c1"), name="cell-20k-64-fp64"),
        # the same at an odd count on the large grid with the tensor-core solve
        dict(_case("cell", 4000037, 256, "tf32x3"), name="cell-4M-256-tf32"),
        # a small study ring with an RF cavity, per-turn moments and per-particle tunes
        dict(_case("turn", 20000, 64, lattice="c1", rf=True, tunes=True), name="turn-20k-64-fp64"),
        # the production run: 1e6 particles, 216 locations, split-TF32 solve
        dict(_case("turn", 1000000, 128, "tf32x3"), name="turn-1M-128-tf32"),
        # the same run in float64 throughout
        dict(_case("turn", 1000000, 128), name="turn-1M-128-fp64"),
        # the high-resolution run with bf16 operands
        dict(_case("turn", 4000000, 256, "bf16x3"), name="turn-4M-256-bf16"),
        # the 2.5-D run: 1e7 particles in 32 slices
        dict(_case("turn", 10000000, 128, "tf32x3", slices=32), name="turn-10M-32x128-tf32"),
        # a short study bunch in a conducting pipe: longitudinal kick and Bezier gather
        dict(_case("turn", 300000, 129, "pipe_tf32x3", lattice="c1", slices=16, lon=True, bezier=True),
             name="turn-300k-16x129-pipe"),
        # a tune scan: 16 bunches of 1e4 .. 2e6 particles on 64^2 .. 256^2 grids in one batch
        dict(_case("batch", 2000000, 256, "tf32x3", bunches=16), name="batch-16-tf32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("deposit", "cell", "turn", "turn", "batch", "moments"))
    n = _log(rng, 2000, 6000000) | 1
    lat = rng.choice(("c1", "c2"))
    if kind == "moments":
        return _case("moments", n, 64, lattice=lat)
    if kind == "deposit":
        nz = rng.choice((1, 1, rng.randint(2, 40)))
        return _case("deposit", n, rng.choice((64, 128, 256)), slices=nz, lattice=lat, ordered=nz == 1 and rng.random() < 0.3)
    if kind == "cell":
        prec = rng.choice(("fp64", "tf32x3", "bf16x3", "pipe_fp64", "pipe_tf32x3"))
        g = rng.choice((64, 128, 256)) + (1 if prec.startswith("pipe") else 0)
        return _case("cell", n, g, prec, lattice=lat)
    if kind == "batch":
        return _case("batch", _log(rng, 30000, 1500000), 256, rng.choice(("fp64", "tf32x3")),
                     lattice=lat, bunches=rng.randint(2, 12))
    prec = rng.choice(("fp64", "tf32x3", "bf16x3", "pipe_fp64", "pipe_tf32x3"))
    pipe = prec.startswith("pipe")
    nz = rng.choice((1, 1, rng.randint(2, 24)))
    g = rng.choice((64, 128, 256) if nz == 1 else (64, 128)) + (1 if pipe else 0)
    lon = pipe and nz > 1 and rng.random() < 0.5
    bez = pipe and rng.random() < 0.5
    # float64 potentials and the longitudinal kick cost a few times the plain step
    n = min(n, 500001 if pipe and not prec.endswith("x3") and (lon or bez) else 1500001 if lon or bez else n)
    return _case("turn", n, g, prec, lattice=lat, slices=nz, rf=nz == 1 and rng.random() < 0.3,
                 tunes=nz == 1 and rng.random() < 0.3, lon=lon, bezier=bez)


# ------------------------------------------------------------------ inputs
def _bunch(case, seed, n):
    """Six CUDA float64 arrays of n: the recipe of synth.gaussian_bunch, drawn on the GPU."""
    cfg = synth.CONFIGS[case["lattice"]]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 13)

    def cut_normal(sig):  # a normal cut at 4 sigma, by inverting its distribution
        u = torch.rand(n, dtype=torch.float64, device="cuda", generator=gen) * 2.0 - 1.0
        return torch.erfinv(u * math.erf(4.0 / math.sqrt(2.0))) * (math.sqrt(2.0) * sig)

    st = {"x": cut_normal(cfg["sig_x"]), "px": cut_normal(cfg["sig_px"]),
          "y": cut_normal(cfg["sig_y"]), "py": cut_normal(cfg["sig_py"])}
    if case["slices"] > 1:  # ordered along the bunch, the layout sliced deposits ask for
        st["sigma"] = torch.sort(cut_normal(SIG_Z))[0].contiguous()
    else:
        st["sigma"] = torch.rand(n, dtype=torch.float64, device="cuda", generator=gen) * 20.0 - 10.0
    st["psigma"] = cut_normal(1e-3)
    return st


def _extent(case):
    cfg = synth.CONFIGS[case["lattice"]]
    return synth.grid_extent(cfg["sig_x"], cfg["sig_y"])


def _slices(case):
    return (case["slices"], -4.0 * SIG_Z, 4.0 * SIG_Z) if case["slices"] > 1 else None


def _ring(case, working_point=None):
    """(element table, beam) of the case's ring."""
    if working_point is not None and case["lattice"] == "c2":
        lat = synth.ring_c2(*synth.C4_WORKING_POINTS[working_point % len(synth.C4_WORKING_POINTS)])
    else:
        lat = synth.lattice(case["lattice"])
    if case["rf"]:
        rows = [tuple(r) for r in lat]
        lat = synth.table(rows[:-1] + [synth.elem(synth.RF, volt=4e6, harmonic=4.0), rows[-1]])
    z = _slices(case)
    nl = N_LAMBDA if z is None else N_PPB / ((z[2] - z[1]) / z[0])
    return lat, synth.beam(n_lambda=nl, circumference=float(lat["length"].sum()))


def _cell_steps(case):
    """The first cell of the ring as [(kick length, elements up to the next location)]."""
    lat, b = _ring(case)
    marks = [k for k in range(len(lat)) if lat[k]["type"] == synth.MARK]
    per = {"c1": 2, "c2": 3}[case["lattice"]]
    s = np.concatenate([[0.0], np.cumsum(lat["length"])])
    steps = []
    for k in range(per):  # the locations of the second cell: each has one before it
        m, e, p = marks[per + k], marks[per + k + 1], marks[per + k - 1]
        steps.append((float(s[m] - s[p]), lat[m + 1:e].copy()))
    return steps, b


def _bunch_counts(case):
    """Counts of a batch: equal steps of the logarithm from 1e4 up to n."""
    k = case["bunches"]
    return [int(round(1e4 * (case["n"] / 1e4) ** (i / max(1, k - 1)))) for i in range(k)]


def _tiling(precision, grid, stacked):
    """The variants timing finds for such grids, as a program would keep them."""
    if precision == "pipe_tf32x3":
        return [0, 0, 0, 0] if stacked == 1 else [0, 2, 1, 3]
    if stacked > 1:
        return [0, 1, 3, 2] if stacked * grid <= 1536 else [2, 1, 4, 3]
    return {64: [0, 0, 0, 0], 128: [3, 0, 0, 0], 256: [3, 2, 1, 0]}[grid]


def _grid(case):
    n = case["grid"]
    g = sc.create_grid(n, n, *_extent(case), precision=case["precision"], slices=_slices(case))
    if case["precision"] in ("tf32x3", "bf16x3", "pipe_tf32x3"):
        sc.set_solver_tiling(g, _tiling(case["precision"], n, case["slices"]))
    if case["lon"]:
        sc.set_longitudinal_kick(g)
    if case["bezier"]:
        sc.set_gather(g, "bezier")
    return g


def _twiss():
    return (20.0, 0.0, 15.0, 0.0)


# ------------------------------------------------------------------ one pass
def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "batch":
        counts = _bunch_counts(case)
        s["states"] = [_bunch(case, seed * 1000 + i, n) for i, n in enumerate(counts)]
        rings = [_ring(case, i) for i in range(len(counts))]
        s["lats"], s["beams"] = [r[0] for r in rings], [r[1] for r in rings]
        s["batch"] = sc.create_batch([(synth.c4_grid_size(n),) * 2 + _extent(case) for n in counts], case["precision"])
        if case["precision"] == "tf32x3":
            sc.batch_set_solver_tiling(s["batch"], _tiling("tf32x3", 256, len(counts)))
        return s
    s["bunch"] = _bunch(case, seed, case["n"])
    if case["kind"] == "moments":
        s["out"] = torch.zeros(14, dtype=torch.float64, device="cuda")
        return s
    s["grid"] = _grid(case)
    if case["kind"] == "deposit":
        s["charge"] = sc.charge_tensor(s["grid"])
        s["charge"].owner = s["grid"]  # a view of the grid's memory: the grid lives as long as it does
        if case["ordered"]:
            sc.sort_particles(s["grid"], s["bunch"])
    elif case["kind"] == "cell":
        s["steps"], s["beam"] = _cell_steps(case)
    else:
        s["lat"], s["beam"] = _ring(case)
        if case["tunes"]:
            s["acc"] = torch.zeros(4 * case["n"], dtype=torch.float64, device="cuda")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "deposit":
        sc.deposit(s["grid"], s["bunch"])
        return s["charge"]
    if kind == "moments":
        return sc.moments_noalloc(s["bunch"], s["out"])
    if kind == "cell":
        g = s["grid"]
        for length, elems in s["steps"]:
            sc.deposit(g, s["bunch"])
            sc.solve(g)
            sc.kick_push(g, s["bunch"], s["beam"], length, elems)
        return dict(s["bunch"])
    if kind == "batch":
        sc.batch_track_turns(s["batch"], s["states"], s["beams"], s["lats"], 1)
        # each coordinate of all bunches, one after another
        return {k: torch.cat([st[k] for st in s["states"]]) for k in KEYS}
    if case["tunes"]:  # moments and phase advances with the turn
        sc.tune_setup(s["grid"], s["bunch"], _twiss(), s["acc"])
        mom = sc.track_turns(s["grid"], s["bunch"], s["beam"], s["lat"], 1, diag=True)
        return {**s["bunch"], "advance": s["acc"][2 * case["n"]:], "moments": mom}
    sc.track_turns(s["grid"], s["bunch"], s["beam"], s["lat"], 1)
    return dict(s["bunch"])


# ------------------------------------------------------------------ work
# float64 operations of one particle: deposit, gather and kick, and each element
_FLOPS = {synth.DRIFT: 19, synth.QUAD: 40, synth.SEXT: 9, synth.RF: 20, synth.MARK: 0}


def _step_work(case, n, nodes, elems):
    """One space-charge location: every location needs the charge of the whole bunch before
    its solve, so each passes over the particles once: six coordinates read and the five
    that change written (88 bytes), the fields of every node read once, the charge written."""
    doubled = 4 * nodes
    solve = 2 * 5 * doubled * math.log2(max(2, doubled // case["slices"]))
    f32 = case["precision"].endswith("x3")
    field = (3 if case["lon"] or case["bezier"] else 2) * (4 if f32 else 8)
    flops = n * (18 + 16 + sum(_FLOPS[int(e["type"])] for e in elems)) + solve
    return 88 * n + nodes * (field + 8), flops


def _ring_work(case, n, grid):
    lat, _ = _ring(case)
    nodes = grid * grid * case["slices"]
    kicks = int((lat["type"] == synth.MARK).sum())
    one, _ = _step_work(case, n, nodes, [])
    _, fl = _step_work(case, n, nodes, [])
    return kicks * one, kicks * fl + n * sum(_FLOPS[int(t)] for t in lat["type"])


def work(case):
    n, grid = case["n"], case["grid"]
    nodes = grid * grid * case["slices"]
    if case["kind"] == "moments":
        return {"bytes": 48 * n + 112, "flops": 28 * n}
    if case["kind"] == "deposit":  # two coordinates (three when sliced) read, the charge written
        return {"bytes": (24 if case["slices"] > 1 else 16) * n + 8 * nodes, "flops": 18 * n}
    if case["kind"] == "cell":
        steps, _ = _cell_steps(case)
        w = [_step_work(case, n, nodes, e) for _, e in steps]
        return {"bytes": sum(v[0] for v in w), "flops": sum(v[1] for v in w)}
    if case["kind"] == "batch":
        w = [_ring_work(case, c, synth.c4_grid_size(c)) for c in _bunch_counts(case)]
        return {"bytes": sum(v[0] for v in w), "flops": sum(v[1] for v in w)}
    b, f = _ring_work(case, n, grid)
    if case["tunes"]:
        b, f = b + n * 96, f + n * 100
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ the same in plain torch, 64 bits
class _Exact:
    """The space-charge step in float64 torch operations: charge by cloud-in-cell with
    2^-20 weights, potential by Hockney's doubled grid (or the pipe's sine series), centred
    differences, bilinear or Bezier gather, and the ring's maps in closed form."""

    def __init__(self, grid, extent, precision, slices=None, lon=False, bezier=False):
        self.n = grid
        self.x0, x1, self.y0, y1 = extent
        self.hx, self.hy = (x1 - self.x0) / (grid - 1), (y1 - self.y0) / (grid - 1)
        self.slices, self.lon, self.bezier = slices, lon, bezier
        self.nz = slices[0] if slices else 1
        self.pipe = precision.startswith("pipe")
        self.fixed = precision.endswith("x3")  # gathers with the charge's 2^-20 weights
        f = dict(dtype=torch.float64, device="cuda")
        if self.pipe:
            m = grid - 2
            k = torch.arange(1, m + 1, **f)
            self.S = torch.sin(math.pi / (m + 1) * torch.outer(k, k))
            ex = torch.sin(math.pi * k / (2 * (m + 1))) ** 2
            self.lam = -4.0 * (ex[None, :] / self.hx ** 2 + ex[:, None] / self.hy ** 2)
        else:
            M = 2 * grid
            d = torch.arange(M, **f)
            d = torch.where(d <= grid, d, d - M)
            r2 = (d[None, :] * self.hx) ** 2 + (d[:, None] * self.hy) ** 2
            r2[0, 0] = 1.0
            G = -0.5 * torch.log(r2)
            a, b = 0.5 * self.hx, 0.5 * self.hy
            G[0, 0] = -(a * b * (math.log(a * a + b * b) - 3.0) + a * a * math.atan(b / a)
                        + b * b * math.atan(a / b)) / (2.0 * a * b)
            self.GF = torch.fft.rfft2(G)

    def locate(self, st):
        xi, et = (st["x"] - self.x0) * (1.0 / self.hx), (st["y"] - self.y0) * (1.0 / self.hy)
        n = self.n
        ok = (xi >= 0) & (xi < n - 1) & (et >= 0) & (et < n - 1)
        k = torch.zeros_like(xi)
        if self.slices:
            nz, z0, z1 = self.slices
            z = (st["sigma"] - z0) * (1.0 / ((z1 - z0) / nz))
            ok &= (z >= 0) & (z < nz)
            k = torch.floor(z)
        zero = torch.zeros_like(xi)
        xi, et, k = torch.where(ok, xi, zero), torch.where(ok, et, zero), torch.where(ok, k, zero)
        i, j = torch.floor(xi), torch.floor(et)
        return ok, i.long(), j.long(), k.long(), xi - i, et - j

    def charge(self, at):
        ok, i, j, k, fx, fy = at
        one = 1 << 20
        ax, ay = torch.round(fx * one).long(), torch.round(fy * one).long()
        Q = torch.zeros(self.nz * self.n * self.n, dtype=torch.int64, device="cuda")
        c = (k * self.n + j) * self.n + i
        w = ok.long()
        for di, wx in ((0, one - ax), (1, ax)):
            for dj, wy in ((0, one - ay), (1, ay)):
                Q.index_add_(0, c + dj * self.n + di, wx * wy * w)
        return Q.view(self.nz, self.n, self.n)

    def potential(self, Q, count):
        """phi with the ring of nodes outside the grid: [nz, n + 2, n + 2]."""
        q = Q.double() * (2.0 ** -40 / count)
        n = self.n
        if self.pipe:
            m = n - 2
            F = q[:, 1:-1, 1:-1] * (-2.0 * math.pi / (self.hx * self.hy))
            u = self.S @ ((self.S @ F @ self.S) / self.lam) @ self.S * (2.0 / (m + 1)) ** 2
            phi = torch.zeros(self.nz, n + 2, n + 2, dtype=torch.float64, device="cuda")
            phi[:, 2:-2, 2:-2] = u
            phi[:, 0, :], phi[:, -1, :] = -phi[:, 2, :], -phi[:, -3, :]
            phi[:, :, 0], phi[:, :, -1] = -phi[:, :, 2], -phi[:, :, -3]
            return phi
        pad = torch.zeros(self.nz, 2 * n, 2 * n, dtype=torch.float64, device="cuda")
        pad[:, :n, :n] = q
        phi = torch.fft.irfft2(torch.fft.rfft2(pad) * self.GF, s=(2 * n, 2 * n))
        return torch.roll(phi, (1, 1), (1, 2))[:, :n + 2, :n + 2].contiguous()

    def kick(self, st, at, phi, kl, klz):
        ok, i, j, k, fx, fy = at
        if self.fixed:
            fx, fy = torch.round(fx * 2.0 ** 20) * 2.0 ** -20, torch.round(fy * 2.0 ** 20) * 2.0 ** -20
        W = self.n + 2
        base = (k * W + j + 1) * W + i + 1
        flat = phi.reshape(-1)
        if self.bezier:
            def weights(f):
                t = (1.0 + f) / 3.0
                u = 1.0 - t
                return ((u ** 3, 3 * t * u * u, 3 * t * t * u, t ** 3),
                        (-3 * u * u, 3 * u * u - 6 * t * u, 6 * t * u - 3 * t * t, 3 * t * t))
            (bx, dx), (by, dy) = weights(fx), weights(fy)

            def surface(shift, wx, wy):
                r = torch.zeros_like(fx)
                for b in range(4):
                    for a in range(4):
                        r = r + flat[(base + shift + (b - 1) * W + a - 1).clamp(0, flat.numel() - 1)] * wx[a] * wy[b]
                return r
            gx, gy = -surface(0, dx, by) / (3 * self.hx), -surface(0, bx, dy) / (3 * self.hy)
            value = lambda shift: surface(shift, bx, by)  # noqa: E731
        else:
            ex = -(phi[:, 1:-1, 2:] - phi[:, 1:-1, :-2]) / (2 * self.hx)
            ey = -(phi[:, 2:, 1:-1] - phi[:, :-2, 1:-1]) / (2 * self.hy)
            c = (k * self.n + j) * self.n + i

            def bil(v, at0, w):
                v = v.reshape(-1)
                g = lambda o: v[(at0 + o).clamp(0, v.numel() - 1)]  # noqa: E731
                lo, hi = g(0) + fx * (g(1) - g(0)), g(w) + fx * (g(w + 1) - g(w))
                return lo + fy * (hi - lo)
            gx, gy = bil(ex, c, self.n), bil(ey, c, self.n)
            value = lambda shift: bil(phi, base + shift, W)  # noqa: E731
        w = ok.double()
        st["px"] = st["px"] + kl * gx * w
        st["py"] = st["py"] + kl * gy * w
        if self.lon:
            up = value(W * W) * (k + 1 < self.nz)
            dn = value(-W * W) * (k > 0)
            st["psigma"] = st["psigma"] - klz * (up - dn) * w

    def step(self, st, b, length, elems):
        kk = 2.0 * b["r_p"] * b["n_lambda"] / (b["beta0"] ** 2 * b["gamma0"] ** 3)
        at = self.locate(st)
        phi = self.potential(self.charge(at), st["x"].numel())
        klz = 0.0
        if self.lon:
            nz, z0, z1 = self.slices
            klz = kk * length * b["gamma0"] / (2.0 * (z1 - z0) / nz)
        self.kick(st, at, phi, kk * length, klz)
        push(st, b, elems)


def push(st, b, elems):
    """Drift, thick quadrupole, thin sextupole and RF cavity in closed form."""
    b2, ig2 = b["beta0"] ** 2, 1.0 / b["gamma0"] ** 2
    for e in elems:
        x, px, y, py, sg, ps = (st[k] for k in KEYS)
        L, t = float(e["length"]), int(e["type"])
        if t == synth.DRIFT:
            pz = torch.sqrt(1.0 + 2.0 * ps + b2 * ps * ps - px * px - py * py)
            st["x"], st["y"] = x + L * px / pz, y + L * py / pz
            st["sigma"] = sg + L * (1.0 - (1.0 + b2 * ps) / pz)
        elif t == synth.QUAD:
            k1, c = float(e["k1"]), 1.0 - ps
            w = torch.sqrt(abs(k1) * c)
            a = torch.sqrt(c / abs(k1))
            C, S, ch, sh = torch.cos(w * L), torch.sin(w * L), torch.cosh(w * L), torch.sinh(w * L)
            foc = lambda u, p: (C * u + a * S * p, C * p - S / a * u)  # noqa: E731
            dfc = lambda u, p: (ch * u + a * sh * p, ch * p + sh / a * u)  # noqa: E731
            (x1, px1), (y1, py1) = (foc(x, px), dfc(y, py)) if k1 > 0 else (dfc(x, px), foc(y, py))
            S2 = c * (px * px + py * py) + k1 * (x * x - y * y)
            D = (x1 * px1 - x * px) + (y1 * py1 - y * py)
            st["sigma"] = sg + ps * (L * ig2) - (L * S2 + D) / (4.0 * c)
            st["x"], st["px"], st["y"], st["py"] = x1, px1, y1, py1
        elif t == synth.SEXT:
            k = float(e["k2l"])
            st["px"], st["py"] = px - 0.5 * k * (x * x - y * y), py + k * x * y
        elif t == synth.RF:
            v = float(e["volt"]) / (b2 * b["gamma0"] * b["mass_ev"])
            st["psigma"] = ps + v * torch.sin(float(e["lag"]) - 2.0 * math.pi * float(e["harmonic"]) / b["circumference"] * sg)


def _exact_turn(X, st, lat, b):
    marks = [k for k in range(len(lat)) if lat[k]["type"] == synth.MARK]
    s = np.concatenate([[0.0], np.cumsum(lat["length"])])
    push(st, b, lat[:marks[0]])
    for q, m in enumerate(marks):
        prev = s[marks[q - 1]] if q else s[marks[-1]] - s[-1]
        X.step(st, b, float(s[m] - prev), lat[m + 1:marks[q + 1] if q + 1 < len(marks) else len(lat)])


def _moments(st):
    m = [st[k].mean() for k in KEYS]
    d = [st[k] - v for k, v in zip(KEYS, m)]
    pairs = ((0, 0), (0, 1), (1, 1), (2, 2), (2, 3), (3, 3), (4, 4), (5, 5))
    return torch.stack(m + [(d[a] * d[c]).mean() for a, c in pairs])


def _phases(st):
    bx, ax, by, ay = _twiss()
    return (torch.atan2(-(ax * st["x"] + bx * st["px"]), st["x"]), torch.atan2(-(ay * st["y"] + by * st["py"]), st["y"]))


def exact(case, seed):
    if case["kind"] == "deposit":
        return None  # whole numbers
    if case["kind"] == "batch":
        counts = _bunch_counts(case)
        if sum(counts) * (216 if case["lattice"] == "c2" else 48) > 3e9:
            return None
        sts = [_bunch(case, seed * 1000 + i, n) for i, n in enumerate(counts)]
        for i, (n, st) in enumerate(zip(counts, sts)):
            _exact_turn(_Exact(synth.c4_grid_size(n), _extent(case), case["precision"]), st, *_ring(case, i))
        return {k: torch.cat([st[k] for st in sts]) for k in KEYS}
    st = _bunch(case, seed, case["n"])
    if case["kind"] == "moments":
        return _moments(st)
    X = _Exact(case["grid"], _extent(case), case["precision"], _slices(case), case["lon"], case["bezier"])
    if case["kind"] == "cell":
        steps, b = _cell_steps(case)
        for length, elems in steps:
            X.step(st, b, length, elems)
        return dict(st)
    lat, b = _ring(case)
    if not case["tunes"]:
        _exact_turn(X, st, lat, b)
        return dict(st)
    mom, p0 = _moments(st), _phases(st)
    _exact_turn(X, st, lat, b)
    adv = torch.cat([torch.remainder(q - p, 2.0 * math.pi) for p, q in zip(p0, _phases(st))])
    return {**st, "advance": adv, "moments": mom[None, :]}
