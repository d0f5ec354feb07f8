"""Performance cases of the ideal-MHD block update, measured through the public
binding (``paper_2303_03026_gb300.amrvac.State``).

A "step" case advances a prepared state by ``steps`` full time steps and reads
the conserved state back into a device tensor; the state keeps evolving from
pass to pass, as in a simulation loop.  A "regrid" case evaluates the
refinement criterion of a state, plans the new block list on the device and
fills a state that already stands on that list.

``exact`` advances the same inputs in plain torch, in 64 bits, with the formulas
of the method (limited reconstruction of primitives, glm interface solve, HLL /
HLLD, strong-stability-preserving Runge-Kutta, CFL step, AMR ghost operators,
flux correction at level changes).
"""
import math
import random

import torch

from paper_2303_03026_gb300 import amrvac
from paper_2303_03026_gb300 import workloads as wl

NV = 9
DEV = "cuda:0"
GAMMA = 5.0 / 3.0


# ------------------------------------------------------------------ the cases

def _case(name, problem, ndim, size, precision, flux, limiter, time, steps=1, block=16,
          pressure="ff", reflux=False):
    return {"name": name, "problem": problem, "ndim": ndim, "size": size, "block": block,
            "precision": precision, "flux": flux, "limiter": limiter, "time": time,
            "pressure": pressure, "reflux": reflux, "steps": steps}


def listed():
    return [
        # the smallest call: a 1D shock tube of 512 cells in one block (a method
        # or teaching test), two stages a step, four steps between two reads
        _case("riemann_1d_512", "riemann", 1, 512, "fp64", "hll", "vanleer", "ssprk2", steps=4,
              block=512),
        # a convergence test on a small square: 16 blocks, one step a call
        _case("alfven_2d_64", "alfven", 2, 64, "fp64", "hlld", "koren", "ssprk3"),
        # the 1024^2 Orszag-Tang vortex at its usual 64-bit precision
        _case("orszag_tang_2d_1024", "vortex", 2, 1024, "fp64", "hlld", "koren", "ssprk3"),
        # a 2D adaptive mesh of blocks that are not 16 wide (12^2 cells), open
        # boundaries: the general per-block kernels
        _case("amr_2d_b12", "blob", 2, 24, "fp64", "hlld", "vanleer", "ssprk3", block=12),
        # 256 independent squares of 64^2 .. 512^2 cells advanced together, each
        # with its own time step (a parameter study)
        _case("instances_2d_256", "instances", 2, 256, "fp32", "hlld", "vanleer", "ssprk3"),
        # a small 3D box: 5^3 blocks, fewer than the chip has processors
        _case("turbulence_3d_80", "turbulence", 3, 80, "fp32", "hlld", "vanleer", "ssprk3",
              pressure="fp64"),
        # 256^3 turbulence at low plasma beta, the uniform-mesh production run
        _case("turbulence_3d_256", "turbulence", 3, 256, "fp32", "hlld", "vanleer", "ssprk3"),
        # the block-adaptive 3D blast of the benchmark: 18,304 blocks, 75 M cells
        _case("blast_3d_amr_6", "blast", 3, 6, "fp32", "hlld", "vanleer", "ssprk3"),
        # the same problem on a coarser base mesh in 64 bits throughout
        _case("blast_3d_amr_2_fp64", "blast", 3, 2, "fp64", "hlld", "vanleer", "ssprk3"),
        # with a fifth-order limiter (three ghost layers)
        _case("blast_3d_amr_3_mp5", "blast", 3, 3, "fp32", "hlld", "mp5", "ssprk3"),
        # conservative to round-off: flux correction at the level changes, the
        # binding's default pressure recovery and a four-stage scheme
        _case("blast_3d_amr_3_reflux", "blast", 3, 3, "fp32", "hll", "woodward", "ssprk43",
              pressure="fp64", reflux=True),
        # one regrid of an evolved blast on density and pressure
        _case("regrid_3d_4", "regrid", 3, 4, "fp32", "hlld", "vanleer", "ssprk3"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["riemann", "alfven", "vortex", "blob", "instances", "turbulence", "blast",
                       "regrid"])
    two = rng.choice(["vanleer", "koren", "minmod", "woodward"])
    five = rng.choice(["mp5", "weno5"])
    pressure = rng.choice(["ff", "fp64"])
    precision = rng.choice(["fp32", "fp64"])
    flux = rng.choice(["hlld", "hll"])
    if kind == "riemann":
        n = _log_int(rng, 100, 4000)
        return _nameless("riemann", 1, n, "fp64", "hll", two, "ssprk2", steps=rng.randint(1, 6),
                         block=n)
    if kind in ("alfven", "vortex"):
        n = 16 * _log_int(rng, 3, 72)
        lim = rng.choice([two, two, five])
        return _nameless(kind, 2, n, precision, flux, lim, rng.choice(["ssprk3", "ssprk2"]),
                         steps=rng.randint(1, 2), pressure=pressure)
    if kind == "blob":
        block = rng.choice([8, 10, 12, 14, 20, 24])
        return _nameless("blob", 2, rng.randint(6, 28), precision, flux, two, "ssprk3",
                         block=block, pressure=pressure)
    if kind == "instances":
        return _nameless("instances", 2, _log_int(rng, 5, 280), "fp32", flux, two, "ssprk3",
                         pressure=pressure)
    if kind == "turbulence":
        small = precision == "fp64"
        n = 16 * rng.randint(3, 8 if small else 16)
        return _nameless("turbulence", 3, n, precision, flux, two, "ssprk3", pressure=pressure)
    if kind == "blast":
        lim = rng.choice([two, two, five]) if precision == "fp32" else two
        base = 2 if precision == "fp64" else rng.randint(2, 5)
        return _nameless("blast", 3, base, precision, flux, lim,
                         rng.choice(["ssprk3", "ssprk43"]), pressure=pressure,
                         reflux=rng.random() < 0.3)
    return _nameless("regrid", 3, rng.randint(2, 5), "fp32", "hlld", "vanleer", "ssprk3",
                     pressure=pressure)


def _nameless(*a, **k):
    c = _case("", *a, **k)
    del c["name"]
    return c


# ------------------------------------------------------------------ mesh, plan

def _shell_mesh(base, levels=4):
    """Blocks refined where they meet the shell 0.2 <= r <= 0.3, graded 2:1."""
    def refine(level, i, j, k):
        h = 1.0 / (base << level)
        lo, hi = (i * h, j * h, k * h), ((i + 1) * h, (j + 1) * h, (k + 1) * h)
        near = far = 0.0
        for a, b in zip(lo, hi):
            a, b = a - 0.5, b - 0.5
            near += a * a if a > 0 else b * b if b < 0 else 0.0
            far += max(a * a, b * b)
        return near <= 0.3 * 0.3 and far >= 0.2 * 0.2
    return wl.amr_meta(3, (base,) * 3, levels - 1, refine)


def _blob_mesh(base):
    """2D, three levels, refined around a point off the centre, open boundaries."""
    def refine(level, i, j, k):
        h = 1.0 / (base << level)
        r = math.hypot((i + 0.5) * h - 0.43, (j + 0.5) * h - 0.56)
        return level < 2 and r < (0.3, 0.17)[level]
    return wl.amr_meta(2, (base, base, 1), 2, refine, periodic=False)


def _plan(case):
    """Scheme, instances and block list of a case."""
    p, nd, n, b = case["problem"], case["ndim"], case["size"], case["block"]
    open_bc = p in ("riemann", "blob")
    cfg = wl.Config(ndim=nd, block_nx=tuple(b if d < nd else 1 for d in range(3)),
                    flux=case["flux"], limiter=case["limiter"], time=case["time"],
                    precision=case["precision"], glm=nd > 1, reflux=case["reflux"],
                    bc=((("outflow", "outflow") if open_bc else ("periodic", "periodic")),) * 3)
    if p == "instances":
        r = random.Random(n)
        insts, metas = [], []
        for q in range(n):
            m = max(4, round(math.exp(r.uniform(math.log(64), math.log(512))) / b))
            insts.append(wl.Instance(base_blocks=(m, m, 1), gamma=r.choice([GAMMA, 1.4])))
            metas.append(torch.from_numpy(wl.uniform_meta((m, m, 1), q)))
        return cfg, insts, torch.cat(metas).numpy()
    if p in ("blast", "regrid"):
        meta, base = _shell_mesh(n), (n, n, n)
    elif p == "blob":
        meta, base = _blob_mesh(n), (n, n, 1)
    else:
        base = tuple(n // b if d < nd else 1 for d in range(3))
        meta = wl.uniform_meta(base)
    return cfg, [wl.Instance(base_blocks=base, gamma=GAMMA)], meta


# ------------------------------------------------------------------ inputs

def _coords(cfg, insts, meta):
    """Cell centres x, y, z, each [nblocks, ncell] (the axes of a dimension that
    is not there are 0), float64 on the GPU."""
    m = torch.as_tensor(meta, dtype=torch.int64, device=DEV)
    nx = cfg.block_nx
    c = torch.arange(nx[0] * nx[1] * nx[2], device=DEV)
    loc = (c % nx[0], (c // nx[0]) % nx[1], c // (nx[0] * nx[1]))
    out = []
    for d in range(3):
        if d >= cfg.ndim:
            out.append(torch.zeros(m.shape[0], c.numel(), dtype=torch.float64, device=DEV))
            continue
        nb = torch.tensor([i.base_blocks[d] for i in insts], device=DEV)[m[:, 0]] << m[:, 1]
        idx = m[:, 2 + d:3 + d] * nx[d] + loc[d][None]
        out.append((idx + 0.5) / (nb * nx[d])[:, None].double())
    return out


def _conserved(g, rho, v, p, B, psi=None):
    e = p / (g - 1.0) + 0.5 * rho * (v[0] ** 2 + v[1] ** 2 + v[2] ** 2) \
        + 0.5 * (B[0] ** 2 + B[1] ** 2 + B[2] ** 2)
    return torch.stack([rho, rho * v[0], rho * v[1], rho * v[2], e, B[0], B[1], B[2],
                        torch.zeros_like(rho) if psi is None else psi])


def _modes(r, count, x, y, z, kmax=3):
    """A smooth periodic field |f| <= 1: ``count`` random Fourier modes."""
    f = torch.zeros_like(x)
    for _ in range(count):
        k = [r.randint(-kmax, kmax) for _ in range(3)]
        f += r.uniform(-1, 1) * torch.sin(2 * math.pi * (k[0] * x + k[1] * y + k[2] * z)
                                          + r.uniform(0, 2 * math.pi))
    return f / count


def _solenoidal(n, seed):
    """Random-phase divergence-free velocity on an n^3 grid, |v_k| ~ k^-2 on
    shells 1 .. 16, rms 1; [3, z, y, x]."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    k1 = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device=DEV)
    kz, ky, kx = torch.meshgrid(k1, k1, k1[: n // 2 + 1], indexing="ij")
    k2 = kx * kx + ky * ky + kz * kz
    kk = k2.sqrt()
    amp = torch.where((kk >= 0.5) & (kk < min(16, n // 4) + 0.5), 1.0 / k2.clamp(min=1.0), 0.0)
    vh = []
    for _ in range(3):
        ph = 2 * math.pi * torch.rand(kk.shape, dtype=torch.float64, device=DEV, generator=gen)
        a = amp * torch.randn(kk.shape, dtype=torch.float64, device=DEV, generator=gen)
        vh.append(torch.polar(a.abs(), ph))
    dot = (kx * vh[0] + ky * vh[1] + kz * vh[2]) / k2.clamp(min=1.0)
    v = torch.stack([torch.fft.irfftn(vh[c] - k * dot, s=(n, n, n))
                     for c, k in enumerate((kx, ky, kz))])
    return v / (v * v).sum(0).mean().sqrt()


def _inputs(case, seed, cfg, insts, meta):
    """Initial conserved state [9, nblocks, ncell] in the state's precision."""
    r = random.Random(seed)
    p = case["problem"]
    x, y, z = _coords(cfg, insts, meta)
    zero, one = torch.zeros_like(x), torch.ones_like(x)
    tp = 2.0 * math.pi
    if p == "riemann":  # random states on both sides of x = 1/2
        left = x < 0.5
        side = lambda lo, hi: torch.where(left, r.uniform(lo, hi), r.uniform(lo, hi))  # noqa: E731
        rho, pr, by = side(0.1, 1.0), side(0.1, 1.0), side(-1.0, 1.0)
        U = _conserved(GAMMA, rho, (zero, zero, zero), pr, (0.75 * one, by, zero))
    elif p == "alfven":  # circularly polarised wave along (1, 1), random phase
        s2, amp = 1.0 / math.sqrt(2.0), r.uniform(0.08, 0.12)
        ph = tp * (x + y) + r.uniform(0, tp)
        sn, cs = amp * torch.sin(ph), amp * torch.cos(ph)
        U = _conserved(GAMMA, one, (-s2 * sn, s2 * sn, cs), 0.1 * one,
                       (s2 - s2 * sn, s2 + s2 * sn, cs))
    elif p == "vortex":  # Orszag-Tang with random offsets
        b0 = 1.0 / math.sqrt(4.0 * math.pi)
        a, b = r.uniform(0, 1), r.uniform(0, 1)
        xs, ys = x + a, y + b
        U = _conserved(GAMMA, 25.0 / (36.0 * math.pi) * one,
                       (-torch.sin(tp * ys), torch.sin(tp * xs), zero),
                       5.0 / (12.0 * math.pi) * one,
                       (-b0 * torch.sin(tp * ys), b0 * torch.sin(2 * tp * xs), zero))
    elif p == "blob":  # dense hot spot in a sheared, magnetised flow
        d2 = (x - 0.43) ** 2 + (y - 0.56) ** 2
        w = r.uniform(0.06, 0.1)
        rho = 1.0 + 2.0 * torch.exp(-d2 / w ** 2) + 0.1 * _modes(r, 3, x, y, zero)
        pr = 0.7 + 3.0 * torch.exp(-d2 / (0.7 * w) ** 2)
        U = _conserved(GAMMA, rho, (0.3 * torch.sin(tp * y), 0.2 * _modes(r, 3, x, y, zero),
                                    0.05 * one), pr,
                       (0.4 + 0.1 * torch.sin(tp * y), 0.3 + 0.1 * torch.sin(tp * x), 0.2 * one),
                       0.01 * torch.sin(tp * x))
    elif p == "instances":  # at most four modes a field, another problem each
        gen = torch.Generator().manual_seed(seed)
        q = torch.as_tensor(meta[:, 0], dtype=torch.int64, device=DEV)
        ni = len(insts)
        ks = torch.randint(-3, 4, (6, 4, ni, 2), generator=gen).double().to(DEV)
        am = torch.empty(6, 4, ni, dtype=torch.float64).uniform_(-1, 1, generator=gen).to(DEV) / 4
        ph = torch.empty(6, 4, ni, dtype=torch.float64).uniform_(0, tp, generator=gen).to(DEV)
        bz = torch.empty(ni, dtype=torch.float64).uniform_(-0.5, 0.5, generator=gen).to(DEV)
        g = torch.tensor([i.gamma for i in insts], dtype=torch.float64, device=DEV)[q][:, None]

        def arg(f, m):
            k = ks[f, m][q]
            return tp * (k[:, :1] * x + k[:, 1:] * y) + ph[f, m][q][:, None], k
        fld = [sum(am[f, m][q][:, None] * torch.sin(arg(f, m)[0]) for m in range(4))
               for f in range(5)]
        bx, by = zero.clone(), zero.clone()
        for m in range(4):
            t, k = arg(5, m)
            c = 0.05 * tp * am[5, m][q][:, None] * torch.cos(t)
            bx += c * k[:, 1:]
            by -= c * k[:, :1]
        vm = 0.5 / math.sqrt(3.0)
        U = _conserved(g, 1.0 + 0.5 * fld[0], [vm * f for f in fld[2:5]], 1.0 + 0.5 * fld[1],
                       (bx, by, bz[q][:, None] + zero))
    elif p == "turbulence":  # Mach 1, beta 0.01
        n, b = case["size"], case["block"]
        v = _solenoidal(n, seed).reshape(3, n // b, b, n // b, b, n // b, b)
        v = v.permute(0, 1, 3, 5, 2, 4, 6).reshape(3, -1, b ** 3)
        U = _conserved(GAMMA, one, v, one / GAMMA,
                       (zero, zero, math.sqrt(2.0 / GAMMA / 0.01) * one))
    else:  # an over-pressured ball in a magnetised medium
        c = [0.5 + (r.uniform(-0.01, 0.01) if p == "blast" else 0.0) for _ in range(3)]
        rr = ((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2).sqrt()
        a = r.uniform(0, tp)
        B = (math.cos(a) * one, math.sin(a) * one, zero)
        if p == "blast":  # at its start, the medium slightly uneven
            rho = 1.0 + 0.05 * _modes(r, 2, x, y, z)
            v = [0.05 * _modes(r, 1, x, y, z) for _ in range(3)]
            U = _conserved(GAMMA, rho, v, torch.where(rr < 0.1, r.uniform(60.0, 100.0), 1.0), B)
        else:  # evolved: a swept-up shell around a hot cavity, quiet outside, in
            # random units of density and pressure (the criterion is free of units,
            # so the planned mesh stays the same)
            ur, up = r.uniform(0.5, 2.0), r.uniform(0.5, 2.0)
            s = (rr / 0.24).clamp(max=1.0)
            inside = rr < 0.24
            rho = ur * torch.where(inside, 0.05 + 3.0 * s ** 9, 1.0)
            v = [math.sqrt(up / ur) * torch.where(inside, 2.0 * s * (t - t0), 0.0)
                 for t, t0 in zip((x, y, z), c)]
            U = _conserved(GAMMA, rho, v, up * torch.where(inside, 4.0 + 4.0 * s ** 8, 1.0),
                           [math.sqrt(up) * b for b in B])
    return U.to(torch.float64 if case["precision"] == "fp64" else torch.float32).contiguous()


REFINE, RATIO, DEEPEST = 0.05, 0.2, 3
WEIGHTS = [0.5, 0, 0, 0, 0.5, 0, 0, 0, 0]  # density and pressure


def prepare(case, seed):
    cfg, insts, meta = _plan(case)
    S = amrvac.State(cfg, insts, meta, device=DEV, pressure=case["pressure"])
    S.set_conserved(_inputs(case, seed, cfg, insts, meta))
    if case["problem"] != "regrid":
        return {"S": S, "steps": case["steps"],
                "out": torch.empty(S.shape, dtype=S.dtype, device=DEV)}
    # the state on the planned mesh stands ready, as between two regrids
    S.regrid_estimate(REFINE, RATIO, DEEPEST, weights=WEIGHTS)
    D = amrvac.State(cfg, insts, S.regrid_plan(), device=DEV, pressure=case["pressure"])
    return {"S": S, "D": D, "out": torch.empty(D.shape, dtype=D.dtype, device=DEV)}


def run(state):
    S = state["S"]
    if "D" not in state:
        S.step(state["steps"])
        return S.get_conserved(out=state["out"])
    est, flags = S.regrid_estimate(REFINE, RATIO, DEEPEST, weights=WEIGHTS)
    meta = S.regrid_plan()
    # the transfer runs on the source state's stream
    S.stream.wait_stream(state["D"].stream)
    S.regrid_transfer(state["D"])
    state["D"].stream.wait_stream(S.stream)
    return {"est": est, "flags": flags, "meta": meta,
            "U": state["D"].get_conserved(out=state["out"])}


# ------------------------------------------------------------------ work

STAGES = {"ssprk2": 2, "ssprk3": 3, "ssprk43": 4}


def work(case):
    """Bytes: the state read once and written once a step (and, for a regrid,
    the old state read and the new one written).  Flops: the arithmetic of the
    formulas, each division and square root counted once: per cell and stage a
    primitive recovery (30) and update (3 a variable and dimension), per face
    the limited slopes of one cell's nine variables (8 each, 40 with five
    points) with two face states, and the Riemann solve (HLL 150, HLLD 290)."""
    cfg, insts, meta = _plan(case)
    cells = meta.shape[0] * case["block"] ** case["ndim"]
    size = 8 if case["precision"] == "fp64" else 4
    if case["problem"] == "regrid":
        # per cell and dimension 12 operations a weighted quantity, twice
        return {"bytes": 2 * NV * size * cells, "flops": cells * (30 + 2 * (3 * 12 + 4))}
    five = case["limiter"] in ("mp5", "weno5", "wenoz5", "wenozp5")
    face = NV * ((2 * 40 if five else 8) + 4) + (290 if case["flux"] == "hlld" else 150)
    per = 30 + case["ndim"] * (face + 3 * NV)
    return {"bytes": 2 * NV * size * cells * case["steps"],
            "flops": per * cells * STAGES[case["time"]] * case["steps"]}


# ------------------------------------------------------------------ in 64 bits

REFINED, COARSER = -1, -2


class _Mesh:
    """Block maps of a case and the ghost operators on them, in torch."""

    def __init__(self, cfg, insts, meta):
        self.nd, self.nx = cfg.ndim, cfg.block_nx
        self.open = cfg.bc[0][0] == "outflow"
        self.meta = torch.as_tensor(meta, dtype=torch.int64, device=DEV)
        self.nb = self.meta.shape[0]
        self.levels = int(self.meta[:, 1].max()) + 1
        base = torch.tensor([i.base_blocks for i in insts], device=DEV)
        sh = torch.tensor([1 if d < self.nd else 0 for d in range(3)], device=DEV)
        lev = torch.arange(self.levels + 1, device=DEV)
        self.n = base[:, None, :] << (lev[None, :, None] * sh)       # blocks [inst, level, 3]
        cnt = self.n.prod(2).reshape(-1)
        self.off = (torch.cumsum(cnt, 0) - cnt).reshape(len(insts), -1)
        self.map = torch.full((int(cnt.sum()),), COARSER, device=DEV)
        q, L, p = self.meta[:, 0], self.meta[:, 1], self.meta[:, 2:]
        self.map[self._at(q, L, p)] = torch.arange(self.nb, device=DEV)
        for up in range(1, self.levels):
            m = L >= up
            self.map[self._at(q[m], L[m] - up, p[m] >> (up * sh))] = REFINED
        nxt = torch.tensor(self.nx, device=DEV)
        self.dx = 1.0 / (self.n[q, L] * nxt).double()                # [block, 3]
        self.gamma = torch.tensor([i.gamma for i in insts], dtype=torch.float64, device=DEV)
        self.sh, self.nxt, self.ni = sh, nxt, len(insts)

    def _at(self, q, L, p):
        n = self.n[q, L]
        return self.off[q, L] + (p[:, 2] * n[:, 1] + p[:, 1]) * n[:, 0] + p[:, 0]

    def find(self, q, L, p):
        """Wrapped or clamped cell p of level L: (map code, cell in the block)."""
        N = self.n[q, L] * self.nxt
        p = torch.minimum(p.clamp(min=0), N - 1) if self.open else p % N
        b = p // self.nxt
        c = p - b * self.nxt
        return p, self.map[self._at(q, L, b)], (c[:, 2] * self.nx[1] + c[:, 1]) * self.nx[0] + c[:, 0]

    def value(self, U, q, L, p):
        """Level-L value of cell p: leaf, mean of the finer cells, or coarse value
        with minmod slopes.  [9, n]"""
        p, code, cell = self.find(q, L, p)
        out = U[:, code.clamp(min=0), cell]
        m = code == REFINED
        if bool(m.any()):
            acc = 0.0
            kids = [(a, b, c) for c in range(2 if self.nd > 2 else 1)
                    for b in range(2 if self.nd > 1 else 1) for a in range(2)]
            for k in kids:
                o = torch.tensor(k, device=DEV)
                acc = acc + self.value(U, q[m], L[m] + 1, (p[m] << self.sh) + o)
            out[:, m] = acc / len(kids)
        m = code == COARSER
        if bool(m.any()):
            qq, LL, pp = q[m], L[m] - 1, p[m]
            c = pp >> self.sh
            mid = self.value(U, qq, LL, c)
            acc = mid.clone()
            for d in range(self.nd):
                e = torch.zeros(3, dtype=torch.int64, device=DEV)
                e[d] = 1
                a, b = mid - self.value(U, qq, LL, c - e), self.value(U, qq, LL, c + e) - mid
                s = torch.where(a * b > 0, torch.where(a > 0, torch.minimum(a, b),
                                                       torch.maximum(a, b)), 0.0)
                acc += torch.where(pp[:, d] % 2 == 1, 0.25, -0.25) * s
            out[:, m] = acc
        return out

    def padded(self, U, blocks, G):
        """U of some blocks with G ghost layers on their faces [9, n, z, y, x]."""
        nx, nd = self.nx, self.nd
        g = [G if d < nd else 0 for d in range(3)]
        n = blocks.numel()
        P = torch.zeros(NV, n, nx[2] + 2 * g[2], nx[1] + 2 * g[1], nx[0] + 2 * g[0],
                        dtype=torch.float64, device=DEV)
        P[:, :, g[2]:g[2] + nx[2], g[1]:g[1] + nx[1], g[0]:g[0] + nx[0]] = \
            U[:, blocks].reshape(NV, n, nx[2], nx[1], nx[0])
        P[0] += (P[0] == 0) * 1.0   # corners are never used
        for d in range(nd):
            for side in (0, 1):
                rng = [torch.arange(nx[e], device=DEV) for e in range(3)]
                rng[d] = torch.arange(-G, 0, device=DEV) if side == 0 \
                    else torch.arange(nx[d], nx[d] + G, device=DEV)
                kk, jj, ii = torch.meshgrid(rng[2], rng[1], rng[0], indexing="ij")
                loc = torch.stack([ii, jj, kk], -1).reshape(-1, 3)
                p = (self.meta[blocks, 2:] * self.nxt)[:, None] + loc[None]
                q = self.meta[blocks, 0][:, None].expand(-1, loc.shape[0]).reshape(-1)
                L = self.meta[blocks, 1][:, None].expand(-1, loc.shape[0]).reshape(-1)
                v = self.value(U, q, L, p.reshape(-1, 3)).reshape(NV, n, *kk.shape)
                sl = [slice(g[e], g[e] + nx[e]) for e in range(3)]
                sl[d] = slice(0, G) if side == 0 else slice(g[d] + nx[d], None)
                P[:, :, sl[2], sl[1], sl[0]] = v
        return P


def _prims(U, g):
    v = U[1:4] / U[0]
    p = (g - 1.0) * (U[4] - 0.5 * (U[1:4] * v).sum(0) - 0.5 * (U[5:8] ** 2).sum(0))
    return torch.cat([U[:1], v, p[None], U[5:]])


def _minmod(a, b):
    return torch.where(a * b > 0, torch.sign(a) * torch.minimum(a.abs(), b.abs()), 0.0)


def _five(lim, a, b, c, d, e):
    """Face value at i+1/2 from five cells."""
    if lim == "mp5":
        vor = (2 * a - 13 * b + 47 * c + 27 * d - 3 * e) / 60
        vmp = c + _minmod(d - c, 4 * (c - b))
        djm, dj, djp = a - 2 * b + c, b - 2 * c + d, c - 2 * d + e

        def mm4(w, x, y, z):
            lo = torch.minimum(torch.minimum(w, x), torch.minimum(y, z))
            hi = torch.maximum(torch.maximum(w, x), torch.maximum(y, z))
            return torch.where(lo > 0, lo, torch.where(hi < 0, hi, 0.0))
        dp, dm = mm4(4 * dj - djp, 4 * djp - dj, dj, djp), mm4(4 * dj - djm, 4 * djm - dj, dj, djm)
        vul, vmd = c + 4 * (c - b), 0.5 * (c + d) - 0.5 * dp
        vlc = c + 0.5 * (c - b) + 4.0 / 3.0 * dm
        mn, mx = torch.minimum, torch.maximum
        vmin = mx(mn(mn(c, d), vmd), mn(mn(c, vul), vlc))
        vmax = mn(mx(mx(c, d), vmd), mx(mx(c, vul), vlc))
        return torch.where((vor - c) * (vor - vmp) <= 0, vor, vor + _minmod(vmin - vor, vmax - vor))
    b0 = 13 / 12 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2
    b1 = 13 / 12 * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2
    b2 = 13 / 12 * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2
    w0, w1, w2 = 0.1 / (1e-6 + b0) ** 2, 0.6 / (1e-6 + b1) ** 2, 0.3 / (1e-6 + b2) ** 2
    return (w0 * (2 * a - 7 * b + 11 * c) / 6 + w1 * (-b + 5 * c + 2 * d) / 6
            + w2 * (2 * c + 5 * d - e) / 6) / (w0 + w1 + w2)


def _half_slope(lim, dm, dp):
    """Increments to the low and the high face of a cell (magnitudes with sign)."""
    if lim == "vanleer":
        s = torch.where(dm * dp > 0, dm * dp / torch.where(dm * dp > 0, dm + dp, 1.0), 0.0)
        return s, s
    am, ap, sg = dm.abs(), dp.abs(), torch.where(dm * dp > 0, torch.sign(dp), 0.0)
    mn = torch.minimum
    if lim == "minmod":
        s = 0.5 * sg * mn(am, ap)
        return s, s
    if lim == "woodward":
        s = 0.5 * sg * mn(mn(2 * am, 0.5 * (am + ap)), 2 * ap)
        return s, s
    hi = 0.5 * sg * mn(mn(2 * am, (am + 2 * ap) / 3), 2 * ap)   # koren
    lo = 0.5 * sg * mn(mn(2 * ap, (ap + 2 * am) / 3), 2 * am)
    return lo, hi


def _fast(g, q, bn):
    a2 = g * q[4] / q[0]
    bt = q[6] ** 2 + q[7] ** 2
    bb = (bn ** 2 + bt) / q[0]
    return (0.5 * (a2 + bb + ((a2 - bb) ** 2 + 4 * a2 * bt / q[0]).sqrt())).sqrt()


def _state_flux(g, q, bx):
    rho, u, v, w, p, _, by, bz = q
    b2 = bx ** 2 + by ** 2 + bz ** 2
    pt = p + 0.5 * b2
    e = p / (g - 1) + 0.5 * rho * (u ** 2 + v ** 2 + w ** 2) + 0.5 * b2
    U = [rho, rho * u, rho * v, rho * w, e, bx, by, bz]
    F = [rho * u, rho * u * u + pt - bx * bx, rho * u * v - bx * by, rho * u * w - bx * bz,
         (e + pt) * u - bx * (u * bx + v * by + w * bz), torch.zeros_like(rho),
         by * u - bx * v, bz * u - bx * w]
    return U, F, pt, e


def _hlld_star(q, e, pt, s, sm, pts, bx):
    rho, u, v, w, _, _, by, bz = q
    su, isd = s - u, 1.0 / (s - sm)
    rs, big = rho * su * isd, rho * su * (s - sm)
    den = big - bx * bx
    flat = den.abs() <= 1e-8 * torch.maximum(big.abs(), bx * bx)
    iden = 1.0 / torch.where(flat, 1.0, den)
    tv, tb = bx * (sm - u) * iden, (rho * su * su - bx * bx) * iden
    vs, ws = torch.where(flat, v, v - by * tv), torch.where(flat, w, w - bz * tv)
    bys, bzs = torch.where(flat, by, by * tb), torch.where(flat, bz, bz * tb)
    vb = u * bx + v * by + w * bz
    es = (su * e - pt * u + pts * sm + bx * (vb - (sm * bx + vs * bys + ws * bzs))) * isd
    return [rs, rs * sm, rs * vs, rs * ws, es, bx, bys, bzs], vs, ws, bys, bzs


def _riemann(flux, g, ql, qr, bx):
    UL, FL, ptl, el = _state_flux(g, ql, bx)
    UR, FR, ptr, er = _state_flux(g, qr, bx)
    cl, cr = _fast(g, ql, bx), _fast(g, qr, bx)
    ul, ur = ql[1], qr[1]
    if flux == "hll":
        sl, sr = torch.minimum(ul - cl, ur - cr), torch.maximum(ul + cl, ur + cr)
        mid = [(sr * a - sl * b + sl * sr * (d - c)) / (sr - sl)
               for a, b, c, d in zip(FL, FR, UL, UR)]
        return [torch.where(sl >= 0, a, torch.where(sr <= 0, b, m))
                for a, b, m in zip(FL, FR, mid)]
    cm = torch.maximum(cl, cr)
    sl, sr = torch.minimum(ul, ur) - cm, torch.maximum(ul, ur) + cm
    al, ar = (sl - ul) * ql[0], (sr - ur) * qr[0]
    sm = (ar * ur - al * ul - ptr + ptl) / (ar - al)
    pts = (ar * ptl - al * ptr + ar * al * (ur - ul)) / (ar - al)
    SL, vl, wl_, byl, bzl = _hlld_star(ql, el, ptl, sl, sm, pts, bx)
    SR, vr, wr_, byr, bzr = _hlld_star(qr, er, ptr, sr, sm, pts, bx)
    a, b = SL[0].sqrt(), SR[0].sqrt()
    ssl, ssr, sb = sm - bx.abs() / a, sm + bx.abs() / b, torch.sign(bx)
    vss, wss = (a * vl + b * vr + (byr - byl) * sb) / (a + b), (a * wl_ + b * wr_ + (bzr - bzl) * sb) / (a + b)
    bys = (a * byr + b * byl + a * b * (vr - vl) * sb) / (a + b)
    bzs = (a * bzr + b * bzl + a * b * (wr_ - wl_) * sb) / (a + b)
    vb = sm * bx + vss * bys + wss * bzs
    el2 = SL[4] - a * (sm * bx + vl * byl + wl_ * bzl - vb) * sb
    er2 = SR[4] + b * (sm * bx + vr * byr + wr_ * bzr - vb) * sb
    left = sm >= 0
    outer = torch.where(left, sl > 0, sr < 0)
    single = torch.where(left, ssl >= 0, ~(ssr >= 0))
    s1, s2 = torch.where(left, sl, sr), torch.where(left, ssl, ssr)
    out = []
    for c in range(8):
        U, F, S = (torch.where(left, x[c], y[c]) for x, y in ((UL, UR), (FL, FR), (SL, SR)))
        T = S if c in (0, 1, 5) else \
            {2: _times(SL, SR, left, vss), 3: _times(SL, SR, left, wss),
             4: torch.where(left, el2, er2), 6: bys, 7: bzs}[c]
        f1 = F + s1 * (S - U)
        out.append(torch.where(outer, F, torch.where(single, f1, f1 + s2 * (T - S))))
    return out


def _times(SL, SR, left, v):
    return torch.where(left, SL[0], SR[0]) * v


def _face_flux(case, cfg, W, d, g, ch):
    """Fluxes of every face along d of padded primitives W [9, n, z, y, x]."""
    nd, nx = cfg.ndim, cfg.block_nx
    G = 3 if case["limiter"] in ("mp5", "weno5") else 2
    for e in range(nd):  # no ghost layers across the other directions
        if e != d:
            W = W.narrow(4 - e, G, nx[e])
    s = lambda o: W.narrow(4 - d, o, nx[d] + 1)  # noqa: E731  cells f - G + o of face f
    if G == 3:
        c = [s(o) for o in range(6)]
        l, r = _five(case["limiter"], *c[:5]), _five(case["limiter"], *c[:0:-1])
        b, c = c[2], c[3]
    else:
        a, b, c, e = (s(o) for o in range(4))
        l = b + _half_slope(case["limiter"], b - a, c - b)[1]
        r = c - _half_slope(case["limiter"], c - b, e - c)[0]
    bad = (l[0] <= 0) | (l[4] <= 0) | (r[0] <= 0) | (r[4] <= 0)
    l, r = torch.where(bad, b, l), torch.where(bad, c, r)
    t1, t2 = (d + 1) % 3, (d + 2) % 3
    bn, psi = 0.5 * (l[5 + d] + r[5 + d]), torch.zeros_like(l[8])
    if cfg.glm:
        bn = bn - (r[8] - l[8]) / (2 * ch)
        psi = 0.5 * (l[8] + r[8]) - 0.5 * ch * (r[5 + d] - l[5 + d])
    pick = lambda w: [w[0], w[1 + d], w[1 + t1], w[1 + t2], w[4], bn, w[5 + t1], w[5 + t2]]  # noqa: E731
    f = _riemann(case["flux"], g, pick(l), pick(r), bn)
    F = torch.empty_like(l)
    F[0], F[1 + d], F[1 + t1], F[1 + t2], F[4] = f[:5]
    F[5 + d], F[5 + t1], F[5 + t2] = psi, f[6], f[7]
    F[8] = ch * ch * bn if cfg.glm else 0.0
    return F


def _cfl(mesh, U, cfg):
    """Per instance (dt, c_h)."""
    smax = torch.zeros(mesh.ni, dtype=torch.float64, device=DEV)
    cmax = torch.zeros_like(smax)
    for blocks in torch.arange(mesh.nb, device=DEV).split(_CHUNK(mesh)):
        q = mesh.meta[blocks, 0]
        g = mesh.gamma[q][:, None]
        w = _prims(U[:, blocks], g)
        s, m = 0.0, torch.zeros_like(w[0])
        for d in range(cfg.ndim):
            o = [(d + k) % 3 for k in range(3)]
            spd = w[1 + d].abs() + _fast(g, [w[0], 0, 0, 0, w[4], 0, w[5 + o[1]], w[5 + o[2]]],
                                         w[5 + d])
            s = s + spd / mesh.dx[blocks, d][:, None]
            m = torch.maximum(m, spd)
        smax.scatter_reduce_(0, q, s.amax(1), "amax")
        cmax.scatter_reduce_(0, q, m.amax(1), "amax")
    return cfg.courant / smax, cmax


def _CHUNK(mesh):
    cells = mesh.nx[0] * mesh.nx[1] * mesh.nx[2]
    return max(1, 4_000_000 // cells)


def _euler(case, cfg, mesh, U, dt, ch, c):
    """U + c dt L(U) with psi damped, on every block."""
    G = 3 if case["limiter"] in ("mp5", "weno5") else 2
    nx, nd = cfg.block_nx, cfg.ndim
    out = torch.empty_like(U)
    face = {}
    if case["reflux"]:
        area = [nx[1] * nx[2], nx[0] * nx[2], nx[0] * nx[1]]
        face = {(d, s): torch.empty(NV, mesh.nb, area[d], dtype=torch.float64, device=DEV)
                for d in range(nd) for s in (0, 1)}
    for blocks in torch.arange(mesh.nb, device=DEV).split(_CHUNK(mesh)):
        q = mesh.meta[blocks, 0]
        col = lambda t: t[:, None, None, None]  # noqa: E731
        g, h, dtb = col(mesh.gamma[q]), col(ch[q]), col(dt[q] * c)
        W = _prims(mesh.padded(U, blocks, G), g)
        acc = 0.0
        for d in range(nd):
            F = _face_flux(case, cfg, W, d, g, h)
            acc = acc + torch.diff(F, dim=4 - d) / col(mesh.dx[blocks, d])
            for s in (0, 1):
                if face:
                    face[d, s][:, blocks] = F.select(4 - d, -s).reshape(NV, blocks.numel(), -1)
        out[:, blocks] = (U[:, blocks].reshape(NV, blocks.numel(), *acc.shape[2:])
                          - dtb * acc).reshape(NV, blocks.numel(), -1)
    if face:
        _reflux(cfg, mesh, out, face, dt, c)
    if cfg.glm:
        dxm = mesh.dx[:, :nd].amin(1)
        q = mesh.meta[:, 0]
        out[8] *= torch.exp(-cfg.glm_alpha * ch[q] * dt[q] * c / dxm)[:, None]
    return out


def _reflux(cfg, mesh, out, face, dt, c):
    """The coarse side of a level change takes the mean of the fine fluxes."""
    nx, nd = cfg.block_nx, cfg.ndim
    q, L = mesh.meta[:, 0], mesh.meta[:, 1]
    shape = out.shape
    out = out.view(NV, mesh.nb, nx[2], nx[1], nx[0])
    for (d, s), F in face.items():
        t = [e for e in range(nd) if e != d]
        nxt = [nx[e] for e in t]
        far = mesh.meta[:, 2:] * mesh.nxt
        far[:, d] += nx[d] if s else -1
        code = mesh.find(q, L, far)[1]
        b = torch.nonzero(code == REFINED).reshape(-1)
        grids = torch.meshgrid(*[torch.arange(n, device=DEV) for n in reversed(nxt)], indexing="ij")
        loc = torch.zeros(grids[0].numel(), 3, dtype=torch.int64, device=DEV)
        for e, gr in zip(reversed(t), grids):
            loc[:, e] = gr.reshape(-1)
        mean = 0.0
        for k in range(1 << len(t)):
            p = ((mesh.meta[b, 2:] * mesh.nxt)[:, None] + loc[None]) * 2
            for i, e in enumerate(t):
                p[..., e] += (k >> i) & 1
            p[..., d] = (2 * (mesh.meta[b, 2 + d] + s) * nx[d] - (0 if s else 1))[:, None]
            n = loc.shape[0]
            p, fb, cell = mesh.find(q[b].repeat_interleave(n), L[b].repeat_interleave(n) + 1,
                                    p.reshape(-1, 3))
            ijk = (cell % nx[0], (cell // nx[0]) % nx[1], cell // (nx[0] * nx[1]))
            at = ijk[t[1]] * nxt[0] + ijk[t[0]] if len(t) == 2 else ijk[t[0]]
            mean = mean + face[d, 1 - s][:, fb, at].reshape(NV, b.numel(), n)
        dF = (F[:, b] - mean / (1 << len(t))) / mesh.dx[b, d][:, None]
        edge = out.select(4 - d, -s)
        edge[:, b] += ((1 if s else -1) * (dt[q[b]] * c)[:, None] * dF) \
            .reshape(NV, b.numel(), *edge.shape[2:])
    return out.view(shape)


#: u0, input, output registers and (a, b, c) of each stage: out = a u0 + b (in + c dt L(in))
SCHEME = {"ssprk2": [(0, 1, 0, 1, 1), (1, 0, .5, .5, 1)],
          "ssprk3": [(0, 1, 0, 1, 1), (1, 2, .75, .25, 1), (2, 0, 1 / 3, 2 / 3, 1)],
          "ssprk43": [(0, 1, 0, 1, .5), (1, 2, 0, 1, .5), (2, 1, 2 / 3, 1 / 3, .5),
                      (1, 0, 0, 1, .5)]}


def exact(case, seed):
    cfg, insts, meta = _plan(case)
    U = _inputs(case, seed, cfg, insts, meta).double()
    mesh = _Mesh(cfg, insts, meta)
    if case["problem"] == "regrid":
        return {"est": _estimate(mesh, U), "flags": None, "meta": None, "U": None}
    dt, ch = _cfl(mesh, U, cfg)
    for _ in range(case["steps"]):
        reg = [U, None, None]
        for i, o, a, b, c in SCHEME[case["time"]]:
            e = _euler(case, cfg, mesh, reg[i], dt, ch, c)
            reg[o] = e if a == 0 else a * reg[0] + b * e
        U = reg[0]
        dt, ch = _cfl(mesh, U, cfg)
    return U


def _estimate(mesh, U):
    """Block maxima of the weighted normalised second derivatives."""
    out = torch.empty(mesh.nb, dtype=torch.float64, device=DEV)
    nx = mesh.nx
    for blocks in torch.arange(mesh.nb, device=DEV).split(_CHUNK(mesh)):
        W = _prims(mesh.padded(U, blocks, 1), mesh.gamma[mesh.meta[blocks, 0]][:, None, None, None])
        tot = 0.0
        for v, w in enumerate(WEIGHTS):
            if w == 0:
                continue
            num = den = 0.0
            for d in range(mesh.nd):
                q = W[v]
                for e in range(mesh.nd):
                    if e != d:
                        q = q.narrow(3 - e, 1, nx[e])
                m, c, p = (q.narrow(3 - d, o, nx[d]) for o in range(3))
                num = num + (p - 2 * c + m) ** 2
                den = den + ((p - c).abs() + (c - m).abs()
                             + 0.01 * (p.abs() + 2 * c.abs() + m.abs())) ** 2
            tot = tot + w * torch.where(den > 0, num / den, 0.0).sqrt()
        out[blocks] = tot.reshape(blocks.numel(), -1).amax(1)
    return out
