"""The calls that a user of this framework makes, as timed cases.

A case is a plain dict.  ``kind`` says which public entry point it goes through:

  run      ``Run.advance`` over whole EM periods: the state goes in, the run
           advances, the fields of both meshes come out
  watch    the same in quarters of a period without CUDA graphs, two fields read
           after each quarter (a monitor or a movie)
  batch    ``Batch.advance``: many runs of uneven sizes together
  adjoint  ``dmr_density`` forward and backward: the density at the end and its
           gradients with respect to E0, the ionization scale and the seed map

Every pass of ``run`` and ``watch`` starts from the same state (fields, currents
and density written back first), so passes do the same work; a batch takes its
densities back, and so does a run with absorbing layers, whose layer fields a
program cannot write.  The states are what a run meets under way: an incident wave of
some MV/m, scattered waves of a few per cent of it, Gaussian plasmas below the
density at which the rectangle would grow.

``exact`` evaluates the same calls in 64 bits with plain torch operations.
"""
import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2105_13276_gb300 import adjoint as A
from paper_2105_13276_gb300 import dmr as D

C0 = 299792458.0
MU0 = 1.25663706212e-6
EPS0 = 8.8541878128e-12
QE = 1.602176634e-19
ME = 9.1093837015e-31
FREQ = 110e9
LAM = C0 / FREQ
DEVICE = "cuda"

EVOLVING = ("Ex", "Ey", "Hz", "vx", "vy", "n")   # what a pass writes
OUTPUTS = EVOLVING + ("erms",)                   # what a pass reads, per mesh
COLLECTED = ("Ey", "n", "erms")                  # what a batch collects, per run and mesh
WATCHED = ("Ey", "n")                            # what a monitor reads


def _case(name, kind, nx, ny, r, n_lambda, rect=None, **kw):
    c = dict(name=name, kind=kind, nx=nx, ny=ny, r=r, n_lambda=n_lambda, precision=1, boundary=0,
             coupling=0, growth=1, periods=1, E0=5e6, p=700.0, plasmas=1, n_lo=1e15, n_hi=1e15)
    i0, j0, i1, j1 = rect if rect else (0, 0, 0, 0)
    c.update(i0=i0, j0=j0, i1=i1, j1=j1)
    c.update(kw)
    return c


def listed():
    return [
        # the front-velocity experiment (1.5 x 1.5 wavelengths) at its start,
        # watched four times per period: the smallest calls
        _case("front96_r2_watch", "watch", 96, 96, 2, 64, (73, 40, 89, 56), E0=5.5e6, p=760.0,
              n_lo=1e16, n_hi=1e16),
        # the same experiment at r = 4 under way (threshold lines, the density
        # alone going back): the rectangle covers a quarter of the domain
        _case("front96_r4_density_back", "run", 96, 96, 4, 64, (41, 24, 93, 72), E0=5.5e6, p=760.0,
              coupling=1, growth=2, periods=2, n_lo=1e16, n_hi=1e17),
        # the plain uniform mesh of the paper's kind, FP64
        _case("uniform256_f64", "run", 256, 256, 1, 64, precision=0, periods=2),
        # the uniform fine mesh that the DMR run below replaces
        _case("uniform1024_f32", "run", 1024, 1024, 1, 64),
        # the headline run: 16 x 16 wavelengths, a patch of 64 x 64 fine cells
        _case("dmr512_r2_f32", "run", 512, 512, 2, 32, (240, 240, 272, 272), periods=4),
        # the same with every field in FP64
        _case("dmr512_r2_f64", "run", 512, 512, 2, 32, (240, 240, 272, 272), precision=0),
        # odd sizes, r = 3, absorbing layers around the domain; the density alone
        # goes back (the reading without a growing mode, for long runs)
        _case("cpml301x187_r3_f32", "run", 301, 187, 3, 32, (101, 61, 164, 110), boundary=1, coupling=1,
              periods=2, plasmas=2),
        # filament arrays on a 64 x 32 wavelength domain, the rectangle at a
        # quarter of it, r = 2 and r = 4 (the largest calls)
        _case("large2048_r2_f32", "run", 2048, 1024, 2, 32, (480, 232, 1504, 744), plasmas=8, n_lo=1e14,
              n_hi=1e16),
        _case("large2048_r4_f32", "run", 2048, 1024, 4, 32, (480, 232, 1504, 744), plasmas=8, n_lo=1e14,
              n_hi=1e16),
        # a parameter study: 16 runs of uneven sizes in one batch
        _case("batch16_f32", "batch", 1024, 1024, 2, 32, runs=16, periods=2),
        # gradients through a recorded run, FP32 and (a small one) FP64
        _case("adjoint512_r2_f32", "adjoint", 512, 512, 2, 32, (240, 240, 272, 272), periods=8, keep=4),
        _case("adjoint40_r2_f64", "adjoint", 40, 32, 2, 16, (12, 10, 24, 20), precision=0, periods=4,
              keep=2, growth=0, n_lo=3e17, n_hi=3e17),
    ]


def _rect(rng, nx, ny, margin, frac):
    """A rectangle of about frac of the domain, at least 4 coarse cells wide and
    `margin` cells inside; sometimes at a side."""
    w = min(max(4, round((nx - 2 * margin) * frac * rng.uniform(0.7, 1.3))), nx - 2 * margin)
    h = min(max(4, round((ny - 2 * margin) * frac * rng.uniform(0.7, 1.3))), ny - 2 * margin)
    i0 = rng.choice([margin, nx - margin - w]) if rng.random() < 0.15 else rng.randint(margin, nx - margin - w)
    j0 = rng.choice([margin, ny - margin - h]) if rng.random() < 0.15 else rng.randint(margin, ny - margin - h)
    return i0, j0, i0 + w, j0 + h


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))
    while True:
        kind = rng.choice(["run", "run", "run", "run", "watch", "batch", "adjoint"])
        precision = 1 if rng.random() < 0.7 else 0
        r = rng.choice([1, 2, 2, 2, 3, 4])
        n_lambda = rng.choice([16, 32, 32, 64])
        E0, p = rng.uniform(3e6, 6e6), rng.uniform(400.0, 760.0)
        extra = dict(precision=precision, E0=E0, p=p, plasmas=rng.randint(1, 6), n_lo=1e14, n_hi=1e16)
        if kind == "batch":
            c = _case("", kind, rng.choice([256, 512, 1024]), 1024, 2, 32, runs=rng.randint(4, 20),
                      periods=rng.randint(1, 2), **dict(extra, precision=1))
        else:
            hi = {"run": 2048, "watch": 512, "adjoint": 400}[kind]
            nx, ny = round(log(40, hi)), round(log(32, min(hi, 1200)))
            boundary = 1 if kind != "adjoint" and min(nx, ny) >= 64 and rng.random() < 0.15 else 0
            rect = _rect(rng, nx, ny, 10 if boundary else 0, log(0.05, 0.6)) if r > 1 else None
            if kind == "adjoint":
                extra.update(periods=rng.randint(1, 3), keep=1)
            else:
                extra.update(periods=1 if kind == "watch" else rng.randint(1, 4),
                             coupling=1 if boundary else int(rng.random() < 0.2), growth=0)
            c = _case("", kind, nx, ny, r, n_lambda, rect, boundary=boundary, **extra)
        c.pop("name")
        if c["kind"] == "adjoint" and _tape_bytes(c) > 12e9:
            continue
        if _cost(c) <= _cost(_LARGEST):
            return c


# ---------------------------------------------------------------------------
# What a user's program has in hand
# ---------------------------------------------------------------------------
def _rect_of(c):
    return (c["i0"], c["j0"], c["i1"], c["j1"]) if c["r"] > 1 else None


def _cfg(c):
    return dict(nx=c["nx"], ny=c["ny"], r=c["r"], n_lambda=c["n_lambda"], steps_per_period=2 * c["n_lambda"],
                freq=FREQ, E0=c["E0"], p_torr=c["p"], growth=c["growth"], m_ex=32, m_ey=16,
                boundary=c["boundary"], coupling=c["coupling"], precision=c["precision"])


def _dtype(c):
    return torch.float32 if c["precision"] == 1 else torch.float64


def _sub_cases(c, seed):
    """The runs of a batch: sizes, fields, pressures and patches drawn from the
    seed of the study (the sizes from the case alone, so that its work is fixed)."""
    size = np.random.RandomState(13276 + c["runs"])
    g = np.random.RandomState(seed)
    subs = []
    for _ in range(c["runs"]):
        nx = int(size.choice([s for s in (128, 256, 512, 1024) if s <= c["nx"]]))
        ic, jc = (int(round(g.uniform(0.25, 0.75) * nx)) for _ in range(2))
        i0, j0 = (min(max(q - 16, 0), nx - 32) for q in (ic, jc))
        subs.append(dict(c, nx=nx, ny=nx, i0=i0, j0=j0, i1=i0 + 32, j1=j0 + 32, E0=float(g.uniform(3e6, 6e6)),
                         p=float(g.uniform(400.0, 760.0))))
    return subs


def _inputs(c, seed, quiet=False):
    """The state of both meshes as FP64 tensors, from the seed alone: four
    scattered plane waves, the drift that goes with them, Gaussian plasmas of
    lambda/8 inside the rectangle.  quiet: the waves left out (a run at t = 0)."""
    g = np.random.RandomState(seed)
    dev = torch.device(DEVICE)
    nx, ny, L = c["nx"], c["ny"], c["n_lambda"]
    dx = LAM / L
    amp = 0.0 if quiet else 0.02 * c["E0"]
    waves = [(amp * a, t, f) for a, t, f in zip(g.uniform(0.5, 1.0, 4), g.uniform(0, 2 * math.pi, 4),
                                                g.uniform(0, 2 * math.pi, 4))]
    rc = _rect_of(c) or (nx // 4, ny // 4, nx - nx // 4, ny - ny // 4)
    # centres where the plasma stays clear of the rectangle's growth zone
    mx, my = ((b - a) / 2 - max(0.0, (b - a) / 2 - 16 * L / 32) for a, b in ((rc[0], rc[2]), (rc[1], rc[3])))
    plasmas = [(math.exp(g.uniform(math.log(c["n_lo"]), math.log(c["n_hi"]))) * g.uniform(0.9, 1.0),
                g.uniform(rc[0] + mx, rc[2] - mx + 1e-9), g.uniform(rc[1] + my, rc[3] - my + 1e-9))
               for _ in range(c["plasmas"])]
    nu_m = 5.3e9 * c["p"]
    k0 = 2 * math.pi / LAM
    meshes = [(0.0, 0.0, dx, nx, ny)]
    if c["r"] > 1:
        i0, j0, i1, j1 = _rect_of(c)
        r = c["r"]
        meshes.append((i0 * dx, j0 * dx, dx / r, r * (i1 - i0), r * (j1 - j0)))
    out = []
    for x0, y0, h, mx_, my_ in meshes:
        def at(sx, sy, cols, rows):
            x = x0 + h * (torch.arange(cols, dtype=torch.float64, device=dev) + sx)
            y = y0 + h * (torch.arange(rows, dtype=torch.float64, device=dev) + sy)
            return x[None, :], y[:, None]

        def field(which, sx, sy, cols, rows):
            x, y = at(sx, sy, cols, rows)
            v = torch.zeros(rows, cols, dtype=torch.float64, device=dev)
            for a, t, f in waves:
                f = f - math.pi / (2 * L) if which == "H" else f
                s = {"x": -math.sin(t), "y": math.cos(t), "H": EPS0 * C0}[which]
                v += a * s * torch.cos(k0 * (math.cos(t) * x + math.sin(t) * y) + f)
            return v
        m = {"Ex": field("x", 0.5, 0.0, mx_, my_ + 1), "Ey": field("y", 0.0, 0.5, mx_ + 1, my_),
             "Hz": field("H", 0.5, 0.5, mx_, my_)}
        m["vx"], m["vy"] = (-QE / (ME * nu_m) * m[q] for q in ("Ex", "Ey"))
        x, y = at(0.0, 0.0, mx_ + 1, my_ + 1)
        n = torch.zeros(my_ + 1, mx_ + 1, dtype=torch.float64, device=dev)
        for n0, ic, jc in plasmas:
            n += n0 * torch.exp(-(((x - ic * dx) / (LAM / 8)) ** 2 + ((y - jc * dx) / (LAM / 8)) ** 2).clamp(max=60.0))
        m["n"] = n
        out.append({q: v.to(_dtype(c)).contiguous() for q, v in m.items()})
    if c["r"] > 1:
        # the coarse nodes under the rectangle carry the fine density
        out[0]["n"][j0:j1 + 1, i0:i1 + 1] = out[1]["n"][::r, ::r]
    return out


def _levels(c):
    return range(2 if c["r"] > 1 else 1)


def _adjoint_inputs(c, seed):
    """Seed map (a perturbed Gaussian on the mesh that carries it) and target."""
    g = torch.Generator().manual_seed(seed)
    n = _inputs(c, seed, quiet=True)[-1]["n"]
    jitter = 1.0 + 0.05 * torch.randn(n.shape, generator=g, dtype=torch.float64)
    target = torch.randn(c["ny"] + 1, c["nx"] + 1, generator=g, dtype=torch.float64)
    dt = _dtype(c)
    return (n.double() * jitter.to(DEVICE)).to(dt), (c["n_lo"] * (1.0 + 0.1 * target.to(DEVICE))).to(dt)


def _buffers(c, names):
    nx, ny, r = c["nx"], c["ny"], c["r"]
    dims = [(nx, ny)] + ([(r * (c["i1"] - c["i0"]), r * (c["j1"] - c["j0"]))] if r > 1 else [])
    shape = {"Ex": (1, 0), "vx": (1, 0), "Ey": (0, 1), "vy": (0, 1), "Hz": (0, 0)}
    out = []
    for a, b in dims:
        out.append({q: torch.empty(b + shape.get(q, (1, 1))[0], a + shape.get(q, (1, 1))[1], dtype=_dtype(c),
                                   device=DEVICE) for q in names})
    return out


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "adjoint":
        n, target = _adjoint_inputs(c, seed)
        torch.cuda.synchronize()
        dt = _dtype(c)
        return dict(c=c, cfg=_cfg(c), n=n.requires_grad_(True), target=target,
                    E0=torch.tensor(c["E0"], dtype=dt, device=DEVICE, requires_grad=True),
                    s=torch.tensor(1.0, dtype=dt, device=DEVICE, requires_grad=True))
    if kind == "batch":
        subs = _sub_cases(c, seed)
        b = D.Batch([_cfg(s) for s in subs])
        state = dict(c=c, batch=b, subs=subs, n=[], out={})
        sizes = [_buffers(s, COLLECTED) for s in subs]
        for q in COLLECTED:
            # every run's maps one after another in one tensor
            state["out"][q] = torch.empty(sum(m[q].numel() for s in sizes for m in s), dtype=_dtype(c), device=DEVICE)
        state["part"] = []
        used = dict.fromkeys(COLLECTED, 0)
        for k, (s, run) in enumerate(zip(subs, b.runs)):
            run.set_patch(_rect_of(s))
            state["n"].append([m["n"] for m in _inputs(s, seed + 7919 * k, quiet=True)])
            parts = []
            for m in sizes[k]:
                part = {}
                for q in COLLECTED:
                    part[q] = state["out"][q][used[q]:used[q] + m[q].numel()]
                    used[q] += m[q].numel()
                parts.append(part)
            state["part"].append(parts)
        torch.cuda.synchronize()
        _write_density(state)
        b.autotune()
        return state
    run = D.Run(_cfg(c))
    if c["r"] > 1:
        run.set_patch(_rect_of(c))
    state = dict(c=c, run=run, fields=_inputs(c, seed), out=_buffers(c, OUTPUTS))
    if c["r"] > 1:
        state["mask"] = torch.empty(c["ny"] + 1, c["nx"] + 1, dtype=torch.uint8, device=DEVICE)
    torch.cuda.synchronize()
    _write_state(state, EVOLVING)
    if kind == "watch":
        state["seen"] = [[{q: torch.empty_like(m[q]) for q in WATCHED} for m in state["out"]] for _ in range(3)]
        torch.cuda.synchronize()
    else:
        run.set_graphs(True)
        run.autotune()
    return state


def _write_state(state, names):
    for level, m in enumerate(state["fields"]):
        for q in names:
            state["run"].write_from(q, level, m[q])


def _write_density(state):
    for run, maps in zip(state["batch"].runs, state["n"]):
        for level, n in enumerate(maps):
            run.write_from("n", level, n)


def run(state):
    c = state["c"]
    if c["kind"] == "adjoint":
        n_t = c["n_lambda"] * 2
        n = A.dmr_density(state["E0"], state["s"], state["n"], state["cfg"], _rect_of(c), c["periods"] * n_t,
                          c["keep"] * n_t)
        loss = (((n - state["target"]) / c["n_lo"]) ** 2).mean()
        gE0, gs, gn = torch.autograd.grad(loss, (state["E0"], state["s"], state["n"]))
        return {"n": n.detach(), "dE0": gE0, "ds": gs, "dn": gn}
    if c["kind"] == "batch":
        _write_density(state)
        state["batch"].advance(c["periods"] * 2 * c["n_lambda"])
        for k, sim in enumerate(state["batch"].runs):
            for level, part in enumerate(state["part"][k]):
                for q, t in part.items():
                    sim.read_into(q, level, t)
        return state["out"]
    sim = state["run"]
    _write_state(state, ("n",) if c["boundary"] else EVOLVING)
    steps = c["periods"] * 2 * c["n_lambda"]
    if c["kind"] == "watch":
        for quarter in range(4):
            sim.advance(steps // 4)
            if quarter < 3:
                for level, m in enumerate(state["seen"][quarter]):
                    for q, t in m.items():
                        sim.read_into(q, level, t)
    else:
        sim.advance(steps)
    for level, m in enumerate(state["out"]):
        for q, t in m.items():
            sim.read_into(q, level, t)
    out = {"fields": state["out"]}
    if c["r"] > 1:
        sim.read_into("mask", 0, state["mask"])
        out["mask"] = state["mask"]
    if c["kind"] == "watch":
        out["seen"] = state["seen"]
    return out


# ---------------------------------------------------------------------------
# Work
# ---------------------------------------------------------------------------
def work(case):
    """Bytes and operations of one pass.  A time step needs the whole state of the
    step before it: each EM step of a mesh reads Ex, Ey, Hz, vx, vy and n and
    writes the first five once, and adds its E^2 sample to an FP64 sum read and
    written once; 37 operations per node.  A gradient is a forward with the
    recomputation from its checkpoints and a reverse sweep that reads the tape
    (E, v) and reads and writes the adjoint state."""
    c = case
    if c["kind"] == "batch":
        parts = [work(dict(s, kind="run")) for s in _sub_cases(c, 0)]
        return {q: float(sum(p[q] for p in parts)) for q in ("bytes", "flops")}
    es = 4 if c["precision"] == 1 else 8
    n_t, r = 2 * c["n_lambda"], c["r"]
    node_steps = float(n_t * (c["nx"] + 1) * (c["ny"] + 1))
    if r > 1:
        node_steps += float(n_t * r * (r * (c["i1"] - c["i0"]) + 1) * (r * (c["j1"] - c["j0"]) + 1))
    node_steps *= c["periods"]
    b, f = node_steps * (11 * es + 16), node_steps * 37
    if c["kind"] == "adjoint":
        b, f = 2 * b + node_steps * (4 * es + 4 * es + 13 * es), 2 * f + node_steps * 80
    return {"bytes": b, "flops": f}


_LARGEST = next(c for c in listed() if c["name"] == "large2048_r4_f32")


def _cost(c):
    """Work of a pass with what a step costs at least, as bytes (for draw)."""
    steps = c["periods"] * 2 * c["n_lambda"] * (c["r"] + 1) * c.get("runs", 1) * (6 if c["kind"] == "adjoint" else 1)
    return work(c)["bytes"] * (4 if c["precision"] == 0 else 1) + 4e6 * steps


def _tape_bytes(c):
    es = 4 if c["precision"] == 1 else 8
    nodes = (c["nx"] + 65) * (c["ny"] + 1) + c["r"] * (c["r"] * (c["i1"] - c["i0"]) + 65) * (c["r"] * (c["j1"] - c["j0"]) + 1)
    return 2.0 * c["keep"] * 2 * c["n_lambda"] * nodes * 4 * es


# ---------------------------------------------------------------------------
# The same in 64 bits, with plain torch operations
# ---------------------------------------------------------------------------
def _coefficients(c, rr):
    dx, dt = LAM / (rr * c["n_lambda"]), 1.0 / (FREQ * rr * 2 * c["n_lambda"])
    h = 0.5 * 5.3e9 * c["p"] * dt
    return dict(dx=dx, ch=dt / (MU0 * dx), ce=dt / (EPS0 * dx), cj=dt * QE / (2 * EPS0), va=(1 - h) / (1 + h),
                vb=QE * dt / ME / (1 + h), mur=(C0 * dt - dx) / (C0 * dt + dx), N=rr * 2 * c["n_lambda"])


def _incident(c, q, level, x, E0):
    """The incident Ey at node columns x (a row vector) and an E level of the mesh."""
    k, ph = 2 * math.pi / LAM, 2 * math.pi * (level % q["N"]) / q["N"]
    return E0 * (math.sin(ph) * torch.cos(k * x) - math.cos(ph) * torch.sin(k * x))


class _Layers:
    """The absorbing layers of a coarse mesh: 8 cells, a cubic conductivity."""

    def __init__(self, c, q, dev):
        eta, depth = math.sqrt(MU0 / EPS0), 8
        dt = 1.0 / (FREQ * q["N"])

        def coef(extent, shift, count):
            at = torch.arange(count, dtype=torch.float64, device=dev) + shift
            d = torch.maximum(depth - at, at - (extent - depth)).clamp(min=0) / depth
            b = torch.exp(-0.8 * 4 / (eta * q["dx"]) * d ** 3 * dt / EPS0)
            return b
        nx, ny = c["nx"], c["ny"]
        self.bxh, self.byh = coef(nx, 0.5, nx)[None, :], coef(ny, 0.5, ny)[:, None]
        self.bxn, self.byn = coef(nx, 0.0, nx + 1)[None, 1:-1], coef(ny, 0.0, ny + 1)[1:-1, None]
        self.hx = self.hy = self.ex = self.ey = 0.0


def _em(m, q, inc, sides, layers=None):
    """One EM step of a mesh from E at a level and H, v half a step before it.
    sides: per side "mur", "pec" or the new tangential E."""
    dey, dex = m["Ey"][:, 1:] - m["Ey"][:, :-1], m["Ex"][1:] - m["Ex"][:-1]
    if layers is not None:
        layers.hx = layers.bxh * layers.hx + (layers.bxh - 1) * dey
        layers.hy = layers.byh * layers.hy + (layers.byh - 1) * dex
        dey, dex = dey + layers.hx, dex + layers.hy
    H = m["Hz"] - q["ch"] * (dey - dex)
    vx = q["va"] * m["vx"] - q["vb"] * m["Ex"]
    vy = q["va"] * m["vy"] - q["vb"] * (m["Ey"] + inc)
    dhy, dhx = H[1:] - H[:-1], H[:, 1:] - H[:, :-1]
    if layers is not None:
        layers.ex = layers.byn * layers.ex + (layers.byn - 1) * dhy
        layers.ey = layers.bxn * layers.ey + (layers.bxn - 1) * dhx
        dhy, dhx = dhy + layers.ex, dhx + layers.ey
    n = m["n"]
    ix = m["Ex"][1:-1] + q["ce"] * dhy + q["cj"] * (n[1:-1, :-1] + n[1:-1, 1:]) * vx[1:-1]
    iy = m["Ey"][:, 1:-1] - q["ce"] * dhx + q["cj"] * (n[:-1, 1:-1] + n[1:, 1:-1]) * vy[:, 1:-1]

    def edge(side, old_b, old_1, new_1):
        if isinstance(side, str):
            return old_1 + q["mur"] * (new_1 - old_b) if side == "mur" else torch.zeros_like(old_b)
        return side
    lo = edge(sides["bottom"], m["Ex"][0], m["Ex"][1], ix[0])
    hi = edge(sides["top"], m["Ex"][-1], m["Ex"][-2], ix[-1])
    le = edge(sides["left"], m["Ey"][:, 0], m["Ey"][:, 1], iy[:, 0])
    ri = edge(sides["right"], m["Ey"][:, -1], m["Ey"][:, -2], iy[:, -1])
    return dict(m, Ex=torch.cat([lo[None], ix, hi[None]]), Ey=torch.cat([le[:, None], iy, ri[:, None]], 1), Hz=H,
                vx=vx, vy=vy)


def _sample(m, inc):
    """|E_total|^2 at the nodes: the mean of the squares of the edges that meet there."""
    def nodes(sq, dim):
        a, b = (sq.narrow(dim, s, sq.shape[dim] - 1) for s in (0, 1))
        return torch.cat([sq.narrow(dim, 0, 1), 0.5 * (a + b), sq.narrow(dim, sq.shape[dim] - 1, 1)], dim)
    return nodes(m["Ex"] ** 2, 1) + nodes((m["Ey"] + inc) ** 2, 0)


def _line(old, new, start, count, r, frac):
    """A coarse tangential E line at the r fine samples of each of its cells."""
    s = torch.arange(count, device=old.device)
    num = 2 * s + 1 - r
    cell = torch.div(num, 2 * r, rounding_mode="floor")
    w = (num - cell * 2 * r).double() / (2 * r)
    i = start + cell
    w = torch.where(i < 0, torch.zeros_like(w), torch.where(i > len(old) - 2, torch.ones_like(w), w))
    i = i.clamp(0, len(old) - 2)
    at = [v[i] * (1 - w) + v[i + 1] * w for v in (old, new)]
    return (1 - frac) * at[0] + frac * at[1]


def _rates(c, m, S, N, s_nu):
    nu_m, w = 5.3e9 * c["p"], 2 * math.pi * FREQ
    x = torch.sqrt(S / N / (1 + (w / nu_m) ** 2)) / (100.0 * c["p"])
    pos = x > 0
    nu = torch.where(pos, s_nu * 5.14e11 * c["p"] * torch.exp(-73.0 * torch.where(pos, x, torch.ones_like(x)) ** -0.44),
                     torch.zeros_like(x))
    De = 0.1 * 760.0 / c["p"]
    wp2 = m["n"] * (QE * QE / (ME * EPS0))
    den = nu * nu_m + wp2
    safe = torch.where(den == 0, torch.ones_like(den), den)
    return nu, torch.where(den == 0, torch.full_like(den, De), (nu * nu_m * De + wp2 * De / 100) / safe)


def _density(c, n, nu, Df, dx):
    fx = 0.5 * (Df[:, 1:] + Df[:, :-1]) * (n[:, 1:] - n[:, :-1])
    fy = 0.5 * (Df[1:] + Df[:-1]) * (n[1:] - n[:-1])
    pad = torch.nn.functional.pad
    lap = pad(fx, (0, 1)) - pad(fx, (1, 0)) + pad(fy, (0, 0, 0, 1)) - pad(fy, (0, 0, 1, 0))
    return n + (lap / dx ** 2 + nu * n - 1e-13 * n * n) / FREQ


def _along(v, start, count, r):
    """A line of node values at the fine nodes of a side."""
    i = start + torch.div(torch.arange(count, device=v.device), r, rounding_mode="floor")
    w = (torch.arange(count, device=v.device) % r).double() / r
    w = torch.where(i > len(v) - 2, torch.ones_like(w), w)
    i = i.clamp(0, len(v) - 2)
    return v[i] * (1 - w) + v[i + 1] * w


def _steps(c, meshes, S, m0, m1, E0, layers):
    """Coarse steps m0 .. m1 - 1 of a period; S: the running E^2 sums per mesh."""
    r, (nx, ny) = c["r"], (c["nx"], c["ny"])
    qc, qf = _coefficients(c, 1), _coefficients(c, r)
    dev = meshes[0]["n"].device
    xc = qc["dx"] * torch.arange(nx + 1, dtype=torch.float64, device=dev)[None]
    outer = dict.fromkeys(("left", "right", "bottom", "top"), "pec" if c["boundary"] else "mur")
    co, fi, S = meshes[0], meshes[1] if r > 1 else None, list(S)
    if r > 1:
        i0, j0, i1, j1 = _rect_of(c)
        nfx, nfy = r * (i1 - i0), r * (j1 - j0)
        xf = qf["dx"] * (r * i0 + torch.arange(nfx + 1, dtype=torch.float64, device=dev))[None]
    for m in range(m0, m1):
        new = _em(co, qc, _incident(c, qc, m, xc, E0), outer, layers)
        if r > 1:
            for k in range(1, r + 1):
                sides = {}
                for sd, on, o, n_, start, count in (
                        ("left", i0 > 0, co["Ey"][:, i0], new["Ey"][:, i0], j0, nfy),
                        ("right", i1 < nx, co["Ey"][:, i1], new["Ey"][:, i1], j0, nfy),
                        ("bottom", j0 > 0, co["Ex"][j0], new["Ex"][j0], i0, nfx),
                        ("top", j1 < ny, co["Ex"][j1], new["Ex"][j1], i0, nfx)):
                    sides[sd] = _line(o, n_, start, count, r, k / r) if on else "mur"
                fi = _em(fi, qf, _incident(c, qf, r * m + k - 1, xf, E0), sides)
                S[1] = S[1] + _sample(fi, _incident(c, qf, r * m + k, xf, E0))
            if c["coupling"] == 0:
                jl, jh = j0 + (j0 > 0), j1 + 1 - (j1 < ny)
                il, ih = i0 + (i0 > 0), i1 + 1 - (i1 < nx)
                ex = fi["Ex"][r * (jl - j0):r * (jh - 1 - j0) + 1:r].reshape(jh - jl, i1 - i0, r).mean(2)
                ey = fi["Ey"][:, r * (il - i0):r * (ih - 1 - i0) + 1:r].reshape(j1 - j0, r, ih - il).mean(1)
                Ex, Ey = new["Ex"].clone(), new["Ey"].clone()
                Ex[jl:jh, i0:i1] = ex
                Ey[j0:j1, il:ih] = ey
                new = dict(new, Ex=Ex, Ey=Ey)
        co = new
        S[0] = S[0] + _sample(co, _incident(c, qc, m + 1, xc, E0))
    return [co] + ([fi] if r > 1 else []), S


def _period_end(c, meshes, S, s_nu):
    r, (nx, ny) = c["r"], (c["nx"], c["ny"])
    new, erms = [], []
    for m, s, rr in zip(meshes, S, (1, r)):
        q = _coefficients(c, rr)
        nu, Df = _rates(c, m, s, q["N"], s_nu)
        new.append(_density(c, m["n"], nu, Df, q["dx"]))
        erms.append(torch.sqrt(s / q["N"]))
    if r > 1:
        i0, j0, i1, j1 = _rect_of(c)
        nc, nf = new[0], new[1].clone()
        rows, cols = nf.shape
        if i1 < nx:
            nf[:, -1] = _along(nc[:, i1], j0, rows, r)
        if i0 > 0:
            nf[:, 0] = _along(nc[:, i0], j0, rows, r)
        if j1 < ny:
            nf[-1] = _along(nc[j1], i0, cols, r)
        if j0 > 0:
            nf[0] = _along(nc[j0], i0, cols, r)
        nc = nc.clone()
        nc[j0:j1 + 1, i0:i1 + 1] = nf[::r, ::r]
        new = [nc, nf]
    return [dict(m, n=n) for m, n in zip(meshes, new)], erms


def _zeros(meshes):
    return [torch.zeros_like(m["n"]) for m in meshes]


def _doubles(meshes):
    return [{q: v.double() for q, v in m.items()} for m in meshes]


def _exact_run(c, meshes, seen=None):
    n_t = 2 * c["n_lambda"]
    dev = meshes[0]["n"].device
    layers = _Layers(c, _coefficients(c, 1), dev) if c["boundary"] else None
    erms = None
    for _ in range(c["periods"]):
        S = _zeros(meshes)
        for quarter in range(4):
            a, b = quarter * n_t // 4, (quarter + 1) * n_t // 4
            meshes, S = _steps(c, meshes, S, a, b, c["E0"], layers)
            if seen is not None and quarter < 3:
                seen.append([{q: m[q] for q in WATCHED} for m in meshes])
        meshes, erms = _period_end(c, meshes, S, 1.0)
    return [dict({q: m[q] for q in EVOLVING}, erms=e) for m, e in zip(meshes, erms)]


def _exact_adjoint(c, seed):
    n_t = 2 * c["n_lambda"]
    n, target = (v.double() for v in _adjoint_inputs(c, seed))
    n.requires_grad_(True)
    E0 = torch.tensor(c["E0"], dtype=torch.float64, device=DEVICE, requires_grad=True)
    s = torch.ones((), dtype=torch.float64, device=DEVICE, requires_grad=True)
    meshes = [{q: torch.zeros_like(v, dtype=torch.float64) for q, v in m.items()} for m in _inputs(c, seed, quiet=True)]
    meshes[-1]["n"] = n
    if c["r"] > 1:
        i0, j0, i1, j1 = _rect_of(c)
        nc = meshes[0]["n"].clone()
        nc[j0:j1 + 1, i0:i1 + 1] = n[::c["r"], ::c["r"]]
        meshes[0]["n"] = nc
    quarter = n_t // 4
    names = [(k, q) for k in _levels(c) for q in EVOLVING]

    def part(m0, E0_, *flat):
        ms = [{} for _ in _levels(c)]
        for (k, q), v in zip(names, flat):
            ms[k][q] = v
        ms, S_ = _steps(c, ms, list(flat[len(names):]), m0, m0 + quarter, E0_, None)
        return tuple(ms[k][q] for k, q in names) + tuple(S_)
    for _ in range(c["periods"]):
        S = _zeros(meshes)
        for a in range(4):
            flat = torch.utils.checkpoint.checkpoint(part, a * quarter, E0, *[meshes[k][q] for k, q in names], *S,
                                                     use_reentrant=False)
            meshes = [{q: flat[names.index((k, q))] for q in EVOLVING} for k in _levels(c)]
            S = list(flat[len(names):])
        meshes, _ = _period_end(c, meshes, S, s)
    out = meshes[0]["n"]
    loss = (((out - target) / c["n_lo"]) ** 2).mean()
    gE0, gs, gn = torch.autograd.grad(loss, (E0, s, n))
    return {"n": out.detach(), "dE0": gE0, "ds": gs, "dn": gn}


def exact(case, seed):
    c = case
    if c["kind"] == "adjoint":
        if c["periods"] * c["n_lambda"] * c["nx"] * c["ny"] > 8 * 32 * 512 * 512:
            return None   # the tape of the plain evaluation takes too long
        return _exact_adjoint(c, seed)
    with torch.no_grad():
        if c["kind"] == "batch":
            got = {q: [] for q in COLLECTED}
            for k, s in enumerate(_sub_cases(c, seed)):
                for m in _exact_run(s, _doubles(_inputs(s, seed + 7919 * k, quiet=True))):
                    for q in COLLECTED:
                        got[q].append(m[q].reshape(-1))
            return {q: torch.cat(v) for q, v in got.items()}
        seen = [] if c["kind"] == "watch" else None
        out = {"fields": _exact_run(c, _doubles(_inputs(c, seed)), seen)}
        if c["r"] > 1:
            out["mask"] = None
        if seen is not None:
            out["seen"] = seen
        return out
