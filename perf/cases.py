"""The work a user of this package has it do, as cases that can be timed and compared.

Each case is one pass through the public entry points (`Context`, `BatchContext`) on
inputs made on the GPU from a seed.  The shapes come from the package's own workloads
(the uniform-field test, the 128^3 and 256^3 Alfven runs, the differentiable run, the
batch of boxes, the sub-cycled step) and from ragged grids and odd packet counts around
them.  Units: c = q = m = dx = 1, so c~ is the ratio c~/c and dt = 0.2 / c~ moves a
packet at most 0.2 cells.

Kinds of pass:
  step      a sort, then four steps (field source, zeroed feedback, fused push), the
            cycle every long run repeats; with "sorted" false the order-free push
  moments   the state-moment grid and the FP64 totals of a set two steps after its sort
  losses    the catastrophic-loss decay with a gathered gas density, on such a set
  subcycle  one global step with per-packet sub-cycling, tiled or order-free
  batch     a sort, then four steps of many independent boxes
  gradient  the checkpointed differentiable run and its gradients
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2111_14704_gb300 as rs

STEPS = 4      # steps between sorts
VA = 1e-4      # Alfven speed
ADV = 0.2      # c~ dt / dx


# ---------------------------------------------------------------------------
# cases

def _step(name, grid, n, **kw):
    c = {"kind": "step", "nx": grid[0], "ny": grid[1], "nz": grid[2], "n": n, "shape": 2,
         "precision": 32, "deterministic": False, "modes": 64, "c_tilde": 0.1, "p_max": 100.0,
         "beam": 0.0, "sorted": True}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    cube = lambda e: (e, e, e)
    return [
        # the smallest runs: one small box, a few thousand packets, all latency and launches
        _step("small_tsc_16", cube(16), 1 << 12, modes=8),
        # the plain method at its test size: FP64, CIC, static uniform fields
        _step("uniform_cic_fp64_32", cube(32), 1 << 18, shape=1, precision=64, modes=0),
        # a box that no tile divides, an odd packet count, linear kernel
        _step("ragged_cic_61x45x97", (61, 45, 97), 1000003, shape=1, modes=16, c_tilde=1 / 30),
        # reproducible deposits, as kept for regression runs
        _step("deterministic_tsc_64", cube(64), 1 << 21, deterministic=True),
        # the FP64 build on the Alfven workload, for checks of the FP32 one
        _step("alfven_tsc_fp64_64", cube(64), 1 << 21, precision=64),
        # the headline run: 128^3, 8 packets per cell, 64 Alfven modes
        _step("alfven_tsc_128", cube(128), 1 << 24),
        # the largest run: a streaming beam in 256^3
        _step("beam_tsc_256", cube(256), 1 << 27, c_tilde=1 / 30, p_max=1000.0, beam=0.3),
        # diagnostics between steps
        {"name": "moments_tsc_128", "kind": "moments", "nx": 128, "ny": 128, "nz": 128,
         "n": 1 << 24, "shape": 2, "precision": 32, "c_tilde": 0.1},
        # the loss term of a run with gas
        {"name": "losses_tsc_128", "kind": "losses", "nx": 128, "ny": 128, "nz": 128,
         "n": 1 << 24, "shape": 2, "precision": 32, "c_tilde": 0.1},
        # a global step at the c~ Courant limit, packets sub-cycled to 0.2 of their limits
        {"name": "subcycle_tiled_128", "kind": "subcycle", "nx": 128, "ny": 128, "nz": 128,
         "n": 1 << 24, "shape": 2, "precision": 32, "c_tilde": 0.1, "tiled": True},
        # a sweep of independent boxes of uneven sizes
        {"name": "batch_512", "kind": "batch", "boxes": 512, "edge_lo": 16, "edge_hi": 64,
         "n_lo": 1 << 12, "n_hi": 1 << 18, "shape": 2, "precision": 32, "shapes": 5},
        # gradients with respect to the fields and the mode amplitudes
        {"name": "gradient_64", "kind": "gradient", "nx": 64, "ny": 64, "nz": 64, "n": 1 << 20,
         "shape": 2, "precision": 32, "c_tilde": 0.1, "modes": 64, "steps": 64, "every": 8},
    ]


def draw(rng):
    def logi(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def grid_n(lo, hi, n_max):
        g = {a: logi(lo, hi) for a in ("nx", "ny", "nz")}
        nodes = g["nx"] * g["ny"] * g["nz"]
        g["n"] = max(1 << 12, min(n_max, int(nodes * math.exp(rng.uniform(math.log(2), math.log(20))))))
        return g

    kind = rng.choice(["step"] * 6 + ["moments", "losses", "subcycle", "batch", "gradient"])
    shape = rng.choice([1, 2, 2])
    ct = math.exp(-rng.uniform(0.0, math.log(100.0)))
    if kind == "step":
        precision = rng.choice([32, 32, 32, 64])
        g = grid_n(12, 200 if precision == 32 else 64, 1 << 25 if precision == 32 else 1 << 22)
        beam = rng.choice([0.0, 0.0, 0.3])
        return {"kind": kind, **g, "shape": shape, "precision": precision,
                "deterministic": rng.random() < 0.2, "modes": rng.choice([0, 8, 32, 64]),
                "c_tilde": ct, "p_max": 1000.0 if beam else 100.0, "beam": beam,
                "sorted": rng.random() < 0.85}
    if kind in ("moments", "losses"):
        return {"kind": kind, **grid_n(12, 160, 1 << 24), "shape": shape,
                "precision": rng.choice([32, 32, 64]), "c_tilde": ct}
    if kind == "subcycle":
        return {"kind": kind, **grid_n(12, 128, 1 << 23), "shape": shape, "precision": 32,
                "c_tilde": ct, "tiled": rng.random() < 0.7}
    if kind == "batch":
        return {"kind": kind, "boxes": logi(8, 384), "edge_lo": 12, "edge_hi": 64, "n_lo": 1 << 12,
                "n_hi": 1 << 18, "shape": shape, "precision": 32, "shapes": rng.randrange(1000)}
    return {"kind": kind, **grid_n(12, 64, 1 << 20), "shape": 2, "precision": rng.choice([32, 32, 64]),
            "c_tilde": ct, "modes": rng.choice([0, 16, 64]), "steps": rng.randrange(8, 33),
            "every": rng.randrange(4, 9)}


# ---------------------------------------------------------------------------
# inputs

def _dtype(precision):
    return torch.float32 if precision == 32 else torch.float64


def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000003 + stream)
    return g


def _packets(grid, n, precision, seed, p_max=100.0, beam=0.0):
    """Uniform positions (offsets exact in FP32), |u| ~ p^-4.5 on [1, p_max], isotropic,
    boosted by `beam` along x; unit weights.  grid: three ints, or three (n,) tensors."""
    dt = _dtype(precision)
    g = _gen(seed, 1)
    rand = lambda: torch.rand(n, dtype=torch.float64, device="cuda", generator=g)
    packed = torch.zeros(n, dtype=torch.int64, device="cuda")
    for a in range(3):
        na = grid[a]
        i = (rand() * na).long()
        hi = na - 1
        i = torch.minimum(i, hi) if isinstance(hi, torch.Tensor) else i.clamp_(max=hi)
        packed |= i << (10 * a)
    off = [torch.rand(n, dtype=torch.float32, device="cuda", generator=g).to(dt) for _ in range(3)]
    p = (1.0 + rand() * (p_max ** -3.5 - 1.0)).pow_(-1.0 / 3.5)
    mu = 2.0 * rand() - 1.0
    phi = 2.0 * math.pi * rand()
    st = torch.sqrt((1.0 - mu * mu).clamp_(min=0.0))
    u = [p * mu, p * st * torch.cos(phi), p * st * torch.sin(phi)]
    if beam:
        gd = 1.0 / math.sqrt(1.0 - beam * beam)
        u[0] = gd * (u[0] + beam * torch.sqrt(1.0 + p * p))
    u = [x.float().to(dt) for x in u]
    return rs.Particles(packed.to(torch.int32), off, u, torch.ones(n, dtype=dt, device="cuda"))


def _modes(n_modes, grid, seed, rms=0.1):
    """Alfven modes: integer wave vectors 0 < |k| <= min(16, edge / 2), equal amplitudes."""
    if not n_modes:
        return None
    r = np.random.default_rng(seed * 7919 + 17)
    kmax = max(1, min(16, min(grid) // 2))
    k = r.integers(-kmax, kmax + 1, size=(64 * n_modes, 3))
    k2 = (k * k).sum(1)
    k = k[(k2 > 0) & (k2 <= kmax * kmax)][:n_modes].astype(np.float64)
    kk = k / np.array(grid)
    e = np.stack([np.zeros(n_modes), kk[:, 2], -kk[:, 1]], 1)
    norm = np.sqrt((e * e).sum(1))
    e = np.where(norm[:, None] > 0, e / np.maximum(norm, 1e-300)[:, None], [0.0, 1.0, 0.0])
    return {"n": k, "e": e, "amp": np.full(n_modes, rms * math.sqrt(2.0 / n_modes)),
            "phase": 2 * math.pi * r.random(n_modes), "sigma": np.where(r.random(n_modes) < 0.5, -1.0, 1.0)}


def _gas(case):
    """Static runs have a uniform gas drift (so E is not 0), the waves carry their own."""
    return (0.0, 0.0, 0.0) if case.get("modes") else (0.0, 0.01, 0.0)


def _grid(case):
    return case["nx"], case["ny"], case["nz"]


def _context(case):
    return rs.Context(rs.Params(*_grid(case), shape=case["shape"], precision=case["precision"],
                                deterministic=int(case.get("deterministic", False)),
                                c_tilde=case["c_tilde"]))


def _boxes(case):
    r = np.random.default_rng(case["shapes"])
    logi = lambda lo, hi: np.rint(np.exp(r.uniform(math.log(lo), math.log(hi), case["boxes"]))).astype(np.int64)
    edge, count = logi(case["edge_lo"], case["edge_hi"]), logi(case["n_lo"], case["n_hi"])
    ct = np.exp(-r.uniform(0.0, math.log(100.0), case["boxes"]))
    rms = r.uniform(0.01, 0.3, case["boxes"])
    return edge, count, ct, rms


def _box_of(count):
    return torch.repeat_interleave(torch.arange(len(count), device="cuda"),
                                   torch.as_tensor(count, device="cuda"))


def _gas_density(case, seed):
    nx, ny, nz = _grid(case)
    return (0.5 + torch.rand((nz, ny, nx), dtype=torch.float64, device="cuda",
                             generator=_gen(seed, 3))).to(_dtype(case["precision"]))


def _feedback_like(case, seed):
    nx, ny, nz = _grid(case)
    return torch.randn((nz, ny, nx, 8), dtype=torch.float64, device="cuda",
                       generator=_gen(seed, 4)).to(_dtype(case["precision"]))


def prepare(case, seed):
    kind, prec = case["kind"], case["precision"]
    s = {"case": dict(case)}
    if kind == "batch":
        edge, count, ct, rms = _boxes(case)
        off = np.concatenate([[0], np.cumsum(count)])
        e = torch.as_tensor(edge, device="cuda")[_box_of(count)]
        s["P"] = _packets((e, e, e), int(off[-1]), prec, seed)
        s["Q"] = rs.Particles.empty(s["P"].n, prec)
        s["ctx"] = rs.BatchContext(rs.Params(2, 2, 2, shape=case["shape"], precision=prec),
                                   np.stack([edge] * 3, 1), ct, ADV / ct, off)
        s["F"], s["fb"] = s["ctx"].grid_tensor(), s["ctx"].grid_tensor()
        for b in range(case["boxes"]):
            m = _modes(64, (int(edge[b]),) * 3, seed * 1009 + b, float(rms[b]))
            s["ctx"].alfven_fields(b, m, 0.0, 1.0, VA, (0.0, 0.0, 0.0), s["F"])
        return s
    ctx = s["ctx"] = _context(case)
    s["P"] = _packets(_grid(case), case["n"], prec, seed, case.get("p_max", 100.0), case.get("beam", 0.0))
    s["modes"] = _modes(case.get("modes", 64), _grid(case), seed)
    s["dt"], s["t"] = ADV / case["c_tilde"], 0.0
    if kind == "gradient":
        s["out"] = {}
        if s["modes"] is None:
            s["F"] = ctx.grid_tensor()
            ctx.alfven_fields(_modes(16, _grid(case), seed), 0.0, 1.0, VA, (0.0, 0.0, 0.0), s["F"])
        return s
    s["Q"] = rs.Particles.empty(case["n"], prec)
    s["F"], s["fb"] = ctx.grid_tensor(), ctx.grid_tensor()
    ctx.alfven_fields(s["modes"], 0.0, 1.0, VA, _gas(dict(case, modes=case.get("modes", 64))), s["F"])
    if kind == "subcycle":
        s["levels"] = torch.zeros(case["n"], dtype=torch.uint8, device="cuda")
    elif kind in ("moments", "losses"):
        ctx.sort(s["P"], s["Q"])
        for _ in range(2):
            ctx.push_gather(s["Q"], s["F"], s["dt"], s["fb"])
        s["fb"] = _feedback_like(case, seed) if kind == "moments" else None
        s["M"] = ctx.grid_tensor() if kind == "moments" else None
        s["nn"] = _gas_density(case, seed) if kind == "losses" else None
    return s


# ---------------------------------------------------------------------------
# one pass

def _set(P):
    return {"cell": P.cell, "off": P.off, "u": P.u, "w": P.w}


def run(state):
    s, case = state, state["case"]
    kind, ctx = case["kind"], s["ctx"]
    if kind == "step":
        if case["sorted"]:
            ctx.sort(s["P"], s["Q"])
            s["P"], s["Q"] = s["Q"], s["P"]
        for _ in range(STEPS):
            if s["modes"] is not None:
                ctx.alfven_fields(s["modes"], s["t"], 1.0, VA, (0.0, 0.0, 0.0), s["F"])
            s["fb"].zero_()
            ctx.push_gather(s["P"], s["F"], s["dt"], s["fb"])
            s["t"] += s["dt"]
        return {**_set(s["P"]), "feedback": s["fb"]}
    if kind == "batch":
        ctx.sort(s["P"], s["Q"])
        s["P"], s["Q"] = s["Q"], s["P"]
        for _ in range(STEPS):
            s["fb"].zero_()
            ctx.push_gather(s["P"], s["F"], s["fb"])
        return {**_set(s["P"]), "feedback": s["fb"]}
    if kind == "moments":
        s["M"].zero_()
        ctx.deposit(s["Q"], s["M"])
        return {"moments": s["M"], "totals": ctx.moments(s["Q"], s["fb"])}
    if kind == "losses":
        ctx.losses(s["Q"], 1e-4, s["dt"], nn=s["nn"])
        return {"w": s["Q"].w}
    if kind == "subcycle":
        s["fb"].zero_()
        dt = 1.0 / case["c_tilde"]
        if not case["tiled"]:
            ctx.push_subcycled(s["P"], s["F"], dt, 0.2, s["fb"], s["levels"])
            return {**_set(s["P"]), "levels": s["levels"], "feedback": s["fb"]}
        counts = ctx.sort_push_subcycled(s["P"], s["Q"], s["F"], dt, 0.2, s["fb"])
        s["P"], s["Q"] = s["Q"], s["P"]
        return {**_set(s["P"]), "levels": counts, "feedback": s["fb"]}
    kw = {"fields": s["F"]} if s["modes"] is None else {"modes": s["modes"], "vA": VA}
    return ctx.gradient(s["P"], case["steps"], s["dt"], checkpoint_every=case["every"], out=s["out"], **kw)


# ---------------------------------------------------------------------------
# bytes and operations

def work(case):
    """Per call: each packet array and each grid read and written once.  Operations: the
    stencil's multiply-adds (gather 6, deposit 8 values per node) and about 200 for the push."""
    kind, es = case["kind"], case["precision"] // 8
    ns = 8 if case["shape"] == 1 else 27
    if kind == "batch":
        edge, count, _, _ = _boxes(case)
        n, nodes = int(count.sum()), int((edge ** 3).sum())
    else:
        n, nodes = case["n"], case["nx"] * case["ny"] * case["nz"]
    read, write, grid = 4 + 7 * es, 4 + 6 * es, 14 * es
    push = n * (read + write) + nodes * grid
    flops = n * (ns * 28 + 200.0)
    sort = n * 2 * read
    if kind in ("step", "batch"):
        b, f = STEPS * push + (sort if case.get("sorted", True) else 0), STEPS * flops
        f += STEPS * nodes * 14.0 * case.get("modes", 0)
    elif kind == "moments":
        b, f = n * (read + 4 * es) + nodes * 16 * es, n * (ns * 16 + 60.0)
    elif kind == "losses":
        b, f = n * (read + es) + nodes * es, n * (ns * 2 + 60.0)
    elif kind == "subcycle":
        b, f = push + (sort if case["tiled"] else 0), 5.0 * flops  # 4 to 8 sub-steps a packet
    else:
        m = case["steps"]
        b = m * (2 * push + n * 12 * es + nodes * 12 * es)
        f = m * (3.0 * flops + n * ns * 54.0 + nodes * 28.0 * case["modes"])
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------------
# the same results in plain torch, FP64

def _axis(f, shape):
    """First stencil node relative to the cell, and the weights along one axis."""
    if shape == 1:
        return torch.zeros_like(f, dtype=torch.int64), [1.0 - f, f]
    hi = f >= 0.5
    d = torch.where(hi, f - 1.0, f)
    return hi.long() - 1, [0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2]


def _stencil(cell, off, dims, base, shape):
    """(node index, weight) of every stencil node of every packet."""
    ax = []
    for a in range(3):
        first, w = _axis(off[a], shape)
        ax.append([((cell[a] + first + k) % dims[a], w[k]) for k in range(len(w))])
    for kz, wz in ax[2]:
        for ky, wy in ax[1]:
            row = (kz * dims[1] + ky) * dims[0] + base
            wyz = wy * wz
            for kx, wx in ax[0]:
                yield row + kx, wx * wyz


def _cross(a, b):
    return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]


def _dot(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]


def _push(cell, off, u, w, F, dims, base, shape, h, adv, scale=1.0):
    """One step: (cell, off, u) after it, the stencil, and the eight densities."""
    st = list(_stencil(cell, off, dims, base, shape))
    f = 0.0
    for node, W in st:
        f = f + W[:, None] * F.index_select(0, node)
    E, B = [f[:, q] for q in range(3)], [f[:, 3 + q] for q in range(3)]
    um = [u[q] + h * E[q] for q in range(3)]
    igm = 1.0 / torch.sqrt(1.0 + _dot(um, um))
    t = [h * igm * B[q] for q in range(3)]
    sf = 2.0 / (1.0 + _dot(t, t))
    cr = _cross(um, t)
    upr = [um[q] + cr[q] for q in range(3)]
    cr = _cross(upr, [sf * t[q] for q in range(3)])
    up = [um[q] + cr[q] for q in range(3)]
    u1 = [up[q] + h * E[q] for q in range(3)]
    ig1 = 1.0 / torch.sqrt(1.0 + _dot(u1, u1))
    sm = [up[q] + um[q] for q in range(3)]
    bb = _cross([0.5 * igm * sm[q] for q in range(3)], B)
    wq = w * scale
    g0 = torch.sqrt(1.0 + _dot(u, u))
    Q = torch.stack([wq] + [wq * u1[q] * ig1 for q in range(3)] + [-wq * (E[q] + bb[q]) for q in range(3)] +
                    [-wq * _dot(E, sm) / (1.0 / ig1 + g0)], 1)
    off1, cell1 = [], []
    for a in range(3):
        o = off[a] + adv * u1[a] * ig1
        k = torch.floor(o.detach())
        off1.append(o - k)
        cell1.append((cell[a] + k.long()) % dims[a])
    return cell1, off1, u1, st, Q


def _unpack(P):
    c = P.cell.long() & 0xFFFFFFFF
    return ([(c >> (10 * a)) & 1023 for a in range(3)], [x.double() for x in P.off],
            [x.double() for x in P.u], P.w.double())


def _sorted(cell, off, u, w, dims, bin0, edge, shape):
    """Stable order by bin-major anchor key (bins of edge^3 nodes, from bin number bin0)."""
    a = [(cell[q] + (off[q] >= 0.5).long()) % dims[q] if shape == 2 else cell[q] for q in range(3)]
    nb = [(d + edge - 1) // edge for d in dims]
    b, l = [x // edge for x in a], [x % edge for x in a]
    key = (((b[2] * nb[1] + b[1]) * nb[0] + b[0]) + bin0) * edge ** 3 + (l[2] * edge + l[1]) * edge + l[0]
    p = torch.argsort(key, stable=True)
    return [x[p] for x in cell], [x[p] for x in off], [x[p] for x in u], w[p], p


def _fields(grid, modes, t, gas):
    nx, ny, nz = grid
    ar = lambda n: torch.arange(n, dtype=torch.float64, device="cuda")
    z, y, x = ar(nz)[:, None, None], ar(ny)[None, :, None], ar(nx)[None, None, :]
    one = torch.ones((nz, ny, nx), dtype=torch.float64, device="cuda")
    B = [one.clone(), 0.0 * one, 0.0 * one]
    v = [gas[a] * one for a in range(3)]
    if modes is not None:
        amp = modes["amp"]
        for m in range(len(amp)):
            k, e = modes["n"][m].tolist(), modes["e"][m].tolist()
            sg, phase = float(modes["sigma"][m]), float(modes["phase"][m])
            om = sg * 2 * math.pi * k[0] / nx * VA
            ph = 2 * math.pi * (k[0] * x / nx + k[1] * y / ny + k[2] * z / nz) - om * t + phase
            co = (amp[m] if isinstance(amp, torch.Tensor) else float(amp[m])) * torch.cos(ph)
            for a in range(3):
                B[a] = B[a] + e[a] * co
                v[a] = v[a] - sg * VA * e[a] * co
    cr = _cross(v, B)
    return torch.stack([-cr[0], -cr[1], -cr[2], *B], -1).reshape(-1, 6)


CHUNK = 1 << 21  # packets at a time


def _cuts(n):
    return [slice(i, min(n, i + CHUNK)) for i in range(0, n, CHUNK)]


def _cut(v, c):
    return [x[c] if isinstance(x, torch.Tensor) else x for x in v]


def _steps(cell, off, u, w, fields_at, dims, base, shape, steps, nodes):
    """`steps` steps; returns the momenta and the last step's feedback grid."""
    for k in range(steps):
        F = fields_at(k)
        G = torch.zeros((nodes, 8), dtype=torch.float64, device="cuda")
        new = []
        for c in _cuts(w.numel()):
            b = base[c] if isinstance(base, torch.Tensor) else base
            c1, o1, u1, st, Q = _push(_cut(cell, c), _cut(off, c), _cut(u, c), w[c], F, _cut(dims, c), b,
                                      shape, 0.5 * ADV, ADV)
            if k == steps - 1:
                for node, W in st:
                    G.index_add_(0, node, W[:, None] * Q)
            new.append((c1, o1, u1))
        cell, off, u = ([torch.cat([x[i][a] for x in new]) for a in range(3)] for i in range(3))
    return cell, off, u, G


def exact(case, seed):
    kind = case["kind"]
    nodes = case.get("nx", 0) * case.get("ny", 0) * case.get("nz", 0)
    with torch.no_grad():
        if kind == "batch":
            return _exact_batch(case, seed)
        if kind == "gradient":
            return _exact_gradient(case, seed, nodes)
        if case["n"] > 1 << 25:
            return None
        grid, shape = _grid(case), case["shape"]
        P = _packets(grid, case["n"], case["precision"], seed, case.get("p_max", 100.0), case.get("beam", 0.0))
        cell, off, u, w = _unpack(P)
        modes = _modes(case.get("modes", 64), grid, seed)
        dt = ADV / case["c_tilde"]
        gshape = (case["nz"], case["ny"], case["nx"], 8)
        edge = 8 if case["precision"] == 32 else 4
        F0 = _fields(grid, modes, 0.0, _gas(dict(case, modes=case.get("modes", 64))))
        if kind == "step":
            if case["sorted"]:
                cell, off, u, w, _ = _sorted(cell, off, u, w, grid, 0, edge, shape)
            at = (lambda k: F0) if modes is None else (lambda k: _fields(grid, modes, k * dt, (0.0, 0.0, 0.0)))
            _, _, u, G = _steps(cell, off, u, w, at, grid, 0, shape, STEPS, nodes)
            # cells and offsets jump where a packet sits on a face: no values for them
            return {"cell": None, "off": [None] * 3, "u": u, "w": w, "feedback": G.reshape(gshape)}
        if kind == "subcycle":
            return {"cell": None, "off": [None] * 3, "u": [None] * 3, "w": None, "levels": None,
                    "feedback": _exact_subcycle(case, cell, off, u, w, F0, nodes).reshape(gshape)}
        cell, off, u, w, _ = _sorted(cell, off, u, w, grid, 0, edge, shape)
        cell, off, u, _ = _steps(cell, off, u, w, lambda k: F0, grid, 0, shape, 2, nodes)
        if kind == "moments":
            G = torch.zeros((nodes, 8), dtype=torch.float64, device="cuda")
            g = torch.sqrt(1.0 + _dot(u, u))
            Q = torch.stack([w] + [w * x for x in u] + [w * g] + [w * x / g for x in u], 1)
            for c in _cuts(w.numel()):
                for node, W in _stencil(_cut(cell, c), _cut(off, c), grid, 0, shape):
                    G.index_add_(0, node, W[:, None] * Q[c])
            tot = torch.cat([Q.sum(0), _feedback_like(case, seed).double().reshape(-1, 8).sum(0)])
            return {"moments": G.reshape(gshape), "totals": tot.cpu().numpy()}
        nn = _gas_density(case, seed).double().reshape(-1)
        out = []
        for c in _cuts(w.numel()):
            dens = sum(W * nn[node] for node, W in _stencil(_cut(cell, c), _cut(off, c), grid, 0, shape))
            uu = _dot(_cut(u, c), _cut(u, c))
            out.append(w[c] * torch.exp(-case["c_tilde"] * 1e-4 * dt * torch.sqrt(uu / (1.0 + uu)) * dens))
        return {"w": torch.cat(out)}


def _exact_subcycle(case, cell, off, u, w, F, nodes):
    """Feedback of one global step: levels from the gyration and crossing limits at its
    start, 2^level sub-steps each.  (A packet whose limit lies within rounding of a power
    of two may take another level in FP32, so the packets themselves have no exact value.)"""
    ct, grid, shape, dt = case["c_tilde"], _grid(case), case["shape"], 1.0 / case["c_tilde"]
    G = torch.zeros((nodes, 8), dtype=torch.float64, device="cuda")
    for c in _cuts(w.numel()):
        ce, o, v, ww = _cut(cell, c), _cut(off, c), _cut(u, c), w[c]
        B = 0.0
        for node, W in _stencil(ce, o, grid, 0, shape):
            B = B + W[:, None] * F.index_select(0, node)[:, 3:]
        g = torch.sqrt(1.0 + _dot(v, v))
        lim = torch.minimum(g / (ct * B.norm(dim=1)), g / torch.sqrt(_dot(v, v)) / ct) * 0.2
        level = torch.ceil(torch.log2(dt / lim)).clamp_(0, 8).long()
        for k in range(9):
            sel = torch.nonzero(level == k).reshape(-1)
            if not sel.numel():
                continue
            a, b, d, ws = _cut(ce, sel), _cut(o, sel), _cut(v, sel), ww[sel]
            sc = 2.0 ** -k
            for _ in range(1 << k):
                a, b, d, st, Q = _push(a, b, d, ws, F, grid, 0, shape, 0.5 * sc, sc, sc)
                for node, W in st:
                    G.index_add_(0, node, W[:, None] * Q)
    return G


def _exact_batch(case, seed):
    edge, count, ct, rms = _boxes(case)
    off0 = np.concatenate([[0], np.cumsum(edge ** 3)])
    box = _box_of(count)
    at = lambda v: torch.as_tensor(v, device="cuda")[box]
    e = at(edge)
    P = _packets((e, e, e), int(count.sum()), case["precision"], seed)
    nb = (edge + 7) // 8
    cell, off, u, w, p = _sorted(*_unpack(P), (e, e, e), at(np.concatenate([[0], np.cumsum(nb ** 3)])[:-1]),
                                 8, case["shape"])
    e, base = e[p], at(off0[:-1])[p]
    F = torch.cat([_fields((int(edge[b]),) * 3, _modes(64, (int(edge[b]),) * 3, seed * 1009 + b, float(rms[b])),
                           0.0, (0.0, 0.0, 0.0)) for b in range(case["boxes"])])
    _, _, u, G = _steps(cell, off, u, w, lambda k: F, (e, e, e), base, case["shape"], STEPS, int(off0[-1]))
    return {"cell": None, "off": [None] * 3, "u": u, "w": w, "feedback": G}


def _exact_gradient(case, seed, nodes):
    grid, shape, steps = _grid(case), case["shape"], case["steps"]
    cell, off, u, w = _unpack(_packets(grid, case["n"], case["precision"], seed))
    modes = _modes(case["modes"], grid, seed)
    dt = ADV / case["c_tilde"]
    static = _fields(grid, _modes(16, grid, seed), 0.0, (0.0, 0.0, 0.0)) if modes is None else None
    with torch.enable_grad():
        dF = torch.zeros((nodes, 6), dtype=torch.float64, device="cuda", requires_grad=True)
        amp = None
        if modes is not None:
            amp = torch.tensor(modes["amp"], device="cuda", requires_grad=True)

        def fields(k):
            m = static if modes is None else _fields(grid, dict(modes, amp=amp), k * dt, (0.0, 0.0, 0.0))
            return m + dF

        def one(k, cell, o, v, F):
            c1, o1, u1, st, Q = _push(cell, o, v, w, F, grid, 0, shape, 0.5 * ADV, ADV)
            G = torch.zeros((nodes, 8), dtype=torch.float64, device="cuda")
            for node, W in st:
                G = G.index_add(0, node, W[:, None] * Q)
            return c1, o1, u1, G

        # forward without a graph, keeping every step's start
        starts, total = [], torch.zeros((nodes, 8), dtype=torch.float64, device="cuda")
        with torch.no_grad():
            for k in range(steps):
                starts.append((cell, off, u))
                cell, off, u, G = one(k, cell, off, u, fields(k))
                total += G
        L = total[:, 4:7].norm()
        gbar = torch.zeros_like(total)
        gbar[:, 4:7] = total[:, 4:7] / L
        bar = [torch.zeros_like(x) for x in off + u]
        f_bar = torch.zeros((nodes, 6), dtype=torch.float64, device="cuda")
        a_bar = None if amp is None else torch.zeros_like(amp)
        for k in reversed(range(steps)):  # step by step, from the last
            c0, o0, u0 = starts[k]
            x = [t.detach().requires_grad_() for t in o0 + u0]
            with torch.no_grad():
                Fk = fields(k)
            Fk = Fk.detach().requires_grad_()
            _, o1, u1, G = one(k, c0, x[:3], x[3:], Fk)
            got = torch.autograd.grad(o1 + u1 + [G], x + [Fk], bar + [gbar])
            bar = list(got[:6])
            f_bar += got[6]
            if amp is not None:
                a_bar += torch.autograd.grad(fields(k), amp, got[6])[0]
    gshape = (case["nz"], case["ny"], case["nx"], 8)
    out = {"feedback": total.reshape(gshape), "loss": torch.stack([L, 1.0 / L]).detach(),
           "field_bar": torch.cat([f_bar, torch.zeros_like(f_bar[:, :2])], 1).reshape(gshape)}
    if amp is not None:
        out["amp_bar"] = a_bar
    return out
