"""Performance cases of the framework: what a streamer code asks of it.

Each case is a dict of plain values.  ``listed()`` holds the named ones, ``draw(rng)`` gives
another of the same ranges, ``prepare`` makes what a user's program has in hand (inputs on the
GPU, a solver with its mesh, coefficient table and captured plans), ``run`` is one pass through
the public entry points, ``work`` the bytes and operations a pass cannot do without, and
``exact`` the outputs in 64 bits from plain torch where a short independent form exists.

Kinds of case
  boxes    many independent single-box solves, the allocation-free entry point
  uniform  one Poisson solve on a uniform cube of 8^3 boxes (FMG, or V-cycles from phi = 0)
  tree     one octree around a streamer head: an FMG solve, a Heun step, both with the field
           and the time step (the benchmark's step), the fluid kernels alone, or a regrid
  quad     a Heun step of the 2-D / axisymmetric form on its quadtree
  batch    many independent uniform solves of uneven size advanced together
  network  training passes of the warm-start network over recorded samples
"""
import ctypes
import math

import numpy as np
import torch

import paper_1708_08434_gb300 as pkg

Q_E, EPS0 = 1.602176634e-19, 8.8541878128e-12
LENGTH, RADIUS, Z_HEAD, VOLTAGE = 0.016, 0.5e-3, 8.5e-3, 25e3
MOST_BOXES = 230000      # boxes of the largest mesh (the paper's 1e8 cells)
MOST_BATCH = 132000000   # cells of the largest batch
MAX_CYCLES = 50

# boundary types and values by face (-x, +x, -y, +y, -z, +z): the plate gap of the streamer
# runs, a grounded box, a corner of grounded walls, one wall at a voltage
WALLS = {
    "plates": ((0, 0, 0, 0, 1, 1), (0.0, 0.0, 0.0, 0.0, 0.0, 1.0)),
    "box": ((1, 1, 1, 1, 1, 1), (0.0, 0.0, 0.0, 0.0, 0.0, 0.0)),
    "corner": ((1, 0, 1, 0, 1, 0), (0.0, 0.0, 0.0, 0.0, 0.0, 0.0)),
    "wall": ((0, 1, 0, 0, 0, 0), (0.0, 2.0, 0.0, 0.0, 0.0, 0.0)),
}


class _Domain:
    def __init__(self, length, nb, max_level, bc_type, bc_val, dims=3, geom=0):
        self.length, self.nb, self.max_level, self.geom = length, nb, max_level, geom
        self.bc_type, self.bc_val, self.origin = bc_type, bc_val, (0.0,) * dims
        self.lbase = nb.bit_length() - 1


def _tree(name, call, nb, levels, width, reach, tol=1e-8, cycles=MAX_CYCLES, mixed=False, nu1=2, nu2=2):
    return {"name": name, "kind": "tree", "call": call, "nb": nb, "levels": levels, "width": width, "reach": reach,
            "tol": tol, "cycles": cycles, "mixed": mixed, "nu1": nu1, "nu2": nu2}


def listed():
    return [
        # an embedder's smallest call: the potential of a few dozen single boxes, launch and latency alone
        {"name": "boxes_64", "kind": "boxes", "n": 64},
        # a small solve, as in set-up code and convergence studies
        {"name": "uniform32_fmg", "kind": "uniform", "call": "fmg", "side": 32, "walls": "plates", "tol": 1e-8,
         "mixed": False, "nu1": 2, "nu2": 2},
        # the uniform 64^3 configuration: V(2,2) cycles from phi = 0 to 1e-10
        {"name": "uniform64_v22", "kind": "uniform", "call": "solve", "side": 64, "walls": "plates", "tol": 1e-10,
         "mixed": False, "nu1": 2, "nu2": 2},
        # one time step of a small refined mesh (about 200 boxes): early in a run, or a parameter scan
        _tree("small_heun", "heun", 2, 3, 2.0, 6e-3),
        # the benchmark's step on 2.4e6 leaf cells: initial FMG solve, field, time step, one Heun step
        _tree("streamer6_step", "step", 8, 6, 10.0, 4.2e-3),
        # the explicit half of a time step on the same mesh: field, time step, one Euler stage
        _tree("streamer6_fluid", "fluid", 8, 6, 10.0, 4.2e-3),
        # adapting the mesh: criterion, one more level at the head, and the derefinement that takes it back
        _tree("streamer6_regrid", "regrid", 8, 6, 10.0, 4.2e-3),
        # the mixed-precision form at its own configuration (2e7 cells)
        _tree("streamer8_mixed", "fmg", 8, 8, 16.0, 12e-3, mixed=True),
        # the paper's largest mesh (1e8 cells): the potential update of a Heun step
        _tree("streamer9_heun", "heun", 16, 9, 25.0, 12.5e-3),
        # the batched configuration: 256 uneven solves, 32^3 to 128^3
        {"name": "batch_256", "kind": "batch", "n": 256, "lo": 32, "hi": 128, "multiple": 8, "walls": "plates",
         "tol": 1e-8, "nu1": 2, "nu2": 2},
        # an axisymmetric time step with the paper's schedule (two V-cycles per potential update)
        {"name": "axi_heun", "kind": "quad", "geom": 1, "nb": 64, "levels": 8, "width": 12.0, "reach": 8e-3,
         "tol": 0.0, "cycles": 2},
        # training the warm-start network on the samples of a run
        {"name": "network_train", "kind": "network", "n": 4096, "batch": 256, "epochs": 1},
    ]


def _log(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def draw(rng):
    kind = rng.choice(["boxes", "uniform", "uniform", "tree", "tree", "tree", "tree", "quad", "quad", "batch", "batch",
                       "network"])
    nu1, nu2 = rng.choice([(2, 2), (2, 2), (2, 2), (1, 1), (1, 2), (3, 2)])
    if kind == "boxes":
        return {"kind": kind, "n": int(round(_log(rng, 1, 1024)))}
    if kind == "uniform":
        call = rng.choice(["fmg", "solve"])
        return {"kind": kind, "call": call, "side": rng.choice([16, 32, 64, 128]), "walls": rng.choice(sorted(WALLS)),
                "tol": _log(rng, 1e-10, 1e-6), "mixed": rng.random() < 0.25, "nu1": nu1, "nu2": nu2}
    if kind == "tree":
        call = rng.choice(["fmg", "heun", "heun", "step", "fluid", "regrid"])
        tol, cycles = rng.choice([(1e-8, MAX_CYCLES), (_log(rng, 1e-9, 1e-6), MAX_CYCLES), (0.0, 2)])
        while True:
            c = _tree("", call, rng.choice([2, 4, 8, 8, 16]), rng.randint(1, 9), _log(rng, 2.0, 25.0),
                      _log(rng, 2e-3, 12.5e-3), tol, cycles, rng.random() < 0.2, nu1, nu2)
            del c["name"]
            if call == "fmg" and tol == 0.0:
                c["tol"] = 1e-8
            if 60 <= _tree_boxes(c) and _capacity(c) <= MOST_BOXES // (4 if call == "regrid" else 1):
                return c
    if kind == "quad":
        tol, cycles = rng.choice([(1e-8, MAX_CYCLES), (0.0, 2)])
        return {"kind": kind, "geom": rng.choice([0, 1]), "nb": rng.choice([4, 8, 16, 32, 64]),
                "levels": rng.randint(2, 8), "width": _log(rng, 2.0, 12.0), "reach": _log(rng, 2e-3, 8e-3), "tol": tol,
                "cycles": cycles}
    if kind == "batch":
        lo = rng.choice([16, 24, 32, 48, 64])
        hi = min(128, lo * rng.choice([1, 2, 4]))
        c = {"kind": kind, "n": int(round(_log(rng, 1, 256))), "lo": lo, "hi": hi, "multiple": rng.choice([2, 4, 8, 8]),
             "walls": rng.choice(sorted(WALLS)), "tol": _log(rng, 1e-9, 1e-6), "nu1": nu1, "nu2": nu2}
        while int((_batch_sides(c).astype(np.int64) ** 3).sum()) > MOST_BATCH:
            c["n"] = max(1, c["n"] // 2)
        return c
    n = int(round(_log(rng, 200, 4096)))
    return {"kind": kind, "n": n, "batch": min(n, rng.choice([64, 128, 256, 1024])), "epochs": 1}


# ---------------------------------------------------------------------------
# the synthetic streamer: a channel hanging from the top electrode with a
# round head, refined around its surface and towards its tip
# ---------------------------------------------------------------------------
def _surface(da, z, radius=RADIUS, z_head=Z_HEAD):
    """Signed distance to the streamer at distance da from its axis and height z (numpy or torch)."""
    lib = torch if isinstance(da, torch.Tensor) else np
    return lib.where(z >= z_head, da - radius, lib.sqrt(da * da + (z - z_head) ** 2) - radius)


def _near(centres, axis, hb, k, width, reach):
    """Which boxes of side hb (k levels above the base) are to be refined."""
    da = np.sqrt(((centres[:, :-1] - axis) ** 2).sum(1))
    z = centres[:, -1]
    half = math.sqrt(centres.shape[1]) * hb / 2
    tip = np.sqrt(da ** 2 + (z - (Z_HEAD - RADIUS)) ** 2)
    return ((np.abs(_surface(da, z)) < half + width * hb / 8) & (tip < half + reach * 2.0 ** -k)).astype(np.int8)


def _flags(case, dims, axis, level, ijk):
    hb = LENGTH / 2 ** level
    return _near((ijk.astype(np.float64) + 0.5) * hb, axis, hb, level - (case["nb"].bit_length() - 1), case["width"],
                 case["reach"])


def _tree_boxes(case, dims=3):
    """Boxes of the mesh, not counting the requests that proper nesting drops."""
    nb, lbase = case["nb"], case["nb"].bit_length() - 1
    axis = LENGTH / 2 if dims == 3 or not case.get("geom") else 0.0
    total = sum((1 << l) ** dims for l in range(lbase + 1))
    ijk = np.stack(np.meshgrid(*[np.arange(nb)] * dims, indexing="ij"), -1).reshape(-1, dims)
    off = np.stack(np.meshgrid(*[np.arange(2)] * dims, indexing="ij"), -1).reshape(1, -1, dims)
    for level in range(lbase, lbase + case["levels"]):
        ijk = (2 * ijk[_flags(case, dims, axis, level, ijk) > 0][:, None, :] + off).reshape(-1, dims)
        total += len(ijk)
        if not len(ijk) or total > 2 * MOST_BOXES:
            break
    return total


def _capacity(case):
    """Boxes a tree case needs room for: a regrid adds a level."""
    return _tree_boxes(dict(case, levels=case["levels"] + 1) if case["call"] == "regrid" else case)


def _rng(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)


def _centres(level, ij):
    """Cell-centre coordinates of the boxes, one [n, 8^d] tensor per axis (x fastest)."""
    dims = ij.shape[1]
    level, ij = torch.from_numpy(level).cuda(), torch.from_numpy(np.ascontiguousarray(ij)).cuda().double()
    h = LENGTH / (8.0 * torch.pow(2.0, level.double()))
    cell = torch.arange(8 ** dims, device="cuda")
    return [(ij[:, d:d + 1] * 8 + ((cell >> 3 * d) & 7)[None, :] + 0.5) * h[:, None] for d in range(dims)]


def _densities(tables, axis, seed, dims):
    """Electron and ion densities of a streamer whose radius, head and density vary with the seed, over a
    noisy background of 1e13 m^-3."""
    g = _rng(seed)
    j = torch.rand(4, generator=g, device="cuda", dtype=torch.float64).cpu().numpy()
    radius, z_head = RADIUS * (0.95 + 0.1 * j[0]), Z_HEAD + 1e-4 * (j[1] - 0.5)
    x = _centres(tables["level"], tables["ijk" if dims == 3 else "ij"])
    z = x.pop()
    da = (x[0] - axis).abs() if dims == 2 else torch.sqrt((x[0] - axis) ** 2 + (x[1] - axis) ** 2)
    s = _surface(da, z, radius, z_head)
    e = ((s + 50e-6) / 50e-6).clamp(0.0, 1.0)
    ne = 1e19 * (0.9 + 0.2 * j[2]) * (1.0 - e * e * (3.0 - 2.0 * e))
    ne += 2e13 * torch.rand(ne.shape, generator=g, device="cuda", dtype=torch.float64)
    head = (z < z_head) & (s < 0.0) & (s >= -20e-6)
    return ne, ne + torch.where(head, 1e20 * (0.9 + 0.2 * j[3]), 0.0)


def _coefficients():
    e = np.arange(1000) * (35e6 / 999)
    alpha = np.zeros(1000)
    alpha[1:] = 4.3e5 * np.exp(-2e7 / e[1:])
    return {"e_max": 35e6, "mu": np.full(1000, 0.03), "diff": np.full(1000, 0.1), "alpha": alpha}


# ---------------------------------------------------------------------------
# prepare
# ---------------------------------------------------------------------------
def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, seed)


def _prepare_boxes(case, seed):
    n, g = case["n"], _rng(seed)
    f = torch.randn(n, 512, generator=g, device="cuda", dtype=torch.float64)
    bt = torch.randint(0, 2, (n, 6), generator=g, device="cuda", dtype=torch.int32)
    bt[:, 5] |= (bt.sum(1) == 0).int()  # one Dirichlet face at least
    bv = torch.randn(n, 6, generator=g, device="cuda", dtype=torch.float64)
    return {"case": case, "f": f, "bt": bt, "bv": bv, "phi": torch.empty_like(f), "lib": pkg.load()}


def _uniform_rho(case, seed):
    """A Gaussian charge at a seeded place plus 1e-3 noise, as [z][y][x] on the unit cube's cells."""
    n, g = case["side"], _rng(seed)
    c = 0.4 + 0.2 * torch.rand(3, generator=g, device="cuda", dtype=torch.float64)
    x = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n
    e = [torch.exp(-(x - c[d]) ** 2 / (2 * 0.05 ** 2)) for d in range(3)]
    rho = e[2][:, None, None] * e[1][None, :, None] * e[0][None, None, :]
    return rho + 1e-3 * torch.rand(n, n, n, generator=g, device="cuda", dtype=torch.float64)


def _morton_boxes(nb):
    """(i, j, k) of the nb^3 boxes of a uniform level in Morton order (x in bit 0)."""
    m = np.arange(nb ** 3)
    out = np.zeros((nb ** 3, 3), np.int64)
    for b in range(nb.bit_length()):
        for d in range(3):
            out[:, d] |= ((m >> (3 * b + d)) & 1) << b
    return out


def _to_boxes(grid):
    """[z][y][x] cells as [box][cell] in Morton order."""
    nb = grid.shape[0] // 8
    b = grid.view(nb, 8, nb, 8, nb, 8).permute(0, 2, 4, 1, 3, 5).reshape(nb, nb, nb, 512)
    i = torch.from_numpy(_morton_boxes(nb)).cuda()
    return b[i[:, 2], i[:, 1], i[:, 0]].contiguous()


def _solver(dom, boxes, case):
    g = pkg.Solver(dom, boxes, case["nu1"], case["nu2"], pkg.MIXED if case["mixed"] else pkg.FP64)
    g.build_octree()
    return g


def _prepare_uniform(case, seed):
    nb = case["side"] // 8
    g = _solver(_Domain(1.0, nb, 0, *WALLS[case["walls"]]), sum((1 << 3 * l) for l in range(nb.bit_length())), case)
    g.var(pkg.RHO)[-nb ** 3:].copy_(_to_boxes(_uniform_rho(case, seed)))
    return {"case": case, "g": g, "leaves": nb ** 3}


def _prepare_tree(case, seed):
    regrid = case["call"] == "regrid"
    dom = _Domain(LENGTH, case["nb"], case["levels"] + regrid, (0, 0, 0, 0, 1, 1), (0.0, 0.0, 0.0, 0.0, 0.0, VOLTAGE))
    g = _solver(dom, _capacity(case), case)
    for level in range(dom.lbase, dom.lbase + case["levels"]):
        ijk = g.level_ijk(level)
        if not len(ijk):
            break
        g.refine_level(level, _flags(case, 3, LENGTH / 2, level, ijk))
    g.set_table(_coefficients())
    ne, ni = _densities(g.tables(), LENGTH / 2, seed, 3)
    s = {"case": case, "g": g, "ne": ne, "ni": ni}
    if case["call"] in ("fmg", "step"):
        return s
    # the state of a run between two steps: potential solved, field and time step known
    g.var(pkg.NE).copy_(ne)
    g.var(pkg.NI).copy_(ni)
    g.charge_rhs(Q_E, EPS0)
    g.fmg(1e-8, MAX_CYCLES)
    g.compute_field()
    s.update(phi=g.var(pkg.PHI).clone(), emag=g.var(pkg.EMAG).clone(), dt=g.dt_limit(Q_E, EPS0))
    if regrid:
        s["grow"], s["back"] = _regrid_flags(g, case)
    return s


def _regrid_flags(g, case):
    """Flags that refine the leaves around the streamer by one level, and those that take it back: -1 on
    the boxes this adds.  Leaves g on its first mesh."""
    old = g.tables()
    grow = np.zeros(len(old["level"]), np.int8)
    for level in range(case["nb"].bit_length() - 1, len(old["level_offset"]) - 1):
        at = slice(*old["level_offset"][level:level + 2])
        grow[at] = _flags(dict(case, width=2.0), 3, LENGTH / 2, level, old["ijk"][at])
    grow[old["child"][:, 0] >= 0] = 0
    g.regrid(grow)
    new = g.tables()
    had = {(int(l), int(m)) for l, m in zip(old["level"], old["morton"])}
    back = np.array([0 if (int(l), int(m)) in had else -1 for l, m in zip(new["level"], new["morton"])], np.int8)
    g.regrid(back)
    if g.n_boxes != len(old["level"]):
        raise RuntimeError("the regrid was not taken back")
    return grow, back


def _prepare_quad(case, seed):
    axis = 0.0 if case["geom"] else LENGTH / 2
    dom = _Domain(LENGTH, case["nb"], case["levels"], (0, 0, 1, 1), (0.0, 0.0, 0.0, VOLTAGE), 2, case["geom"])
    g = pkg.Quad(dom, _tree_boxes(case, 2))
    for level in range(dom.lbase, dom.lbase + case["levels"]):
        ij = g.level_ij(level)
        if not len(ij):
            break
        g.refine_level(level, _flags(case, 2, axis, level, ij))
    g.set_table(_coefficients())
    ne, ni = _densities(g.tables(), axis, seed, 2)
    g.view(pkg.NE).copy_(ne)
    g.view(pkg.NI).copy_(ni)
    g.charge_rhs(Q_E, EPS0)
    g.fmg(1e-8, MAX_CYCLES)
    g.compute_field()
    return {"case": case, "g": g, "ne": ne, "ni": ni, "phi": g.view(pkg.PHI).clone(), "emag": g.view(pkg.EMAG).clone(),
            "dt": g.dt_limit(Q_E, EPS0)}


def _batch_sides(case):
    """Cells per side of each solve, log-uniform: multiples of case["multiple"] that halve down to a side of
    at most 16."""
    ok = [n for n in range(case["lo"], case["hi"] + 1, 2) if n % case["multiple"] == 0 and _coarsest(n) <= 16]
    u = np.random.default_rng(case["n"] * 1009 + case["lo"]).random(case["n"])
    want = case["lo"] * (case["hi"] / case["lo"]) ** u
    return np.array([min(ok, key=lambda n: abs(n - w)) for w in want], np.int32)


def _coarsest(n):
    while n % 2 == 0 and n > 8:
        n //= 2
    return n


def _batch_rho(n, g):
    """Up to eight Gaussian blobs of charge on the unit cube, [z][y][x]."""
    u = torch.rand(8, 6, generator=g, device="cuda", dtype=torch.float64)
    x = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n
    e = torch.exp(-(x - 0.2 - 0.6 * u[:, :3, None]) ** 2 / (2 * (0.03 + 0.07 * u[:, 3, None, None]) ** 2))
    amp = (0.5 + 0.5 * u[:, 4]) * (u[:, 5] < 0.6)
    amp[0] = 1.0
    return torch.einsum("b,bz,by,bx->zyx", amp, e[:, 2], e[:, 1], e[:, 0])


def _prepare_batch(case, seed):
    b = pkg.Batch(_batch_sides(case), 1.0, *WALLS[case["walls"]], nu1=case["nu1"], nu2=case["nu2"])
    g = _rng(seed)
    for s, n in enumerate(b.sides):
        b.grid(b.rhs, s).copy_(-_batch_rho(int(n), g))
    b.tune(1)
    return {"case": case, "b": b}


def _network_params(r):
    parts = []
    for co, ci in ((16, 2), (16, 16), (1, 16)):
        parts += [r.standard_normal(co * ci * 27) * math.sqrt(2.0 / (ci * 27)), np.zeros(co)]
    return np.concatenate(parts).astype(np.float32)


def _prepare_network(case, seed):
    r, n = np.random.default_rng(seed), case["n"]
    net = pkg.Network(n, n)
    x = r.random((n, 1000, 2), np.float32) * 2 - 1
    net.load_samples(x, 0.3 * r.standard_normal((n, 512), np.float32))
    return {"case": case, "net": net, "p": _network_params(r)}


# ---------------------------------------------------------------------------
# run
# ---------------------------------------------------------------------------
def run(state):
    return globals()["_run_" + state["case"]["kind"]](state, state["case"])


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def _run_boxes(s, case):
    rc = s["lib"].sm_box_solve_noalloc(1.0, case["n"], _ptr(s["bt"]), _ptr(s["bv"]), _ptr(s["f"]), _ptr(s["phi"]),
                                       ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    if rc:
        raise RuntimeError("sm_box_solve_noalloc: %d" % rc)
    return s["phi"]


def _run_uniform(s, case):
    g = s["g"]
    g.charge_rhs(1.0, 1.0, True)
    phi = g.var(pkg.PHI)
    if case["call"] == "fmg":
        g.fmg(case["tol"], MAX_CYCLES)
    else:
        phi.zero_()
        g.solve(case["tol"], MAX_CYCLES)
    return {"phi": phi[-s["leaves"]:], "coarse": phi[:-s["leaves"]]}


def _fields(g, view):
    return {"phi": view(pkg.PHI), "ne": view(pkg.NE), "ni": view(pkg.NI), "emag": view(pkg.EMAG)}


def _restore(s, view):
    view(pkg.NE).copy_(s["ne"])
    view(pkg.NI).copy_(s["ni"])
    if "phi" in s:
        view(pkg.PHI).copy_(s["phi"])
        view(pkg.EMAG).copy_(s["emag"])


def _run_tree(s, case):
    g, call = s["g"], case["call"]
    _restore(s, g.var)
    if call == "fluid":
        g.compute_field()
        dt = g.dt_limit(Q_E, EPS0)
        g.fluid_stage(dt)
        return dict(_fields(g, g.var), dt=dt)
    if call == "regrid":
        flags = g.refine_flags()
        g.regrid(s["grow"])
        grown = {k: v.clone() for k, v in _fields(g, g.var).items()}
        g.regrid(s["back"])
        return dict(_fields(g, g.var), grown=grown, flags=flags)
    if call != "heun":
        g.charge_rhs(Q_E, EPS0)
        g.fmg(case["tol"], case["cycles"])
        if call == "fmg":
            return {"phi": g.var(pkg.PHI)}
        g.compute_field()
        dt = g.dt_limit(Q_E, EPS0)
    else:
        dt = s["dt"]
    _, dt_next, _, _ = g.advance(dt, Q_E, EPS0, case["tol"], case["cycles"])
    return dict(_fields(g, g.var), dt=dt, dt_next=dt_next)


def _run_quad(s, case):
    g = s["g"]
    _restore(s, g.view)
    _, dt_next, _, _ = g.advance(s["dt"], Q_E, EPS0, case["tol"], case["cycles"])
    return dict(_fields(g, g.view), dt_next=dt_next)


def _run_batch(s, case):
    b = s["b"]
    b.phi.zero_()
    b.solve(case["tol"], MAX_CYCLES)
    return [b.phi]


def _run_network(s, case):
    net = s["net"]
    net.set_params(s["p"])
    loss = net.train(case["epochs"], case["batch"], 1e-3)
    return {"params": net.get_params(), "loss": loss}


# ---------------------------------------------------------------------------
# work: inputs read once, outputs written once; operations of the method on
# the leaf cells (a V-cycle: per sweep 8, residual and restriction 10,
# prolongation 4; 8/7 for the coarser levels of a uniform grid)
# ---------------------------------------------------------------------------
def _vcycle_flops(cells, nu):
    return cells * (8.0 * nu + 14.0)


def work(case):
    kind = case["kind"]
    if kind == "boxes":
        return {"bytes": case["n"] * (512 * 16 + 72), "flops": case["n"] * 512 * 6 * 16.0}
    if kind == "uniform":
        cells, nu = case["side"] ** 3, case["nu1"] + case["nu2"]
        cycles = -math.log10(case["tol"]) * (0.6 if case["call"] == "fmg" else 1.0)
        return {"bytes": 16.0 * cells, "flops": max(1.0, cycles) * _vcycle_flops(cells * 8 / 7, nu)}
    if kind == "tree":
        cells, nu = 512.0 * _tree_boxes(case), case["nu1"] + case["nu2"]
        solve = 0.6 * -math.log10(case["tol"]) if case["tol"] else case["cycles"]
        solves = {"fmg": 1, "heun": 2, "step": 3, "fluid": 0, "regrid": 0}[case["call"]]
        stages = {"fmg": 0, "heun": 2, "step": 2, "fluid": 1, "regrid": 0}[case["call"]]
        arrays = {"fmg": 3, "heun": 7, "step": 6, "fluid": 6, "regrid": 12}[case["call"]]
        return {"bytes": 8.0 * arrays * cells, "flops": solves * solve * _vcycle_flops(cells, nu) + 80.0 * stages * cells}
    if kind == "quad":
        cells = 64.0 * _tree_boxes(case, 2)
        solve = 0.6 * -math.log10(case["tol"]) if case["tol"] else case["cycles"]
        return {"bytes": 56.0 * cells, "flops": 2 * solve * _vcycle_flops(cells, 4) + 120.0 * cells}
    if kind == "batch":
        cells = float((_batch_sides(case).astype(np.int64) ** 3).sum())
        return {"bytes": 16.0 * cells, "flops": -math.log10(case["tol"]) * _vcycle_flops(cells * 8 / 7, case["nu1"] + case["nu2"])}
    return {"bytes": case["epochs"] * case["n"] * (2000 * 2 + 512 * 4.0), "flops": case["epochs"] * case["n"] * 512 * 16416 * 3.0}


# ---------------------------------------------------------------------------
# exact: the discrete Poisson problem on a uniform cube in the eigenvectors
# of the one-dimensional second difference.  An adaptive mesh's composite
# problem and Adam's steps in a shuffled order have no such short form.
# ---------------------------------------------------------------------------
def _axis_matrix(n, lo, hi):
    """n x n second difference with ghosts -phi (Dirichlet, 1) or phi (Neumann, 0), unit spacing."""
    a = torch.diag(torch.full((n,), -2.0, dtype=torch.float64))
    i = torch.arange(n - 1)
    a[i, i + 1] = a[i + 1, i] = 1.0
    a[0, 0] += -1.0 if lo else 1.0
    a[-1, -1] += -1.0 if hi else 1.0
    return a


def _poisson(f, h, types, values, eig):
    """phi with (7-point Laplacian) phi = f on one cube, f as [z][y][x]."""
    n = f.shape[0]
    f = f * h * h
    for face in range(6):
        if types[face]:
            d = 2 - face // 2
            f.select(d, n - 1 if face & 1 else 0).sub_(2.0 * values[face])
    lam, vec = [], []
    for a in (2, 1, 0):  # z, y, x
        key = (n, types[2 * a], types[2 * a + 1])
        if key not in eig:
            w, v = torch.linalg.eigh(_axis_matrix(*key))
            eig[key] = w.cuda(), v.cuda()
        lam.append(eig[key][0])
        vec.append(eig[key][1])
    t = _transform(f, vec, True)
    t /= lam[0][:, None, None] + lam[1][None, :, None] + lam[2][None, None, :]
    return _transform(t, vec, False)


def _transform(t, vec, forward):
    for v in vec:  # the first axis moves to the end; three turns restore the order
        t = torch.tensordot(t, v if forward else v.t(), dims=([0], [0]))
    return t


def exact(case, seed):
    kind, eig = case["kind"], {}
    if kind == "boxes":
        s = _prepare_boxes(case, seed)
        bt, bv = s["bt"].cpu().tolist(), s["bv"].cpu().tolist()
        return torch.stack([_poisson(s["f"][p].view(8, 8, 8), 1.0 / 8, bt[p], bv[p], eig).reshape(512)
                            for p in range(case["n"])])
    if kind == "uniform":
        n = case["side"]
        types, values = WALLS[case["walls"]]
        return {"phi": _to_boxes(_poisson(-_uniform_rho(case, seed), 1.0 / n, types, values, eig)), "coarse": None}
    if kind == "batch":
        g, out, end = _rng(seed), [], 0
        types, values = WALLS[case["walls"]]
        for n in _batch_sides(case).tolist():
            out.append(_poisson(-_batch_rho(n, g), 1.0 / n, types, values, eig).reshape(-1))
            end = -(-end // 32) * 32 + n ** 3
            out.append(torch.zeros(-end % 32, dtype=torch.float64, device="cuda"))
        return [torch.cat(out[:-1])]
    return None
