"""The work a user of this library has it do, as measurable cases.

A coupled CFD-DEM program calls one coupling step per time step, so most
cases are whole steps over the range of beds, grid ratios, precisions and
options in use; the rest are the batched step, the step and the training of
the learned drag closure, and the maps between grids that are not nested.

``listed()`` gives the cases, ``draw(rng)`` one more of the same ranges,
``prepare`` the inputs and handles a program holds before the call, ``run``
one pass through the public entry points with all its outputs, ``work`` the
bytes and operations a pass cannot do without, and ``exact`` the same
outputs in 64 bits from plain torch.

Beds (drawn on the GPU from the seed; lengths in units where the longest
lateral side of the domain is 1):
  uniform    spheres uniform in the box, N(0, 0.05) velocities, a
             Taylor-Green fluid field;
  packed     a jittered lattice of four spheres per bulk cell and axis,
             filled from the bottom, in lattice order, porosity about 0.44,
             upward inflow with noise;
  clustered  log-normal spheres in 200 Gaussian clusters, in random order,
             over-packed cluster cores, upward inflow, gravity.
"""
import math
import random

import torch

import paper_1807_11834_gb300 as cg

RHO_F, MU_F, RHO_P = 1000.0, 1.0e-3, 2500.0   # water and glass
EPS_SWITCH, EPS_MIN = 0.8, 0.1
DI_FELICE, ERGUN = cg.CG_DRAG_DI_FELICE, cg.CG_DRAG_ERGUN_WEN_YU
DEV = "cuda"


# ------------------------------------------------------------------ cases
def _step(bed, n, fine, ratio, **kw):
    """A coupling step.  order: "caller" (cg_step) or "sorted"
    (cg_step_sorted, two particle buffers used in turn); move: the particles
    are advanced by the step; graph: the step is replayed as a CUDA graph;
    cell: cell values in place of the trilinear interpolation."""
    c = dict(kind="step", bed=bed, n=n, nx=fine[0], ny=fine[1], nz=fine[2], ratio=ratio, fp64=False,
             law=ERGUN if bed == "packed" else DI_FELICE, order="caller", move=True, graph=False, cell=False,
             eps_fine=True, sums=False, implicit=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: ten thousand spheres on a unit cube in double
        # precision, fluid iterations on particles at rest; launches and latency
        dict(_step("uniform", 10_000, (32, 32, 32), 4, fp64=True, move=False, sums=True), name="tiny_fp64"),
        # a small DEM loop that keeps its particles in cell order and replays
        # its step as a graph, as a time loop with fixed buffers does
        dict(_step("clustered", 500_000, (128, 128, 64), 4, order="sorted", graph=True, sums=True),
             name="small_clustered_sorted_graph"),
        # odd sizes throughout: ratio 3, a ragged particle count, uneven axes
        dict(_step("uniform", 700_001, (183, 147, 129), 3), name="ragged_ratio3"),
        # double precision at a middle size, the other correlation, moving
        dict(_step("packed", 1_000_000, (160, 160, 320), 4, fp64=True, sums=True), name="packed_fp64"),
        # the 4M packed bed between two moves of its particles
        dict(_step("packed", 4_000_000, (256, 256, 512), 4, move=False), name="packed_bed"),
        # semi-implicit exchange coefficients for the fluid solver, coarse
        # ratio 2, moving
        dict(_step("packed", 2_000_003, (128, 128, 256), 2, implicit=True), name="packed_implicit"),
        # a DEM code that keeps its own (random) particle order
        dict(_step("clustered", 4_000_000, (256, 256, 128), 4, sums=True), name="medium_clustered_caller"),
        # the largest single-GPU bed, kept in cell order
        dict(_step("clustered", 32_000_000, (512, 512, 256), 4, order="sorted", sums=True), name="clustered_sorted"),
        # a parameter sweep: uneven small instances stepped together
        dict(kind="batch", count=16, n_min=10_000, n_max=1_000_000, plan=0, graph=True, name="batch_16"),
        # a step with the learned closure between two refreshes of its record
        dict(kind="learned", n=2_000_000, nx=192, ny=192, nz=384, ratio=4, act="relu", age=3, name="learned_step"),
        # closure training: minibatches of one pass over the sampled rows
        dict(kind="train", rows=65_536, batches=4, act="gelu", name="closure_train"),
        # both maps between a bulk grid and an offset fine grid
        dict(kind="map", bx=64, by=64, bz=128, fx=250, fy=250, fz=500, comps=3, fp64=False, name="map_offset"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid(rng, cells):
    """Bulk cells per axis of about this many cells, uneven, at least 4."""
    e = cells ** (1.0 / 3.0)
    a, b = _log(rng, 0.7, 1.4), _log(rng, 0.7, 1.4)
    return [max(4, int(round(v))) for v in (e * a, e * b, e / (a * b))]


def draw(rng):
    kind = rng.choices(["step", "batch", "learned", "train", "map"], [8, 1, 1, 1, 1])[0]
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(4, 24), n_min=10_000, n_max=int(_log(rng, 50_000, 1_000_000)),
                    plan=rng.randrange(1 << 30), graph=rng.random() < 0.5)
    if kind == "train":
        return dict(kind=kind, rows=int(_log(rng, 1_000, 100_000)), batches=rng.randint(1, 6),
                    act=rng.choice(["gelu", "relu"]))
    if kind == "map":
        b = [rng.randint(20, 96) for _ in range(3)]
        f = [int(round(v * _log(rng, 1.3, 4.3))) for v in b]
        return dict(kind=kind, bx=b[0], by=b[1], bz=b[2], fx=f[0], fy=f[1], fz=f[2], comps=rng.randint(1, 4),
                    fp64=rng.random() < 0.25)
    if kind == "learned":
        n = int(_log(rng, 50_000, 4_000_000))
        r = rng.choice([2, 4])
        nb = _grid(rng, min(2 ** 19, n / _log(rng, 8, 40)))
        return dict(kind=kind, n=n, nx=nb[0] * r, ny=nb[1] * r, nz=nb[2] * r, ratio=r,
                    act=rng.choice(["gelu", "relu"]), age=rng.randint(1, 9))
    bed = rng.choice(["uniform", "packed", "clustered"])
    fp64 = rng.random() < 0.25
    r = rng.choices([2, 3, 4, 5, 8], [3, 1, 8, 1, 2])[0]
    n = int(_log(rng, 10_000, 2_000_000 if fp64 else 16_000_000))
    # spheres per bulk cell from dilute to dense, and at most 40M fine cells
    cells = max(64.0, min(n / _log(rng, 4, 60), 4.0e7 / r ** 3, 2.0 ** 20))
    nb = _grid(rng, cells)
    order = rng.choice(["caller", "sorted"])
    return _step(bed, n, [v * r for v in nb], r, fp64=fp64, order=order,
                 move=order == "sorted" or rng.random() < 0.7, law=rng.choice([DI_FELICE, ERGUN]),
                 cell=rng.random() < 0.1, eps_fine=rng.random() < 0.7, sums=fp64,
                 implicit=order == "caller" and rng.random() < 0.15)


# ------------------------------------------------------------------ inputs
def _gen(seed, k=0):
    return torch.Generator(device=DEV).manual_seed(1000 * int(seed) + k)


def _desc(c):
    """The coupling problem of a case: cubic bulk cells, the longer lateral side 1."""
    r = c["ratio"]
    h = 1.0 / max(c["nx"], c["ny"])
    return dict(origin=(0.0, 0.0, 0.0), extent=(h * c["nx"], h * c["ny"], h * c["nz"]),
                fine_n=(c["nx"], c["ny"], c["nz"]), ratio=r, fp64=c.get("fp64", False), law=c.get("law", DI_FELICE),
                interp=cg.CG_INTERP_CELL if c.get("cell") else cg.CG_INTERP_TRILINEAR, rho_f=RHO_F, mu_f=MU_F,
                rho_p=RHO_P, eps_switch=EPS_SWITCH, eps_min=EPS_MIN,
                gravity=(0.0, 0.0, -9.81) if c.get("bed") == "clustered" else (0.0, 0.0, 0.0))


def _taylor_green(d):
    nx, ny, nz = d["fine_n"]
    ax = [(torch.arange(m, device=DEV, dtype=torch.float64) + 0.5) * (L / m) for m, L in zip(d["fine_n"], d["extent"])]
    sx, cx, sy, cy, cz = ax[0].sin(), ax[0].cos(), ax[1].sin(), ax[1].cos(), ax[2].cos()
    u = torch.zeros(3, nz, ny, nx, device=DEV, dtype=torch.float64)
    u[0] = 0.1 * cz[:, None, None] * cy[None, :, None] * sx[None, None, :]
    u[1] = -0.1 * cz[:, None, None] * sy[None, :, None] * cx[None, None, :]
    return u.reshape(3, -1)


def _inflow(d, gen, dtype):
    n = d["fine_n"][0] * d["fine_n"][1] * d["fine_n"][2]
    u = torch.randn(3, n, device=DEV, dtype=dtype, generator=gen).mul_(0.02)
    u[2] += 0.5
    return u


def _particles(bed, n, d, gen, move):
    """(pos_d [n][4], vel [n][4], time step) in float64."""
    f64 = dict(device=DEV, dtype=torch.float64)
    L = torch.tensor(d["extent"], **f64)
    H = d["extent"][0] * d["ratio"] / d["fine_n"][0]
    pos = torch.empty(n, 4, **f64)
    vel = torch.zeros(n, 4, **f64)
    if bed == "uniform":
        dm = 0.08 * H
        pos[:, :3] = torch.rand(n, 3, generator=gen, **f64) * L
        pos[:, 3] = dm
        vel[:, :3] = torch.randn(n, 3, generator=gen, **f64) * 0.05
    elif bed == "packed":
        nb = [m // d["ratio"] for m in d["fine_n"]]
        s = 4   # lattice sites per bulk cell and axis; more when the bed would not fit
        while n > (s ** 3) * nb[0] * nb[1] * nb[2]:
            s += 1
        dm = 1.024 * H / s
        q = torch.arange(n, device=DEV)
        ijk = torch.stack([q % (nb[0] * s), q // (nb[0] * s) % (nb[1] * s), q // (nb[0] * nb[1] * s * s)], 1)
        jit = (torch.rand(n, 3, generator=gen, **f64) * 2 - 1) * 0.75
        pos[:, :3] = torch.minimum(((ijk + 0.5 + jit) * (H / s)).clamp_(min=0.0), L)
        pos[:, 3] = dm
        if move:
            vel[:, :3] = torch.randn(n, 3, generator=gen, **f64) * 0.02
    else:
        dm = 0.256 * H
        centres = torch.rand(200, 3, generator=gen, **f64) * L
        at = centres[torch.randint(0, 200, (n,), device=DEV, generator=gen)]
        xyz = at + torch.randn(n, 3, generator=gen, **f64) * 0.05
        bad = ((xyz < 0) | (xyz > L)).any(1).nonzero()[:, 0]
        while bad.numel():
            xyz[bad] = at[bad] + torch.randn(bad.numel(), 3, generator=gen, **f64) * 0.05
            bad = bad[((xyz[bad] < 0) | (xyz[bad] > L)).any(1)]
        pos[:, :3] = xyz
        pos[:, 3] = dm * torch.exp(0.3 * torch.randn(n, generator=gen, **f64))
        # a developed bed: the particles already move with the flow
        vel[:, :3] = torch.randn(n, 3, generator=gen, **f64) * 0.02
        vel[:, 2] += 0.3
    # a time step that keeps the explicit advance of the smallest spheres in
    # over-packed cells stable however many steps are taken
    return pos, vel, 0.02 * dm if move else 0.0


def _bed(c, seed):
    d = _desc(c)
    T = torch.float64 if c["fp64"] else torch.float32
    gen = _gen(seed)
    pos, vel, dt = _particles(c["bed"], c["n"], d, gen, c["move"])
    u = (_taylor_green(d) if c["bed"] == "uniform" else _inflow(d, gen, T)).to(T).contiguous()
    return d, pos.to(T), vel.to(T), u, dt


def _batch_sizes(c):
    """(fine edge, ratio, particles, diameter) per instance, the sweep's plan."""
    rng = random.Random(c["plan"])
    return [(rng.choice([32, 64, 96, 128]), rng.choice([2, 4, 8]), int(_log(rng, c["n_min"], c["n_max"])),
             rng.uniform(0.002, 0.01)) for _ in range(c["count"])]


def _batch_instances(c, seed):
    """(desc, pos, vel, u) per instance."""
    out = []
    for k, (edge, ratio, n, dia) in enumerate(_batch_sizes(c)):
        d = _desc(dict(nx=edge, ny=edge, nz=edge, ratio=ratio))
        pos, vel, _ = _particles("uniform", n, d, _gen(seed, k + 1), False)
        pos[:, 3] = dia
        out.append((d, pos.float(), vel.float(), _taylor_green(d).float().contiguous()))
    return out


FEAT_LO = (0.0, 0.0, 0.0, -2000.0, -2000.0, -2000.0, -0.01)
FEAT_HI = (1.0, 6.0, 4.0, 2000.0, 2000.0, 2000.0, 0.1)


def _network(gen):
    """Closure parameters (float32): small corrections, as trained ones are."""
    def u(*s, b):
        return ((torch.rand(*s, generator=gen, device=DEV, dtype=torch.float64) * 2 - 1) * b).float()
    return dict(W1=u(16, 64, b=0.9), b1=u(64, b=0.1), W2=u(64, 64, b=0.3), b2=u(64, b=0.1), w3=u(64, b=0.02),
                b3=u(1, b=0.01))


def _handle(p, act):
    return cg.Mlp(cg.mlp_pack({k: v.cpu().numpy() for k, v in p.items()}), FEAT_LO, FEAT_HI, activation=act)


def _learned_inputs(c, seed):
    """A moving packed bed, the field of the last refresh and today's field."""
    d, pos, vel, u0, dt = _bed(dict(c, bed="packed", fp64=False, law=ERGUN, move=True), seed)
    gen = _gen(seed, 7)
    u1 = u0 + 0.02 * torch.randn(u0.shape, device=DEV, generator=gen)
    return d, pos, vel, u0, u1, dt, _network(gen)


def _rows(c, seed):
    """Minibatches of closure features (inside the box) and targets."""
    gen = _gen(seed, 3)
    lo, hi = torch.tensor(FEAT_LO, device=DEV), torch.tensor(FEAT_HI, device=DEV)
    out = []
    for _ in range(c["batches"]):
        x = torch.rand(c["rows"], 7, device=DEV, generator=gen)
        f = torch.zeros(c["rows"], 8, device=DEV)
        f[:, :7] = lo + (hi - lo) * x
        t = (2.0 * x[:, 0] - x[:, 1]).sin() + 0.1 * torch.randn(c["rows"], device=DEV, generator=gen)
        out.append((f, t))
    return out, _network(gen)


def _map_grids(c):
    """The bulk box and a fine box that covers it from a small offset."""
    h = 1.0 / max(c["bx"], c["by"])
    L = [h * c[k] for k in ("bx", "by", "bz")]
    return ((0.0, 0.0, 0.0), tuple(L), (c["bx"], c["by"], c["bz"])), \
        (tuple(-0.004 * v for v in L), tuple(1.008 * v for v in L), (c["fx"], c["fy"], c["fz"]))


def _map_fields(c, seed):
    T = torch.float64 if c["fp64"] else torch.float32
    gen = _gen(seed, 5)
    nb, nf = c["bx"] * c["by"] * c["bz"], c["fx"] * c["fy"] * c["fz"]
    return (torch.randn(c["comps"], nf, device=DEV, dtype=T, generator=gen) * 0.1 + 0.5,
            torch.randn(c["comps"], nb, device=DEV, dtype=T, generator=gen))


# ------------------------------------------------------------------ prepare
def prepare(case, seed):
    return dict(step=_prepare_step, batch=_prepare_batch, learned=_prepare_learned, train=_prepare_train,
                map=_prepare_map)[case["kind"]](case, seed)


def _prepare_step(c, seed):
    d, pos, vel, u, dt = _bed(c, seed)
    stream = torch.cuda.Stream() if c["graph"] else None
    g = cg.Grids(d, stream=stream)
    out = g.alloc_outputs(c["n"], eps_fine=c["eps_fine"], implicit=c["implicit"], implicit_fine=c["implicit"])
    if not c["sums"]:
        out["sums"] = None
    s = dict(kind="step", grids=g, bufs=[(pos, vel)], u=u, out=out, dt=dt, turn=0, graphs=None)
    if c["order"] == "sorted":
        out["perm"] = torch.empty(c["n"], device=DEV, dtype=torch.int32)
        s["bufs"].append((torch.empty_like(pos), torch.empty_like(vel)))
    if c["graph"]:
        # one eager call sizes the handle's buffers, then one graph per buffer;
        # the particles go back to their first state
        first = pos.clone(), vel.clone()
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            _call_step(s)
        torch.cuda.synchronize()
        graphs = []
        for _ in range(2):
            gr = torch.cuda.CUDAGraph()
            with torch.cuda.graph(gr, stream=stream):
                _call_step(s)
            graphs.append(gr)
        torch.cuda.synchronize()
        for b, a in zip(s["bufs"][s["turn"]], first):
            b.copy_(a)
        s["graphs"], s["at"] = graphs, 0
        torch.cuda.synchronize()
    return s


def _call_step(s):
    pos, vel = s["bufs"][s["turn"]]
    if len(s["bufs"]) == 1:
        s["grids"].cg_step(pos, vel, s["u"], s["out"], dt=s["dt"])
        return pos, vel
    s["turn"] ^= 1
    po, vo = s["bufs"][s["turn"]]
    s["grids"].cg_step_sorted(pos, vel, po, vo, s["u"], s["out"], dt=s["dt"])
    return po, vo


BATCH_FIELDS = ("eps_bulk", "u_bulk", "var_bulk", "S_bulk", "force", "S_fine", "eps_fine")


def _batch_shapes(d, n):
    """Shape of every output field of an instance."""
    nf = math.prod(d["fine_n"])
    nb = nf // d["ratio"] ** 3
    return dict(eps_bulk=(nb,), u_bulk=(3, nb), var_bulk=(nb,), S_bulk=(3, nb), force=(3, n), S_fine=(3, nf),
                eps_fine=(nf,))


def _pad4(m):
    return (m + 3) // 4 * 4


def _prepare_batch(c, seed):
    """The outputs of a sweep: one array per field, the instances one after
    another in it (each starting at a multiple of four values)."""
    inst = _batch_instances(c, seed)
    shapes = [_batch_shapes(d, pos.shape[0]) for d, pos, _, _ in inst]
    outs = {k: torch.zeros(sum(_pad4(math.prod(s[k])) for s in shapes), device=DEV,
                           dtype=torch.float64 if k == "eps_bulk" else torch.float32) for k in BATCH_FIELDS}
    at = dict.fromkeys(BATCH_FIELDS, 0)
    items = []
    for (d, pos, vel, u), shape in zip(inst, shapes):
        o = {}
        for k in BATCH_FIELDS:
            m = math.prod(shape[k])
            o[k] = outs[k][at[k]:at[k] + m].view(shape[k])
            at[k] += _pad4(m)
        items.append((d, pos, vel, u, o))
    b = cg.Batch(items)
    b.use_graph(c["graph"])
    return dict(kind="batch", batch=b, outs=outs)


def _prepare_learned(c, seed):
    d, pos, vel, u0, u1, dt, net = _learned_inputs(c, seed)
    g = cg.Grids(d)
    out = g.alloc_outputs(c["n"], eps_fine=True)
    out["sums"] = None
    g.cg_average_fine_to_bulk(u0, out["u_bulk"], out["var_bulk"])   # the record of the last refresh
    return dict(kind="learned", grids=g, mlp=_handle(net, c["act"]), pos=pos, vel=vel, u=u1, out=out, dt=dt,
                age=c["age"])


def _prepare_train(c, seed):
    rows, net = _rows(c, seed)
    return dict(kind="train", mlp=_handle(net, c["act"]), rows=rows, loss=torch.zeros(len(rows), device=DEV))


def _prepare_map(c, seed):
    bulk, fine = _map_grids(c)
    u, S = _map_fields(c, seed)
    return dict(kind="map", map=cg.Map(bulk, fine, fp64=c["fp64"]), u=u, S=S,
                ub=u.new_empty(u.shape[0], S.shape[1]), Sf=u.new_empty(u.shape))


# ------------------------------------------------------------------ run
def run(state):
    return dict(step=_run_step, batch=_run_batch, learned=_run_learned, train=_run_train, map=_run_map)[state["kind"]](state)


def _run_step(s):
    if s["graphs"]:
        s["graphs"][s["at"]].replay()
        s["at"] ^= 1
        s["turn"] ^= 1
        pos, vel = s["bufs"][s["turn"]]
    else:
        pos, vel = _call_step(s)
    r = dict(s["out"])
    if s["dt"] > 0.0 or len(s["bufs"]) == 2:
        r["pos"], r["vel"] = pos, vel
    return r


def _run_batch(s):
    s["batch"].step()
    return s["outs"]


def _run_learned(s):
    s["grids"].cg_step_learned(s["pos"], s["vel"], s["u"], s["out"], s["mlp"], s["age"], dt=s["dt"])
    return dict(s["out"], pos=s["pos"], vel=s["vel"])


def _run_train(s):
    """One pass over the minibatches, then the weights as a checkpoint or a
    stopping rule reads them (the last batch's gradient beside them)."""
    m = s["mlp"]
    for k, (f, t) in enumerate(s["rows"]):
        m.train_step(f, t, 1e-4, s["loss"][k:k + 1])
    p, g = m.params(grads=True)
    return dict(params=p, grads=g, loss=s["loss"])


def _run_map(s):
    s["map"].average(s["u"], s["ub"])
    s["map"].project(s["S"], s["Sf"])
    return dict(u_bulk=s["ub"], S_fine=s["Sf"])


# ------------------------------------------------------------------ work
def work(case):
    c, k = case, case["kind"]
    T = 8 if c.get("fp64") else 4
    if k == "train":
        n = c["rows"] * c["batches"]
        return dict(bytes=36.0 * n + 8 * 5313 * c["batches"], flops=6.0 * (7 * 64 + 64 * 64 + 64) * n)
    if k == "map":
        nb, nf = c["bx"] * c["by"] * c["bz"], c["fx"] * c["fy"] * c["fz"]
        return dict(bytes=2.0 * T * c["comps"] * (nb + nf), flops=4.0 * c["comps"] * nf)
    if k == "batch":
        n = nf = nb = 0
        for edge, ratio, m, _ in _batch_sizes(c):
            n, nf, nb = n + m, nf + edge ** 3, nb + (edge // ratio) ** 3
        return dict(bytes=44.0 * n + 28.0 * nf + 36.0 * nb, flops=200.0 * n + 40.0 * nf)
    n, nf = c["n"], c["nx"] * c["ny"] * c["nz"]
    nb = nf // c["ratio"] ** 3
    if k == "learned":
        return dict(bytes=76.0 * n + 28.0 * nf + 40.0 * nb, flops=(2.0 * (7 * 64 + 64 * 64 + 64) + 300) * n + 40.0 * nf)
    b = n * (11.0 * T + (8 * T if c["move"] or c["order"] == "sorted" else 0) + (4 if c["order"] == "sorted" else 0))
    b += nf * T * (6.0 + (1 if c["eps_fine"] else 0) + (4 if c["implicit"] else 0))
    b += nb * (8.0 + 7 * T + (4 * T if c["implicit"] else 0))
    return dict(bytes=b, flops=200.0 * n + 40.0 * nf)


# ------------------------------------------------------------------ exact
def exact(case, seed):
    return dict(step=_exact_step, batch=_exact_batch, learned=_exact_learned, train=_exact_train,
                map=_exact_map)[case["kind"]](case, seed)


CHUNK = 1 << 22


def _cells(d, xyz):
    """Linear bulk cell of each point."""
    nb = [m // d["ratio"] for m in d["fine_n"]]
    i = []
    for a in range(3):
        H = d["extent"][a] / nb[a]
        i.append(torch.floor((xyz[:, a] - d["origin"][a]) / H).clamp_(0, nb[a] - 1).long())
    return i[0] + nb[0] * (i[1] + nb[1] * i[2])


def _stencil(d, xyz):
    """Per axis: lower centre, weight of the upper one, and whether the point
    lies beyond the outer centres."""
    out = []
    for a in range(3):
        m = d["fine_n"][a] // d["ratio"]
        xi = (xyz[:, a] - d["origin"][a]) / (d["extent"][a] / m) - 0.5
        i0 = torch.floor(xi).clamp_(0, m - 2)
        t = xi - i0
        out.append((i0.long(), t.clamp(0.0, 1.0), (t < 0) | (t > 1)))
    return out


def _corners(d, st, field):
    """The eight stencil values [8][...] of a bulk field [cells][k], corner bits x, y, z."""
    nbx, nby = d["fine_n"][0] // d["ratio"], d["fine_n"][1] // d["ratio"]
    (i, _, _), (j, _, _), (k, _, _) = st
    return [field[(i + (q & 1)) + nbx * ((j + (q >> 1 & 1)) + nby * (k + (q >> 2)))] for q in range(8)]


def _trilinear(d, xyz, field):
    if d["interp"] == cg.CG_INTERP_CELL:
        return field[_cells(d, xyz)]
    st = _stencil(d, xyz)
    tx, ty, tz = (s[1][:, None] for s in st)
    v = _corners(d, st, field)
    x = [v[q] + tx * (v[q + 1] - v[q]) for q in (0, 2, 4, 6)]
    y = [x[q] + ty * (x[q + 1] - x[q]) for q in (0, 2)]
    return y[0] + tz * (y[1] - y[0])


def _eps_gradient(d, xyz, eps):
    st = _stencil(d, xyz)
    v = _corners(d, st, eps[:, None])
    g = []
    for a in range(3):
        o = [b for b in range(3) if b != a]
        acc = 0.0
        for q in range(8):
            if q >> a & 1:
                continue
            w = 1.0
            for b in o:
                w = w * (st[b][1] if q >> b & 1 else 1.0 - st[b][1])
            acc = acc + w * (v[q | 1 << a] - v[q])[:, 0]
        H = d["extent"][a] * d["ratio"] / d["fine_n"][a]
        g.append(torch.where(st[a][2], torch.zeros_like(acc), acc / H))
    return torch.stack(g, 1)


def _beta(law, eps, dia, s):
    """Drag factor of a sphere: force = beta slip."""
    if law == DI_FELICE:
        red = RHO_F * eps * dia / MU_F
        Re = red * s
        cds = (0.63 * s.sqrt() + 4.8 / red.sqrt()) ** 2
        chi = torch.where(Re > 0, 3.7 - 0.65 * torch.exp(-0.5 * (1.5 - torch.log10(Re.clamp(min=1e-300))) ** 2),
                          torch.full_like(Re, 3.7))
        return 0.5 * cds * RHO_F * (math.pi / 4) * dia ** 2 * eps ** (2.0 - chi)
    vp = math.pi / 6 * dia ** 3
    ergun = (150.0 * (1 - eps) * MU_F / (eps * dia ** 2) + 1.75 * RHO_F * s / dia) * vp
    eRe = eps * RHO_F * dia * s / MU_F
    cds = torch.where(eRe < 1000.0, 24.0 * MU_F / (eps * RHO_F * dia) * (1 + 0.15 * eRe ** 0.687), 0.44 * s)
    wenyu = 0.75 * cds * eps * RHO_F * eps ** -2.65 / dia * vp
    return torch.where(eps < EPS_SWITCH, ergun, wenyu)


def _average(d, u):
    """Mean and summed variance over the nested fine cells: [3][n_b], [n_b]."""
    r = d["ratio"]
    nb = [m // r for m in d["fine_n"]]
    ub, var = [], 0.0
    for c in range(3):
        v = u[c].double().view(nb[2], r, nb[1], r, nb[0], r)
        m = v.mean((1, 3, 5), keepdim=True)
        var = var + ((v - m) ** 2).mean((1, 3, 5)).reshape(-1)
        ub.append(m.reshape(-1))
    return torch.stack(ub), var


def _project(d, B):
    """Bulk fields [k][n_b] at the fine centres: [k][n_f]."""
    r = d["ratio"]
    nb = [m // r for m in d["fine_n"]]
    out = []
    for b in B:
        v = b.reshape(nb[2], nb[1], nb[0])
        for dim, a in ((2, 0), (1, 1), (0, 2)):
            f = torch.arange(d["fine_n"][a], device=DEV)
            if d["interp"] == cg.CG_INTERP_CELL:
                v = v.index_select(dim, f // r)
                continue
            xi = (f.double() + 0.5) / r - 0.5
            i0 = torch.floor(xi).clamp(0, nb[a] - 2)
            t = (xi - i0).clamp(0.0, 1.0)
            shape = [1, 1, 1]
            shape[dim] = -1
            lo, hi = v.index_select(dim, i0.long()), v.index_select(dim, i0.long() + 1)
            v = lo + t.view(shape) * (hi - lo)
        out.append(v.reshape(-1))
    return torch.stack(out)


def _porosity(d, cell, dia):
    nb = [m // d["ratio"] for m in d["fine_n"]]
    VB = math.prod(d["extent"][a] / nb[a] for a in range(3))
    phi = torch.zeros(math.prod(nb), device=DEV, dtype=torch.float64).index_add_(0, cell, math.pi / 6 * dia ** 3)
    return 1.0 - phi / VB, VB


def _net(p, x, act):
    """The closure on scaled inputs [n][7]."""
    f = torch.nn.functional.gelu if act == "gelu" else torch.relu
    a = f(x @ p["W1"][:7] + p["b1"])
    return f(a @ p["W2"] + p["b2"]) @ p["w3"] + p["b3"]


def _advance(d, x, v, F, dt):
    dia = x[:, 3:]
    u = v[:, :3] + dt * (F / (RHO_P * math.pi / 6 * dia ** 3) + torch.tensor(d["gravity"], device=DEV).double())
    q = x[:, :3] + dt * u
    for a in range(3):
        lo, hi = d["origin"][a], d["origin"][a] + d["extent"][a]
        under, over = q[:, a] < lo, q[:, a] > hi
        q[:, a] = torch.where(under, 2 * lo - q[:, a], torch.where(over, 2 * hi - q[:, a], q[:, a]))
        u[:, a] = torch.where(under | over, -u[:, a], u[:, a])
    return torch.cat([q, dia], 1), torch.cat([u, v[:, 3:]], 1)


def _full_step(d, pos, vel, u, dt, *, eps_fine, sums=False, implicit=False, order="caller", moved=False, record=None,
               net=None, age=0):
    """One coupling step in 64 bits; record and net: with the learned closure
    on that record (u_bulk, var_bulk)."""
    n = pos.shape[0]
    cell = torch.cat([_cells(d, pos[a:a + CHUNK, :3].double()) for a in range(0, n, CHUNK)])
    eps, VB = _porosity(d, cell, pos[:, 3].double())
    ub, var = _average(d, u)
    fresh = torch.cat([eps[:, None], ub.T], 1)
    if record is not None:
        ub, var = record
    b4 = torch.cat([eps[:, None], ub.T], 1)
    nb = eps.numel()
    f64 = dict(device=DEV, dtype=torch.float64)
    F = torch.empty(3, n, **f64)
    P, V = (torch.empty(n, 4, **f64) for _ in range(2)) if moved else (None, None)
    S, A = torch.zeros(nb, 3, **f64), torch.zeros(nb, 4, **f64)
    tot = torch.zeros(cg.CG_NSUMS, **f64)
    for a in range(0, n, CHUNK):
        x, v, cl = pos[a:a + CHUNK].double(), vel[a:a + CHUNK].double(), cell[a:a + CHUNK]
        b = _trilinear(d, x[:, :3], b4)
        e = b[:, 0].clamp(min=EPS_MIN)
        s = b[:, 1:] - v[:, :3]
        smag = s.norm(dim=1)
        beta = _beta(d["law"], e, x[:, 3], smag)
        f = beta[:, None] * s
        if net is not None:
            lo, hi = torch.tensor(FEAT_LO, **f64), torch.tensor(FEAT_HI, **f64)
            Re = RHO_F * e * x[:, 3] * smag / MU_F
            feat = torch.cat([e[:, None], torch.log10(1 + Re)[:, None], smag[:, None],
                              _eps_gradient(d, x[:, :3], eps), _trilinear(d, x[:, :3], var[:, None])], 1)
            q = (feat - lo) / (hi - lo)
            ok = ((q >= 0) & (q <= 1)).all(1, keepdim=True)
            r = _net({k: w.double() for k, w in net[0].items()}, q, net[1])
            sf = _trilinear(d, x[:, :3], fresh)[:, 1:] - v[:, :3]
            plain = _beta(d["law"], e, x[:, 3], sf.norm(dim=1))[:, None] * sf
            f = torch.where(ok, (1 + age * r)[:, None] * f, plain)
        F[:, a:a + CHUNK] = f.T
        S.index_add_(0, cl, f)
        if implicit:
            A.index_add_(0, cl, beta[:, None] * torch.cat([torch.ones_like(v[:, :1]), v[:, :3]], 1))
        x1, v1 = _advance(d, x, v, f, dt) if dt > 0 else (x, v)
        if moved:
            P[a:a + CHUNK], V[a:a + CHUNK] = x1, v1
        if sums:
            vp = math.pi / 6 * x[:, 3] ** 3
            tot[0] += vp.sum()
            tot[2:5] += f.sum(0)
            tot[11] += (beta * smag).sum()
            tot[12:15] += (RHO_P * vp[:, None] * v1[:, :3]).sum(0)
            tot[15] += (b[:, 0] < EPS_MIN).sum()
    S, A = (S / -VB).T, (A / VB).T
    Sf = _project(d, S)
    o = dict(eps_bulk=eps, u_bulk=ub, var_bulk=var, S_bulk=S, force=F, S_fine=Sf,
             eps_fine=_project(d, eps[None])[0] if eps_fine else None, sums=None)
    if sums:
        tot[1] = ((1 - eps) * VB).sum()
        tot[5:8] = S.sum(1) * VB
        tot[8:11] = Sf.sum(1) * VB / d["ratio"] ** 3
        o["sums"] = tot
    if implicit:
        o["implicit_bulk"], o["implicit_fine"] = A, _project(d, A)
    if order == "sorted":
        perm = torch.sort(cell, stable=True)[1]
        o["perm"] = None
        P, V = P[perm], V[perm]
    if moved:
        o["pos"], o["vel"] = P, V
    return o


def _exact_step(c, seed):
    d, pos, vel, u, dt = _bed(c, seed)
    return _full_step(d, pos, vel, u, dt, eps_fine=c["eps_fine"], sums=c["sums"], implicit=c["implicit"],
                      order=c["order"], moved=c["move"] or c["order"] == "sorted")


def _exact_batch(c, seed):
    outs = {k: [] for k in BATCH_FIELDS}
    for d, pos, vel, u in _batch_instances(c, seed):
        o = _full_step(d, pos, vel, u, 0.0, eps_fine=True)
        for k in BATCH_FIELDS:
            v = o[k].reshape(-1)
            outs[k].append(torch.nn.functional.pad(v, (0, _pad4(v.numel()) - v.numel())))
    return {k: torch.cat(v) for k, v in outs.items()}


def _exact_learned(c, seed):
    d, pos, vel, u0, u1, dt, net = _learned_inputs(c, seed)
    return _full_step(d, pos, vel, u1, dt, eps_fine=True, moved=True, record=_average(d, u0), net=(net, c["act"]),
                      age=c["age"])


def _exact_train(c, seed):
    rows, net = _rows(c, seed)
    p = {k: v.double().requires_grad_() for k, v in net.items()}
    lo, hi = torch.tensor(FEAT_LO, device=DEV).double(), torch.tensor(FEAT_HI, device=DEV).double()
    names = ("W1", "b1", "W2", "b2", "w3", "b3")
    m = {k: torch.zeros_like(p[k]) for k in names}
    v = {k: torch.zeros_like(p[k]) for k in names}
    losses = []
    for t, (f, y) in enumerate(rows, 1):
        x = (f[:, :7].double() - lo) / (hi - lo)
        loss = ((_net(p, x, c["act"]) - y.double()) ** 2).mean()
        g = dict(zip(names, torch.autograd.grad(loss, [p[k] for k in names])))
        losses.append(loss.detach())
        with torch.no_grad():
            for k in names:
                m[k] = 0.9 * m[k] + 0.1 * g[k]
                v[k] = 0.999 * v[k] + 0.001 * g[k] ** 2
                p[k] -= 1e-4 * (m[k] / (1 - 0.9 ** t)) / ((v[k] / (1 - 0.999 ** t)).sqrt() + 1e-8)
    flat = lambda q: torch.cat([q[k].detach().reshape(-1) for k in names])   # noqa: E731
    return dict(params=flat(p), grads=flat(g), loss=torch.stack(losses))


def _overlap(R, C, a):
    """Overlap lengths [cells of R][cells of C] along an axis."""
    def edges(G):
        return G[0][a] + torch.arange(G[2][a] + 1, device=DEV, dtype=torch.float64) * (G[1][a] / G[2][a])
    r, q = edges(R), edges(C)
    return (torch.minimum(r[1:, None], q[None, 1:]) - torch.maximum(r[:-1, None], q[None, :-1])).clamp(min=0.0)


def _exact_map(c, seed):
    bulk, fine = _map_grids(c)
    u, S = _map_fields(c, seed)
    W = [_overlap(bulk, fine, a) for a in range(3)]

    def apply(f, shape, M):
        v = f.double().reshape(-1, shape[2], shape[1], shape[0]) @ M[0].T
        v = M[1] @ v
        return torch.einsum("zk,ckyx->czyx", M[2], v).reshape(f.shape[0], -1)
    vol = (W[2].sum(1)[:, None, None] * W[1].sum(1)[:, None] * W[0].sum(1)).reshape(-1)
    Vf = math.prod(fine[1][a] / fine[2][a] for a in range(3))
    return dict(u_bulk=apply(u, fine[2], W) / vol, S_fine=apply(S, bulk[2], [w.T for w in W]) / Vf)
