"""The incremental binning's branches at their edges, and the porosity formed
while binning: arrivals around the limit of the lists, a change from the
sorted to the caller's order without movers, and spheres outside the
accumulators' fast range."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import TOL_FP32, TOL_FP64, assert_close, inputs, to_dev, to_np

pytestmark = pytest.mark.gpu

FIELDS = ("eps_bulk", "u_bulk", "force", "S_bulk", "S_fine", "eps_fine")


def _fresh(cg, desc, pos, vel, uf, dt=0.0):
    import torch
    g = cg.Grids(desc)
    out = g.alloc_outputs(pos.shape[0], eps_fine=True, bins=True)
    g.cg_step(pos.clone(), vel.clone(), uf, out, dt=dt)
    torch.cuda.synchronize()
    g.close()
    return out


@pytest.mark.parametrize("sorted_step", [False, True])
@pytest.mark.parametrize("k", [1, 31, 32, 33, 34, 300])
def test_arrivals_around_the_list_limit(cuda_lib, k, sorted_step):
    """k particles move into one cell, with a few others elsewhere: the bins
    are the oracle's and the fields a fresh handle's bit for bit, whichever
    side of the limit the cell lies on."""
    import torch
    cg = cuda_lib
    w = synth.tiny(seed=3, n=20_011, fp64=False)
    pos, vel, uf = inputs(w)
    g = cg.Grids(w.desc)
    out = g.alloc_outputs(w.n, eps_fine=True, bins=True)
    po, vo = torch.empty_like(pos), torch.empty_like(vel)
    if sorted_step:
        g.cg_step_sorted(pos, vel, po, vo, uf, out)
        pos, vel = po, vo
    else:
        g.cg_step(pos, vel, uf, out)
    gen = torch.Generator(device="cuda").manual_seed(k)
    idx = torch.randperm(w.n, device="cuda", generator=gen)
    pos[idx[:k], :3] = 0.40 + 0.01 * torch.rand(k, 3, device="cuda", generator=gen)
    pos[idx[k:k + 50], :3] = torch.rand(50, 3, device="cuda", generator=gen)
    if sorted_step:
        p2, v2 = torch.empty_like(pos), torch.empty_like(vel)
        g.cg_step_sorted(pos, vel, p2, v2, uf, out)
    else:
        g.cg_step(pos, vel, uf, out)
    torch.cuda.synchronize()
    cell, perm, cs, _ = oracle.bin(w.desc, to_np(pos))
    assert np.array_equal(to_np(out["cell"]), cell)
    assert np.array_equal(to_np(out["perm"]), perm)
    assert np.array_equal(to_np(out["cell_start"]), cs)
    ref = _fresh(cg, w.desc, pos, vel, uf)
    for f in FIELDS:
        assert torch.equal(out[f], ref[f]), f
    g.close()


def test_caller_order_after_a_sorted_step_without_movers(cuda_lib):
    """A sorted step leaves out the inverse permutation; a step in the caller's
    order that then finds no mover must not use a stale one."""
    import torch
    cg = cuda_lib
    w = synth.small_clustered_bed(seed=4)
    pos, vel, uf = inputs(w)
    g = cg.Grids(w.desc)
    out = g.alloc_outputs(w.n, eps_fine=True, bins=True)
    po, vo = torch.empty_like(pos), torch.empty_like(vel)
    g.cg_step(pos, vel, uf, out)                       # a binning with another inverse
    g.cg_step_sorted(pos, vel, po, vo, uf, out)
    g.cg_step_sorted(po, vo, pos, vel, uf, out)        # identity hint: nothing moved
    p2, v2 = pos.clone(), vel.clone()                  # the same particles in other arrays
    g.cg_step(p2, v2, uf, out)
    torch.cuda.synchronize()
    ref = _fresh(cg, w.desc, p2, v2, uf)
    for f in FIELDS + ("cell", "perm", "cell_start"):
        assert torch.equal(out[f], ref[f]), f
    F, S = torch.empty_like(out["force"]), torch.empty_like(out["S_bulk"])
    g.cg_drag(p2, v2, out["eps_bulk"], out["u_bulk"], F, S)
    torch.cuda.synchronize()
    assert torch.equal(F, out["force"]) and torch.equal(S, out["S_bulk"])
    g.close()


def _eps_by_every_path(cg, w):
    """Porosity of w by a binning from scratch, an incremental one in either
    order, the digit sort, and the deposit entry."""
    import torch
    pos, vel, uf = inputs(w)
    res = {}
    g = cg.Grids(w.desc)
    out = g.alloc_outputs(w.n)
    g.cg_step(pos, vel, uf, out)
    res["scratch"] = to_np(out["eps_bulk"]).copy()
    g.cg_step(pos, vel, uf, out)
    res["incremental"] = to_np(out["eps_bulk"]).copy()
    eps = torch.empty(g.n_bulk, device="cuda", dtype=torch.float64)
    g.cg_deposit(cg.CG_DEP_VOLUME, w.n, pos, eps)
    res["deposit"] = to_np(eps).copy()
    po, vo, p2, v2 = (torch.empty_like(pos) for _ in range(4))
    g.cg_step_sorted(pos, vel, po, vo, uf, out)
    g.cg_step_sorted(po, vo, p2, v2, uf, out)
    res["sorted"] = to_np(out["eps_bulk"]).copy()
    g.close()
    d = dict(w.desc)
    d["sort_digits"] = 8
    g = cg.Grids(d)
    g.cg_step(pos, vel, uf, out)
    res["digits"] = to_np(out["eps_bulk"]).copy()
    g.close()
    return res


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("crowd", [False, True])
def test_porosity_of_any_sphere(cuda_lib, fp64, crowd):
    """Diameters from nothing to many cells (the sums' integer pieces change
    form at 1/8 and 1 of a cell's volume and at 2^32 cells), one per cell or all
    in a few cells: every path gives the same bits, within the path's tolerance
    of the oracle."""
    w = synth.tiny(seed=9, n=6_000, fp64=fp64)
    H = 1.0 / 8
    sizes = np.array([0.0, 1e-7, 1e-3, 0.1, 0.6, 0.62, 0.63, 1.2, 1.24, 1.25, 3.0, 2000.0, 2100.0, 1e5, -0.1]) * H
    if crowd:
        w.pos_d[:, :3] = 0.3 + 0.2 * w.pos_d[:, :3]
        w.pos_d[:4000:7, 3] = 0.63 * H
    else:
        w.pos_d[:sizes.size, 3] = sizes
        w.pos_d[:sizes.size, :3] = (np.stack([np.arange(sizes.size) % 8, np.arange(sizes.size) // 8, np.full(sizes.size, 3)], 1) + 0.5) / 8
    cell, perm, cs, _ = oracle.bin(w.desc, w.pos_d)
    want = oracle.deposit_volume(w.desc, w.pos_d, cs, perm)[0]
    res = _eps_by_every_path(cuda_lib, w)
    for name, eps in res.items():
        assert np.array_equal(eps, res["scratch"]), name
    # cell by cell: the largest sphere's cell says nothing of the others
    err = np.abs(res["scratch"] - want) / np.maximum(np.abs(want), 1.0)
    assert err.max() <= (TOL_FP64 if fp64 else TOL_FP32), err.max()
    # FP32: the sums are good to 2^-46 of phi, far below the path's tolerance
    phi = np.abs(1.0 - want)
    assert (np.abs(res["scratch"] - want) <= 2.0 ** -40 * phi + 2.0 ** -48).all()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_porosity_after_a_bad_diameter(cuda_lib, bad):
    """A diameter that is not finite makes its cell's porosity NaN and no
    other's; the next step, without it, is clean."""
    import torch
    w = synth.tiny(seed=2, n=5_000, fp64=False)
    pos, vel, uf = inputs(w)
    good = pos.clone()
    pos[77, 3] = float(bad)
    g = cuda_lib.Grids(w.desc)
    out = g.alloc_outputs(w.n, bins=True)
    eps = []
    for p in (good, pos, good):
        g.cg_step(p, vel, uf, out)
        eps.append(out["eps_bulk"].clone())
    torch.cuda.synchronize()
    c = int(out["cell"][77])
    assert torch.isnan(eps[1][c]) and int(torch.isnan(eps[1]).sum()) == 1
    other = torch.arange(g.n_bulk, device="cuda") != c
    assert torch.equal(eps[1][other], eps[0][other]) and torch.equal(eps[2], eps[0])
    g.close()


@pytest.mark.parametrize("fp64,interp,law", [(False, 0, 0), (False, 0, 1), (False, 1, 0), (True, 0, 1)])
@pytest.mark.parametrize("n,nb", [(1, (2, 2, 2)), (33, (2, 3, 2)), (5_000, (3, 2, 5)), (20_000, (40, 20, 24)),
                                  (60_001, (17, 9, 13)), (400_003, (33, 16, 12))])
def test_sorted_drag_equals_the_drag_in_the_callers_order(cuda_lib, n, nb, fp64, interp, law):
    """The sorted step's fused drag and reaction over grids from two cells per
    axis on, a particle in many cells to thousands in one, rows shorter and
    longer than a staged window: every field, force and record as cg_step's,
    bit for bit, with and without advancing."""
    import torch
    cg = cuda_lib
    r = 2
    desc = synth.make_desc((-0.3, 0.0, 0.1), (1.0, 0.7, 0.9), [r * m for m in nb], r, fp64=fp64, law=law, interp=interp,
                           gravity=(0.0, 1.0, -9.0))
    rng = synth.rng_for(n, 11)
    T = np.float64 if fp64 else np.float32
    pos = np.empty((n, 4), T)
    pos[:, :3] = np.array(desc["origin"]) + rng.random((n, 3)) * np.array(desc["extent"])
    pos[:, 3] = 0.002
    vel = (0.05 * rng.standard_normal((n, 4))).astype(T)
    g, f = cg.Grids(desc), cg.Grids(desc)
    u = to_dev((0.5 + 0.02 * rng.standard_normal((3, g.n_fine))).astype(T))
    pi, vi = to_dev(pos), to_dev(vel)
    oa = g.alloc_outputs(n, eps_fine=True, bins=True, implicit=True)
    ob = f.alloc_outputs(n, eps_fine=True, bins=True, implicit=True)
    for dt in (0.0, 1e-4, 1e-4, 0.0):
        po, vo = torch.empty_like(pi), torch.empty_like(vi)
        pr, vr = pi.clone(), vi.clone()
        g.cg_step_sorted(pi, vi, po, vo, u, oa, dt=dt)
        f.cg_step(pr, vr, u, ob, dt=dt)
        torch.cuda.synchronize()
        perm = oa["perm"].long()
        assert torch.equal(po, pr[perm]) and torch.equal(vo, vr[perm])
        for k in FIELDS + ("cell", "perm", "cell_start", "implicit_bulk"):
            assert torch.equal(oa[k], ob[k]), (dt, k)
        pi, vi = po, vo
    assert g.cg_sync_status()[:2] == f.cg_sync_status()[:2]
    g.close()
    f.close()
