"""The reaction's chunks and the drag's blocks change size with the particle
count: forces summed per cell and the diagnostics, on both sides of every
change, against plain FP64 sums of the forces the step returns."""
import math

import numpy as np
import pytest

import synth
from parity_util import to_dev

pytestmark = pytest.mark.gpu

# chunks change at 2^15, 2^16, 2^17; blocks at 8 SM counts of 32, 64 and 128 threads (152 SMs)
SIZES = (1, 31, 33, 257, 2**15 - 1, 2**15, 8 * 152 * 32, 8 * 152 * 32 + 1, 2**16 - 1, 2**16, 8 * 152 * 64 + 1,
         2**17 - 1, 2**17, 8 * 152 * 128 + 1)


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("fp64,ordered", [(False, False), (False, True), (True, False), (True, True)])
def test_sums_on_both_sides_of_every_size(cuda_lib, n, fp64, ordered):
    import torch
    cg = cuda_lib
    r, nb = 2, (13, 9, 11)
    desc = synth.make_desc((0.0, 0.0, 0.0), (1.3, 0.9, 1.1), [r * m for m in nb], r, fp64=fp64, law=0, interp=0,
                           gravity=(0.0, 0.0, 0.0))
    rng = synth.rng_for(n, 5)
    T = np.float64 if fp64 else np.float32
    pos = np.empty((n, 4), T)
    # half of the particles in one corner: cells of one and of thousands
    pos[:, :3] = np.array(desc["extent"]) * rng.random((n, 3)) * np.where(rng.random((n, 1)) < 0.5, 0.2, 0.999)
    pos[:, 3] = 0.004 + 0.004 * rng.random(n)
    vel = (0.05 * rng.standard_normal((n, 4))).astype(T)
    g = cg.Grids(desc)
    u = to_dev((0.5 + 0.02 * rng.standard_normal((3, g.n_fine))).astype(T))
    p, v = to_dev(pos), to_dev(vel)
    out = g.alloc_outputs(n, bins=True)
    if ordered:
        po, vo = torch.empty_like(p), torch.empty_like(v)
        g.cg_step_sorted(p, v, po, vo, u, out)
    else:
        g.cg_step(p, v, u, out)
    torch.cuda.synchronize()
    F = out["force"].double().reshape(3, n)
    mag = F.abs()
    ulp = 2.0**-53 if fp64 else 2.0**-24
    VB = math.prod(desc["extent"]) / math.prod(nb)
    cell = out["cell"].long()
    want = torch.zeros(3, math.prod(nb), dtype=torch.float64, device="cuda").index_add_(1, cell, F)
    size = torch.zeros_like(want).index_add_(1, cell, mag)
    # a round's scan has five roundings, the running sum is compensated, the
    # division by V_B adds two; FP64: the plain sums here round once per addend
    most = int(torch.bincount(cell).max())
    tol = 10 * ulp if not fp64 else (10 + most) * ulp
    assert bool(((out["S_bulk"].double().reshape(3, -1) * VB + want).abs() <= tol * size).all())
    sums = out["sums"].cpu().numpy()
    # a lane adds its slot of every round of its chunk in turn, the rest is compensated
    tol = (12 + most / 32) * ulp if not fp64 else (12 + n) * ulp
    tot, tm = F.sum(1).cpu().numpy(), mag.sum(1).cpu().numpy()
    assert np.all(np.abs(sums[2:5] - tot) <= tol * tm)
    assert sums[15] == g.cg_sync_status()[2][2]
    g.close()


@pytest.mark.parametrize("r", [2, 3, 5])
@pytest.mark.parametrize("fp64,ordered", [(False, False), (False, True), (True, False)])
def test_fields_without_the_sums_are_the_same(cuda_lib, r, fp64, ordered):
    """A step that is given no place for its sums forms none: every other
    output keeps its bits, and so does the clamped count."""
    import torch
    cg = cuda_lib
    nb, n = (6, 5, 7), 20_011
    desc = synth.make_desc((0.0, 0.0, 0.0), (0.6, 0.5, 0.7), [r * m for m in nb], r, fp64=fp64, law=1, interp=0,
                           gravity=(0.0, 0.0, 0.0))
    rng = synth.rng_for(n, 6)
    T = np.float64 if fp64 else np.float32
    pos = np.empty((n, 4), T)
    pos[:, :3] = np.array(desc["extent"]) * rng.random((n, 3)) * 0.999
    pos[:, 3] = 0.012
    vel = (0.05 * rng.standard_normal((n, 4))).astype(T)
    got = []
    for sums in (True, False):
        g = cg.Grids(desc)
        u = to_dev((0.5 + 0.02 * synth.rng_for(n, 7).standard_normal((3, g.n_fine))).astype(T))
        p, v = to_dev(pos), to_dev(vel)
        out = g.alloc_outputs(n, eps_fine=True, bins=True)
        if not sums:
            out["sums"] = None
        for _ in range(2):
            if ordered:
                g.cg_step_sorted(p, v, torch.empty_like(p), torch.empty_like(v), u, out)
            else:
                g.cg_step(p, v, u, out)
        torch.cuda.synchronize()
        got.append(({k: t.clone() for k, t in out.items() if t is not None and k != "sums"}, g.cg_sync_status()))
        g.close()
    assert got[0][1] == got[1][1]
    for k in got[1][0]:
        assert torch.equal(got[0][0][k], got[1][0][k]), k
