"""Cells that receive many particles in one incremental binning: their lists of
movers are walked up to the limit, merged above it, and sorted by digits where
more than a warp's registers hold moved, in one part or several."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import inputs, to_dev, to_np

pytestmark = pytest.mark.gpu

FIELDS = ("eps_bulk", "u_bulk", "force", "S_bulk", "S_fine", "eps_fine")


@pytest.mark.parametrize("sorted_step", [False, True])
@pytest.mark.parametrize("stay", [0, 1, 100, 3_900, 4_200, 9_000])
@pytest.mark.parametrize("k", [4, 5, 33, 64, 65, 129, 256, 257, 1_500])
def test_movers_into_a_cell(cuda_lib, k, stay, sorted_step):
    """k particles move into a cell of `stay` (ten of which leave it), among
    them ids below, between and above its own; two thousand move elsewhere, so
    that other cells are crowded too; then nothing moves; then a few leave.  The
    bins are the oracle's and the fields a fresh handle's bit for bit."""
    import torch
    cg = cuda_lib
    w = synth.tiny(seed=3, n=20_011, fp64=False)
    rng = np.random.default_rng([k, stay])
    ids = rng.permutation(w.n)
    w.pos_d[:, 0] = 0.5 + 0.49 * w.pos_d[:, 0]                 # none near the cell
    cell = lambda m: (0.26 + 0.1 * rng.random((m, 3))).astype(np.float32)   # noqa: E731
    w.pos_d[ids[:stay], :3] = cell(stay)
    pos, vel, uf = inputs(w)
    g = cg.Grids(w.desc)
    out = g.alloc_outputs(w.n, eps_fine=True, bins=True)
    po, vo = torch.empty_like(pos), torch.empty_like(vel)
    if sorted_step:
        g.cg_step_sorted(pos, vel, po, vo, uf, out)
        pos, vel, po, vo = po, vo, pos, vel
    else:
        g.cg_step(pos, vel, uf, out)

    def at(rows):   # where these particles stand now
        if not sorted_step:
            return torch.from_numpy(rows).cuda()
        inv = torch.empty(w.n, dtype=torch.long, device="cuda")
        inv[out["perm"].long()] = torch.arange(w.n, device="cuda")
        return inv[torch.from_numpy(rows).cuda()]

    def move(k_in, gone, others, place):
        pos[place[stay:stay + k_in], :3] = to_dev(cell(k_in))
        pos[place[:gone], :3] = to_dev((0.7 + 0.2 * rng.random((gone, 3))).astype(np.float32))
        r = place[-others:] if others else place[:0]
        pos[r, :3] = to_dev(np.stack([0.5 + 0.49 * rng.random(others), rng.random(others), rng.random(others)], 1).astype(np.float32))

    place = at(ids)
    for step, (k_in, gone, others) in enumerate([(k, min(10, stay), 2_000), (0, 0, 0), (0, min(3, stay), 5)]):
        move(k_in, gone, others, place)
        if sorted_step:
            now, nv = pos.clone(), vel.clone()
            g.cg_step_sorted(pos, vel, po, vo, uf, out)
        else:
            now, nv = pos, vel
            g.cg_step(pos, vel, uf, out)
        torch.cuda.synchronize()
        c, perm, cs, _ = oracle.bin(w.desc, to_np(now))
        assert np.array_equal(to_np(out["cell"]), c), step
        assert np.array_equal(to_np(out["perm"]), perm), step
        assert np.array_equal(to_np(out["cell_start"]), cs), step
        f = cg.Grids(w.desc)
        ref = f.alloc_outputs(w.n, eps_fine=True)
        f.cg_step(now.clone(), nv.clone(), uf, ref)
        torch.cuda.synchronize()
        f.close()
        for name in FIELDS:
            assert torch.equal(out[name], ref[name]), (step, name)
        if sorted_step:
            place = at(np.arange(w.n))[place]
            pos, vel, po, vo = po, vo, pos, vel
    g.close()
