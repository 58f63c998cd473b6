"""The bin rule of the built kernels on the cells' faces: every face of every
axis, points on it and up to three representable numbers to either side, in
both precisions, over grids whose spacing, origin and magnitude the float filter
and the quotient have to get right; binned from scratch, incrementally, and by
the digit sort."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import to_dev, to_np

pytestmark = pytest.mark.gpu

GRIDS = {
    "unit": ((0.0, 0.0, 0.0), (1.0, 1.0, 1.0), (40, 24, 32)),
    "thirds": ((0.1, -0.7, 1.0 / 3.0), (0.7, 1.9, 1.1), (34, 46, 22)),
    "far": ((1000.1, -2047.3, 513.7), (1.0, 1.0, 1.0), (28, 20, 26)),
    "long": ((-3.0, 0.01, 0.0), (6.0, 0.03, 1e-3), (4096, 6, 4)),
    "tiny": ((1e-30, -1e-31, 0.0), (3e-30, 7e-30, 5e-30), (18, 14, 22)),
    "huge": ((1e30, -3e30, 0.0), (3e30, 7e30, 5e30), (18, 14, 22)),
    "quotient_range": ((0.0, -1e-220, 1e-200), (1e-199, 3e-210, 7e-199), (18, 14, 22)),
}


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("name", GRIDS)
def test_points_on_and_next_to_every_face(cuda_lib, name, fp64):
    import torch
    if name == "quotient_range" and not fp64:
        pytest.skip("below the FP32 range")
    origin, extent, fine = GRIDS[name]
    d = synth.make_desc(origin, extent, fine, 2, fp64=fp64, law=synth.DRAG_DI_FELICE)
    T = np.float64 if fp64 else np.float32
    rng = np.random.default_rng(7)
    pts = []
    mid = [origin[a] + 0.5 * extent[a] for a in range(3)]
    for a in range(3):
        nb = fine[a] // 2
        i = np.arange(nb + 1) if nb < 200 else np.unique(np.concatenate([np.arange(40), rng.integers(0, nb + 1, 200), [nb]]))
        face = (origin[a] + i * (extent[a] / nb)).astype(T)
        for k in range(-3, 4):
            f = face.copy()
            for _ in range(abs(k)):
                f = np.nextafter(f, T(np.inf if k > 0 else -np.inf))
            p = np.empty((f.size, 4), T)
            p[:, :3] = np.array(mid, T)
            p[:, a] = f
            pts.append(p)
    extra = np.zeros((6, 4), T)
    extra[0, :3], extra[1, :3] = 0.0, -0.0
    extra[2:, :3] = np.array(origin, T) + np.array(extent, T) * np.array([[-1.0], [2.0], [1e3], [-1e3]], T)
    pos = np.concatenate(pts + [extra]).astype(T)
    pos[:, 3] = 0.0
    want = oracle.bin(d, pos)
    dev = to_dev(pos)
    for digits in (0, 8):
        g = cuda_lib.Grids(dict(d, sort_digits=digits))
        cell = torch.empty(pos.shape[0], dtype=torch.int32, device="cuda")
        perm, cs = torch.empty_like(cell), torch.empty(g.n_bulk + 1, dtype=torch.int32, device="cuda")
        other = dev[torch.randperm(pos.shape[0], device="cuda")].contiguous()
        for p in (dev, other, dev):       # from scratch, then incrementally from another order
            g.cg_bin_particles(p, cell, perm, cs)
        torch.cuda.synchronize()
        for got, ref in zip((cell, perm, cs), want):
            assert np.array_equal(to_np(got), ref), digits
        counts = g.cg_sync_status()[2]
        assert counts[1] == 0
        g.close()
