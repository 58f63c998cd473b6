"""The averages' means are as exact as compensated sums of the values make
them, whatever the values' sign."""
import numpy as np
import pytest

import synth
from parity_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("r", [3, 5, 6, 7])
def test_mean_of_a_field_of_no_mean(cuda_lib, r, fp64):
    """Cell means far below the values: rounding the compensated sum, and its
    quotient by (or product with the rounded reciprocal of) the count, are 3 u
    of the mean, the sum's own residue below (2 u)^2 r^3 of the mean magnitude."""
    import torch
    nb = (13, 9, 11)
    fine = tuple(r * m for m in nb)
    d = synth.make_desc((0, 0, 0), (1, 1, 1), fine, r, fp64=fp64, law=synth.DRAG_DI_FELICE)
    T, u = (np.float64, 2.0 ** -53) if fp64 else (np.float32, 2.0 ** -24)
    f = (0.02 * synth.rng_for(r, 21).standard_normal((3, fine[2], fine[1], fine[0]))).astype(T)
    g = cuda_lib.Grids(d)
    ub = torch.empty(3, g.n_bulk, device="cuda", dtype=g.dtype)
    var = torch.empty(g.n_bulk, device="cuda", dtype=g.dtype)
    g.cg_average_fine_to_bulk(to_dev(f.reshape(3, -1)), ub, var)
    torch.cuda.synchronize()
    g.close()
    # exact sums: the values as integers (float64 of that scale keeps 53 bits of each)
    cells = f.reshape(3, nb[2], r, nb[1], r, nb[0], r).transpose(0, 1, 3, 5, 2, 4, 6).reshape(3, -1, r ** 3)
    scale = 2.0 ** (70 if fp64 else 50)
    want = np.array([[sum(int(float(x) * scale) for x in c) for c in comp] for comp in cells], dtype=object)
    got = ub.cpu().numpy()
    worst = 0.0
    for c in range(3):
        for i in range(want.shape[1]):
            m = float(want[c, i]) / scale / r ** 3
            err = abs(float(got[c, i]) - m)
            bound = 3.0 * u * abs(m) + (2 * u) ** 2 * r ** 3 * float(np.abs(cells[c, i]).mean())
            worst = max(worst, err / bound)
    assert worst <= 1.0, worst
