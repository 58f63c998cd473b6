"""The maps' means over many values are as exact as over few."""
import numpy as np
import pytest

import synth
from parity_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("rows", [3, 7, 512, 4096])
def test_map_average_over_many_values(cuda_lib, rows, axis):
    """FP32 means of positive values over long columns.  The weights, the
    products and sums of each axis, the coverage and the quotient are 13
    roundings, and the plain chains, of up to 16 terms, hardly all err alike: 18
    u, however many values there are (one chain over 4096 is off by 38 u)."""
    import torch
    n = [2, 3, 2]
    n[axis] = 2 * rows
    bulk = ((0.0, 0.0, 0.0), (1.0, 1.0, 1.0), (2, 2, 2))
    fine = ((0.0, 0.0, 0.0), (1.0, 1.0, 1.0), tuple(n))
    f = (0.5 + synth.rng_for(rows, axis).random((2, n[2], n[1], n[0]))).astype(np.float32)
    m = cuda_lib.Map(bulk, fine, fp64=False)
    ub = torch.empty(2, 8, device="cuda")
    m.average(to_dev(f.reshape(2, -1)), ub)
    torch.cuda.synchronize()
    m.close()
    want = f.astype(np.float64)
    for a in range(3):   # axis a of the field is dimension 3 - a
        e = np.minimum(np.arange(1, n[a] + 1)[None] / n[a], np.array([[0.5], [1.0]]))
        w = np.clip(e - np.maximum(np.arange(n[a])[None] / n[a], np.array([[0.0], [0.5]])), 0.0, None) * 2.0
        want = np.moveaxis(np.tensordot(w, want, (1, 3 - a)), 0, 3 - a)
    err = np.abs(ub.cpu().numpy().astype(np.float64) / want.reshape(2, -1) - 1.0).max()
    assert err <= 18 * 2.0 ** -24, err
