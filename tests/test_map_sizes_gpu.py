"""The maps' kernels at their edges against the FP64 oracle: rows of one and of
several x tiles, a bulk cell over more fine indices than a block has threads,
chunks along z with remainders, single planes and columns, grids that overlap
in part, and every component count."""
import numpy as np
import pytest

import oracle
from parity_util import TOL_FP32, TOL_FP64, assert_close, assert_close_interp, to_dev, to_np

pytestmark = pytest.mark.gpu

UNIT = (1.0, 1.0, 1.0)
CASES = {
    "one_cell": (((0.0, 0.0, 0.0), UNIT, (1, 1, 1)), ((0.0, 0.0, 0.0), UNIT, (1, 1, 1)), 1),
    "wide_cells": (((0.0, 0.0, 0.0), UNIT, (3, 2, 2)), ((0.0, 0.0, 0.0), UNIT, (900, 3, 5)), 2),
    "block_wide": (((0.0, 0.0, 0.0), UNIT, (2, 2, 3)), ((0.0, 0.0, 0.0), UNIT, (512, 4, 7)), 1),
    "many_tiles": (((0.0, 0.0, 0.0), UNIT, (311, 3, 4)), ((-0.01, -0.2, -0.1), (1.02, 1.3, 1.2), (701, 7, 9)), 3),
    "partial": (((0.0, 0.0, 0.0), UNIT, (9, 8, 7)), ((0.4, 0.3, -0.6), (1.5, 0.4, 1.0), (40, 13, 17)), 4),
    "one_plane": (((0.0, 0.0, 0.0), UNIT, (17, 11, 1)), ((0.0, 0.0, 0.0), UNIT, (33, 30, 1)), 5),
    "long_column": (((0.0, 0.0, 0.0), UNIT, (1, 1, 331)), ((0.0, 0.01, 0.0), UNIT, (2, 1, 999)), 8),
    "coarse_fine": (((0.0, 0.0, 0.0), UNIT, (600, 5, 4)), ((0.0, 0.0, 0.0), UNIT, (290, 3, 3)), 3),
}


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("name", CASES)
def test_maps_match_the_oracle(cuda_lib, name, fp64):
    import torch
    cg = cuda_lib
    bulk, fine, nc = CASES[name]
    tol = TOL_FP64 if fp64 else TOL_FP32
    dt = np.float64 if fp64 else np.float32
    rng = np.random.default_rng(11)
    nb, nf = int(np.prod(bulk[2])), int(np.prod(fine[2]))
    u = (0.5 + 0.1 * rng.standard_normal((nc, nf))).astype(dt)
    S = (0.5 + 0.1 * rng.standard_normal((nc, nb))).astype(dt)
    m = cg.Map(bulk, fine, fp64=fp64)
    ub = torch.full((nc, nb), float("nan"), dtype=m.dtype, device="cuda")
    sf = torch.full((nc, nf), float("nan"), dtype=m.dtype, device="cuda")
    m.average(to_dev(u), ub)
    m.project(to_dev(S), sf)
    torch.cuda.synchronize()
    assert_close("u_B", to_np(ub), oracle.map_average(bulk, fine, u), tol)
    ref = oracle.map_project(bulk, fine, S)
    assert_close_interp("S_f", to_np(sf), ref, oracle.map_project(bulk, fine, np.abs(S.astype(np.float64))), tol)
    m.close()
