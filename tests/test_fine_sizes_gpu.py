"""The fine-grid sweeps over ratios and grid sizes: every compiled ratio and
the any-ratio form, uneven axes, grids of one block and grids whose threads
walk several layers with a ragged last segment, both interpolations, with
the path tolerances of the repository."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import TOL_FP32, TOL_FP64, assert_close, assert_close_interp, to_dev, to_np

pytestmark = pytest.mark.gpu

SMALL, LARGE = (5, 7, 3), (34, 41, 43)


@pytest.mark.parametrize("interp", [synth.INTERP_TRILINEAR, synth.INTERP_CELL])
@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("r,nb", [(1, SMALL), (2, SMALL), (3, SMALL), (4, SMALL), (5, SMALL), (6, SMALL), (8, SMALL),
                                  (2, LARGE), (3, LARGE), (4, LARGE), (5, (20, 21, 19)), (8, (18, 13, 11))])
def test_average_and_projection(cuda_lib, r, nb, fp64, interp):
    import torch
    fine = tuple(r * m for m in nb)
    d = synth.make_desc((0.1, -0.2, 0.3), (1.0, 1.3, 0.7), fine, r, fp64=fp64, law=synth.DRAG_DI_FELICE, interp=interp)
    rng = synth.rng_for(5, r)
    T = np.float64 if fp64 else np.float32
    tol = TOL_FP64 if fp64 else TOL_FP32
    nf, n_b = int(np.prod(fine)), int(np.prod(nb))
    u = (0.5 + 0.02 * rng.standard_normal((3, nf))).astype(T)
    S = rng.standard_normal((3, n_b)).astype(T)
    g = cuda_lib.Grids(d)
    kw = dict(device="cuda", dtype=g.dtype)
    ub, var, Sf, Sf1 = (torch.full(s, 7.0, **kw) for s in ((3, n_b), (n_b,), (3, nf), (1, nf)))
    g.cg_average_fine_to_bulk(to_dev(u), ub, var)
    g.cg_project_bulk_to_fine(to_dev(S), Sf)
    g.cg_project_bulk_to_fine(to_dev(S[:1]), Sf1)
    torch.cuda.synchronize()
    want_u, want_v = oracle.average(d, u.reshape((3,) + fine[::-1]))
    assert_close("u_bulk", to_np(ub), want_u, tol, vec=True)
    if r > 1:
        assert_close("var_bulk", to_np(var), want_v, tol)
    else:
        assert np.all(to_np(var) == 0.0)
    want = oracle.project(d, S)
    assert_close_interp("S_fine", to_np(Sf), want, oracle.project(d, np.abs(S)), tol)
    assert torch.equal(Sf1[0], Sf[0])
    g.close()


@pytest.mark.parametrize("r", [2, 3, 4, 5])
def test_projection_sums(cuda_lib, r):
    """The step's sums of S_f V_f and of S_B V_B, formed by the projection
    over several layers per thread, agree with the fields it wrote and read."""
    import torch
    w = synth.tiny(seed=r, n=30_000, fine=36 * r, ratio=r, fp64=True)
    g = cuda_lib.Grids(w.desc)
    out = g.alloc_outputs(w.n)
    g.cg_step(to_dev(w.pos_d), to_dev(w.vel), to_dev(w.u_fine.reshape(3, -1)), out)
    torch.cuda.synchronize()
    Vf = 1.0 / (36 * r) ** 3
    Sf, Sb = out["S_fine"].double(), out["S_bulk"].double()
    scale = (Sb.abs().sum(1) * Vf * r ** 3).max().item()
    got = out["sums"].cpu()
    # plain FP64 sums of 46,656 r^3 values: 1e-12 of the sum of magnitudes
    assert (got[8:11] - (Sf.sum(1) * Vf).cpu()).abs().max().item() <= 1e-12 * scale
    assert (got[5:8] - (Sb.sum(1) * Vf * r ** 3).cpu()).abs().max().item() <= 1e-12 * scale
    g.close()
