"""Porosity and deposited volume of spheres small against their cell: the
cells' whole-number sums keep the volumes' own precision at any size."""
from fractions import Fraction
import math

import numpy as np
import pytest

import synth
from parity_util import to_dev

pytestmark = pytest.mark.gpu

U64 = 2.0 ** -53
PI = Fraction("3.14159265358979323846264338327950288419716939937510")


def _volume(d, n=1):
    """Exact volume of n spheres of diameter d."""
    return n * PI / 6 * Fraction(float(d)) ** 3


def _run(cg, desc, pos, path):
    """(porosity, sums) of a step over the particles by one of the binning paths."""
    import torch
    n = pos.shape[0]
    T = pos.dtype
    nf = math.prod(desc["fine_n"])
    p, v = to_dev(pos), torch.zeros(n, 4, device="cuda", dtype=to_dev(pos).dtype)
    u = to_dev(np.full((3, nf), 0.25, T))
    if path == "batch":
        g = cg.Grids(desc)
        out = g.alloc_outputs(n)
        g.close()
        b = cg.Batch([(desc, p, v, u, out)])
        b.step()
        torch.cuda.synchronize()
        b.close()
        return out["eps_bulk"].cpu().numpy(), out["sums"].cpu().numpy()
    g = cg.Grids(dict(desc, sort_digits=8) if path == "digits" else desc)
    out = g.alloc_outputs(n)
    if path == "sorted":
        po, vo, p2, v2 = (torch.empty_like(p) for _ in range(4))
        g.cg_step_sorted(p, v, po, vo, u, out)
        g.cg_step_sorted(po, vo, p2, v2, u, out)
    else:
        for _ in range(2 if path == "incremental" else 1):
            g.cg_step(p, v, u, out)
    torch.cuda.synchronize()
    if path == "scratch":
        eps = torch.empty_like(out["eps_bulk"])
        g.cg_deposit(cg.CG_DEP_VOLUME, n, p, eps)
        torch.cuda.synchronize()
        assert torch.equal(eps, out["eps_bulk"])
    g.close()
    return out["eps_bulk"].cpu().numpy(), out["sums"].cpu().numpy()


PATHS = ("scratch", "incremental", "sorted", "digits")


@pytest.mark.parametrize("path", PATHS + ("batch",))
@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("d", [0.3, 0.08, 0.0101, 1.03e-3, 1.07e-4])
def test_deposited_volume_of_equal_spheres(cuda_lib, d, fp64, path):
    """Equal spheres of diameter d cells, whose roundings add up: the volume
    deposited is the volume of the spheres.  FP64: the identity's 1e-12.  FP32:
    each volume is a pair good to 2^-46, its cell's sum and product with V_B to
    2^-45, 2^-42 in all."""
    if path == "batch" and fp64:
        pytest.skip("batches are FP32")
    T = np.float64 if fp64 else np.float32
    desc = synth.make_desc((0, 0, 0), (1, 1, 1), (32, 32, 32), 4, fp64=fp64, law=synth.DRAG_DI_FELICE)
    n = 5_000
    pos = np.empty((n, 4), T)
    pos[:, :3] = synth.rng_for(3).random((n, 3)) * 0.999
    pos[:, 3] = d / 8
    _, sums = _run(cuda_lib, desc, pos, path)
    want = float(_volume(pos[0, 3], n))
    assert abs(sums[1] - want) <= (1e-12 if fp64 else 2.0 ** -42) * want, (sums[1] - want) / want
    if fp64:
        assert abs(sums[0] - sums[1]) <= 1e-12 * sums[0], (sums[0] - sums[1]) / sums[0]


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("d", [0.0117, 0.00771, 0.00333])
def test_porosity_of_many_small_spheres(cuda_lib, d, path):
    """Two hundred thousand equal spheres in each of a few cells, FP64: a
    volume carries three roundings and pi / 6 V_B one (V_B is a power of two), so
    the porosity is within 5 phi u of the exact one, and its own rounding u."""
    desc = synth.make_desc((0, 0, 0), (1, 1, 1), (16, 16, 16), 4, fp64=True, law=synth.DRAG_DI_FELICE)
    n = 600_000
    rng = synth.rng_for(8)
    pos = np.empty((n, 4))
    pos[:, :3] = (np.array([[0, 0, 0], [1, 2, 3], [3, 3, 3]])[np.arange(n) % 3] + 0.1 + 0.8 * rng.random((n, 3))) / 4
    pos[:, 3] = d / 4
    eps, _ = _run(cuda_lib, desc, pos, path)
    phi = _volume(pos[0, 3], n // 3) * 4 ** 3
    got = np.sort(eps)[:3]
    err = max(abs(float(Fraction(float(e)) - (1 - phi))) for e in got)
    assert err <= (5 * float(phi) + 1) * U64, err / U64
    assert (np.sort(eps)[3:] == 1.0).all()


@pytest.mark.parametrize("path", PATHS)
@pytest.mark.parametrize("fp64", [False, True])
def test_spheres_far_larger_than_a_cell(cuda_lib, fp64, path):
    """Several spheres of up to just below 2^32 cells in one cell, and beside
    them smaller ones: no sum overflows."""
    T = np.float64 if fp64 else np.float32
    desc = synth.make_desc((0, 0, 0), (1, 1, 1), (32, 32, 32), 4, fp64=fp64, law=synth.DRAG_DI_FELICE)
    n = 4_000
    big = [2010.0, 2010.0, 2010.0, 2010.0, 2010.0, 1500.0, 1.7, 0.4]   # 2016.8 cells: 2^32 cells' volume
    pos = np.empty((n, 4), T)
    pos[:, :3] = 0.2 + 0.75 * synth.rng_for(5).random((n, 3))
    pos[:, 3] = 0.001
    pos[:len(big), :3] = 0.05
    pos[:len(big), 3] = np.array(big) / 8
    eps, sums = _run(cuda_lib, desc, pos, path)
    want = float(1 - sum(_volume(x) for x in pos[:len(big), 3]) * 8 ** 3)
    assert abs(eps[0] - want) <= (1e-15 if fp64 else 2.0 ** -44) * abs(want), (eps[0], want)
