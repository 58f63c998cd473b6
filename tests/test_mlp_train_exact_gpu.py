"""The training kernel's gradient on operands without rounding: inputs, weights
and hidden activations that are BF16 values, sums that are exact in FP32, and
output gradients dZ2 of full FP32 significands, so that the gradient's own
arithmetic (dZ as three BF16 terms, rows in groups of 32) is all that is left."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BLOCKS = ("W1", "b1", "W2", "b2", "w3", "b3")


def _network(rng):
    """Weights of few bits: W1 in quarters, W2 in eighths, biases likewise, w3
    in 64ths."""
    def q(shape, unit, most):
        return rng.integers(-most, most + 1, shape).astype(np.float64) * unit
    W1 = np.zeros((16, 64))
    W1[:7] = q((7, 64), 0.25, 4)
    return dict(W1=W1, b1=q(64, 1 / 32, 16), W2=q((64, 64), 1 / 8, 8), b2=q(64, 1 / 8, 8), w3=q(64, 1 / 64, 31),
                b3=q(1, 1 / 64, 31))


def _bf16(x):
    """FP32 values rounded to BF16 (nearest, ties to even)."""
    u = x.astype(np.float32).view(np.uint32)
    return ((u + 0x7FFF + (u >> 16 & 1)) & 0xFFFF0000).astype(np.uint32).view(np.float32)


@pytest.mark.parametrize("n,rows", [(4, range(4)), (128, range(30, 34)), (128, range(62, 66)), (128, range(124, 128)),
                                    (256, (5, 133, 200, 255)), (8192, (0, 1000, 4111, 8191))])
def test_gradient_of_exact_operands(cuda_lib, n, rows):
    """A few rows with a residual among n (the others have none), so that a
    gradient entry is a sum of up to four terms: within 1e-6 of the sum of their
    magnitudes (truncating FP32 sums of four: 4 x 2^-23 at most), and W1 and b1
    within 4e-6 of that of dA1's terms too (of 64: 64 x 2^-24).  A dZ of two BF16
    terms is off by up to 2^-17, 8e-6, of a term."""
    import torch
    rng = np.random.default_rng([n, len(tuple(rows)), rows[0]])
    p = _network(rng)
    x = np.zeros((n, 8))
    x[:, :7] = rng.integers(0, 5, (n, 7)) / 8.0
    z1 = x[:, :7] @ p["W1"][:7] + p["b1"]
    a1 = np.maximum(z1, 0.0)
    z2 = a1 @ p["W2"] + p["b2"]
    a2 = np.maximum(z2, 0.0)
    c = a2 @ p["w3"] + p["b3"]
    assert np.array_equal(_bf16(a1), a1) and np.array_equal(c.astype(np.float32), c)
    t = c.astype(np.float32)
    rows = np.array(rows)
    t[rows] -= rng.standard_normal(rows.size).astype(np.float32)
    dc = (c.astype(np.float32) - t) * np.float32(2.0 / n)             # exact: n is a power of two
    d2 = (dc[:, None] * p["w3"].astype(np.float32)) * (z2 > 0)        # FP32, one rounding
    d2 = d2.astype(np.float32)
    full = d2[rows][(d2[rows] != 0)]
    assert (np.abs(full - _bf16(full)) > 0).mean() > 0.9              # dZ2 is not a BF16 value
    da = _bf16(d2).astype(np.float64) @ p["W2"].T
    d1 = da * (z1 > 0)
    mag1 = (np.abs(_bf16(d2)).astype(np.float64) @ np.abs(p["W2"]).T) * (z1 > 0)
    want = dict(W1=x[:, :7].T @ d1, b1=d1.sum(0), W2=a1.T @ d2.astype(np.float64), b2=d2.astype(np.float64).sum(0),
                w3=a2.T @ dc.astype(np.float64), b3=np.array([dc.astype(np.float64).sum()]))
    size = dict(W1=x[:, :7].T @ mag1, b1=mag1.sum(0), W2=a1.T @ np.abs(d2).astype(np.float64),
                b2=np.abs(d2).astype(np.float64).sum(0), w3=a2.T @ np.abs(dc).astype(np.float64),
                b3=np.array([np.abs(dc).astype(np.float64).sum()]))
    m = cuda_lib.Mlp(cuda_lib.mlp_pack(p), [0.0] * 7, [1.0] * 7, activation="relu")
    loss = torch.zeros(1, device="cuda")
    m.grads(torch.from_numpy(x.astype(np.float32)).cuda(), torch.from_numpy(t).cuda(), loss)
    got = cuda_lib.mlp_unpack(m.params(grads=True)[1])
    assert m.sync_status()[0] == 0
    assert not np.asarray(got["W1"])[7:].any()
    for k in BLOCKS:
        g = np.asarray(got[k])[:7] if k == "W1" else np.asarray(got[k])
        err = np.abs(g - want[k])
        bound = 4e-6 * size[k] if k in ("W1", "b1") else 1e-6 * size[k]
        assert (err <= bound).all(), (k, (err / np.maximum(size[k], 1e-300)).max())
