"""The training kernels at the sizes where they can go wrong: one row, the
edges of a 128-row tile, one tile more than a wave of CTAs, and the weight
image that a training step updates in place."""
import numpy as np
import pytest

from oracle import mlp as om
from test_mlp_gpu import ACTS, make, random_features, scaled

pytestmark = pytest.mark.gpu

BLOCKS = ("W1", "b1", "W2", "b2", "w3", "b3")


@ACTS
@pytest.mark.parametrize("n", [1, 127, 128, 129, 152 * 128 + 1, 40_000])
def test_gradient_at_tile_edges(cuda_lib, n, act):
    """Each block of the gradient within 2^-8 (norm-wise) of the oracle's: a
    hidden activation or a dZ2 on a rounding boundary may take the
    neighbouring BF16 value, 2^-8 of itself, and in the worst case of one row
    all of a block's weight rests on it."""
    import torch
    m, p = make(cuda_lib, 4, act)
    f = random_features(n, 17)
    t = np.cos(3 * f[:, 0]).astype(np.float32)
    loss = torch.zeros(1, device="cuda")
    m.grads(torch.from_numpy(f).cuda(), torch.from_numpy(t).cuda(), loss)
    got = cuda_lib.mlp_unpack(m.params(grads=True)[1])
    want_loss, want = om.loss_and_grads(p, scaled(f), t.astype(np.float64), bf16_inputs=True, act=act)
    assert m.sync_status()[0] == 0
    # the loss is a mean of (c - t)^2 with c within 2^-8 of itself
    assert abs(loss.item() - want_loss) <= 2.0 ** -7 * max(want_loss, 1e-6)
    for k in BLOCKS:
        w = np.asarray(want[k], np.float64)
        assert np.linalg.norm(got[k].reshape(w.shape) - w) <= 2.0 ** -8 * np.linalg.norm(w), k


@ACTS
def test_training_keeps_the_weight_image(cuda_lib, act):
    """After training steps the closure's forward pass is, bit for bit, that
    of a closure created from its parameters."""
    import torch
    m, _ = make(cuda_lib, 6, act)
    f = torch.from_numpy(random_features(3_000, 2)).cuda()
    t = f[:, 0].contiguous()
    for _ in range(3):
        m.train_step(f, t, 1e-2)
    fresh = cuda_lib.Mlp(m.params(), m.lo, m.hi, activation=act)
    out = [torch.empty(3_000, device="cuda") for _ in range(2)]
    m.forward(f, out[0])
    fresh.forward(f, out[1])
    torch.cuda.synchronize()
    assert torch.equal(out[0], out[1])
