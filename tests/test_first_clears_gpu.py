"""What a new handle counts in is zero before its first step, on whatever
stream that runs, and making a handle waits for none of the caller's work."""
import pytest

import synth
from parity_util import inputs

pytestmark = pytest.mark.gpu

BUSY = 400_000_000   # clock cycles of a one-thread kernel: 0.2 s and more


def test_creation_does_not_wait_for_the_callers_streams(cuda_lib):
    import torch
    w = synth.tiny(seed=1, n=4_000)
    cuda_lib.Grids(w.desc).close()
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    done = torch.cuda.Event(), torch.cuda.Event()
    for s, e in zip((torch.cuda.default_stream(), side), done):
        with torch.cuda.stream(s):
            torch.cuda._sleep(BUSY)
            e.record()
    g = cuda_lib.Grids(w.desc, stream=side)
    waited = [e.query() for e in done]
    torch.cuda.synchronize()
    g.close()
    assert waited == [False, False]


@pytest.mark.parametrize("fp64", [False, True])
def test_first_steps_on_another_stream(cuda_lib, fp64):
    """A handle made on a busy stream and used on another one: 4,000 particles,
    which need no more room than a new handle has."""
    import torch
    cg = cuda_lib
    w = synth.tiny(seed=1, n=4_000, fp64=fp64)
    pos, vel, uf = inputs(w)
    gen = torch.Generator(device="cuda").manual_seed(2)
    beds = [pos] + [pos[torch.randperm(w.n, device="cuda", generator=gen)].contiguous() for _ in range(2)]
    want = []
    for p in beds:
        f = cg.Grids(w.desc)
        out = f.alloc_outputs(w.n, eps_fine=True, bins=True)
        f.cg_step(p.clone(), vel, uf, out)
        torch.cuda.synchronize()
        want.append(out)
        f.close()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(a):
        torch.cuda._sleep(BUSY)
    g = cg.Grids(w.desc, stream=a)
    g.set_stream(b)
    outs = [g.alloc_outputs(w.n, eps_fine=True, bins=True) for _ in beds]
    b.wait_stream(torch.cuda.default_stream())
    for p, out in zip(beds, outs):
        g.cg_step(p, vel, uf, out)
    torch.cuda.synchronize()
    for k, (got, ref) in enumerate(zip(outs, want)):
        for name in ("eps_bulk", "u_bulk", "var_bulk", "force", "S_bulk", "S_fine", "eps_fine", "cell", "perm", "cell_start"):
            assert torch.equal(got[name], ref[name]), (k, name)
    assert g.cg_sync_status()[:2] == (0, 0)
    g.close()
