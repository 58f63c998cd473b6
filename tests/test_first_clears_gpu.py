"""What a handle counts in is zero before a step: the first one, on whatever
stream that runs, and one after a step that failed halfway.  Making a handle
waits for none of the caller's work."""
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


NAMES = ("eps_bulk", "u_bulk", "var_bulk", "force", "S_bulk", "S_fine", "eps_fine", "sums")


@pytest.mark.parametrize("form", ["scratch", "incremental", "sorted", "batch"])
def test_a_step_after_one_whose_launch_failed(cuda_lib, form):
    """Each launch of a step is left out in turn (on the host): the step says
    so, and the next one is a fresh handle's bit for bit."""
    import torch
    cg = cuda_lib
    w = synth.tiny(seed=5, n=20_000, fp64=False)
    pos, vel, uf = inputs(w)

    def fresh():
        if form == "batch":
            f = cg.Grids(w.desc)
            out = f.alloc_outputs(w.n, eps_fine=True)
            f.close()
            h = cg.Batch([(w.desc, pos, vel, uf, out)])
            return h, out, [h.step]
        h = cg.Grids(w.desc)
        out = h.alloc_outputs(w.n, eps_fine=True)
        if form == "sorted":
            ab = pos.clone(), vel.clone(), torch.empty_like(pos), torch.empty_like(vel)
            return h, out, [lambda: h.cg_step_sorted(*ab, uf, out), lambda: h.cg_step_sorted(ab[2], ab[3], ab[0], ab[1], uf, out)]
        return h, out, [lambda: h.cg_step(pos, vel, uf, out)] * (2 if form == "incremental" else 1)

    h, out, calls = fresh()
    for c in calls:
        c()
    torch.cuda.synchronize()
    want = {k: out[k].clone() for k in NAMES}
    h.close()
    try:
        failed = 0
        while True:
            h, out, calls = fresh()
            for c in calls[:-1]:
                c()
            assert cg.lib().cg_debug_fail_launch_after(failed) == 0
            try:
                calls[-1]()
            except cg.CgError as e:
                assert e.code == 2
            else:
                break
            calls[-1]()
            torch.cuda.synchronize()
            for k in NAMES:
                assert torch.equal(out[k], want[k]), (failed, k)
            h.close()
            failed += 1
            assert failed < 60
        assert failed >= 8
        h.close()
        assert cg.lib().cg_debug_fail_launch_after(-2) == 1
    finally:
        cg.lib().cg_debug_fail_launch_after(-1)
