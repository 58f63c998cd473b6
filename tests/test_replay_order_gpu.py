"""Captured and eager steps mixed on one handle: what a captured step leaves
on the device is what the next call starts from, whatever the host did when
the step was captured."""
import pytest

import synth
from parity_util import inputs

pytestmark = pytest.mark.gpu

FIELDS = ("eps_bulk", "u_bulk", "force", "S_bulk", "S_fine", "eps_fine", "implicit_bulk", "implicit_fine")
BINS = ("cell", "perm", "cell_start")


class Mixed:
    """A handle on a stream of its own, with steps called on it or captured."""

    def __init__(self, cg, fp64):
        import torch
        self.cg = cg
        self.w = synth.tiny(seed=6, n=20_000, fp64=True) if fp64 else synth.small_clustered_bed(seed=4)
        self.a, self.va, self.uf = inputs(self.w)
        self.b, self.vb = torch.empty_like(self.a), torch.empty_like(self.va)
        self.stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        self.g = cg.Grids(self.w.desc, stream=self.stream)
        self.out = self.g.alloc_outputs(self.w.n, eps_fine=True, bins=True, implicit=True, implicit_fine=True)

    def step(self, pos, vel):
        self.g.cg_step(pos, vel, self.uf, self.out)

    def sorted(self, pos, vel, po, vo):
        self.g.cg_step_sorted(pos, vel, po, vo, self.uf, self.out)

    def on_stream(self, fn, *args):
        import torch
        torch.cuda.synchronize()   # the inputs come from the default stream
        with torch.cuda.stream(self.stream):
            fn(*args)
        torch.cuda.synchronize()

    def capture(self, fn, *args):
        import torch
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=self.stream):
            fn(*args)
        torch.cuda.synchronize()
        return g

    def replay(self, *graphs):
        import torch
        torch.cuda.synchronize()
        with torch.cuda.stream(self.stream):
            for g in graphs:
                g.replay()
        torch.cuda.synchronize()

    def check(self, pos, vel, what):
        """The last step's outputs are a fresh handle's, bit for bit."""
        import torch
        f = self.cg.Grids(self.w.desc)
        ref = f.alloc_outputs(self.w.n, eps_fine=True, bins=True, implicit=True, implicit_fine=True)
        f.cg_step(pos.clone(), vel.clone(), self.uf, ref)
        torch.cuda.synchronize()
        f.close()
        for k in FIELDS + BINS:
            assert torch.equal(self.out[k], ref[k]), (what, k)

    def poison(self):
        for k in FIELDS:
            self.out[k].fill_(float("nan"))


@pytest.mark.parametrize("fp64", [False, True])
def test_a_captured_step_that_has_not_run_yet(cuda_lib, fp64):
    """A step in the caller's order is captured after sorted steps and called
    before the capture's first replay: nothing of the capture has run."""
    m = Mixed(cuda_lib, fp64)
    m.on_stream(m.sorted, m.a, m.va, m.b, m.vb)     # from an unsorted order
    m.on_stream(m.sorted, m.b, m.vb, m.a, m.va)     # in cell order: nothing crosses a cell
    p, v = m.a.clone(), m.va.clone()
    graph = m.capture(m.step, p, v)
    m.poison()
    m.on_stream(m.step, p, v)
    m.check(p, v, "called")
    m.poison()
    m.replay(graph)
    m.check(p, v, "replayed")
    m.g.close()


@pytest.mark.parametrize("fp64", [False, True])
def test_sorted_replays_between_steps_in_the_callers_order(cuda_lib, fp64):
    """Captured sorted steps, a step with movers, the captured steps again,
    then a step that finds no mover."""
    import torch
    m = Mixed(cuda_lib, fp64)
    m.on_stream(m.sorted, m.a, m.va, m.b, m.vb)
    g1 = m.capture(m.sorted, m.b, m.vb, m.a, m.va)
    g2 = m.capture(m.sorted, m.a, m.va, m.b, m.vb)
    m.replay(g1, g2)
    gen = torch.Generator(device="cuda").manual_seed(1)
    q, vq = (x[torch.randperm(m.w.n, device="cuda", generator=gen)].contiguous() for x in (m.b, m.vb))
    m.poison()
    m.on_stream(m.step, q, vq)
    m.check(q, vq, "movers")
    m.replay(g1, g2)
    p, v = m.b.clone(), m.vb.clone()
    m.poison()
    m.on_stream(m.step, p, v)
    m.check(p, v, "no movers")
    # the drag by itself, from the binning of a replayed sorted step
    m.on_stream(m.step, q, vq)
    m.replay(g1)
    F, S = torch.empty_like(m.out["force"]), torch.empty_like(m.out["S_bulk"])
    want_F, want_S = m.out["force"].clone(), m.out["S_bulk"].clone()
    for _ in range(2):
        m.on_stream(m.g.cg_drag, m.b, m.vb, m.out["eps_bulk"], m.out["u_bulk"], F, S)
        assert torch.equal(F, want_F) and torch.equal(S, want_S)
    m.g.close()


@pytest.mark.parametrize("fp64", [False, True])
def test_a_replayed_step_after_sorted_steps(cuda_lib, fp64):
    """A captured step in the caller's order replayed after eager sorted steps
    over the same arrays."""
    m = Mixed(cuda_lib, fp64)
    m.on_stream(m.step, m.a, m.va)
    graph = m.capture(m.step, m.a, m.va)
    m.replay(graph)
    m.check(m.a, m.va, "unsorted")
    m.on_stream(m.sorted, m.a, m.va, m.b, m.vb)
    m.on_stream(m.sorted, m.b, m.vb, m.a, m.va)
    m.poison()
    m.replay(graph)
    m.check(m.a, m.va, "sorted")
    m.on_stream(m.sorted, m.a, m.va, m.b, m.vb)      # the next sorted step: forces in the caller's order
    m.check(m.a, m.va, "sorted again")
    m.g.close()
