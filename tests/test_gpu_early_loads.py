"""Weights requested ahead of a GEMM's wait for the kernel before it: only what an earlier launch of the handle has waited for.

A call that is only captured has waited for nothing, so the marks of eager writes (a layout, the straddle block) outlive it;
a layout that is captured can be replayed unseen, so eager calls never go ahead after one.  Outputs against the oracle."""
import numpy as np
import pytest
import torch

import helpers
import oracle
from paper_2510_02822_b200 import binding as fx
from paper_2510_02822_b200 import inputs

pytestmark = pytest.mark.gpu


class Case:
    """A linear layer of two K blocks with its oracle, under any group order."""

    def __init__(self, ratio):
        self.dev = torch.device("cuda:0")
        self.c = c = inputs.ranged_linear("early", 200, 256, 80, 16, seed=91, group_structured=True)
        self.perm, self.sxg, _, _ = helpers.prepare_linear(c)
        self.q = oracle.quantize(c.X, c.x_scale)
        self.W = torch.from_numpy(c.Wq).to(self.dev)
        self.X = torch.from_numpy(c.X).to(self.dev)
        self.L = fx.Layer(self.W, torch.from_numpy(c.w_scale).to(self.dev), None, self.perm, self.sxg, c.G)
        self.Y = torch.empty((c.M, c.N), dtype=torch.int32, device=self.dev)
        self.slabs = tuple(torch.empty(c.M * c.K + 16, dtype=t, device=self.dev) for t in (torch.uint8, torch.int8))
        self.L.set_lowbit_ratio(ratio)

    def prologue(self):
        self.L.quantize_lower(self.X, self.c.x_scale, slabs=self.slabs)

    def gemm(self):
        self.L.mixed_gemm(*self.slabs, self.c.M, self.c.x_scale, self.c.y_scale, fx.OUT_ACC_I32, self.Y)
        return fx.flexiq_layer_early_loads(self.L.h)

    def check(self, perm, ratio):
        sw = oracle.weight_positions_linear(self.c.Wq, self.c.G, perm)
        ref = oracle.mixed_gemm_acc(self.q, self.c.Wq, self.c.G, perm, self.sxg[perm].copy(), sw, oracle.n_low(ratio, self.c.K // self.c.G))
        assert np.array_equal(self.Y.cpu().numpy(), ref)
        self.Y.zero_()


def capture(f):
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        r = f()
    return g, r


def test_captured_call_leaves_the_layout_mark():
    k = Case(0.5)                                     # 128 of 256 channels: no straddle block
    k.prologue()
    assert k.gemm() == (True, True)                   # creating the layer has waited for its layout
    other = k.perm[::-1].copy()
    k.L.set_group_perm(k.W, other, k.sxg)
    g, early = capture(lambda: (k.prologue(), k.gemm())[1])
    assert early == (False, False)
    k.prologue()
    assert k.gemm() == (False, False)                 # nothing has waited for the layout yet
    k.check(other, 0.5)
    k.prologue()
    assert k.gemm() == (True, True)
    k.check(other, 0.5)
    g.replay()
    k.check(other, 0.5)
    k.L.close()


def test_captured_call_leaves_the_straddle_mark():
    k = Case(0.25)                                    # 64 channels: inside the first K block
    k.prologue()                                      # writes the straddle block
    k.L.set_lowbit_ratio(1.0)
    slab = torch.empty(k.c.M * k.c.K + 16, dtype=torch.uint8, device=k.dev)

    def whole():
        k.L.quantize_lower(k.X, k.c.x_scale, slabs=(slab, None))
        k.L.mixed_gemm(slab, None, k.c.M, k.c.x_scale, k.c.y_scale, fx.OUT_ACC_I32, k.Y)
    g, _ = capture(whole)
    k.L.set_lowbit_ratio(0.25)
    assert k.gemm() == (True, False)                  # only the captured call came in between
    k.check(k.perm, 0.25)
    assert k.gemm() == (True, True)
    k.check(k.perm, 0.25)
    g.replay()
    k.check(k.perm, 1.0)
    k.L.close()


def test_layout_in_a_graph():
    k = Case(0.25)
    other = k.perm[::-1].copy()

    def relaid():
        k.L.set_group_perm(k.W, other, k.sxg)
        k.prologue()
        first = k.gemm()
        k.prologue()
        return first, k.gemm()
    g, early = capture(relaid)
    assert early == ((False, False), (True, False))   # the capture's own first GEMM waits for its layout; its straddle block is always late
    k.L.set_group_perm(k.W, k.perm, k.sxg)
    for _ in range(2):
        k.prologue()
        assert k.gemm() == (False, False)             # a replay may have rewritten both
        k.check(k.perm, 0.25)
    g.replay()
    k.check(other, 0.25)
    k.prologue()
    assert k.gemm() == (False, False)
    k.check(other, 0.25)
    k.L.close()


def test_layout_alone_in_a_graph():
    k = Case(0.25)
    other = k.perm[::-1].copy()
    g, _ = capture(lambda: k.L.set_group_perm(k.W, other, k.sxg))
    k.prologue()                                      # not replayed yet: the straddle block of the first order
    k.gemm()
    k.check(k.perm, 0.25)
    g.replay()
    k.prologue()
    assert k.gemm() == (False, False)
    k.check(other, 0.25)                              # the block follows the weights that the replay has laid out
    k.L.close()
