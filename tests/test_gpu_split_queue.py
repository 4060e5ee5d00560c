"""The split product's tile queue: tiles are handed out by a device counter that the launch
itself returns to zero, so launches of any tile count, in any order, on one context or on
two streams at once, give the same bits."""
import pytest
import torch

from helpers import gpu_pattern, upload_pairs
from paper_2205_08941_gb300 import cq
from paper_2205_08941_gb300 import inputs as I

pytestmark = pytest.mark.gpu


class Product:
    """L.S on a cell, in split precision and in FP64."""

    def __init__(self, ctx, shape, norb, rS, rL):
        cell = I.diamond_cell(shape, a=10.26, sigma=0.1, seed=5, norb=norb)
        self.ctx = ctx
        self.pL, self.pS, self.pX = (gpu_pattern(ctx, cell, r) for r in (rL, rS, rL + rS))
        self.L = upload_pairs(ctx, self.pL, I.random_blocks(cell, rL, 1, symmetric=False))
        self.S = upload_pairs(ctx, self.pS, I.random_blocks(cell, rS, 2, symmetric=False))

    def __call__(self, prec=cq.CQ_SPLIT_BF16X3):
        C = self.ctx.zeros(self.pX)
        self.ctx.bsmm(1.0, self.pL, self.L, self.pS, self.S, 0.0, self.pX, C, prec)
        return C


# one tile; fewer tiles than SMs; more tiles than SMs; tiles of few K steps
CASES = [((1, 1, 1), 9, 4.0, 4.0), ((2, 2, 1), 4, 6.0, 7.0), ((3, 3, 3), 9, 14.0, 16.0),
         ((4, 3, 3), 4, 5.0, 5.0)]


@pytest.mark.parametrize("case", CASES)
def test_repeated_launches_give_the_same_bits(case):
    ctx = cq.Context(0)
    p, other = Product(ctx, *case), Product(ctx, (2, 2, 2), 9, 8.0, 9.0)
    first = p()
    # the split's error model: 1e-5 of the product's largest values covers every block here
    ref = p(cq.CQ_FP64)
    assert float((first - ref).abs().max()) <= 1e-5 * float(ref.abs().max())
    for _ in range(3):
        other()
        assert torch.equal(p(), first)
    ctx.close()


def test_two_contexts_on_two_streams_do_not_share_the_queue():
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    a = Product(cq.Context(0, stream=s1), (3, 3, 3), 9, 14.0, 16.0)
    b = Product(cq.Context(0, stream=s2), (4, 3, 3), 4, 10.0, 12.0)
    torch.cuda.synchronize()
    want = a(), b()
    torch.cuda.synchronize()
    outs = [(a.ctx.zeros(a.pX), b.ctx.zeros(b.pX)) for _ in range(4)]
    torch.cuda.synchronize()
    for ca, cb in outs:
        for p, c in ((a, ca), (b, cb)):
            p.ctx.bsmm(1.0, p.pL, p.L, p.pS, p.S, 0.0, p.pX, c, cq.CQ_SPLIT_BF16X3)
    torch.cuda.synchronize()
    for ca, cb in outs:
        assert torch.equal(ca, want[0]) and torch.equal(cb, want[1])
    a.ctx.close()
    b.ctx.close()
