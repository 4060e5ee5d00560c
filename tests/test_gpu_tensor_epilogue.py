"""Tensor-core products: the drain's and the epilogue's branches give the same values.  Powers
of two are exact in every step, so scaled operands and coefficients must give bit-equal
results, whichever path they take (ordinary or extreme group exponents; alpha = 1 and beta =
0 or not; C on a 16-byte boundary or not)."""
import pytest
import torch

from helpers import gpu_pattern, upload_pairs
from paper_2205_08941_gb300 import cq
from paper_2205_08941_gb300 import inputs as I

pytestmark = pytest.mark.gpu
PRECS = [cq.CQ_SPLIT_BF16X3, cq.CQ_FP64_EMU]


def product(shape, norb, rA, rB, rC):
    ctx = cq.Context(0)
    cell = I.diamond_cell(shape, a=10.26, sigma=0.1, seed=5, norb=norb)
    pA, pB, pC = (gpu_pattern(ctx, cell, r) for r in (rA, rB, rC))
    A = upload_pairs(ctx, pA, I.random_blocks(cell, rA, 1, symmetric=False))
    B = upload_pairs(ctx, pB, I.random_blocks(cell, rB, 2, symmetric=False))

    def run(A=A, B=B, alpha=1.0, beta=0.0, C=None, prec=cq.CQ_SPLIT_BF16X3):
        C = ctx.zeros(pC) if C is None else C
        ctx.bsmm(alpha, pA, A, pB, B, beta, pC, C, prec)
        ctx.sync()
        return C

    return ctx, pC, A, B, run


# sparse tiles (most slots without a block), full ones, and the 4-orbital layout
SHAPES = [((4, 3, 2), 9, 12.0, 9.0, 7.0), ((2, 2, 2), 9, 8.0, 9.0, 17.0), ((3, 2, 2), 4, 9.0, 8.0, 8.0)]


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("shape", SHAPES)
def test_epilogue_paths_agree_to_the_bit(shape, prec):
    ctx, pC, A, B, run = product(*shape)
    C = run(prec=prec)
    assert float(C.abs().max()) > 0.0
    assert torch.equal(run(alpha=2.0, prec=prec), 2.0 * C)
    assert torch.equal(run(alpha=-0.5, prec=prec), -0.5 * C)
    old = torch.randn(pC.n_values, dtype=torch.float64, device="cuda:0")
    # beta * old + C is one rounding of each value: the same sum in torch
    assert torch.equal(run(beta=1.0, C=old.clone(), prec=prec)[C != 0], (old + C)[C != 0])
    odd = torch.zeros(pC.n_values + 1, dtype=torch.float64, device="cuda:0")[1:]
    assert odd.data_ptr() % 16 == 8 and torch.equal(run(C=odd, prec=prec), C)
    ctx.close()


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("ea,eb", [(60, -60), (80, -80), (-120, 100), (-100, 30), (40, 40)])
def test_emulated_scales_are_exact(shape, ea, eb):
    """Group exponents inside and beyond the range of the drain's single scale factor."""
    ctx, pC, A, B, run = product(*shape)
    C = run(prec=cq.CQ_FP64_EMU)
    S = run(A=A * 2.0 ** ea, B=B * 2.0 ** eb, prec=cq.CQ_FP64_EMU)
    if ea + eb < -60:  # the smallest words of the three-float sums may leave FP32's range
        err = float((S * 2.0 ** -(ea + eb) - C).abs().max())
        assert err <= 2.0 ** -50 * float(C.abs().max())
    else:
        assert torch.equal(S * 2.0 ** -(ea + eb), C)
    ctx.close()
