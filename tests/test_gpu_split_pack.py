"""Packing of 9-orbital operands for the split product: whole blocks staged through shared memory
with 16-byte copies, or 8-byte ones for operands off that boundary.  Both give the same bits, and
the product agrees with the oracle to the split's error, for atom counts around the group sizes
(14 and 7 atoms of a row group, 16 of a tail group) and for operands with few or no blocks in
common."""
import numpy as np
import pytest
import torch

import oracle as O
from helpers import (block_errors, gpu_pattern, layout_index, natural_scale, to_oracle,
                     upload_pairs)
from paper_2205_08941_gb300 import cq
from paper_2205_08941_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def cell_of(n):
    """n atoms of a diamond cell large enough to hold them."""
    full = I.diamond_cell((2, 2, 2), a=10.26, sigma=0.2, seed=17, norb=9)
    return I.Cell(pos=full.pos[:n].copy(), box=full.box.copy(), nb=full.nb[:n].copy())


def shifted(t):
    buf = torch.empty(t.numel() + 2, dtype=t.dtype, device=t.device)
    off = 1 if buf.data_ptr() % 16 == 0 else 0
    out = buf[off:off + t.numel()]
    out.copy_(t)
    assert out.data_ptr() % 16 == 8
    return out


@pytest.mark.parametrize("n,rA,rB", [(1, 5.0, 5.0), (7, 9.0, 9.0), (8, 5.0, 12.0), (14, 12.0, 6.0),
                                     (15, 9.0, 9.0), (16, 20.0, 20.0), (17, 20.0, 1.0),
                                     (33, 8.0, 20.0), (64, 1.0, 12.0), (64, 15.0, 9.0)])
def test_packed_operands(n, rA, rB):
    ctx = cq.Context(0)
    cell = cell_of(n)
    rC = rA + rB
    pA, pB, pC = (gpu_pattern(ctx, cell, x) for x in (rA, rB, rC))
    a = I.random_blocks(cell, rA, 1, symmetric=False)
    b = I.random_blocks(cell, rB, 2, symmetric=False)
    A, B = upload_pairs(ctx, pA, a), upload_pairs(ctx, pB, b)
    want = ctx.bsmm(1.0, pA, A, pB, B, 0.0, pC, ctx.zeros(pC), cq.CQ_SPLIT_BF16X3)
    for x, y in ((shifted(A), B), (A, shifted(B)), (shifted(A), shifted(B))):
        got = ctx.bsmm(1.0, pA, x, pB, y, 0.0, pC, ctx.zeros(pC), cq.CQ_SPLIT_BF16X3)
        assert torch.equal(got, want)
    oA, oB, oC = (O.Pattern.of_cell(cell, x) for x in (rA, rB, rC))
    vA, vB = O.scatter(oA, a), O.scatter(oB, b)
    ref = O.bsmm(1.0, oA, vA, oB, vB, 0.0, oC)
    scale = natural_scale(oA, vA, oB, vB, oC)
    got = to_oracle(want, layout_index(pC, oC))
    # dropped plane products and operand truncation are 3 * 2^-24 of each term; FP32 sums of up
    # to 64 steps between drains add 64 * 2^-24
    err, _ = block_errors(oC, got, ref)
    assert np.all(err <= 67 * 2.0 ** -24 * scale + 1e-300)
    ctx.close()


@pytest.mark.parametrize("rA,rB,rC", [(1.0, 1.0, 18.0), (6.0, 1.0, 25.0), (9.0, 9.0, 40.0)])
def test_tiles_without_work(rA, rB, rC):
    """C reaches farther than the operands: tiles with no K step at all between tiles with some."""
    ctx = cq.Context(0)
    cell = I.diamond_cell((6, 2, 2), a=10.26, sigma=0.2, seed=17, norb=9)
    pA, pB, pC = (gpu_pattern(ctx, cell, x) for x in (rA, rB, rC))
    a = I.random_blocks(cell, rA, 1, symmetric=False)
    b = I.random_blocks(cell, rB, 2, symmetric=False)
    C = ctx.empty(pC).fill_(7.0)
    ctx.bsmm(1.0, pA, upload_pairs(ctx, pA, a), pB, upload_pairs(ctx, pB, b), 0.0, pC, C,
             cq.CQ_SPLIT_BF16X3)
    oA, oB, oC = (O.Pattern.of_cell(cell, x) for x in (rA, rB, rC))
    vA, vB = O.scatter(oA, a), O.scatter(oB, b)
    ref = O.bsmm(1.0, oA, vA, oB, vB, 0.0, oC)
    err, _ = block_errors(oC, to_oracle(C, layout_index(pC, oC)), ref)
    assert np.all(err <= 67 * 2.0 ** -24 * natural_scale(oA, vA, oB, vB, oC) + 1e-300)
    ctx.close()
