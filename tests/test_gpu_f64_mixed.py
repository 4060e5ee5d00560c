"""The FP64 product on mixed bases: blocks sorted by width and tasks by the orbital count of k
give the oracle's product on every combination -- one atom per count, rare counts, a batch
whose cells differ, and products of few and of many rows."""
import numpy as np
import pytest
import torch

import oracle as O
from helpers import assert_product_close, gpu_pattern, layout_index, natural_scale, to_oracle, upload_pairs
from paper_2205_08941_gb300 import cq
from paper_2205_08941_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,counts,r", [
    ((1, 1, 1), (1, 2, 3, 6, 7, 11, 15, 16), 6.0),   # every atom its own count
    ((2, 2, 2), (5, 9, 13), 9.0),
    ((2, 2, 2), (4, 9), 12.0),
    ((3, 2, 2), (13,), 8.0),                          # uniform, but on the general kernel
    ((3, 3, 2), (9, 9, 9, 9, 9, 9, 9, 16), 8.0)])     # one rare count
def test_mixed_products_match_the_oracle(shape, counts, r):
    ctx = cq.Context(0)
    cell = I.diamond_cell(shape, a=10.26, sigma=0.2, seed=11, norb=9)
    cell.nb = np.resize(np.array(counts, dtype=np.int32), cell.n_atoms)
    rA, rB, rC = r, 0.8 * r, 1.3 * r
    pA, pB, pC = (gpu_pattern(ctx, cell, x) for x in (rA, rB, rC))
    A, B = (I.random_blocks(cell, x, k, symmetric=False) for x, k in ((rA, 1), (rB, 2)))
    oA, oB, oC = (O.Pattern.of_cell(cell, x) for x in (rA, rB, rC))
    C = ctx.zeros(pC)
    ctx.bsmm(1.0, pA, upload_pairs(ctx, pA, A), pB, upload_pairs(ctx, pB, B), 0.0, pC, C)
    vA, vB = O.scatter(oA, A), O.scatter(oB, B)
    ref = O.bsmm(1.0, oA, vA, oB, vB, 0.0, oC)
    scale = natural_scale(oA, vA, oB, vB, oC)
    assert_product_close(oC, to_oracle(C, layout_index(pC, oC)), ref, scale)
    ctx.close()
