"""The FP64 product's vector loads and paired launches: operands off the 16-byte boundary give the
aligned product's bits, and the LNV evaluation (whose products go two to a launch) gives the sums
of single products."""
import numpy as np
import pytest
import torch

from helpers import gpu_pattern, upload_pairs
from paper_2205_08941_gb300 import cq
from paper_2205_08941_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def shifted(t):
    """A copy of t that starts 8 bytes after a 16-byte boundary."""
    buf = torch.empty(t.numel() + 2, dtype=t.dtype, device=t.device)
    off = 1 if buf.data_ptr() % 16 == 0 else 0
    out = buf[off:off + t.numel()]
    out.copy_(t)
    assert out.data_ptr() % 16 == 8
    return out


@pytest.mark.parametrize("shape,norb,r", [((1, 1, 1), 9, 5.0), ((2, 2, 2), 9, 11.0),
                                          ((1, 1, 1), 4, 5.0), ((3, 2, 2), 4, 12.0)])
@pytest.mark.parametrize("beta", [0.0, 0.5])
def test_operands_off_the_16_byte_boundary(shape, norb, r, beta):
    ctx = cq.Context(0)
    cell = I.diamond_cell(shape, a=10.26, sigma=0.2, seed=3, norb=norb)
    pA, pB, pC = (gpu_pattern(ctx, cell, x) for x in (r, 0.8 * r, 1.3 * r))
    A, B, C0 = (upload_pairs(ctx, p, I.random_blocks(cell, x, k, symmetric=False))
                for p, x, k in ((pA, r, 1), (pB, 0.8 * r, 2), (pC, 1.3 * r, 3)))
    want = C0.clone()
    ctx.bsmm(1.5, pA, A, pB, B, beta, pC, want)
    for a, b in ((shifted(A), B), (A, shifted(B)), (shifted(A), shifted(B))):
        got = shifted(C0)
        ctx.bsmm(1.5, pA, a, pB, b, beta, pC, got)
        assert torch.equal(got, want)
    ctx.close()


@pytest.mark.parametrize("shape,counts", [((1, 1, 1), (9,)), ((2, 2, 1), (9,)), ((2, 2, 2), (4,)),
                                          ((1, 1, 2), (1, 4, 9, 13))])
def test_lnv_evaluation_equals_single_products(shape, counts):
    ctx = cq.Context(0)
    cell = I.diamond_cell(shape, a=10.26, sigma=0.2, seed=5, norb=9)
    cell.nb = np.resize(np.array(counts, dtype=np.int32), cell.n_atoms)
    rS, rL = 6.0, 8.0
    pS, pL = gpu_pattern(ctx, cell, rS), gpu_pattern(ctx, cell, rL)
    pX, pU = gpu_pattern(ctx, cell, rS + rL), gpu_pattern(ctx, cell, 2 * rS + rL)
    S = upload_pairs(ctx, pS, I.random_blocks(cell, rS, 1))
    H = upload_pairs(ctx, pS, I.random_blocks(cell, rS, 2))
    L = upload_pairs(ctx, pL, I.random_blocks(cell, rL, 4))
    ne = float(np.sum(cell.nb))
    lnv = ctx.lnv(pS, S, H, pL, L, ne, cq.CQ_FP64)  # corrects L towards the electron count
    rep = lnv.state()

    def prod(pa, a, pb, b, pc):
        c = ctx.zeros(pc)
        ctx.bsmm(1.0, pa, a, pb, b, 0.0, pc, c)
        return c
    X, Y = prod(pL, L, pS, S, pX), prod(pL, L, pS, H, pX)
    U = prod(pS, S, pX, X, pU)
    R1, R3 = prod(pU, U, pX, Y, pL), prod(pU, U, pX, X, pL)
    for got, p, q, r in ((rep["energy"], X, Y, R1), (rep["n_elec"], X, X, R3)):
        t2, t3 = ctx.trace_prod(pX, p, pX, q), ctx.trace_prod(pL, L, pL, r)
        # the same products bit for bit; only the two traces' sums and this combination round
        assert abs(got - 2.0 * (3.0 * t2 - 2.0 * t3)) <= 1e-12 * (abs(t2) + abs(t3))
    ctx.close()
