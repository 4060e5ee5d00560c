"""Emulated-FP64 products whose scale factors are large: groups of one scalar row of A and one
scalar column of B whose large values meet only small partners, so that 2^(E_A + E_B) is far
above the product.  Every value lies on its group's digit grid and every sum fits 53 bits, so
the emulated product equals the FP64 one to the bit."""
import pytest
import torch

from helpers import gpu_pattern
from paper_2205_08941_gb300 import cq
from paper_2205_08941_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def blocks(p, nb, gen, col, E, small):
    """Blocks whose K orbital 0 holds +-(2 or 3) 2^(E - 2) and whose other K orbitals hold
    +-(1, 2 or 3) 2^small (col: K runs over columns, as in A), or the other way round for
    the right-hand operand, whose orbital 0 is small and whose other orbitals are large."""
    n = p.n_blocks
    rnd = lambda lo: torch.randint(lo, 4, (n, nb, nb), generator=gen, dtype=torch.float64)
    sgn = 2.0 * torch.randint(0, 2, (n, nb, nb), generator=gen, dtype=torch.float64) - 1.0
    big, little = rnd(2) * 2.0 ** (E - 2), rnd(1) * 2.0 ** small
    first = torch.zeros(nb, dtype=torch.bool)
    first[0] = True
    first = first[None, None, :] if col else ~first[None, :, None]
    v = torch.where(first, big, little) * sgn
    out = torch.zeros(n, p.n_values // n, dtype=torch.float64)
    out[:, :nb * nb] = v.reshape(n, -1)
    return out.reshape(-1).cuda()


@pytest.mark.parametrize("shape,nb,rA,rB,rC", [((2, 2, 2), 9, 8.0, 9.0, 12.0), ((3, 2, 2), 4, 9.0, 8.0, 8.0)])
@pytest.mark.parametrize("EA,EB", [(60, 60), (81, 60), (82, 60), (88, 60), (88, 59), (60, 88), (120, 20)])
def test_large_scales_of_small_products(shape, nb, rA, rB, rC, EA, EB):
    ctx = cq.Context(0)
    cell = I.diamond_cell(shape, a=10.26, sigma=0.1, seed=5, norb=nb)
    pA, pB, pC = (gpu_pattern(ctx, cell, r) for r in (rA, rB, rC))
    gen = torch.Generator().manual_seed(7)
    # orbital 0: about 2^(EA + EB - 36); the others 2^(EA + EB - 64) (digits 0 and 4, 7 and 0)
    A = blocks(pA, nb, gen, True, EA, EA - 63)
    B = blocks(pB, nb, gen, False, EB, EB - 36)
    want = ctx.bsmm(1.0, pA, A, pB, B, 0.0, pC, ctx.zeros(pC))
    got = ctx.bsmm(1.0, pA, A, pB, B, 0.0, pC, ctx.zeros(pC), cq.CQ_FP64_EMU)
    ctx.sync()
    assert 2.0 ** (EA + EB - 40) < float(want.abs().max()) < 2.0 ** 120
    assert torch.equal(got, want)
    ctx.close()
