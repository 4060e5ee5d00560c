"""The order of a reduction's sums is that of 1024 CTAs of eight warps (warp w of CTA c takes blocks
8 c + w, 8 c + w + 8192, ..., a lane every 32nd value of a block), whatever the basis: traces, dots
and residual norms against a NumPy emulation of that order, to the bit.  The operands have 26
significant bits, so their products are exact and a multiply and an add round like an FMA.
And the per-cell reductions of uniform batches against each cell alone."""
import numpy as np
import pytest
import torch

from helpers import gpu_pattern, upload_pairs
from paper_2205_08941_gb300 import cq
from paper_2205_08941_gb300 import inputs as I

pytestmark = pytest.mark.gpu
CTAS, WARPS, LANES = 1024, 8, 32


def tree(v):
    """Sums over the last axis (a power of two long) as a warp's xor shuffles form them."""
    while v.shape[-1] > 1:
        h = v.shape[-1] // 2
        v = v[..., :h] + v[..., h:]
    return v[..., 0]


def ordered_sum(terms):
    """terms: (blocks, values of a block) of exact products, zeros where there is nothing to add."""
    n, e = terms.shape
    passes, chunks = -(-n // (CTAS * WARPS)), -(-e // LANES)
    t = np.zeros((passes * CTAS * WARPS, chunks * LANES))
    t[:n, :e] = terms
    t = t.reshape(passes, CTAS, WARPS, chunks, LANES)
    s = np.zeros((CTAS, WARPS, LANES))
    for p in range(passes):
        for c in range(chunks):
            s = s + t[p, :, :, c, :]
    part = tree(tree(s))  # warps, then the eight warp sums
    lane = np.zeros(256)
    for k in range(CTAS // 256):
        lane = lane + part[256 * k:256 * (k + 1)]
    return tree(tree(lane.reshape(8, 32)))


class Side:
    """A pattern and its blocks on the host: row, column and place of every block."""

    def __init__(self, ctx, cell, r):
        self.p, self.nb = gpu_pattern(ctx, cell, r), cell.nb
        rp, self.col, self.off, _ = (x.cpu().numpy() for x in self.p.export())
        self.row = np.repeat(np.arange(cell.n_atoms), np.diff(rp))
        self.at = {(i, j): b for b, (i, j) in enumerate(zip(self.row, self.col))}

    def values(self, seed):
        """26-bit values from 1 to 2: every sum of their products rounds."""
        rng = np.random.default_rng(seed)
        return rng.integers(2 ** 25, 2 ** 26, size=self.p.n_values) / 2.0 ** 25

    def block(self, v, b):
        ni, nj = self.nb[self.row[b]], self.nb[self.col[b]]
        return v[self.off[b]:self.off[b] + ni * nj].reshape(ni, nj)


def up(v):
    return torch.tensor(v, device="cuda:0")


# few blocks, more than one CTA's four partials hold, more than one pass of 8192 blocks
CASES = [((1, 1, 1), (9,), 4.0), ((3, 3, 3), (9,), 9.0), ((3, 3, 3), (4,), 12.0), ((5, 5, 5), (4,), 9.0),
         ((1, 1, 1), (13,), 4.0), ((3, 3, 3), (13,), 9.0), ((5, 5, 5), (5,), 9.0), ((2, 2, 2), (16,), 9.0),
         ((3, 3, 2), (5, 9, 13), 9.0), ((3, 3, 2), (1, 16, 4), 9.0)]


@pytest.mark.parametrize("shape,counts,r", CASES)
def test_sums_are_those_of_1024_ctas(shape, counts, r):
    ctx = cq.Context(0)
    cell = I.diamond_cell(shape, a=10.26, sigma=0.2, seed=21, norb=9)
    cell.nb = np.resize(np.array(counts, dtype=np.int32), cell.n_atoms)
    a, b = Side(ctx, cell, r), Side(ctx, cell, 0.8 * r)
    A, A2, B = a.values(1), a.values(2), b.values(3)
    words = int(cell.nb.max()) ** 2
    dot, trace = np.zeros((a.p.n_blocks, words)), np.zeros((a.p.n_blocks, words))
    for k, (i, j) in enumerate(zip(a.row, a.col)):
        x = a.block(A, k)
        dot[k, :x.size] = (x * a.block(A2, k)).ravel()
        partner = b.at.get((j, i))
        if partner is not None:
            trace[k, :x.size] = (x * b.block(B, partner).T).ravel()
    assert ctx.dot(a.p, up(A), up(A2)) == ordered_sum(dot)
    assert ctx.trace_prod(a.p, up(A), b.p, up(B)) == ordered_sum(trace)
    # the residual of a Hotelling step from T = I: ||S - I||_F over P_S + P_T (a square root
    # hides about half of the differences in a last place, so several S)
    v, T = Side(ctx, cell, 1.8 * r), np.zeros(b.p.n_values)
    for i, n in enumerate(cell.nb):
        b.block(T, b.at[(i, i)])[...] = np.eye(n)
    for seed in range(4, 10):
        S, frob = a.values(seed), np.zeros((v.p.n_blocks, words))
        for k, (i, j) in enumerate(zip(v.row, v.col)):
            s = a.at.get((i, j))
            if s is not None:
                x = a.block(S, s) - (np.eye(cell.nb[i]) if i == j else 0.0)
                frob[k, :x.size] = (x * x).ravel()
        assert ctx.hotelling_step(a.p, up(S), b.p, up(T)) == np.sqrt(ordered_sum(frob))
    ctx.close()


@pytest.mark.parametrize("norb", [9, 4, 13])
def test_uniform_batches_reduce_like_their_cells(norb):
    """Row sums (to the bit) and LNV sums (to rounding) of two cells of unequal sizes."""
    ctx = cq.Context(0)
    cells = [I.diamond_cell(s, a=10.26, sigma=0.1, seed=k, norb=norb)
             for k, s in enumerate([(2, 1, 1), (3, 2, 2)])]
    rS, rL = 7.0, 9.0
    pos, nb, start, boxes = I.concat_cells(cells)
    pos, nb = torch.tensor(pos, device="cuda:0"), torch.tensor(nb, dtype=torch.int32, device="cuda:0")
    qS, qL = (ctx.pattern_batch(pos, start, boxes, nb, [r, r]) for r in (rS, rL))
    matrices = I.overlap_hamiltonian_species if norb == 13 else I.overlap_hamiltonian
    S, H, L, one = [], [], [], []
    for k, c in enumerate(cells):
        pS, pL = gpu_pattern(ctx, c, rS), gpu_pattern(ctx, c, rL)
        s, h = matrices(c, I.silicon_model(rS))
        one.append((pS, pL))
        S.append(upload_pairs(ctx, pS, s))
        H.append(upload_pairs(ctx, pS, h))
        L.append(0.02 * upload_pairs(ctx, pL, I.random_blocks(c, rL, 50 + k)))
    ctx.sync()
    ne = [4.0 * c.n_atoms for c in cells]
    T = ctx.hotelling_init(qS, torch.cat(S), qL, ctx.zeros(qL))
    Tc = torch.cat([ctx.hotelling_init(pS, S[c], pL, ctx.zeros(pL)) for c, (pS, pL) in enumerate(one)])
    ctx.sync()
    assert torch.equal(T, Tc)
    lb = ctx.lnv_cells(qS, torch.cat(S), torch.cat(H), qL, torch.cat(L), ne)
    batch = [lb.state()] + [lb.step() for _ in range(3)]
    for c, (pS, pL) in enumerate(one):
        l1 = ctx.lnv(pS, S[c], H[c], pL, L[c].clone(), ne[c])
        for got, want in zip(batch, [l1.state()] + [l1.step() for _ in range(3)]):
            # the bound of the same comparison on mixed bases
            assert got[c]["energy"] == pytest.approx(want["energy"], rel=1e-13)
            assert got[c]["n_corr"] == want["n_corr"]
        l1.close()
    ctx.close()
