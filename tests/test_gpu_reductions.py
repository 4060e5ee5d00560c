"""One-launch reductions: traces, dots, residual norms and Gershgorin row sums against NumPy on
every basis path (9, 4, 13 orbitals, mixed), from fewer blocks than one CTA takes to more than
the whole grid takes at once, with partners absent and with NaN in the padding words."""
import numpy as np
import pytest
import torch

from helpers import gpu_pattern, upload_pairs
from paper_2205_08941_gb300 import cq
from paper_2205_08941_gb300 import inputs as I

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


def dense(pairs, cell):
    off = np.concatenate([[0], np.cumsum(cell.nb)])
    m = np.zeros((off[-1], off[-1]))
    for p in range(pairs.n_pairs):
        i, j = pairs.i[p], pairs.j[p]
        m[off[i]:off[i + 1], off[j]:off[j + 1]] = \
            pairs.values[pairs.off[p]:pairs.off[p + 1]].reshape(cell.nb[i], cell.nb[j])
    return m


def make(shape, counts):
    cell = I.diamond_cell(shape, a=10.26, sigma=0.2, seed=21, norb=9)
    cell.nb = np.resize(np.array(counts, dtype=np.int32), cell.n_atoms)
    return cell


CASES = [((1, 1, 1), (9,)), ((2, 2, 1), (9,)), ((3, 3, 3), (9,)), ((1, 1, 1), (4,)),
         ((3, 3, 3), (4,)), ((2, 2, 2), (13,)), ((3, 2, 2), (1, 16, 5, 9)), ((1, 1, 1), (1,))]


@pytest.mark.parametrize("shape,counts", CASES)
@pytest.mark.parametrize("rA,rB", [(4.0, 9.0), (9.0, 4.0)])
def test_trace_and_dot(shape, counts, rA, rB):
    ctx = cq.Context(0)
    cell = make(shape, counts)
    pA, pB = gpu_pattern(ctx, cell, rA), gpu_pattern(ctx, cell, rB)
    a = I.random_blocks(cell, rA, 1, symmetric=False)
    a2 = I.random_blocks(cell, rA, 3, symmetric=False)
    b = I.random_blocks(cell, rB, 2, symmetric=False)
    dA, dA2, dB = (dense(x, cell) for x in (a, a2, b))
    A, A2, B = upload_pairs(ctx, pA, a), upload_pairs(ctx, pA, a2), upload_pairs(ctx, pB, b)
    pad = upload_pairs(ctx, pA, I.PairBlocks(a.i, a.j, a.off, np.ones_like(a.values))) == 0
    if all(c % 2 for c in counts):  # a padding word after every block
        assert int(pad.sum()) == pA.n_blocks
    A[pad], A2[pad] = float("nan"), float("nan")
    for got, want, mag in (
            (ctx.trace_prod(pA, A, pB, B), np.sum(dA * dB.T), np.sum(np.abs(dA * dB.T))),
            (ctx.dot(pA, A, A2), np.sum(dA * dA2), np.sum(np.abs(dA * dA2)))):
        # two orders of the same sum: each adds below a few thousand terms in a chain or a tree
        assert abs(got - want) <= 4096 * EPS * mag
    assert ctx.trace_prod(pA, A, pB, B) == ctx.trace_prod(pA, A, pB, B)
    ctx.close()


def test_more_blocks_than_one_pass_of_the_grid():
    ctx = cq.Context(0)
    cell = make((5, 5, 5), (9,))
    p = gpu_pattern(ctx, cell, 12.0)
    assert p.n_blocks > 1024 * 8
    g = torch.Generator(device="cuda").manual_seed(4)
    A = torch.randn(p.n_values, dtype=torch.float64, device="cuda", generator=g)
    B = torch.randn(p.n_values, dtype=torch.float64, device="cuda", generator=g)
    keep = (torch.arange(p.n_values, device="cuda") % 82) < 81
    want, mag = (A * B * keep).sum().item(), (A * B * keep).abs().sum().item()
    assert abs(ctx.dot(p, A, B) - want) <= 4096 * EPS * mag
    ctx.close()


@pytest.mark.parametrize("shape,counts", CASES)
def test_row_sums_and_residual(shape, counts):
    ctx = cq.Context(0)
    cell = make(shape, counts)
    r = 6.0
    pS, pT = gpu_pattern(ctx, cell, r), gpu_pattern(ctx, cell, 8.0)
    s = I.random_blocks(cell, r, 5)
    dS = dense(s, cell)
    S = upload_pairs(ctx, pS, s)
    T = ctx.zeros(pT)
    ctx.hotelling_init(pS, S, pT, T)  # T = I / max_r sum_q |S_rq|
    scale = 1.0 / np.abs(dS).sum(axis=1).max()
    t = ctx.dot(pT, T, T)
    n = float(cell.nb.sum())
    assert abs(t - n * scale * scale) <= 4096 * EPS * n * scale * scale
    v = dS * scale - np.eye(dS.shape[0])
    want = np.sqrt((v * v).sum())
    got = ctx.hotelling_step(pS, S, pT, T)
    assert abs(got - want) <= 4096 * EPS * want
    ctx.close()
