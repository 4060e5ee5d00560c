"""Learned start: the per-row descriptor kernel and the tensor-core training step at the sizes
where they branch -- rows cached in shared memory and rows too long for it, cells without a
neighbour or with atoms on the pair axis only, batches off the tile and chunk sizes."""
import numpy as np
import pytest
import torch

import oracle as O
from helpers import gpu_pattern
from oracle import guess as G
from paper_2205_08941_gb300 import cq
from paper_2205_08941_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# a 1-cell row with few atoms, an ordinary one, a perfect lattice (ties, on-axis atoms), a row
# of 2744 atoms (not cached)
@pytest.mark.parametrize("shape,norb,sigma,r,checked", [
    ((1, 1, 1), 9, 0.1, 3.0, 8), ((3, 2, 2), 4, 0.1, 12.0, 40), ((2, 2, 2), 9, 0.0, 8.0, 40),
    ((7, 7, 7), 4, 0.1, 70.0, 6)])
def test_descriptors_match_the_oracle(shape, norb, sigma, r, checked):
    ctx = cq.Context(0)
    cell = I.diamond_cell(shape, a=10.26, sigma=sigma, seed=3, norb=norb)
    pg = gpu_pattern(ctx, cell, r)
    g = cq.Guess(ctx, seed=1)
    desc, frames, pairs = (v.cpu().numpy() for v in g.descriptors(pg))
    po = O.Pattern.of_cell(cell, r)
    ref = G.pairs_of(po)
    assert np.array_equal(pairs, ref)
    rng = np.random.default_rng(0)
    for q in rng.choice(len(ref), size=min(checked, len(ref)), replace=False):
        F, f = G.frame_and_descriptor(po, ref[q])
        if sigma == 0.0:
            # a perfect lattice: the third atom is one of several at equal distance, and
            # rounding picks it; what does not depend on the choice agrees, and the frame is one
            R, iso = frames[q].reshape(3, 3), np.r_[0:10, 10:64:9]
            assert np.allclose(R @ R.T, np.eye(3), atol=4e-6) and np.linalg.det(R) > 0.99
            assert np.allclose(desc[q][iso], f[iso], rtol=1e-5, atol=1e-5 * max(1.0, np.abs(f).max()))
            continue
        assert np.allclose(frames[q].reshape(3, 3), F, atol=2e-6)
        assert np.allclose(desc[q], f, rtol=1e-5, atol=1e-5 * max(1.0, np.abs(f).max()))
    g.close()
    ctx.close()


@pytest.mark.parametrize("rows", [1, 15, 16, 17, 127, 128, 129, 257, 4097])
def test_training_step_gradients(rows):
    """BF16 operands against the FP64 network: the tolerances of the existing BF16 test."""
    ctx = cq.Context(0)
    rng = np.random.default_rng(rows)
    g = cq.Guess(ctx, seed=3)
    X = rng.normal(size=(rows, 64)).astype(np.float32)
    T = rng.normal(size=(rows, 81)).astype(np.float32)
    sc = [rng.normal(size=64), 1 + rng.random(64), rng.normal(size=81), 1 + rng.random(81)]
    sc = [v.astype(np.float32) for v in sc]
    g.set_scale(*sc)
    w, b = g.params()
    b = (rng.normal(size=b.shape) * 0.1).astype(np.float32)
    g.set_params(w, b)
    Xg, Tg = torch.tensor(X, device="cuda:0"), torch.tensor(T, device="cuda:0")
    loss, gw, gb = g.train_step(Xg, Tg, 0.0, grads=True)
    lo, gwo, gbo = G.loss_and_grads(w, b, X, T, *sc)
    assert loss == pytest.approx(lo, rel=1e-2)
    assert np.abs(gw - gwo).max() <= 3e-2 * np.abs(gwo).max()
    assert np.abs(gb - gbo).max() <= 3e-2 * np.abs(gbo).max()
    # a smaller batch after a larger one uses the same buffers
    g.train_step(torch.cat([Xg, Xg]), torch.cat([Tg, Tg]), 0.0)
    again = g.train_step(Xg, Tg, 0.0, grads=True)
    assert again[0] == loss and np.array_equal(again[1], gw) and np.array_equal(again[2], gb)
    g.close()
    ctx.close()
