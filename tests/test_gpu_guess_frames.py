"""Pair frames where the third atom lies just outside the environment radius of 8 bohr."""
import numpy as np
import pytest

import oracle as O
from helpers import gpu_pattern
from oracle import guess as G
from paper_2205_08941_gb300 import cq
from paper_2205_08941_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_third_atom_just_outside_the_environment():
    """Atoms 2 and 3 lie 8.0063 bohr from the midpoint of atoms 0 and 1 and nobody is nearer.
    Rounded to FP32, the squared distance of the nearer one (3) is the larger."""
    pos = np.array([[0, 0, 0], [60.125 * 2 ** 30, 20.25 * 2 ** 30, 20.5 * 2 ** 30],
                    [40594601882, 10392815028, 8877514925],
                    [40616999052, 8936365396, 10205348138]]) / 2.0 ** 30
    cell = I.Cell(pos=pos, box=np.full(3, 200.0), nb=np.full(4, 4, dtype=np.int32))
    w2 = [float(((pos[k] - 0.5 * pos[1]) ** 2).sum()) for k in (2, 3)]
    assert 64.0 < w2[1] < w2[0] < 64.2
    ctx = cq.Context(0)
    pg, po = gpu_pattern(ctx, cell, 80.0), O.Pattern.of_cell(cell, 80.0)
    g = cq.Guess(ctx, seed=1)
    desc, frames, pairs = (v.cpu().numpy() for v in g.descriptors(pg))
    assert np.array_equal(pairs, G.pairs_of(po))
    q = next(q for q, b in enumerate(pairs) if (po.row[b], po.col[b]) == (0, 1))
    F, f = G.frame_and_descriptor(po, pairs[q])
    assert np.allclose(frames[q].reshape(3, 3), F, atol=2e-6)
    assert np.allclose(desc[q], f, rtol=1e-5, atol=1e-5)
    g.close()
    ctx.close()
