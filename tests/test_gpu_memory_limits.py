"""Calls under the context's memory limit: a call that is refused leaves the state as it was, and
later calls go on from there."""
import numpy as np
import pytest
import torch

from paper_2205_08941_gb300 import cq

pytestmark = pytest.mark.gpu


def batch(rows, seed=1):
    rng = np.random.default_rng(seed)
    put = lambda n: torch.tensor(rng.normal(size=(rows, n)).astype(np.float32), device="cuda:0")
    return put(64), put(81)


@pytest.mark.parametrize("fp32", [False, True])
def test_refused_growth_of_the_networks_buffers(fp32):
    """A larger batch that does not fit is refused; a batch of the old size then allocates again
    (or is refused in its turn) and gives the old results."""
    ctx = cq.Context(0)
    g = cq.Guess(ctx, seed=3, fp32_weights=fp32)
    X, T = batch(257)
    Xl, Tl = batch(4097, seed=2)
    out = g.forward(X)
    loss, gw, gb = g.train_step(X, T, 0.0, grads=True)
    used = ctx.mem_used()
    ctx.set_mem_limit(used)
    for refused in (lambda: g.forward(Xl), lambda: g.train_step(Xl, Tl, 0.0)):
        with pytest.raises(cq.CQError) as e:
            refused()
        assert e.value.status == 3
        assert torch.equal(g.forward(X), out)
        again = g.train_step(X, T, 0.0, grads=True)
        assert again[0] == loss and np.array_equal(again[1], gw) and np.array_equal(again[2], gb)
        assert ctx.mem_used() <= used
    # nothing fits any more: both are refused, and both work once they are allowed to
    with pytest.raises(cq.CQError):
        g.forward(Xl)
    ctx.set_mem_limit(1)
    for call in (lambda: g.forward(X), lambda: g.train_step(X, T, 0.0)):
        with pytest.raises(cq.CQError) as e:
            call()
        assert e.value.status == 3
    ctx.set_mem_limit(0)
    assert torch.equal(g.forward(X), out)
    assert g.train_step(X, T, 0.0) == loss
    g.close()
    ctx.close()


@pytest.mark.parametrize("fp32", [False, True])
def test_refused_training_step_is_no_step(fp32):
    """Adam's step count advances with the weights only."""
    X, T = batch(300)

    def train(refusals):
        ctx = cq.Context(0)
        g = cq.Guess(ctx, seed=3, fp32_weights=fp32)
        for _ in range(3):
            if refusals:
                ctx.set_mem_limit(1)
                Xl, Tl = batch(5000, seed=2)
                with pytest.raises(cq.CQError) as e:
                    g.train_step(Xl, Tl, 1e-3)
                assert e.value.status == 3
                ctx.set_mem_limit(0)
            g.train_step(X, T, 1e-3)
        w, b = g.params()
        g.close()
        ctx.close()
        return w, b

    for x, y in zip(train(True), train(False)):
        assert np.array_equal(x, y)


def test_fp64_probe_needs_no_memory():
    ctx = cq.Context(0)
    ctx.set_mem_limit(max(1, ctx.mem_used()))
    assert ctx.peak_fp64() > 1e11
    ctx.close()
