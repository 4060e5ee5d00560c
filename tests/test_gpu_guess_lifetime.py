"""A learned start that outlives its context: its calls are refused and it can be destroyed."""
import pytest
import torch

from paper_2205_08941_gb300 import cq

pytestmark = pytest.mark.gpu


def test_guess_outlives_its_context():
    ctx = cq.Context(0)
    kept, gone = cq.Guess(ctx, seed=1), cq.Guess(ctx, seed=2)
    x = torch.zeros((20, 64), device="cuda:0")
    t = torch.zeros((20, 81), device="cuda:0")
    kept.train_step(x, t, 1e-3)
    gone.close()
    cq.lib().cq_ctx_destroy(ctx.h)  # not Context.close, which closes the objects first
    ctx.h = None
    for call in (lambda: kept.forward(x), lambda: kept.train_step(x, t, 1e-3), lambda: kept.params(),
                 lambda: kept.loss_sum(), lambda: kept.fit_scale(x, t)):
        with pytest.raises(cq.CQError) as e:
            call()
        assert e.value.status == 1
    kept.close()
    other = cq.Context(0)
    g = cq.Guess(other, seed=1)
    assert g.forward(x).shape == (20, 81)
    g.close()
    other.close()
