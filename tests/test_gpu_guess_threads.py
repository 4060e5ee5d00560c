"""Learned start from several host threads, each with its own context and stream, on cells whose
rows need different amounts of shared memory."""
import ctypes
import threading

import pytest
import torch

from helpers import gpu_pattern
from paper_2205_08941_gb300 import cq
from paper_2205_08941_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_descriptors_of_short_and_long_rows_side_by_side():
    """Rows of about 800 neighbours (more shared memory than a launch gets by default) beside rows
    of a few."""
    jobs = 4 * [((6, 5, 5), 30.0, 400)] + 8 * [((1, 1, 1), 3.0, 10 ** 6)]
    errors, done, ready = [], threading.Event(), threading.Barrier(len(jobs), timeout=100)

    def work(shape, r, passes):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                ctx = cq.Context(0, stream=torch.cuda.current_stream())
                cell = I.diamond_cell(shape, a=10.26, sigma=0.1, seed=3, norb=4)
                p = gpu_pattern(ctx, cell, r)
                g = cq.Guess(ctx, seed=1)
                ref = g.descriptors(p)
                out = [torch.zeros_like(x) for x in ref]
                torch.cuda.current_stream().synchronize()
                args = [ctx.h, p.h] + [ctypes.c_void_p(x.data_ptr()) for x in out]
                call = cq.lib().cq_guess_descriptors
                ready.wait()  # every thread is set up: from here on they run side by side
                for n in range(passes):
                    ctx._check(call(*args))
                    if n and done.is_set():
                        break
                ctx.sync()
                assert all(torch.equal(x, y) for x, y in zip(out, ref))
                g.close()
                ctx.close()
        except Exception as e:  # noqa: BLE001  (reported by the test's thread)
            errors.append((shape, repr(e)))
            ready.abort()
        if shape != (1, 1, 1):
            done.set()

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
