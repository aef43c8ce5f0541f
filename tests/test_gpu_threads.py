"""Host threads, each with a context and a stream of its own, whose calls run
the same kernels with different amounts of shared memory: no call may be
refused, and every result is that of the same call alone (FP64 to 1e-9 of the
largest value: the forces are summed by atomics)."""
import threading

import numpy as np
import pytest

from paper_1803_07491_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

THREADS = 4


@pytest.fixture(scope="module")
def bop():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1803_07491_gb300 import build, bop as b
    build.build()
    return b


def _pair(model, small, large):
    return [I.with_run(I.small_bcc(*c, 0.05, 31, model=model), n_mom=m) for c, m in (small, large)]


@pytest.mark.parametrize("ws,runs", [
    (_pair(I.MODEL_S, ((2, 2, 2), 3), ((3, 3, 3), 9)), 1500),    # the structure alone
    (_pair(I.MODEL_S, ((2, 2, 2), 5), ((3, 3, 3), 9)), 400),
    (_pair(I.MODEL_SD, ((2, 2, 2), 5), ((3, 2, 2), 7)), 400)], ids=["structure", "s", "sd"])
def test_threads_of_different_sizes(bop, ws, runs):
    def call(ctx, w):
        if runs > 1000:
            st = ctx.build(w.pos, w.cell, w.pbc)
            return np.array([st["n_sites"], st["n_adj"], st["moment_products"]], float)
        r = ctx.evaluate(w.pos, w.cell, w.pbc)
        return np.concatenate([r.forces.cpu().numpy().ravel(), [r.e_total]])

    ref = []
    for w in ws:
        ctx = bop.Context(w.model, w.run, "fp64")
        ref.append(call(ctx, w))
        ctx.close()
    errors = []

    def work(w, r):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                ctx = bop.Context(w.model, w.run, "fp64")
                for _ in range(runs):
                    if np.max(np.abs(call(ctx, w) - r)) > 1e-9 * max(1.0, np.abs(r).max()):
                        errors.append("result differs")
                ctx.close()
        except bop.BopError as e:
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(ws[q % 2], ref[q % 2])) for q in range(THREADS)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]
