"""Several batches alive at once, of different widths: each goes on as if it
were alone."""
import numpy as np
import pytest

from paper_2306_10379_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _batch(p, seed):
    n = np.array([4 * p + 37, 3 * p + 50, 200], np.int32)
    return I.er_batch(3, I.SEED_BASE + seed, sizes=(n, np.full(3, p, np.int32)))


@pytest.mark.parametrize("use_graph", [False, True])
def test_wide_batch_outlives_a_narrow_one(torch_cuda, use_graph):
    from paper_2306_10379_gb300 import gsi
    widths = (32, 4, 16)
    inputs = [_batch(p, 60 + p) for p in widths]

    def run(b):
        if use_graph:
            b.solve(check=False)
        else:
            b.step(6)
        return [b.basis(i) for i in range(3)]

    alone = []
    for B in inputs:
        with gsi.Batch(B, tol=1e-12, max_iters=6) as b:
            alone.append(run(b))
    live = [gsi.Batch(B, tol=1e-12, max_iters=6) for B in inputs]  # the narrow ones are created after the wide one
    for b, ref in zip(live, alone):
        for (X, ev), (Xr, er) in zip(run(b), ref):
            assert np.array_equal(X, Xr) and np.array_equal(ev, er)
    for b in live:
        b.close()
