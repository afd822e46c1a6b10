"""Contexts of several host threads at once: kernels whose shared memory depends on the grid are
launched by all of them, and every call gives the rates that it gives alone."""
import threading

import numpy as np
import pytest

from paper_2306_16493_gb300 import epwi, synth

pytestmark = pytest.mark.gpu

# grids of few and many axis points and q2 groups: different shared memory of one kernel
GRIDS = [(6, 4, 5), (64, 4, 3), (5, 3, 40), (18, 15, 20), (48, 10, 11)]


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16x3"])
def test_grids_of_different_layouts_together(precision):
    s = synth.al_like_system()
    ctxs, want, err = [], [], []
    for grid in GRIDS:
        ctx = epwi.Context(precision=precision)
        ctx.setup(s)
        ctx.eigs(grid)
        mu = 0.5 * sum(ctx.band_range())
        ctx.scatter_rates(300.0, mu, 0.05, mu - 0.5, mu + 0.5)
        ctxs.append((ctx, mu))
        want.append(ctx.rates()[2])

    def work(i):
        ctx, mu = ctxs[i]
        try:
            for _ in range(150):
                ctx.scatter_rates(300.0, mu, 0.05, mu - 0.5, mu + 0.5)
                assert np.array_equal(ctx.rates()[2], want[i])
        except Exception as e:                    # noqa: BLE001 (reported by the main thread)
            err.append((GRIDS[i], repr(e)))

    th = [threading.Thread(target=work, args=(i,)) for i in range(len(GRIDS))]
    for t in th:
        t.start()
    for t in th:
        t.join()
    for ctx, _ in ctxs:
        ctx.close()
    assert not err, err
