"""The autotuner's tiles, which the library keeps for the whole process, used by batches of several host
threads at once."""
import threading

import numpy as np
import pytest

from oracle import epwi_oracle as O
from paper_2306_16493_gb300 import epwi, synth

pytestmark = pytest.mark.gpu


def _together(n, work):
    err = []

    def run(i):
        try:
            work(i)
        except BaseException as e:                # noqa: BLE001 (reported by the main thread)
            err.append(repr(e))
    th = [threading.Thread(target=run, args=(i,)) for i in range(n)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not err, err


def test_batches_planned_by_several_threads():
    """Each thread plans and runs batches of shapes that the others plan as well: the rates are those of a
    single batch with the same tiles."""
    systems = [synth.tiny_system(1), synth.tiny_system(2), synth.al_like_system(), synth.al_like_ws_system()]
    grids = [(4, 4, 5), (5, 4, 3), (3, 4, 4), (4, 3, 3)]
    mus = np.array([O.Grids(s, g).band_centre() for s, g in zip(systems, grids)])

    def rates(order, tiles=None):
        b = epwi.Batch()
        b.setup([systems[x] for x in order], [grids[x] for x in order])
        for x, t in enumerate(tiles or []):
            b.set_tile(x, t[0], t[1])
        mu = mus[order]
        b.plan(300.0, mu, 0.08, mu - 2.0, mu + 2.0, autotune=tiles is None)
        b.run()
        out = {x: (b.tile(i)[:2], b.rates(i)[2]) for i, x in enumerate(order)}
        b.close()
        return out
    got = [[] for _ in range(4)]

    def work(i):
        for j in range(4):
            got[i].append(rates([(i + j + x) % 4 for x in range(3)]))
    _together(4, work)
    for run in sum(got, []):
        order = list(run)
        want = rates(order, [run[x][0] for x in order])
        for x in order:
            assert np.array_equal(run[x][1], want[x][1]), x
