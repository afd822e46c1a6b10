"""Tiles that the batch autotuner keeps for the process: a class is the shape together with the form of
the R_p sum, so a set that is no cube (direct sum) is tuned for itself."""
import dataclasses

import numpy as np
import pytest

from oracle import epwi_oracle as O
from paper_2306_16493_gb300 import epwi, synth

pytestmark = pytest.mark.gpu
TUNED, CACHED = 1, 2


def test_a_cube_and_a_reordered_cube_are_two_classes():
    s = synth.tiny_system(3)
    # three Wannier functions: a shape that nothing else plans
    s = dataclasses.replace(s, nw=3, H=np.ascontiguousarray(s.H[:, :3, :3]),
                            g=np.ascontiguousarray(s.g[..., :3, :3]))
    p = np.roll(np.arange(len(s.Rp)), 1)
    t = dataclasses.replace(s, Rp=s.Rp[p].copy(), wp=s.wp[p].copy(), Phi=s.Phi[p].copy(),
                            g=np.ascontiguousarray(s.g[:, p]))
    grid = (4, 5, 3)
    mu = O.Grids(s, grid).band_centre()
    got = []
    for x in (s, t, s, t):
        b = epwi.Batch()
        b.setup([x], [grid])
        assert b.plan(300.0, [mu], 0.08, [mu - 2.0], [mu + 2.0], autotune=True) > 0
        got.append(b.tile(0)[2])
        b.close()
    assert got == [TUNED, TUNED, CACHED, CACHED]
