"""The window's k-points and states in order, on grids that fill, just miss and just pass a block of the
kernel that counts them (4096 points), and on one of many blocks."""
import numpy as np
import pytest

from oracle import epwi_oracle as O
from paper_2306_16493_gb300 import epwi, synth
from tests.models import tb_dp_system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make,grid,half", [
    (tb_dp_system, (16, 16, 16), 0.3), (tb_dp_system, (13, 15, 21), 0.3), (tb_dp_system, (16, 16, 17), 9.0),
    (synth.al_like_system, (16, 16, 16), 20.0),       # every band of every point
    (synth.al_like_system, (30, 24, 20), 0.2),
])
def test_states_in_order(make, grid, half):
    s = make()
    gr = O.Grids(s, grid)
    mu = gr.band_centre()
    ik, n = gr.window_states(mu - half, mu + half)
    o = np.lexsort((n, ik))
    ctx = epwi.Context(precision="fp32")
    ctx.setup(s)
    ctx.eigs(grid)
    ns, _ = ctx.scatter_rates(300.0, mu, 0.005, mu - half, mu + half)
    k, b, _ = ctx.rates()
    assert ns == len(ik) > 0
    assert np.array_equal(k, ik[o]) and np.array_equal(b, n[o])
    assert np.array_equal(ctx.sieve()[0], np.unique(ik))
    ctx.close()
