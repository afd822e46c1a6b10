"""The batch kernel's units (pairs of one q1, a block of columns): fewer columns than lanes, columns
beyond a whole block, tiles that end inside a run or inside a warp's share, single pairs, and
R_p sets that are no cube (direct sum).  Against each system's FP64 path within the mixed-precision
bound of the batch, 1e-4."""
import numpy as np
import pytest

from oracle import epwi_oracle as O
from paper_2306_16493_gb300 import epwi, synth
from tests.models import tb_dp_system

pytestmark = pytest.mark.gpu
T, ETA, TOL = 300.0, 0.08, 1e-4

SYSTEMS = [
    (lambda: tb_dp_system(r=1), (9, 5, 4)),              # 3 columns: ten pairs side by side
    (lambda: tb_dp_system(r=2), (4, 7, 5)),
    (lambda: synth.tiny_system(1), (1, 6, 7)),           # one q1: runs longer than a unit
    (lambda: synth.batch_system(15)[0], (3, 3, 2)),      # 432 columns: four blocks, the last ragged
    (lambda: synth.al_like_ws_system(), (4, 4, 5)),      # no cube
]


@pytest.mark.parametrize("mt", [1, 13, 64])
def test_units_match_the_fp64_path(mt):
    systems = [make() for make, _ in SYSTEMS]
    grids = [g for _, g in SYSTEMS]
    mu = np.array([O.Grids(s, g).band_centre() for s, g in zip(systems, grids)])
    lo, hi = mu - 2.0, mu + 2.0
    b = epwi.Batch()
    b.setup(systems, grids)
    for s in range(len(systems)):
        b.set_tile(s, min(mt, 13) if s == 3 else mt, 8)
    assert b.plan(T, mu, ETA, lo, hi, autotune=False) > 0
    b.run()
    for s, (sysm, grid) in enumerate(zip(systems, grids)):
        k, n, r = b.rates(s)
        ctx = epwi.Context(precision="fp64", device=0)
        ctx.setup(sysm)
        ctx.eigs(grid)
        ctx.scatter_rates(T, mu[s], ETA, lo[s], hi[s])
        k2, n2, r2 = ctx.rates()
        ctx.close()
        assert np.array_equal(k, k2) and np.array_equal(n, n2) and r2.max() > 0
        assert np.abs(r - r2).max() <= TOL * r2.max(), s
