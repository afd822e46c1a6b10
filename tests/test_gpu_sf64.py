"""Sum-factorised FP64 rates (scatter_sf64.cu) against the oracle at 1e-10 (FP64 rounding of sums of
some 10^4 terms): ragged plane blocks, several q2 groups, one to eight bands, R_p sets that are
no cube, and the Gamma capture of the iterative BTE."""
import numpy as np
import pytest

from oracle import epwi_oracle as O
from paper_2306_16493_gb300 import epwi, synth
from tests.models import tb_dp_system
from tests.parity import compare_rates, gpu_run, oracle_run

pytestmark = pytest.mark.gpu
TOL = 1e-10


def _system(name):
    if name.startswith("one_band"):
        return tb_dp_system(r=int(name[-1]))
    return getattr(synth, f"{name}_system")()


@pytest.mark.parametrize("name,grid,half,eta", [
    ("one_band_1", (7, 6, 5), None, 0.05),
    ("one_band_2", (5, 17, 19), None, 0.05),
    ("tiny", (3, 4, 5), None, 0.05),
    ("tiny", (2, 33, 40), 0.4, 0.03),             # six plane blocks, many q2 per block
    ("al_like", (6, 18, 17), 0.3, 0.04),
    ("al_like", (4, 260, 1), 0.3, 0.05),          # N3 = 1: 256 q2 values in a plane block
    ("al_like_ws", (9, 20, 15), 0.3, 0.04),
    ("si_like", (6, 5, 4), None, 0.05),
])
def test_rates_match_the_oracle(name, grid, half, eta):
    s = _system(name)
    gr = O.Grids(s, grid)
    mu = gr.band_centre()
    lo, hi = (-1e9, 1e9) if half is None else (mu - half, mu + half)
    ref = oracle_run(gr, 300.0, mu, eta, lo, hi)
    out = gpu_run(s, grid, 300.0, mu, eta, lo, hi)
    assert out["n_pairs"] == ref["n_pairs"]
    err, n = compare_rates(out, ref, gr.eps, TOL)
    assert n > 0 and err <= TOL, err
    out["ctx"].close()


def test_gamma_rows_of_skipped_bands_are_zero():
    """Final bands out of reach are not written by the capture: after one step from F0 = v tau the
    mean free paths equal the oracle's, also when the Gamma buffer held another run's values."""
    s, grid = synth.tiny_system(), (6, 5, 7)
    gr = O.Grids(s, grid)
    mu = gr.band_centre()
    ctx = epwi.Context()
    ctx.setup(s)
    ctx.eigs(grid)
    for eta, lo, hi in ((0.08, -1e9, 1e9), (0.03, mu - 1.0, mu + 1.0)):
        ctx.ibte(300.0, mu, eta, lo, hi, max_iter=1, tol=0.0)
    ref = O.ibte(gr, 300.0, mu, 0.03, mu - 1.0, mu + 1.0, max_iter=1, tol=0.0)
    F = ctx.mfp()
    assert np.abs(F - ref["F"]).max() <= TOL * np.abs(ref["F"]).max()
    ctx.close()
