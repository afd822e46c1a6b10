"""The sum-factorised rates read the sieve's decision mask: items of two runs that hold more than
256 pairs together, several q2 groups per plane block, one and two axis-1 points, odd column counts,
and the list positions of the Gamma capture in later groups.  FP32 against the FP64 path (itself
pinned to the oracle) within the fp32 mode's 1e-5 for rates and 1e-4 for mean free paths, which is
what its other tests allow."""
import numpy as np
import pytest

from oracle import epwi_oracle as O
from paper_2306_16493_gb300 import epwi, synth
from tests.models import tb_dp_system

pytestmark = pytest.mark.gpu


def _system(name):
    if name.startswith("one_band"):
        return tb_dp_system(r=int(name[-1]))
    return getattr(synth, f"{name}_system")()


@pytest.mark.parametrize("name,grid,half,eta", [
    ("tiny", (3, 17, 19), None, 0.3),             # full runs: 256 + 256 pairs in one item
    ("al_like", (1, 5, 7), None, 0.05),
    ("al_like", (2, 16, 32), None, 0.2),          # both self-paired items, whole plane blocks
    ("al_like", (5, 260, 1), 0.5, 0.05),          # 256 q2 in a plane block
    ("one_band_2", (9, 17, 19), None, 0.1),
    ("si_like", (4, 12, 6), None, 0.05),          # W = 8: one q2 per group
])
def test_rates_and_capture(name, grid, half, eta):
    s = _system(name)
    gr = O.Grids(s, grid)
    mu = gr.band_centre()
    lo, hi = (-1e9, 1e9) if half is None else (mu - half, mu + half)
    out = {}
    for prec in ("fp64", "fp32"):
        ctx = epwi.Context(precision=prec, device=0)
        ctx.setup(s)
        ctx.eigs(grid)
        _, npairs = ctx.scatter_rates(300.0, mu, eta, lo, hi)
        rate = ctx.rates()[2]
        ctx.ibte(300.0, mu, eta, lo, hi, max_iter=2, tol=0.0)
        out[prec] = (npairs, rate, ctx.mfp())
        ctx.close()
    (na, ra, fa), (nb, rb, fb) = out["fp64"], out["fp32"]
    assert na == nb and ra.max() > 0
    assert np.abs(ra - rb).max() <= 1e-5 * ra.max()
    assert np.abs(fa - fb).max() <= 1e-4 * np.abs(fa).max()
