"""A delta cut-off that no energy difference reaches (sieve_c infinite, or c eta beyond FP32): every q
with a kept mode is a pair of every window k-point, and nothing else is, on grids whose planes do
not fill their last block; the rates are those of a finite cut-off that keeps the same pairs."""
import numpy as np
import pytest

from oracle import epwi_oracle as O
from paper_2306_16493_gb300 import epwi, synth

pytestmark = pytest.mark.gpu
T, ETA = 300.0, 0.02


def _rates(s, grid, mu, half, c, precision):
    ctx = epwi.Context(precision=precision, sieve_c=c)
    ctx.setup(s)
    ctx.eigs(grid)
    ns, npairs = ctx.scatter_rates(T, mu, ETA, mu - half, mu + half)
    out = ctx.sieve()[1], npairs, ctx.rates()[2], ctx.stats()["n_kpoints"]
    ctx.close()
    return out


@pytest.mark.parametrize("c", [np.inf, 1e300, 1e41])
@pytest.mark.parametrize("name,grid,half,precision", [
    ("al_like", (18, 15, 20), 0.3, "fp32"),       # columns of k-points; 300 points a plane
    ("al_like", (18, 15, 20), 0.3, "fp64"),
    ("si_like", (20, 15, 16), 2.0, "fp32"),
    ("tiny", (6, 5, 7), 0.5, "fp64"),             # a k-point at a time
])
def test_no_cutoff(name, grid, half, precision, c):
    s = getattr(synth, f"{name}_system")()
    gr = O.Grids(s, grid)
    mu = gr.band_centre() if not s.n_valence else gr.band_edges(s.n_valence)[1] + half
    counts, npairs, r, nkp = _rates(s, grid, mu, half, c, precision)
    kept = int((gr.hw.max(axis=1) >= 1e-4).sum())
    assert (counts == kept).all() and npairs == kept * nkp
    # 20 keV: above any difference of the energies, within FP32
    ref = _rates(s, grid, mu, half, 1e6, precision)
    assert ref[1] == npairs and np.array_equal(ref[2], r)
