"""Sieve count by (k2, k3) columns (k_sieve_count_cols): pair counts of sampled k-points equal the
oracle's, and the rates over the decision mask are bitwise those of the re-evaluating fill (which
decides every candidate by itself), on grids of one and two passes over a column, with partial
plane blocks, both block sizes, and smearings on either side of the phonon energies."""
import numpy as np
import pytest

from oracle import epwi_oracle as O
from paper_2306_16493_gb300 import epwi, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,grid,half,eta", [
    ("al_like", (18, 15, 20), 0.3, 0.02),         # two plane blocks, the second one partial
    ("al_like", (18, 15, 20), 0.5, 0.002),        # c eta below the phonon energies: exact per-mode test
    ("al_like", (48, 10, 11), 1.5, 0.01),         # up to 48 k-points per column: three passes, several bands
    ("al_like", (70, 9, 9), 0.4, 0.02),           # beyond 64 axis-1 points: 128 threads
    ("si_like", (20, 15, 16), 2.0, 0.01),         # eight bands
    ("si_like", (72, 8, 9), 2.0, 0.003),
])
def test_counts_and_mask(name, grid, half, eta, monkeypatch):
    s = getattr(synth, f"{name}_system")()
    gr = O.Grids(s, grid)
    mu = gr.band_centre() if not s.n_valence else gr.band_edges(s.n_valence)[1] + half
    lo, hi = mu - half, mu + half
    ctx = epwi.Context(precision="fp32")
    ctx.setup(s)
    ctx.eigs(grid)
    ns, npairs = ctx.scatter_rates(300.0, mu, eta, lo, hi)
    assert ctx.stats()["n_kpoints"] * gr.nk >= 1 << 23     # the size from which the column kernel runs
    k, counts = ctx.sieve()
    r = ctx.rates()[2]
    ik, n = gr.window_states(lo, hi)
    assert len(np.unique(ik)) == len(k) and counts.sum() == npairs
    for p in np.random.default_rng(0).choice(len(k), 40, replace=False):
        assert counts[p] == len(O.sieve_k(gr, int(k[p]), n[ik == k[p]], eta)), int(k[p])
    monkeypatch.setenv("EPWI_SIEVE_MASK_MAX_BYTES", "0")
    assert ctx.scatter_rates(300.0, mu, eta, lo, hi) == (ns, npairs)
    assert np.array_equal(ctx.rates()[2], r)
    ctx.close()
