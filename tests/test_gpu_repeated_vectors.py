"""Lattice-vector sets that list a vector more than once: its terms add up in every Fourier sum, so
splitting a vector's weight over two or four entries changes neither the bands nor the phonons."""
import dataclasses

import numpy as np
import pytest

from paper_2306_16493_gb300 import epwi, synth

pytestmark = pytest.mark.gpu


def repeated(s, copies=2):
    """s with the weight of R = 0 and of one pair +-R of each set spread over `copies` entries."""
    def spread(R, w):
        lut = {tuple(v): i for i, v in enumerate(R.tolist())}
        i = next(i for v, i in lut.items() if v != (0, 0, 0) and tuple(-x for x in v) in lut)
        pick = [lut[(0, 0, 0)], i, lut[tuple(-R[i])]]
        idx = np.concatenate([np.arange(len(R))] + [pick] * (copies - 1))
        w2 = w[idx].copy()
        w2[np.isin(idx, pick)] /= copies
        return idx, w2
    ie, we = spread(s.Re, s.we)
    ip, wp = spread(s.Rp, s.wp)
    return dataclasses.replace(s, Re=s.Re[ie].copy(), we=we, H=s.H[ie].copy(), Rp=s.Rp[ip].copy(), wp=wp,
                               Phi=s.Phi[ip].copy(), g=np.ascontiguousarray(s.g[ie][:, ip]))


@pytest.mark.parametrize("name,grid,copies", [("tiny", (6, 5, 4), 2), ("al_like", (6, 7, 5), 4), ("si_like", (4, 4, 5), 2)])
def test_bands_and_phonons(name, grid, copies):
    s = getattr(synth, f"{name}_system")()
    out = []
    for x in (s, repeated(s, copies)):
        ctx = epwi.Context()
        ctx.setup(x)
        ctx.eigs(grid)
        eps, _, vel = ctx.bands()
        out.append((eps, vel.sum(axis=1), ctx.phonons()[0] ** 2))
        ctx.close()
    # sums of up to 343 terms and the eigensolver: rounding of FP64 times their number.  The velocities are
    # summed over the bands: that is the trace of dH/dk, whatever the basis of degenerate bands
    for x, y in zip(*out):
        assert np.abs(x - y).max() <= 1e-12 * np.abs(x).max()


# nw = 4, 3 modes, R_p within |n| <= 2; twice the bounds of the modes' parity with the oracle
@pytest.mark.parametrize("precision,tol", [("fp64", 2e-10), ("fp32", 2e-5), ("fp16x3", 2e-4), ("bf16x3", 2e-4),
                                           ("tf32x3", 2e-4)])
@pytest.mark.parametrize("copies", [2, 8])
def test_rates(precision, tol, copies):
    s = synth.al_like_system()
    out = []
    for x in (s, repeated(s, copies)):
        ctx = epwi.Context(precision=precision)
        ctx.setup(x)
        ctx.eigs((10, 9, 8))
        mu = 0.5 * sum(ctx.band_range())
        ctx.scatter_rates(300.0, mu, 0.05, mu - 0.4, mu + 0.4)
        out.append(ctx.rates())
        ctx.close()
    (k, n, r), (k2, n2, r2) = out
    assert np.array_equal(k, k2) and np.array_equal(n, n2)
    assert np.abs(r2 - r).max() <= tol * r.max()
