"""Eigensolvers (jacobi.cuh) against NumPy's on whole grids: eigenvalues, the gauge-invariant
projectors of well separated states, and orthonormality, all at 1e-12 of the matrix scale (FP64
rounding of the Fourier sums and a few sweeps), for the compile-time sizes (1, 3, 4, 6, 8), the
runtime ones and the warp solver, with exact degeneracies (a crystal with the cubic point group, on
a grid that holds its high-symmetry points and lines)."""
import numpy as np
import pytest

from oracle import epwi_oracle as O
from paper_2306_16493_gb300 import epwi, synth
from tests.models import tb_dp_system

pytestmark = pytest.mark.gpu
TOL = 1e-12


def _bands(nw, nat=1, r=1):
    lat, tau = {1: synth.fcc_cell, 2: synth.diamond_cell}[nat](5.0) if nat <= 2 else synth.cubic_cell(nat)
    return synth.make_system("x", lat, tau, 27.0, nw, r, r >= 2, 7 + nw, 0.040)


@pytest.mark.parametrize("make,grid", [
    (lambda: tb_dp_system(), (8, 8, 8)),
    (lambda: _bands(2), (6, 5, 4)),
    (lambda: _bands(3, nat=2), (6, 5, 4)),
    (lambda: synth.al_like_system(), (11, 10, 9)),
    (lambda: synth.al_like_sym_system(), (48, 48, 48)),
    (lambda: _bands(5, nat=2), (7, 6, 5)),
    (lambda: _bands(8, nat=2), (9, 8, 7)),
    (lambda: _bands(9, nat=4), (4, 3, 5)),            # the warp solver, odd size
    (lambda: _bands(24, nat=6), (3, 4, 3)),
])
def test_bands_and_modes(make, grid):
    s = make()
    ctx = epwi.Context()
    ctx.setup(s)
    ctx.eigs(grid)
    eps, V, _ = ctx.bands()
    hw, u = ctx.phonons()
    ctx.close()
    frac = O.grid_frac(grid)
    ref, Vr = O.bands(s, frac)
    scale = np.abs(ref).max()
    assert np.abs(eps - ref).max() <= TOL * scale
    eye = np.einsum("kin,kim->knm", V.conj(), V)
    assert np.abs(eye - np.eye(s.nw)).max() <= TOL
    gap = np.full(ref.shape, np.inf)
    if s.nw > 1:
        d = np.diff(ref, axis=1)
        gap[:, :-1], gap[:, 1:] = d, np.minimum(gap[:, 1:], d)
        gap[:, 1:-1] = np.minimum(d[:, 1:], d[:, :-1])
    overlap = np.abs(np.einsum("kin,kin->kn", V.conj(), Vr))
    far = gap > 1e-3 * scale                          # 1 - |<v|v'>| ~ (rounding / gap)^2
    assert np.abs(overlap[far] - 1).max() <= TOL
    lam = np.linalg.eigvalsh(O.dynmat_q(s, frac)) * O.HBAR2_AMU_A2
    assert np.abs(np.sign(hw) * hw ** 2 - lam).max() <= TOL * np.abs(lam).max()
    # sum over the kept modes of omega |u><u|: (hbar^2 / 2) M^-1/2 P M^-1/2, P = 1 minus dropped modes
    m = np.sqrt(np.repeat(s.mass, 3))
    e = u * m[None, :, None] * np.sqrt(2 * np.abs(hw) / O.HBAR2_AMU_A2)[:, None, :]
    keep = hw >= 1e-4
    gram = np.einsum("qin,qim->qnm", e.conj(), e)
    want = np.einsum("qn,nm->qnm", keep.astype(float), np.eye(s.nm))
    assert np.abs(gram - want).max() <= 10 * TOL
