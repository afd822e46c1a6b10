"""Close levels and opposite wave vectors: H(k) V = V eps and D(q) e = e lambda at every point, with
orthonormal V, at 1e-12 of the matrix scale, for a crystal whose exact degeneracies are split by a
small Hermitian perturbation (the solver finishes such matrices by its series, by further sweeps or by
both, depending on the splitting), and for grids with one, two, even and odd numbers of points
per axis (q and -q come from one solve)."""
import dataclasses

import numpy as np
import pytest

from oracle import epwi_oracle as O
from paper_2306_16493_gb300 import epwi, synth

pytestmark = pytest.mark.gpu
TOL = 1e-12


def _check(s, grid):
    ctx = epwi.Context()
    ctx.setup(s)
    ctx.eigs(grid)
    eps, V, _ = ctx.bands()
    hw, u = ctx.phonons()
    ctx.close()
    frac = O.grid_frac(grid)
    H = O.hamiltonian_k(s, frac)
    scale = np.abs(H).max()
    assert np.abs(H @ V - V * eps[:, None, :]).max() <= TOL * scale
    assert np.abs(np.einsum("kin,kim->knm", V.conj(), V) - np.eye(s.nw)).max() <= TOL
    D = O.dynmat_q(s, frac) * O.HBAR2_AMU_A2
    lam = np.sign(hw) * hw ** 2
    e = u * np.sqrt(np.repeat(s.mass, 3))[None, :, None] * np.sqrt(2 * np.abs(hw) / O.HBAR2_AMU_A2)[:, None, :]
    assert np.abs(D @ e - e * lam[:, None, :]).max() <= TOL * np.abs(D).max()


@pytest.mark.parametrize("split", [0.0, 1e-12, 1e-9, 1e-6, 1e-4])
@pytest.mark.parametrize("copies", [1, 2, 4])          # 4, 8 and 16 bands (the warp solver)
def test_split_degeneracies(split, copies):
    s = synth.al_like_sym_system()
    if copies > 1:                                    # every level copies-fold degenerate
        s = dataclasses.replace(s, nw=copies * s.nw, H=np.kron(np.eye(copies), s.H),
                                g=np.kron(np.eye(copies), s.g))
    rng = np.random.default_rng(3)
    h = rng.normal(size=(s.nw, s.nw)) + 1j * rng.normal(size=(s.nw, s.nw))
    H = s.H.copy()
    H[[i for i, r in enumerate(np.asarray(s.Re).tolist()) if r == [0, 0, 0]][0]] += split * (h + h.conj().T)
    _check(dataclasses.replace(s, H=H), (8, 8, 8))


@pytest.mark.parametrize("nat,nw", [(1, 4), (2, 8), (4, 9)])
@pytest.mark.parametrize("grid", [(1, 5, 4), (2, 1, 6), (5, 4, 1), (6, 3, 2), (1, 1, 1)])
def test_opposite_points(nat, nw, grid):
    lat, tau = {1: synth.fcc_cell, 2: synth.diamond_cell}[nat](5.0) if nat <= 2 else synth.cubic_cell(nat)
    _check(synth.make_system("x", lat, tau, 27.0, nw, 1, False, 7 + nw, 0.040), grid)
