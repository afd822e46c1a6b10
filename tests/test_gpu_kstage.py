"""Re->k sum factorised over the axes (kstage.cuh) in each precision: rates against the FP64 oracle
on ragged grids, and bitwise independence of the k-point chunking (chunks see other columns)."""
import numpy as np
import pytest

from oracle import epwi_oracle as O
from paper_2306_16493_gb300 import synth
from tests.parity import compare_rates, gpu_run, oracle_run

pytestmark = pytest.mark.gpu
#: per degenerate group: FP64 rounding; FP32 interpolation; fp16 hi/lo split (about 22 bits)
TOL = {"fp64": 1e-10, "fp32": 1e-5, "fp16x3": 1e-4}


@pytest.mark.parametrize("name,grid,precision", [
    ("al_like", (12, 7, 9), "fp64"),
    ("al_like", (15, 11, 8), "fp32"),
    ("al_like", (9, 16, 10), "fp16x3"),
    ("al_like_ws", (11, 10, 9), "fp64"),          # R_e not a cube
    ("al_like_ws", (11, 10, 9), "fp32"),
    ("al_like", (20, 20, 1), "fp32"),             # a single k3
    ("al_like", (1, 24, 20), "fp64"),             # a single k1: no sharing along the columns
])
def test_rates_and_chunking(name, grid, precision):
    s = getattr(synth, f"{name}_system")()
    gr = O.Grids(s, grid)
    mu = gr.band_centre()
    args = (s, grid, 300.0, mu, 0.05, mu - 0.4, mu + 0.4)
    out = gpu_run(*args, precision=precision)
    err, n = compare_rates(out, oracle_run(gr, *args[2:]), gr.eps, TOL[precision])
    assert n > 0 and err <= TOL[precision], err
    part = gpu_run(*args, precision=precision, kpoint_chunk=29)
    assert part["stats"]["n_chunks"] > 1 and np.array_equal(part["inv_tau"], out["inv_tau"])
    out["ctx"].close()
    part["ctx"].close()
