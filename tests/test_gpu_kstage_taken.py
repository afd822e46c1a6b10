"""Rates of windows that the rule gives to the factorised Re->k sum, the rule asked for each: a single k3
among them (test_gpu_kstage.py's 20 x 20 x 1 window is small enough for the direct sum)."""
import numpy as np
import pytest

from oracle import epwi_oracle as O
from paper_2306_16493_gb300 import synth
from tests import hostcpp
from tests.parity import compare_rates, gpu_run, oracle_run

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-10, "fp32": 1e-5}       # as in test_gpu_kstage.py

SRC = r"""
#include <cstdio>
#include "kstage.cuh"
int main() {
    int D, nRe, nw, fp64;
    long long nkp, nrow;
    double nk3, ncol;
    if (scanf("%d %d %lld %lf %lf %lld %d %d", &D, &nRe, &nkp, &nk3, &ncol, &nrow, &nw, &fp64) != 8) return 1;
    printf("%d\n", ks_pays(D, nRe, nkp, nk3, ncol, nrow, nw, fp64 != 0));
}
"""


@pytest.mark.parametrize("grid,half,precision", [
    ((24, 24, 1), 0.5, "fp32"),                   # a single k3
    ((24, 1, 24), 0.5, "fp32"),                   # a single k2
    ((9, 13, 7), 0.4, "fp64"),
])
def test_factorised_sum_is_taken(grid, half, precision, tmp_path):
    s = synth.al_like_system()
    gr = O.Grids(s, grid)
    mu = gr.band_centre()
    out = gpu_run(s, grid, 300.0, mu, 0.05, mu - half, mu + half, precision=precision)
    k = out["ctx"].sieve()[0]
    plane = k % (grid[1] * grid[2])
    # without the sieve's own counts the rule takes the largest numbers of k3 and columns
    nk3, ncol = min(grid[2], len(k)), min(grid[1] * grid[2], len(k))
    assert len(np.unique(plane)) <= ncol
    args = (5, len(s.Re), len(k), nk3, ncol, 5 ** 3 * s.nm * s.nw, s.nw, int(precision == "fp64"))
    assert hostcpp.run(tmp_path, SRC, stdin=" ".join(map(str, args))).strip() == "1"
    err, n = compare_rates(out, oracle_run(gr, 300.0, mu, 0.05, mu - half, mu + half), gr.eps, TOL[precision])
    assert n > 0 and err <= TOL[precision], err
    out["ctx"].close()
