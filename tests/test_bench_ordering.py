"""The ordering ablation compares the two orders with the same kind of sums: its crystal is the same one
with a vector listed twice, and the q-batch arm runs the direct sum on it."""
import argparse
import json

import numpy as np
import pytest

import bench
from paper_2306_16493_gb300 import synth


def test_listed_twice_is_the_same_crystal():
    s = synth.tiny_system()
    d = bench.listed_twice(s)
    assert len(d.Re) == len(s.Re) + 1 and len(d.Rp) == len(s.Rp) + 1
    i, j = (int(np.flatnonzero((R == 0).all(axis=1))[0]) for R in (s.Re, s.Rp))
    for R, w, n, x in ((s.Re, s.we, d.we, i), (s.Rp, s.wp, d.wp, j)):
        assert n[x] + n[-1] == w[x] and np.array_equal(np.delete(n[:-1], x), np.delete(w, x))
    assert np.array_equal(d.H[-1], s.H[i]) and np.array_equal(d.Phi[-1], s.Phi[j])
    assert np.array_equal(d.g[:-1, :-1], s.g) and np.array_equal(d.g[-1, :-1], s.g[i])
    assert np.array_equal(d.g[:, -1], d.g[:, j])


@pytest.mark.gpu
def test_arms(capsys):
    bench.run_kbatch(argparse.Namespace(ablation_grid=8, warmup=1, steps=1))
    line = json.loads(capsys.readouterr().out)
    assert line["q_batch"]["tiles"] > 0           # direct sums: 128-pair tiles
    assert line["q_batch_factorised"]["tiles"] == 0
    assert line["max_rel_rate_difference"] <= 1e-10
    assert line["predicted_mac_ratio"] == pytest.approx(4 / line["mean_window_bands_n_k"])
