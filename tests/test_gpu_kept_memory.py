"""Workspaces that a context keeps between calls of one kind (draws, the capture's pair lists, decisions
of a chunk) are given back by the first call of another kind, and by another grid."""
import gc

import pytest

from paper_2306_16493_gb300 import epwi, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _no_garbage():
    gc.collect()                                  # contexts of other tests are gone before the first reading


def _free():
    import torch
    return torch.cuda.mem_get_info(0)[0]


def test_workspaces_are_given_back():
    s = synth.al_like_system()
    ctx = epwi.Context(precision="fp32")
    ctx.setup(s)
    ctx.eigs(24)
    mu = 0.5 * sum(ctx.band_range())
    args = (300.0, mu, 0.05, mu - 0.4, mu + 0.4)
    nk, slack = 24 ** 3, 32 << 20
    _, npairs = ctx.scatter_rates(*args)          # every buffer that stays is there
    nkp = ctx.stats()["n_kpoints"]
    lists, draws = 8 * npairs, 4 * nkp * nk       # pair and offset per pair; a count per (k, q)
    assert lists > 4 * slack and draws > 4 * slack
    ctx.ibte(*args, max_iter=2)
    f0 = _free()
    ctx.ibte(*args, max_iter=2)
    assert abs(_free() - f0) <= slack             # kept from one call to the next
    ctx.scatter_rates(*args)
    assert _free() - f0 >= lists - slack

    def draw():
        ctx.set_precision("fp64")
        ctx.scatter_rates_is(*args, samples_per_k=64, proposal="uniform")

    draw()                                        # the FP64 path's own buffers are there
    ctx.set_precision("fp32")
    ctx.ibte(*args, max_iter=2)
    f0 = _free()
    draw()
    assert abs((f0 - _free()) - (draws - lists)) <= 2 * slack          # draws in, lists out
    f0 = _free()
    draw()
    assert abs(_free() - f0) <= slack
    ctx.eigs((6, 5, 4))
    assert _free() - f0 >= draws - slack
    ctx.close()


def test_decisions_of_a_chunk(monkeypatch):
    s = synth.al_like_system()
    ctx = epwi.Context(precision="fp32")
    ctx.setup(s)
    ctx.eigs(24)
    mu = 0.5 * sum(ctx.band_range())
    args = (300.0, mu, 0.05, mu - 4.0, mu + 4.0)
    monkeypatch.setenv("EPWI_SIEVE_MASK_MAX_BYTES", "0")
    ctx.scatter_rates(*args)
    mask = ctx.stats()["n_kpoints"] * 24 ** 3 // 8 // ctx.stats()["n_chunks"]
    f0 = _free()
    assert mask > 4 << 20
    ctx.eigs((6, 5, 4))
    assert _free() - f0 >= mask - (2 << 20)
    ctx.close()


def test_split_modes_hold_no_run_tables():
    """The run tables (one word per plane block, q1 and k-point) serve the sum-factorised kernels only."""
    s = synth.al_like_system()
    ctx = epwi.Context(precision="fp16x3")
    ctx.setup(s)
    ctx.eigs((1000, 3, 2))
    mu = 0.5 * sum(ctx.band_range())
    args = (300.0, mu, 0.05, mu - 0.4, mu + 0.4)
    _, npairs = ctx.scatter_rates(*args)
    runs = 4 * 1001 * ctx.stats()["n_kpoints"]
    assert runs > 12 << 20
    ctx.ibte(*args, max_iter=2)
    f0 = _free()
    ctx.scatter_rates(*args)                      # gives the capture's lists back
    assert abs(_free() - f0 - 8 * npairs) <= 6 << 20
    ctx.close()
