"""Statistics of an FP64 rates call: flops and tiles are those of the kernel that ran."""
import pytest

from paper_2306_16493_gb300 import epwi, synth
from tests.test_gpu_repeated_vectors import repeated

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,direct", [("al_like", False), ("al_like", True), ("si_like", False)])
def test_fp64_flops_and_tiles(name, direct):
    s = getattr(synth, f"{name}_system")()
    r = int(abs(s.Rp).max())
    if direct:
        s = repeated(s)                           # a vector listed twice: the direct sum over R_p
    ctx = epwi.Context()
    ctx.setup(s)
    ctx.eigs((7, 6, 8))
    lo, hi = ctx.band_range()
    ctx.scatter_rates(300.0, 0.5 * (lo + hi), 0.05, lo, lo + 0.4 * (hi - lo))
    st = ctx.stats()
    nbar = st["n_states"] / st["n_kpoints"]
    per = 8.0 * len(s.Rp) * s.nm * s.nw if direct else \
        4.0 * 2 * r * s.nm * s.nw + 8.0 * (s.nw * s.nm + s.nm ** 2)
    assert st["n_pairs"] > 0
    assert st["scatter_flops"] == pytest.approx(per * st["n_pairs"] * nbar, rel=1e-12)
    assert (st["n_tiles"] > 0) == direct
    ctx.close()
