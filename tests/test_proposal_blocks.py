"""Launches of the learned proposal's network, on the CPU: every (state, cell) is in one launch, and no
launch has more rows (cells times modes) than the kernel's 32-bit indices and 1 GiB of outputs, up
to one cell for each of the 2^31 - 1 points of the largest grid."""
import numpy as np

from tests import hostcpp

SRC = r"""
#include <cstdio>
#include "epwi_internal.cuh"
#include "mlp.cuh"
int main() {
    long long ns, ncell, nm;
    while (scanf("%lld %lld %lld", &ns, &ncell, &nm) == 3) {
        const PropBlock b = prop_block(ns, ncell, (int)nm);
        printf("%lld %lld\n", (long long)b.states, (long long)b.cells);
    }
}
"""


def test_launch_blocks(tmp_path):
    rng = np.random.default_rng(1)
    cases = [(1, 2 ** 31 - 1, 3), (5, 2 ** 31 - 1, 18), (3, 715827883, 3), (1, 1, 3), (7, 2 ** 28 // 3, 3), (7, 2 ** 28 // 3 + 1, 3)]
    cases += [(int(np.exp(rng.uniform(0, 12))), int(np.exp(rng.uniform(0, np.log(2 ** 31 - 1)))), int(rng.integers(1, 7)) * 3)
              for _ in range(500)]
    out = hostcpp.run(tmp_path, SRC, stdin="\n".join(" ".join(map(str, c)) for c in cases)).split()
    for (ns, ncell, nm), s, x in zip(cases, map(int, out[::2]), map(int, out[1::2]), strict=True):
        assert 1 <= s <= ns and 1 <= x <= ncell and s * x * nm <= 2 ** 28
        assert x == ncell or s == 1               # part of the cells: of one state only
        assert s in (1, ns) or (s + 1) * x * nm > 2 ** 28
