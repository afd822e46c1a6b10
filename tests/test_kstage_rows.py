"""Workspace of the factorised Re->k sum, on the CPU: the blocks of rows stay within 4 GiB for every
number of columns that a grid can have, as long as one row does, and cover the rows."""
import numpy as np

from tests import hostcpp

SRC = r"""
#include <cstdio>
#include "kstage.cuh"
int main() {
    long long D, nk3, ncol, nrow, W, elem;
    while (scanf("%lld %lld %lld %lld %lld %lld", &D, &nk3, &ncol, &nrow, &W, &elem) == 6)
        printf("%lld\n", (long long)ks_block_rows(D, nk3, ncol, nrow, (int)W, (size_t)elem, kKsThreads));
}
"""


def test_blocks_of_rows(tmp_path):
    rng = np.random.default_rng(5)
    cases = [(7, 1024, 1 << 20, 1944, 24, 16), (5, 1, 1 << 20, 1500, 4, 8), (13, 4096, 4096, 3, 1, 8),
             (5, 48, 2304, 1500, 4, 8), (7, 100, 3000, 16464, 8, 8)]
    for _ in range(4000):
        nk3 = int(np.exp(rng.uniform(0, np.log(4097))))
        cases.append((int(rng.choice([1, 3, 5, 7, 9, 11, 13])), nk3, int(np.exp(rng.uniform(np.log(nk3), np.log(2 ** 20)))),
                      int(np.exp(rng.uniform(np.log(3), np.log(1e6)))), int(rng.integers(1, 25)), int(rng.choice([8, 16]))))
    out = hostcpp.run(tmp_path, SRC, stdin="\n".join(" ".join(map(str, c)) for c in cases)).split()
    small = 0
    for (D, nk3, ncol, nrow, W, elem), rows in zip(cases, map(int, out), strict=True):
        per_row = (D * D * nk3 + D * ncol) * W * elem
        assert 1 <= rows <= nrow
        assert rows * per_row <= 2 ** 32 or rows == 1
        assert rows == nrow or rows % 128 == 0 or per_row * 128 > 2 ** 32     # whole CTAs where they fit
        small += rows < min(nrow, 128)
    assert small > 20                             # shapes that 128 rows would take beyond 4 GiB
