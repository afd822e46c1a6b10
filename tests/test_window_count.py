"""The counts that place the k-points and states of a window, on the CPU: running sums up to the
largest grid that epwi_eigs takes (2^31 - 1 points) with every band of 24 in the window."""
from tests import hostcpp

SRC = r"""
#include <cstdio>
#include "sieve.cuh"
int main() {
    // blocks of points as the scan's block sums hold them, then the exclusive sums point by point
    const int64_t nk = ((int64_t)1 << 31) - 1, per = 4096;
    for (int64_t w : {1, 24}) {
        WindowCount run{};
        for (int64_t k = 0; k < nk; k += per) {
            const int64_t m = nk - k < per ? nk - k : per;
            if (run.kpoints != k || run.states != k * w) return printf("off at %lld\n", (long long)k), 1;
            run += WindowCount{m, m * w};
        }
        const WindowCount last = run - WindowCount{1, w};
        if ((last + WindowCount{1, w}).kpoints != nk) return 1;
        printf("%lld %lld\n", (long long)run.kpoints, (long long)run.states);
    }
}
"""


def test_counts_of_the_largest_windows(tmp_path):
    nk = 2 ** 31 - 1
    assert hostcpp.run(tmp_path, SRC).split() == [str(x) for w in (1, 24) for x in (nk, nk * w)]
