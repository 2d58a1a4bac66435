"""The node a persistent block takes (node_at in nmc_internal.h) lies in the batch whatever the order buffer holds.

The kernels' own function, compiled for the host; no GPU is needed.
"""

import subprocess

from paper_2601_00976_gb300 import _build

PROGRAM = r"""
#include <limits.h>
#include <stdio.h>
#include "nmc_internal.h"
int main() {
    const int order[8] = {3, 0, INT_MIN, -1, 4, 5, INT_MAX, 1};   // n = 5: entries 2..3 and 5..6 are not of the batch
    for (long long n : {1ll, 5ll, 8ll})
        for (long long k = 0; k < n; ++k) printf("%lld ", nmc::node_at(order, k, n));
    // without an order, and past the end: the index itself, which ends the block's loop
    printf("%lld %lld %lld %lld\n", nmc::node_at(nullptr, 4, 5), nmc::node_at(nullptr, 6, 5), nmc::node_at(order, 5, 5),
           nmc::node_at(order, 1ll << 30, 5));
    return 0;
}
"""


def test_node_stays_in_the_batch(tmp_path):
    src, exe = tmp_path / "node.cu", tmp_path / "node"
    src.write_text(PROGRAM)
    subprocess.run([_build._nvcc(), "-std=c++17", "-I" + _build.INCLUDE, "-I" + _build.CSRC, str(src), "-o", str(exe)],
                   check=True, capture_output=True)
    got = [int(x) for x in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()]
    assert got == [0,
                   3, 0, 0, 0, 4,
                   3, 0, 0, 0, 4, 5, 7, 1,
                   4, 6, 5, 1 << 30]
