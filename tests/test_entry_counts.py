"""Entry counts of the bins' sort buffers and index maps: sums of row or column lengths stay in
32 bits and are above the buffer's size exactly when the true sum is."""
import os
import subprocess

import numpy as np
import pytest

from paper_1503_04500_gb300 import build_ext

PROGRAM = """
#include <cstdio>
#include <cstdlib>
#include "common.cuh"
int main(int argc, char **argv) {  // room, then the lengths on standard input
    const int room = atoi(argv[1]);
    int sum = 0;
    for (long long len; std::scanf("%lld", &len) == 1;) {
        const int c = rsai::counted_entries(len, room);
        if (c < 0 || sum > INT_MAX - c) return 3;  // left 32 bits
        sum += c;
    }
    std::printf("%d", sum > room ? -1 : sum);
    return 0;
}
"""


@pytest.fixture(scope="module")
def count(tmp_path_factory):
    d = tmp_path_factory.mktemp("entry_counts")
    (d / "count.cu").write_text(PROGRAM)
    exe = str(d / "count")
    subprocess.run([build_ext.nvcc(), *build_ext.ARCH, "-std=c++17", "-I", build_ext.SRC, str(d / "count.cu"), "-o", exe],
                   check=True, capture_output=True)

    def run(room, lengths):
        text = " ".join(str(int(x)) for x in lengths)
        return int(subprocess.run([exe, str(room)], input=text, check=True, capture_output=True, text=True,
                                  timeout=60).stdout)

    return run


@pytest.mark.parametrize("room", [128, 4096, 131072])
def test_counted_entries(count, room):
    """-1 for "does not fit", else the exact sum, against 64-bit sums."""
    dense = 2**20
    rng = np.random.default_rng(1)
    cases = [[room], [room + 1], [room // 2, room - room // 2], [room, 1], [0, 0], [dense] * 1024,  # 2^30
             [dense] * 1024 + [1], [dense] * 2048, [dense] * 4096, [2**31 - 1] * 4096, [2**31 - 1]]
    cases += [rng.integers(0, room // 8, 16).tolist() for _ in range(8)]
    for lengths in cases:
        true = sum(lengths)
        assert count(room, lengths) == (true if true <= room else -1), lengths[:4]
