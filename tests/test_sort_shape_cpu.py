"""The radix sort's tile counts over the whole range of an int (csrc/sort_shape.h, compiled
for the host): the last tile is the one that holds the last key, and the later passes'
counts fit the array they lie over (16 bytes per key)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_00444_gb300", "csrc")

SRC = """
#include <climits>
#include <cstdio>
#include <initializer_list>
#include "sort_shape.h"
int main() {
    for (long long n : {1LL, 1023LL, 1024LL, 1025LL, 163840LL, 163841LL, 491520LL, 491521LL, 1048576LL, 1048577LL,
                        4194304LL, 4194305LL, (long long)INT_MAX - 8192, (long long)INT_MAX - 8191,
                        (long long)INT_MAX - 8190, (long long)INT_MAX - 1, (long long)INT_MAX}) {
        long long tile = 0;
        meshgs::sort_shape((int)n, [&](auto th, auto it) { tile = (long long)th.value * it.value; });
        std::printf("%lld %lld %d\\n", n, tile, meshgs::sort_tiles((int)n));
    }
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="no host compiler")
def test_tile_counts_up_to_int_max(tmp_path):
    (tmp_path / "t.cpp").write_text(SRC)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(tmp_path / "t.cpp"), "-o", exe], check=True)
    rows = [list(map(int, x.split())) for x in subprocess.run([exe], capture_output=True, text=True).stdout.splitlines()]
    assert len(rows) == 17
    for n, tile, T in rows:
        assert T == -(-n // tile), (n, tile, T)
        assert T * tile <= 2 ** 31                        # a key's index is an int in the last tile too
        assert T == 1 or 3 * T * 1024 <= 16 * n
