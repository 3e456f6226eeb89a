"""The rule that takes a set to the rank walk (more than so many prefixes a
row), compiled on its own with the host compiler: equal to the exact integers'
over the whole 64-bit range, where least x W x rows wraps."""
import os
import random
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2407_20474_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include "fz_host_math.h"
int main() {
    unsigned long long c, r, w, l;
    while (std::scanf("%llu %llu %llu %llu", &c, &r, &w, &l) == 4)
        std::printf("%d\n", fz::prefixes_exceed(c, r, w, l) ? 1 : 0);
    return 0;
}
"""


def test_prefixes_exceed(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "driver.cpp", tmp_path / "driver"
    src.write_text(DRIVER)
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    rng = random.Random(3)
    cases = [(2 * 10**18 + 4 * 10**6, 2 * 10**18, 4, 3), (2**64 - 1, 2**62, 4, 3), (2**64 - 1, 2**60 + 1, 4, 3),
             (0, 0, 4, 3), (1, 1, 4, 3), (4, 0, 4, 3), (3, 0, 4, 3)]
    for _ in range(4000):
        W, least = rng.choice((1, 4, 16, 64)), rng.choice((1, 3, 10))
        rows = rng.getrandbits(rng.randint(1, 63))
        prefixes = max(0, least * rows + rng.randint(-3, 3)) if rng.random() < 0.5 else rng.getrandbits(rng.randint(1, 62))
        if rows + W * prefixes < 2**64:
            cases.append((rows + W * prefixes, rows, W, least))
    out = subprocess.run([str(exe)], input="\n".join("%d %d %d %d" % c for c in cases) + "\n", capture_output=True,
                         text=True, check=True).stdout.split()
    assert [int(x) for x in out] == [int(c - r >= w and (c - r) // w > l * r) for c, r, w, l in cases]
