"""The 32-bit truncating division by an invariant integer (host build of the
library header) against Python's, at the divisors IntegerSGD clamps to."""
import os
import random
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_trunc_division_matches_python(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "div.cu"
    src.write_text(r'''
#include <cstdio>
#include "nitro_internal.cuh"
int main() {
    unsigned d; int x;
    while (scanf("%u %d", &d, &x) == 2)
        printf("%d %d\n", nitro::FloorDiv32::make(d).trunc_div(x), nitro::FloorDiv32::make(d).floor_div(x));
    return 0;
}
''')
    exe = tmp_path / "div"
    subprocess.run([nvcc, "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2407_11698_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True, capture_output=True)
    rnd = random.Random(5)
    ds = [1, 2, 3, 10, 640, 327680, 25000, 2**31 - 1, 2**31, 2**31 + 1, 2**32 - 1]
    ds += [rnd.randrange(1, 2**32) for _ in range(40)]
    cases = [(d, x) for d in ds for x in [0, 1, -1, 2**31 - 1, -2**31, -2**31 + 1] +
             [rnd.randrange(-2**31, 2**31) for _ in range(40)] +
             [k * d + e for k in (-3, -1, 1, 2) for e in (-1, 0, 1) if -2**31 <= k * d + e < 2**31]]
    out = subprocess.run([str(exe)], input="".join("%d %d\n" % c for c in cases), capture_output=True,
                         text=True, check=True).stdout
    for (d, x), line in zip(cases, out.splitlines()):
        tr, fl = map(int, line.split())
        assert tr == (x // d if x >= 0 else -(-x // d)), (d, x)
        assert fl == x // d, (d, x)
        # a divisor above 2^31 gives what 2^31 + 1 gives
        if d > 2**31:
            assert x // d == x // (2**31 + 1) and abs(x) // d == abs(x) // (2**31 + 1)
