"""The fixed-point records' arithmetic is modulo 2^32 without relying on signed
overflow: the library's helpers compiled for the host with the sanitizer that
aborts on undefined operations, against Python's integers."""
import random
import subprocess

import paper_2603_07321_gb300.buildlib as B

PROGRAM = r"""
#include <stdio.h>
#include "pta_dev.cuh"
int main() {
    long long a, b;
    int shift;
    while (scanf("%lld %lld %d", &a, &b, &shift) == 3)
        printf("%d %d\n", pta::rec_diff((int)a, (int)b), pta::rec_join((int)a, (int)b, shift));
}
"""


def _wrap(v):
    return (v + 2**31) % 2**32 - 2**31


def test_differences_and_sums_wrap(tmp_path):
    src, exe = tmp_path / "t.cu", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([B._nvcc()] + B.ARCH + ["-std=c++17", "-I" + B.INC, "-I" + B.CSRC, "-Xcompiler",
                   "-fsanitize=undefined,-fno-sanitize-recover=all", str(src), "-o", str(exe)],
                   check=True, capture_output=True)
    rng = random.Random(1)
    edge = [-2**31, -2**31 + 1, -1, 0, 1, 2**31 - 1]
    pairs = [(a, b) for a in edge for b in edge]
    pairs += [(rng.randrange(-2**31, 2**31), rng.randrange(-2**31, 2**31)) for _ in range(200)]
    lines = [(a, b, s) for a, b in pairs for s in (0, 1, 14, 19)]
    r = subprocess.run([str(exe)], input="".join("%d %d %d\n" % x for x in lines), text=True,
                       capture_output=True)
    assert r.returncode == 0, r.stderr
    got = [tuple(map(int, x.split())) for x in r.stdout.splitlines()]
    assert got == [(_wrap(a - b), _wrap((a << s) + b)) for a, b, s in lines]
