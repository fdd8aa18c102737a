"""Which row a warp of the sequences' preparing kernel copies (csrc/sequence_rows.h),
run on the host with a trap on division by zero: without x (I = 0) no row is
one of x and nothing may be divided by I."""
import os
import shutil
import subprocess

import pytest

from paper_1911_08020_gb300 import build as darb_build

MAIN = r"""
#include "sequence_rows.h"
#include <cstdio>
#include <cstdlib>
int main(int argc, char **argv) {
    const long H = std::atol(argv[1]), I = std::atol(argv[2]), T = std::atol(argv[3]);
    for (long row = 0; row < H + I * T; ++row) {
        const darb::seq::PrepRow r = darb::seq::prep_row(row, H, I);
        std::printf("%d %ld %ld\n", int(r.of_x), long(r.t), long(r.k));
    }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("rows")
    (d / "main.cc").write_text(MAIN)
    subprocess.run([gxx, "-std=c++17", "-O0", "-fsanitize=integer-divide-by-zero",
                    "-fsanitize-undefined-trap-on-error", "-I", darb_build.CSRC, str(d / "main.cc"),
                    "-o", str(d / "main")], check=True)
    return os.path.join(d, "main")


@pytest.mark.parametrize("H,I,T", [(5, 0, 3), (1, 0, 1), (4, 3, 2), (1, 1, 5)])
def test_rows(program, H, I, T):
    r = subprocess.run([program, str(H), str(I), str(T)], capture_output=True, text=True)
    assert r.returncode == 0, "division by zero"
    got = [tuple(map(int, line.split())) for line in r.stdout.splitlines()]
    assert got == [(0, 0, k) for k in range(H)] + [(1, t, k) for t in range(T) for k in range(I)]
