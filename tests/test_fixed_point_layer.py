"""The integer layer of the fixed-point residual (csrc/dg_fix.cuh), compiled for
the host and compared with exact integers.  No GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2002_04222_gb300", "csrc")


def run_host(tmp_path, body, lines):
    """stdout of a host program whose main() reads the lines' numbers."""
    from paper_2002_04222_gb300.build import nvcc
    src, exe = tmp_path / "probe.cu", tmp_path / "probe"
    src.write_text('#include <cstdio>\n#include "dg_fix.cuh"\nusing namespace dg;\n'
                   "int main() {\n" + body + "\nreturn 0; }\n")
    subprocess.run([nvcc(), "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a",
                    "--expt-relaxed-constexpr", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], input="\n".join(lines), check=True, capture_output=True,
                         text=True).stdout
    return out.split()


def test_shift_rounds_to_the_nearest(tmp_path):
    """Every shift, 63 and beyond among them (a flux that is exactly zero, or
    far below the other terms): nearest, ties up, 0 where |x| < 2^(sh - 1)."""
    xs = [0, 1, -1, 2, -3, 5, (1 << 20) + 7, -(1 << 40) + 1, (1 << 58) - 1, -(1 << 60), (1 << 60)]
    cases = [(x, sh) for x in xs for sh in (0, 1, 2, 31, 32, 58, 60, 61, 62, 63, 64, 400)]
    got = run_host(tmp_path, 'long long x; int s; while (scanf("%lld %d", &x, &s) == 2) '
                             'printf("%lld\\n", (long long)fix_shift(x, s));',
                   [f"{x} {sh}" for x, sh in cases])
    assert len(got) == len(cases)
    for (x, sh), g in zip(cases, got):
        assert int(g) == (2 * x + (1 << sh)) // (2 << sh), (x, sh)
