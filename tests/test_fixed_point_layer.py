"""The integer layer of the fixed-point residual (csrc/dg_fix.cuh), compiled for
the host and compared with exact integers.  No GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2002_04222_gb300", "csrc")


def run_host(tmp_path, body, lines, extra=""):
    """stdout of a host program whose main() reads the lines' numbers."""
    from paper_2002_04222_gb300.build import nvcc
    src, exe = tmp_path / "probe.cu", tmp_path / "probe"
    src.write_text('#include <cstdio>\n#include "dg_fix.cuh"\n' + extra + "using namespace dg;\n"
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


def test_products_round_alike_on_both_signs(tmp_path):
    """v r at a shared exponent, for factors of both signs (a negative
    beta_s makes some): the magnitude is cut off towards 0 to within two units
    of the exact product's, zeros stay 0, and the signs of v and r only change
    the result's sign."""
    from fractions import Fraction
    import random
    import struct
    rng = random.Random(4)

    def expo(v):
        return (struct.unpack("<q", struct.pack("<d", v))[0] >> 52) & 0x7ff

    vs = [0.0, 1.0, 0.75, 2.0 ** -30, 2.0 ** -70] + [rng.uniform(0.1, 1.9) * 2.0 ** -rng.randrange(8)
                                                     for _ in range(20)]
    rs = [1.0, 0.0, 0.3, 1.7e5, 3e-9] + [rng.uniform(0.5, 8.0) for _ in range(5)]
    cases = [(sv * v, sr * r) for v in vs for r in rs for sv in (1, -1) for sr in (1, -1)]
    # an exponent no product exceeds: that of v's largest plus r's
    emax = [expo(2.0) + (expo(r) - 1022 if r else 0) for _, r in cases]
    got = run_host(tmp_path, 'double v, r; int e; while (scanf("%la %la %d", &v, &r, &e) == 3) '
                             'printf("%lld\\n", (long long)to_fix_mul(v, fix_scale(r), e, 58));',
                   [f"{v.hex()} {r.hex()} {e}" for (v, r), e in zip(cases, emax)])
    assert len(got) == len(cases)
    by = {}
    for (v, r), e, g in zip(cases, emax, got):
        exact = abs(Fraction(v) * Fraction(r)) * Fraction(2) ** (58 - (e - 1022))
        x, sign = int(g), (-1 if (v < 0) != (r < 0) else 1)
        assert 0 <= sign * x <= exact + 1 and exact - sign * x < 3, (v, r, x)
        by.setdefault((abs(v), abs(r)), set()).add(sign * x)
    assert all(len(s) == 1 for s in by.values())


def test_the_smallest_scale_is_a_normal_double(tmp_path):
    """One unit of M^-1 B^T W G at the smallest shared exponent, every stage's
    input shifted up as far as it goes (59 places) and two bits kept below the
    last stage's unit, is 2^-1022 at least: fix_to_double has no subnormals (a
    smaller scale borrowed from the sign bit and came out near 2^1000)."""
    inst = ([(2, p, q) for p, q in ((1, 3), (2, 3), (2, 4), (3, 5), (4, 6), (5, 7), (6, 8))]
            + [(3, p, q) for p, q in ((1, 3), (2, 4), (2, 5), (3, 5), (3, 6), (4, 6), (4, 8))])
    got = run_host(tmp_path, 'int d, P, Q; FixTab f; '
                             'while (scanf("%d %d %d", &d, &P, &Q) == 3) { build_fix_tables(P, Q, f); '
                             'printf("%d\\n", FIX_EMIN - 1022 - 58 - 2 - 59 * d + f.eDh + d * f.eA); }',
                   [f"{d} {p} {q}" for d, p, q in inst], extra='#include "dg_fixtab.cu"\n')
    assert len(got) == len(inst)
    for i, g in zip(inst, got):
        assert int(g) >= -1022, (i, g)
