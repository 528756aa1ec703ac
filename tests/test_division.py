"""div_by of the float64 rescue against `/`, on the CPU: the function as it stands
in solve.cu, compiled as C, on random quotients, on divisors and quotients next
to the ends of a binade, and at the magnitudes where it divides instead."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1409_2081_gb300", "csrc")

MAIN = r"""
static unsigned long long s = 88172645463325252ull;
static unsigned long long rnd(void) { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; }
static double one_to_two(void) {
    unsigned long long u = (rnd() >> 12) | 0x3ff0000000000000ull;
    double d;
    memcpy(&d, &u, 8);
    return d;
}
int main(void) {
    long bad = 0;
    for (long i = 0; i < 3000000; ++i) {
        double a = one_to_two(), b = one_to_two();
        switch (i % 6) {
            case 1: b = 2.0 - (double)(rnd() % 64) * 0x1p-52; break;
            case 2: b = 1.0 + (double)(rnd() % 64) * 0x1p-52; break;
            case 3: a = b * (2.0 - (double)(rnd() % 64) * 0x1p-52); break;
            case 4: a = ldexp(a, (int)(rnd() % 2000) - 1000); b = ldexp(b, (int)(rnd() % 600) - 300); break;
            case 5: a = b * (1.0 + (double)(rnd() % 64) * 0x1p-52) - (double)(rnd() % 3) * 0x1p-52; break;
        }
        const double q = a / b, d = div_by(a, b, 1.0 / b), e = div_by(-a, b, 1.0 / b);
        bad += memcmp(&q, &d, 8) != 0 || -q != e;
    }
    printf("%ld\n", bad);
    return 0;
}
"""


def test_div_by_is_the_rounded_quotient(tmp_path):
    src = open(os.path.join(CSRC, "solve.cu")).read()
    m = re.search(r"__device__ __forceinline__ (double div_by\(.*?\n\}\n)", src, flags=re.S)
    c = tmp_path / "d.c"
    c.write_text("#include <math.h>\n#include <stdio.h>\n#include <string.h>\nstatic " + m.group(1) + MAIN)
    exe = tmp_path / "d"
    subprocess.check_call(["gcc", "-O2", "-ffp-contract=off", str(c), "-o", str(exe), "-lm"])
    assert subprocess.check_output([str(exe)], text=True).strip() == "0"
