"""Second differences carry a factor 2^2 in the exponent (csrc/stage_int.cuh, limb_bits).  It has nothing to do with
the field's own exponent, of which 2047 alone means Inf or NaN: a finite field with values near the end of the
range, where e + 2 passes 2047, has second differences that are numbers, zero for a constant, or overflow to
infinity.  The function is compiled for the host; Python's integers give the exact values."""
import subprocess

from paper_2606_02053_gb300 import build as libbuild

SRC = r"""
#include <cstdio>
#include "stage_split.cuh"
int main() {
  long long v; int e, up;
  while (scanf("%lld %d %d", &v, &e, &up) == 3)
    printf("%llu\n", cosmos::limb_bits<true, true>(cosmos::limb_of(v), e, up));
  return 0;
}
"""


def rounded(v, e, up):
    """FP64 bits of v 2^(e + up - 1085) for |v| < 2^53 (no rounding)."""
    if e >= 2047:
        return 0x7FF8000000000000
    if v == 0:
        return 0
    sign, u = (1 << 63 if v < 0 else 0), abs(v)
    n = u.bit_length() - 1
    ex = n + e + up - 1085 + 1023
    if ex >= 2047:
        return sign | 0x7FF0000000000000
    return sign | ex << 52 | (u << (52 - n)) & ((1 << 52) - 1)


def test_the_factor_of_second_differences_is_no_part_of_the_fields_exponent(tmp_path):
    cu, exe = tmp_path / "limbs.cu", tmp_path / "limbs"
    cu.write_text(SRC)
    subprocess.check_call([libbuild.nvcc(), "-std=c++17", "-O1", *libbuild.ARCH, "-I", libbuild.CSRC, "-o", str(exe), str(cu)])
    cases = [(v, e, up) for v in (0, 1, -1, 3 << 40, -(5 << 48), (1 << 53) - 1) for e in (1, 60, 1961, 2044, 2045, 2046, 2047)
             for up in (0, 2) if not (v and e < 80)]
    text = "".join("%d %d %d\n" % c for c in cases)
    got = [int(x) for x in subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout.split()]
    assert len(got) == len(cases)
    for c, g in zip(cases, got):
        assert g == rounded(*c), (c, hex(g), hex(rounded(*c)))
